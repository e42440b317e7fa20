// tc_kernel.cu -- split-precision SP2 chain on the 5th-generation tensor cores.
//
// The activation f(X) = X^2 of every layer (Eq. activ) is evaluated from the
// dual 16-bit representation X = X^(0) + X^(1) as X^(0)X^(0) + X^(0)X^(1) +
// X^(1)X^(0) (the paper's A + B + B^T; the X^(1)X^(1) term is dropped), all
// three products accumulated in one FP32 accumulator in tensor memory:
//   S[i,j] = sum_k hi[i,k] lo[j,k] + lo[i,k] hi[j,k] + hi[i,k] hi[j,k]
// (rows of X; X is symmetric), all three issued from the same staged K block.
// FP16 stores both parts times 2^11 (so lo stays in FP16's normal range): every
// product carries 2^22, removed in the epilogue.  BF16 needs no scaling.
//
// Centred operands and accumulator-bias removal: the FP32 accumulator of the
// tensor cores truncates once per MMA instruction, a relative bias of order
// (K/16) 2^-24 that would make the chain converge to (1 + beta) times the
// projector.  The operands are therefore the split of Y = X - I/2 (near
// convergence Y^2 ~ I/4, so the product error is mostly a multiple of the
// identity), the square is rebuilt as X^2 = Y^2 + X - I/4, and the identity
// component of the error is measured exactly from Tr(Y^2) = ||Y||_F^2 (both
// reduced in FP64) and carried to the next layer as a scalar offset c
// (true X = stored X + c I).
//
// Kernel structure (one persistent launch for the whole chain: cooperative for
// single-CTA tiles, a cluster launch sized to the resident pairs for CTA pairs):
//   warp 0      TMA producer: 2-D tiled bulk copies (128B swizzle) into a ring of
//               stages of one A block (this CTA's rows) and one B block; a square
//               tile takes each K block in two stages, (hi, hi) and (lo, lo), a
//               response tile in four, (X hi, Y hi), (X lo, Y lo), (Y hi, X hi),
//               (Y lo, X lo).  The tensor cores' FP32 accumulator truncates once per
//               MMA instruction; the small cross products of each K block are issued
//               before its hi x hi product.
//   warp 1      tcgen05.mma: the warp walks the ring, one elected lane issues (K=16 per
//               instruction), FP32 accumulator in TMEM, double-buffered so the
//               epilogue of tile t overlaps the MMAs of t+1.
//   warps 2..9  epilogue, two warps per SM sub-partition (the epilogue is bound by
//               instruction latency, so a second warp hides it): warp w reads TMEM
//               lanes 32 (w mod 4) .. +31 and the tile's column half (w - 2) / 4, in
//               16-column chunks; X_{n+1} = S or 2 X_n - S, FP32 master + split
//               operands written for the tile and its mirror (only tiles with rows <=
//               columns are computed; the direct orientation of a chunk above the
//               diagonal leaves as two TMA tensor stores), compensated partials of
//               Tr X and ||X||_F^2 (FP32 pairs, one FP64 record per 256 x 256 pair tile
//               and CTA; with narrower tiles a pass of its own writes the records).
//   warp 10     the decisions of a batch's instances that this CTA owns.
// Between layers (Schedule): a density solve runs without a grid barrier.  With
// several waves of tiles, a tile of layer n + 1 starts its K blocks once the tiles of
// layer n that wrote them have completed; with one wave, once the layer has.  Only the
// epilogue needs the layer's sign and offset, so the statistics and the decision run
// beside the next layer's copies and MMAs.  In a batch each instance advances on its own.
// Responses, adjoints and layer application run in rounds ended by a grid barrier,
// after which every CTA takes the same decision.
// The response / adjoint stream reuses the same machinery with six products per K
// block: (C + C^T)[i,j] = sum_k X[i,k] Y[j,k] + Y[i,k] X[j,k] for symmetric X and Y.
#include "device_common.cuh"
#include "tc_ptx.cuh"

namespace sp2i {

namespace {

// Tile configuration: 128 CG x BN, BN = 256, 128 or 64.  CG = 2: a cluster of two CTAs
// computes the tile with M = 256 MMAs issued by the even CTA; each CTA loads its own 128
// rows of A and half of the B rows.  CG = 1: one CTA, M = 128 MMAs.  An element's
// products and their order are those of its row and column whatever the tile, so every
// shape gives the same X; the host picks one by size (narrow_tiles).
template <int CG, int BN>
struct Cfg {
    static constexpr int BOX = BN / CG < 128 ? BN / CG : 128;             // rows per load box (tc_box_rows)
    static constexpr uint32_t A_BYTES = 128 * TC_BK * 2;                   // 16 KB: own 128 rows
    static constexpr uint32_t B_BYTES = (BN / CG) * TC_BK * 2;             // own B rows
    static constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int STAGES = 196608 / STAGE_BYTES;                    // 4, 6 or 8
    static constexpr uint32_t TX_BYTES = STAGE_BYTES * CG;               // bytes per stage over the pair
    static constexpr int TILE_M = 128 * CG;                              // output rows per tile
    static constexpr uint32_t TMEM_COLS = 2 * BN;                        // two FP32 accumulators
};
constexpr int MAX_STAGES = 8;
constexpr int EPI_WARPS = 8;                              // warps 2..9
constexpr int EPI_CHUNK = 16;                             // accumulator columns per epilogue step
// Per epilogue warp: the transpose buffer of a chunk (32 x (EPI_CHUNK + 1) words) or
// the chunk's hi and lo boxes for the tensor stores, 128-byte aligned.
constexpr uint32_t EPI_T_FLOATS = 576;
static_assert(EPI_CHUNK == EPI_BOX_COLS && EPI_BOX_ROWS == 32, "store box = one warp's chunk");
static_assert(EPI_T_FLOATS >= 32 * (EPI_CHUNK + 1) && EPI_T_FLOATS * 4 >= 2 * EPI_BOX_ROWS * EPI_BOX_COLS * 2 &&
                  (EPI_T_FLOATS * 4) % 128 == 0,
              "epilogue buffer");

struct TcSmemTail {
    uint64_t full[MAX_STAGES];
    uint64_t empty[MAX_STAGES];
    uint64_t tfull[2];
    uint64_t tempty[2];
    uint64_t drain;                  // MMA completion, waited for when the launch aborts
    uint32_t tmem_base;
    uint32_t pad;
    unsigned int issued;             // producer: ring stages this CTA has loaded into
    unsigned int consumed;           // MMA thread (even CTA): stages whose copies it has waited for
    FF red[EPI_WARPS][4];            // per epilogue warp: a record's four partials (compensated pairs)
    double flow_sums[5];             // dataflow: the layer's sums; [4] nonzero: a wait gave up
    struct FlowEntry {               // batch: the decision of a list entry's layer, for the epilogue warps
        int go, flip;
        float cf, alpha;
    } entry[2];
    RoundCtl rc;
    InstDesc desc;                   // a lone instance's descriptor (global loads of it would miss L1
                                     // after every acquire)
};

constexpr size_t STAGE_AREA = 196608;  // 4 x 48 KB, 6 x 32 KB or 8 x 24 KB
static_assert(EPI_WARPS * EPI_T_FLOATS * 4 >= 4 * MAX_BATCH * sizeof(double) + MAX_BATCH * sizeof(int),
              "round sums and decisions reuse the epilogue transpose buffers");
constexpr size_t SMEM_BYTES = 1024 /*alignment slack*/ + STAGE_AREA + (size_t)EPI_WARPS * EPI_T_FLOATS * 4 +
                              sizeof(TcSmemTail);

// Instruction descriptor, kind::f16: FP32 accumulator, A and B of one 16-bit
// type (0 = FP16, 1 = BF16), both K-major, M = 128 * CG, N = BN: idesc_f16_mn.

// ---------------------------------------------------------------------------
// Work description of one tile, identical for the three roles.
// ---------------------------------------------------------------------------
struct TileWork {
    int inst, job, tile, bi, bj;
    int resp;            // 0: square of X (three products per K block), 1: C + C^T of X and Y (six)
    int xslot;           // X operand slot
    int ybuf;            // Y input buffer (resp)
    int flip;            // layer choice is 2X - X^2
    int n;               // forward layer index of the input (square jobs)
    int rec;             // square job recomputing a forward layer in the adjoint's reverse sweep
    float cf;            // offset c of the input X: true X = stored X + c I
    float alpha;         // expansion a of the layer (1 = plain)
};

// Stop this CTA's roles, and for a CTA pair its peer's (so that neither waits for
// signals the other will no longer send).
template <int CG>
__device__ __forceinline__ void tc_abort(RoundCtl &rc, uint32_t peer_abort) {
    rc.abort = 1;
    if (CG == 2) asm volatile("fence.acq_rel.cluster;" ::: "memory");   // after what this CTA has seen
    if (CG == 2) asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_abort), "r"(1) : "memory");
}

__device__ __forceinline__ TileWork describe(const RoundCtl &rc, const RunParams &p, int g) {
    TileWork w;
    map_tile(rc, p.B, rc.inst, g, w.inst, w.job, w.tile);
    const InstDesc &d = rc.inst[w.inst];
    const int2 bt = p.tiles[d.tile_off + w.tile];
    w.bi = bt.x;
    w.bj = bt.y;
    w.rec = 0;
    if (rc.phase == 1 && rc.rec_mode) {  // adjoint reverse, checkpointing: X_{n+1} again from X_n
        const int n = rc.rec_top;
        w.resp = 0;
        w.rec = 1;
        w.xslot = xslot_of(d, n);
        w.ybuf = 0;
        w.flip = rc.chist[n + 1] == SP2_CHOICE_FLIP;
        w.n = n;
        w.cf = (float)rc.chist_c[n];
        w.alpha = rc.chist_a[n + 1];
    } else if (rc.phase == 1) {  // adjoint reverse: G_m from G_{m+1} and X_m
        const int k = rc.layer[0];
        const int m = rc.rev_total - 1 - k;
        w.resp = 1;
        w.xslot = xslot_of(d, m);
        w.ybuf = k & 1;
        w.flip = rc.chist[m + 1] == SP2_CHOICE_FLIP;
        w.n = m;
        w.cf = (float)rc.chist_c[m];
        w.alpha = rc.chist_a[m + 1];
    } else {
        const int n = rc.layer[w.inst];
        w.resp = w.job;
        w.xslot = xslot_of(d, n);
        w.ybuf = n & 1;
        w.flip = rc.choice[w.inst] == SP2_CHOICE_FLIP;
        w.n = n;
        w.cf = (float)rc.coff[w.inst];
        w.alpha = rc.alpha[w.inst];
    }
    return w;
}

// Dataflow schedule: tile g (at bt) of layer r for the producer and the MMA thread (the
// layer's sign and offset are not needed there).
__device__ __forceinline__ TileWork describe_flow(const RoundCtl &rc, int g, int2 bt, int r) {
    TileWork w;
    const InstDesc &d = rc.inst[0];
    w.inst = 0;
    w.job = 0;
    w.tile = g;
    w.bi = bt.x;
    w.bj = bt.y;
    w.resp = 0;
    w.xslot = xslot_of(d, r);
    w.ybuf = 0;
    w.flip = 0;
    w.n = r;
    w.rec = 0;
    w.cf = 0.0f;
    w.alpha = 1.0f;
    return w;
}

// Dataflow schedule, producer.  A 256-column block kt of the operand row blocks pa
// and pb of X_n was written by at most four tiles of the previous layer, each done
// when its counter reaches `target` (EPI_WARPS * CG completions per layer).  The counters are
// read with relaxed loads one block ahead (flow_peek), so their latency hides under
// the current block's copies, and re-polled only while a tile is still running;
// one acquire fence then orders the TMA reads after the tiles' stores.
__device__ __forceinline__ unsigned int ld_relaxed(const unsigned int *p) {
    unsigned int v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void flow_peek(const RunParams &p, int pa, int pb, int kt, unsigned int (&v)[4]) {
    const int *e0 = p.blk_src + (pa * p.nblk + kt) * 2, *e1 = p.blk_src + (pb * p.nblk + kt) * 2;
    const int src[4] = {e0[0], e0[1], e1[0], e1[1]};
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = src[k] < 0 ? 0xFFFFFFFFu : ld_relaxed(p.tile_done + src[k]);
}
__device__ __noinline__ bool flow_wait_block(const RunParams &p, int pa, int pb, int kt, unsigned int target,
                                       unsigned int (&v)[4], const volatile int *abort) {
    const int *e0 = p.blk_src + (pa * p.nblk + kt) * 2, *e1 = p.blk_src + (pb * p.nblk + kt) * 2;
    const int src[4] = {e0[0], e0[1], e1[0], e1[1]};
    const unsigned long long t0 = global_ns();
    for (int k = 0; k < 4; ++k) {
        while (v[k] < target) {
            if (*abort || ld_volatile(p.err) != 0) return false;
            if (global_ns() - t0 > p.timeout_ns) {
                set_error(p.err, SP2_ERR_TIMEOUT);
                return false;
            }
            __nanosleep(32);
            v[k] = ld_relaxed(p.tile_done + src[k]);
        }
    }
    // The tiles' generic-proxy stores, released with their counters, reach the TMA reads.
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    asm volatile("fence.proxy.async.global;" ::: "memory");
    return true;
}

// Dataflow schedule: wait until a counter (epilogue warps done with a tile of layers
// 0 .. r - 1, or records written) has reached `target`; false when the launch is
// stopping or the wait ran out.  Relaxed polls and one acquire load at the end (0.4 us less than a fence).
__device__ __forceinline__ bool flow_wait(const RunParams &p, const unsigned int *counter, unsigned int target,
                                          const volatile int *abort) {
    if (ld_relaxed(counter) < target) {
        const unsigned long long t0 = global_ns();
        for (int i = 0; ld_relaxed(counter) < target; ++i) {
            if ((i & 31) != 31) continue;   // the clock and the flags now and then
            if (*abort || ld_volatile(p.err) != 0) {
                // One more look: the other CTA of a pair ends this one once it has seen the
                // chain's last layer complete, and this one (as CTA 0 it has that decision
                // to write down) may not have looked since.
                asm volatile("fence.acq_rel.cluster;" ::: "memory");
                break;
            }
            if (global_ns() - t0 > p.timeout_ns) {
                set_error(p.err, SP2_ERR_TIMEOUT);
                return false;
            }
            __nanosleep(64);
        }
    }
    return ld_acquire(counter) >= target;
}

// The eight epilogue warps: one partial record from each warp's compensated pairs (fq: half
// of ||X||_F^2, an element above the diagonal counting twice), which
// stay FP32 pairs through the warp and cross-warp sums (FP64 arithmetic is slow on this
// part); one conversion, written by one thread (epilogue warp 0, lane 0).
__device__ __forceinline__ void write_record(FF (&red)[EPI_WARPS][4], Part *out, const FF &ft, const FF &fq,
                                             const FF &fw, const FF &fp, int ew, int lane) {
    const FF q = {2.0f * fq.s, 2.0f * fq.c};
    FF qw = q;
    ff_add_ff(qw, fw);
    const FF r4[4] = {ff_warp_sum(ft), ff_warp_sum(q), ff_warp_sum(qw), ff_warp_sum(fp)};
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < 4; ++k) red[ew][k] = r4[k];
    asm volatile("bar.sync 1, %0;" ::"n"(EPI_WARPS * 32) : "memory");
    if (ew == 0 && lane == 0) {
        FF a4[4] = {red[0][0], red[0][1], red[0][2], red[0][3]};
        for (int k = 1; k < EPI_WARPS; ++k)
#pragma unroll
            for (int c = 0; c < 4; ++c) ff_add_ff(a4[c], red[k][c]);
        Part s4;
        s4.t = ff_value(a4[0]);
        s4.q = ff_value(a4[1]);
        s4.w = ff_value(a4[2]);
        s4.p = ff_value(a4[3]);
        *out = s4;
    }
}

// Narrow tiles, the eight epilogue warps: record u of X_n, the sums over the 128 x 256
// elements that CTA u mod 2 of pair tile u / 2 would own, by the same warps' rows and
// columns and in the same order as that CTA's epilogue adds them.  X_n comes back from
// its FP32 master (lower triangle, coalesced across the warp).  The pass runs once the layer's tiles are complete, beside the next layer's copies and
// MMAs, which need no statistics; only the next epilogue does.
__device__ __forceinline__ void flow_record(FF (&red)[EPI_WARPS][4], const InstDesc &d, const int2 *units, int u, int n,
                                         int ew, int lane) {
    const int np = d.np;
    const int2 bt = units[u >> 1];
    const float *X = xmaster(d, n, false);
    const int rw0 = bt.x * 256 + (u & 1) * 128 + ((ew + 2) & 3) * 32, r = rw0 + lane;
    const int col0 = bt.y * 256 + (ew >> 2) * 128;
    int j0 = 0, j1 = (rw0 < np) ? 128 / EPI_CHUNK : 0;
    while (j1 > 0 && col0 + (j1 - 1) * EPI_CHUNK >= np) --j1;
    while (j0 < j1 && col0 + j0 * EPI_CHUNK + EPI_CHUNK - 1 < rw0) ++j0;
    FF ft = {0.f, 0.f}, fq = {0.f, 0.f}, fp = {0.f, 0.f}, fw = {0.f, 0.f};
    // A short loop, three chunks of loads ahead: the pass is bound by instruction fetch
    // (unrolled over 64 columns it took twice as long) and by the loads' latency.
    const float pd = (j0 < j1 && r < d.n) ? __ldcg(d.pdiag[n & 1] + r) : 0.0f;
    const float *p = X + (size_t)(col0 + j0 * EPI_CHUNK) * np + r;
    const size_t step = (size_t)EPI_CHUNK * np;
    float x[EPI_CHUNK], y[EPI_CHUNK], z[EPI_CHUNK], u3[EPI_CHUNK];
    auto load = [&](int j, float (&v)[EPI_CHUNK]) {
        if (j < j1) {
#pragma unroll
            for (int jj = 0; jj < EPI_CHUNK; ++jj) v[jj] = __ldcg(p + (size_t)jj * np);
        }
        p += step;
    };
    load(j0, x);
    load(j0 + 1, y);
    load(j0 + 2, z);
#pragma unroll 1
    for (int j = j0; j < j1; ++j) {
        load(j + 3, u3);
        const int jd = r - (col0 + j * EPI_CHUNK);   // the diagonal's column in the chunk
        float xd = 0.0f;
        if (col0 + j * EPI_CHUNK > rw0 + 31) {       // strictly above it
#pragma unroll
            for (int jj = 0; jj < EPI_CHUNK; ++jj) ff_add_sq1(fq, x[jj]);
        } else {
#pragma unroll
            for (int jj = 0; jj < EPI_CHUNK; ++jj) {
                ff_add_sq(fq, jj >= jd ? x[jj] : 0.0f, jj == jd ? 0.5f : 1.0f);
                if (jj == jd) xd = x[jj];
            }
        }
        if (jd >= 0 && jd < EPI_CHUNK) {
            ff_add(ft, xd);
            if (r < d.n) {
                ff_add(fp, pd);
                ff_add_sq(fw, xd - 0.5f, 1.0f);
                ff_add_sq(fw, xd, -1.0f);
            }
        }
#pragma unroll
        for (int jj = 0; jj < EPI_CHUNK; ++jj) {
            x[jj] = y[jj];
            y[jj] = z[jj];
            z[jj] = u3[jj];
        }
    }
    write_record(red, d.part[n % 3] + u, ft, fq, fw, fp, ew, lane);
}

// Dataflow schedule of a batch.  Every CTA walks the same fixed list of tiles layer
// after layer, and an instance's tiles start layer n as soon as its own layer n - 1 is
// complete and decided, whatever the others do: no barrier, and a pair's remainder of one
// round overlaps the next.  (Every wait is for a list entry a whole round earlier, so the
// first unfinished entry never waits.)  The decisions of instance i are taken by one
// CTA, i mod grid, in a warp of its own, and published in the instance's control block.

// 1: instance `ctl` runs layer r, 0: its chain has stopped, -1: the launch is stopping.
__device__ __forceinline__ int flow_wait_instance(const RunParams &p, const InstCtl *ctl, int r,
                                                  const volatile int *abort) {
    unsigned int seq = ld_relaxed(&ctl->flow_seq);
    if (seq < (unsigned int)r + 1u) {
        const unsigned long long t0 = global_ns();
        for (int i = 0; (seq = ld_relaxed(&ctl->flow_seq)) < (unsigned int)r + 1u; ++i) {
            if ((i & 31) != 31) continue;
            if (*abort || ld_volatile(p.err) != 0) return -1;
            if (global_ns() - t0 > p.timeout_ns) {
                set_error(p.err, SP2_ERR_TIMEOUT);
                return -1;
            }
            __nanosleep(64);
        }
    }
    return ld_acquire(&ctl->flow_seq) == FLOW_STOPPED ? 0 : 1;
}

// One warp: sums and decides for instances blockIdx.x, blockIdx.x + gridDim.x, ... until
// all of them have stopped.
template <int CG>
__device__ __noinline__ void flow_owner(RoundCtl &rc, const RunParams &p, int lane, const volatile int *abort) {
    int left = 0;
    for (int i = blockIdx.x; i < p.B; i += gridDim.x) ++left;
    unsigned long long t0 = global_ns();
    for (bool first = true; left > 0; first = false) {
        bool progress = false;
        for (int i = blockIdx.x; i < p.B; i += gridDim.x) {
            if (!first && !rc.active[i]) continue;
            InstCtl *ctl = rc.inst[i].ctl;
            const int n = rc.layer[i] + (rc.ran[i] ? 1 : 0);   // the layer whose records come next
            int ready = 1;
            if (!first && lane == 0) {
                const unsigned int target = (unsigned int)(EPI_WARPS * CG * rc.inst[i].ntiles) * (unsigned int)n;
                ready = (ld_relaxed(&ctl->flow_done) >= target && ld_acquire(&ctl->flow_done) >= target) ? 1 : 0;
            }
            if (!warp_waited(ready)) continue;
            double sums[4] = {0.0, 0.0, 0.0, 0.0};
            if (rc.active[i]) sum_layer_partials(rc.inst[i], n, lane, sums);
            int go = 0;
            if (lane == 0) {
                go = decide_instance(rc, p, sums, i, true) > 0 ? 1 : 0;
                ctl->flow_flip = rc.choice[i] == SP2_CHOICE_FLIP;
                ctl->flow_cf = (float)rc.coff[i];
                ctl->flow_alpha = rc.alpha[i];
                asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&ctl->flow_seq),
                             "r"(go ? (unsigned int)n + 1u : FLOW_STOPPED)
                             : "memory");
            }
            __syncwarp();
            progress = true;
            if (!__shfl_sync(0xffffffffu, go, 0)) --left;
        }
        if (progress) {
            t0 = global_ns();
            continue;
        }
        int stop = 0;
        if (lane == 0) {
            if (*abort || ld_volatile(p.err) != 0) stop = 1;
            else if (global_ns() - t0 > p.timeout_ns) {
                set_error(p.err, SP2_ERR_TIMEOUT);
                stop = 1;
            }
        }
        if (__shfl_sync(0xffffffffu, stop, 0)) return;
        __nanosleep(100);
    }
}

// Dataflow schedule, the eight epilogue warps: wait for layer r - 1 (with narrow tiles,
// compute this CTA's record of it and wait for the other CTAs'), the sums of its records
// in a fixed order (a warp per value) and the decision for instance 0; one barrier hands it to
// the others (flow_go by parity: the next decision cannot pass this one's readers, who
// arrive at its barrier first).  Returns false when the chain stopped or the launch is
// stopping.
template <bool NARROW>
__device__ __forceinline__ bool flow_decide(RoundCtl &rc, FF (&red)[EPI_WARPS][4], double *sums, const RunParams &p,
                                         int r, int ew, int lane, unsigned int per_layer, const volatile int *abort) {
    if constexpr (!NARROW) {
        // Wide tiles: one warp does it all, beside the next layer's long K loops (48.2
        // against 51.5 us per layer at N = 2304 with the steps below, no difference in
        // several waves).
        if (ew == 0) {
            int go = 1;
            if (lane == 0 && r > 0) go = flow_wait(p, p.layer_done, per_layer * (unsigned int)r, abort) ? 1 : 0;
            go = warp_waited(go);
            double a[4];
            if (go) sum_layer_partials(rc.inst[0], r, lane, a);
            if (lane == 0) {
                if (ld_volatile(p.err) != 0) go = 0;
                if (go) go = decide_instance(rc, p, a, 0, blockIdx.x == 0) > 0 ? 1 : 0;
                rc.flow_go[r & 1] = go;
            }
        }
        asm volatile("bar.sync 1, %0;" ::"n"(EPI_WARPS * 32) : "memory");
        return rc.flow_go[r & 1] != 0;
    }
    // One thread of a CTA polls (more of them slowed the increments themselves).
    const bool unit = r > 0 && (int)blockIdx.x < p.units;
    if (unit) {
        if (ew == 0 && lane == 0 && !flow_wait(p, p.layer_done, per_layer * (unsigned int)r, abort)) sums[4] = 1.0;
        asm volatile("bar.sync 1, %0;" ::"n"(EPI_WARPS * 32) : "memory");
    }
    // (An aborting launch goes through the same barriers, with whatever X holds.)
    if (unit) flow_record(red, rc.inst[0], p.tiles + rc.inst[0].unit_off, blockIdx.x, r, ew, lane);
    if (r > 0) {
        if (ew == 0 && lane == 0) {
            if (unit) {
                __threadfence();
                atomicAdd(p.stat_done, 1u);
            }
            if (!flow_wait(p, p.stat_done, (unsigned int)p.units * (unsigned int)r, abort)) sums[4] = 1.0;
        }
        asm volatile("bar.sync 1, %0;" ::"n"(EPI_WARPS * 32) : "memory");
    }
    if (ew < 4) {   // warp c sums value c of the records
        const double a = sum_layer_value(rc.inst[0], r, ew, lane);
        if (lane == 0) sums[ew] = a;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(EPI_WARPS * 32) : "memory");
    if (ew == 0 && lane == 0) {
        int go = sums[4] == 0.0 && ld_volatile(p.err) == 0;
        if (go) go = decide_instance(rc, p, sums, 0, blockIdx.x == 0) > 0 ? 1 : 0;
        rc.flow_go[r & 1] = go;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(EPI_WARPS * 32) : "memory");
    return rc.flow_go[r & 1] != 0;
}

template <int PREC, int CG, int BN, int SCHED>
__global__ void __launch_bounds__(TC_THREADS, 1) k_tc_persistent(const __grid_constant__ RunParams p) {
    using C = Cfg<CG, BN>;
    static_assert(C::STAGES <= MAX_STAGES, "ring of stages");
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *stages = smem;
    float *epi_T = (float *)(smem + STAGE_AREA);
    TcSmemTail &tl = *(TcSmemTail *)(epi_T + EPI_WARPS * EPI_T_FLOATS);
    RoundCtl &rc = tl.rc;
    const volatile int *abort = &rc.abort;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = (CG == 2) ? cluster_rank() : 0u;   // position in the CTA pair
    const bool leader = (rank == 0);
    const int cluster_id = blockIdx.x / CG, nclusters = gridDim.x / CG;

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            mbar_init(&tl.full[s], 1);
            mbar_init(&tl.empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&tl.tfull[a], 1);
            mbar_init(&tl.tempty[a], EPI_WARPS * CG);  // one arrival per epilogue warp of the pair
        }
        mbar_init(&tl.drain, 1);
        tl.issued = 0;
        tl.consumed = 0;
        tl.flow_sums[4] = 0.0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (p.B == 1) tl.desc = p.inst[0];
        round_ctl_init(rc, p, p.B == 1 ? &tl.desc : p.inst);
        if (SCHED == RUN_BATCH) {
            rc.prefix[0] = 0;
            for (int i = 0; i < p.B; ++i) rc.prefix[i + 1] = rc.prefix[i] + p.inst[i].ntiles;
        }
    }
    if (warp == 1) {
        if (CG == 2) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&tl.tmem_base)),
                         "r"(C::TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                             smem_u32(&tl.tmem_base)),
                         "r"(C::TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        tc_fence_before();
    }
    __syncthreads();
    if (CG == 2) cluster_sync_all();  // both CTAs' barriers exist before any cross-CTA signal
    tc_fence_after();
    const uint32_t tmem_base = tl.tmem_base;

    // Cluster addresses of the even CTA's barriers (the pair's MMA side) and of the
    // peer's abort flag.
    uint32_t lead_full0 = 0, lead_tempty0 = 0, peer_abort = 0;
    if (CG == 2) {
        lead_full0 = cluster_addr(&tl.full[0], 0);
        lead_tempty0 = cluster_addr(&tl.tempty[0], 0);
        peer_abort = cluster_addr(&rc.abort, rank ^ 1u);
    }

    // Pipeline state, private to each role and carried across tiles and rounds.
    uint32_t stage = 0, phase = 0;      // producer / MMA ring
    uint32_t acc = 0, acc_phase = 0;    // MMA / epilogue accumulators
    int pend[MAX_STAGES];               // producer: parity + 1 of a load not yet released
    for (int s = 0; s < MAX_STAGES; ++s) pend[s] = 0;
    unsigned int issued = 0, consumed = 0;   // producer / MMA thread: ring stages so far
    const uint32_t stage0_lo = sdesc_lo(smem_u32(stages));
    const uint32_t idesc = idesc_f16_mn(PREC == SP2_BF16_SPLIT ? 1u : 0u, C::TILE_M, BN);

    // ---------- per-tile work of the three roles (both schedules below) ----------
    // Producer: every K block of tile w into the ring.  In the dataflow schedule a
    // 256-column block of X_n is loaded only once the tiles of the previous layer
    // that wrote it (and its mirror) have completed.
    int df_round = -1;   // dataflow: layer whose inputs are known to be complete everywhere
    auto produce_tile = [&](const TileWork &w) {
        if (SCHED == RUN_WAVE && w.n > 0) {
            // One wave of tiles: the layer's tiles end together.
            if (!flow_wait(p, p.layer_done, (unsigned int)(EPI_WARPS * CG * rc.inst[0].ntiles * w.n), abort)) {
                tc_abort<CG>(rc, peer_abort);
                return;
            }
            asm volatile("fence.proxy.async.global;" ::: "memory");
        }
        // Dataflow: the column block checked last, the one peeked ahead and its counters.
        int df_kt = -1, df_next = -1;
        unsigned int df_v[4] = {0u, 0u, 0u, 0u};
        bool df_ready = SCHED != RUN_FLOW || w.n == 0 || df_round == w.n;
        if (!df_ready) {
            if (ld_relaxed(p.layer_done) >= (unsigned int)(EPI_WARPS * CG * rc.inst[0].ntiles * w.n)) {
                df_round = w.n;   // every tile of the previous layer is done
                df_ready = true;
            } else {
                // Or every tile that wrote this tile's two operand row blocks is: one pass
                // of relaxed loads (all in flight together), no per-block checks then.
                const int pa = (w.bi * C::TILE_M + (int)rank * 128) / 256, pb = w.bj;
                const int nb = (rc.inst[0].np + 255) / 256;
                unsigned int mn = 0xFFFFFFFFu;
                for (int kt = 0; kt < nb; ++kt) {
                    unsigned int v[4];
                    flow_peek(p, pa, pb, kt, v);
                    mn = min(mn, min(min(v[0], v[1]), min(v[2], v[3])));
                }
                df_ready = mn >= (unsigned int)(EPI_WARPS * CG * w.n);
            }
            if (df_ready) {
                asm volatile("fence.acq_rel.gpu;" ::: "memory");
                asm volatile("fence.proxy.async.global;" ::: "memory");
            }
        }
        const InstDesc &d = rc.inst[w.inst];
        const int nkb = d.np / TC_BK;
        // Successive waves of tiles walk K in opposite directions, so that a
        // wave starts on the K blocks the previous one left in L2.
        const bool kdown = ((w.tile / d.kwave) & 1) != 0;
        const int row_a = w.bi * C::TILE_M + (int)rank * 128;
        const int row_b = w.bj * BN + (CG == 2 ? (int)rank * (BN / 2) : 0);
        // Square tiles: each K block in two consecutive ring slots, (hi, hi) then
        // (lo, lo), which feed all three products.  Response tiles: the six
        // segments one after another, one K block per slot.
        const int nslot = (w.resp ? 4 : 2) * nkb;
        const CUtensorMap *X3 = d.xmap + w.xslot * MAPS_PER_SLOT;   // maps hi, hi, lo
        for (int kb = 0; kb < nslot; ++kb) {
            int kx;
            const CUtensorMap *am, *bm;
            if (w.resp) {
                // Response / adjoint tiles: per K block (X hi, Y hi), (X lo, Y lo),
                // (Y hi, X hi), (Y lo, X lo) -- rows bi on the A side, rows bj on the B
                // side -- feeding X Y^T and Y X^T.
                const CUtensorMap *Y3 = d.ymap + w.ybuf * MAPS_PER_SLOT;
                const int q = kb & 3;
                kx = (kdown ? nkb - 1 - (kb >> 2) : (kb >> 2)) * TC_BK;
                const CUtensorMap *xm = (q & 1) ? X3 + 2 : X3 + 1, *ym = (q & 1) ? Y3 + 2 : Y3 + 1;
                am = (q < 2) ? xm : ym;
                bm = (q < 2) ? ym : xm;
            } else {
                kx = (kdown ? nkb - 1 - (kb >> 1) : (kb >> 1)) * TC_BK;
                am = bm = (kb & 1) ? X3 + 2 : X3 + 1;
            }
            if (!df_ready && kx / 256 != df_kt) {
                // Dataflow: this 256-column block of both operand panels must come
                // from tiles of the previous layer that have completed.
                df_kt = kx / 256;
                const int pa = row_a / 256, pb = row_b / 256;
                if (df_next != df_kt) flow_peek(p, pa, pb, df_kt, df_v);
                if (!flow_wait_block(p, pa, pb, df_kt, (unsigned int)(EPI_WARPS * CG * w.n), df_v, abort)) {
                    tc_abort<CG>(rc, peer_abort);
                    break;
                }
                const int nx = kdown ? df_kt - 1 : df_kt + 1;   // next block of this walk
                df_next = -1;
                if (nx >= 0 && nx * 256 < d.np) {
                    flow_peek(p, pa, pb, nx, df_v);
                    df_next = nx;
                }
            }
            if (!mbar_wait(&tl.empty[stage], phase ^ 1u, abort, p.timeout_ns, p.err)) {
                tc_abort<CG>(rc, peer_abort);
                break;
            }
            pend[stage] = 0;
            uint8_t *sa = stages + (size_t)stage * C::STAGE_BYTES;
            if (CG == 1) {
                mbar_expect_tx(&tl.full[stage], C::TX_BYTES);
#pragma unroll
                for (int q = 0; q < 128; q += C::BOX)
                    tma_load_2d(sa + q * (TC_BK * 2), am, kx, row_a + q, &tl.full[stage]);
#pragma unroll
                for (int q = 0; q < BN; q += C::BOX)
                    tma_load_2d(sa + C::A_BYTES + q * (TC_BK * 2), bm, kx, row_b + q, &tl.full[stage]);
            } else {
                // Both CTAs' bytes complete on the even CTA's barrier.
                if (leader) mbar_expect_tx(&tl.full[stage], C::TX_BYTES);
                const uint32_t fb = lead_full0 + stage * 8u;
#pragma unroll
                for (int q = 0; q < 128; q += C::BOX)
                    tma_load_2d_pair(sa + q * (TC_BK * 2), am, kx, row_a + q, fb);
                tma_load_2d_pair(sa + C::A_BYTES, bm, kx, row_b, fb);   // BN / 2 rows: one box
            }
            pend[stage] = (int)phase + 1;
            *(volatile unsigned int *)&tl.issued = ++issued;
            if (++stage == C::STAGES) {
                stage = 0;
                phase ^= 1u;
            }
        }
    };
    // MMA warp (the leader CTA's, all lanes): tile w's products into the next
    // accumulator; false when a wait gave up (the launch is stopping).
    // One ring slot: its operands' low descriptor word, or 0 when the wait gave up.
    auto mma_slot = [&](uint32_t &slot) -> uint32_t {
        slot = stage;
        if (!mbar_wait_warp(&tl.full[stage], phase, abort, p.timeout_ns, p.err)) {
            tc_abort<CG>(rc, peer_abort);
            return 0;
        }
        ++consumed;
        if (lane == 0) *(volatile unsigned int *)&tl.consumed = consumed;
        if (++stage == C::STAGES) {
            stage = 0;
            phase ^= 1u;
        }
        return stage0_lo + slot * (C::STAGE_BYTES >> 4);
    };
    auto mma_tile = [&](const TileWork &w) -> bool {
        if (!mbar_wait_warp(&tl.tempty[acc], acc_phase ^ 1u, abort, p.timeout_ns, p.err)) {
            tc_abort<CG>(rc, peer_abort);
            return false;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * BN;
        constexpr uint32_t B_OFF = C::A_BYTES >> 4;
        bool ok = true;
        // Per K block, a square: the (hi, hi) and (lo, lo) slots, then hi lo, lo hi (the
        // small cross terms first) and hi hi.  A response: the slots (X hi, Y hi),
        // (X lo, Y lo) for X Y^T, released as soon as those products are issued, then
        // (Y hi, X hi), (Y lo, X lo) for Y X^T; cross terms before hi x hi in each.
        const int nslots = rc.inst[w.inst].np / TC_BK * (w.resp ? 2 : 1);
        for (int kb = 0; kb < nslots; ++kb) {
            uint32_t st_h, st_l;
            const uint32_t sh = mma_slot(st_h);
            const uint32_t sl = sh ? mma_slot(st_l) : 0u;
            if (!sl) {
                ok = false;
                break;
            }
            tc_fence_after();
#pragma unroll
            for (int k = 0; k < TC_BK / 16; ++k)   // hi x lo
                umma_f16<CG>(d_tmem, sh + 2 * k, sl + B_OFF + 2 * k, idesc, (kb | k) != 0 ? 1u : 0u);
#pragma unroll
            for (int k = 0; k < TC_BK / 16; ++k)   // lo x hi
                umma_f16<CG>(d_tmem, sl + 2 * k, sh + B_OFF + 2 * k, idesc, 1u);
#pragma unroll
            for (int k = 0; k < TC_BK / 16; ++k)   // hi x hi
                umma_f16<CG>(d_tmem, sh + 2 * k, sh + B_OFF + 2 * k, idesc, 1u);
            umma_commit<CG>(&tl.empty[st_h]);
            umma_commit<CG>(&tl.empty[st_l]);
        }
        umma_commit<CG>(&tl.tfull[acc]);
        if (++acc == 2) {
            acc = 0;
            acc_phase ^= 1u;
        }
        return ok;
    };
    const int ew = warp - 2;                  // epilogue warp 0 .. EPI_WARPS - 1
    const int quarter = warp & 3;             // TMEM lanes this warp may access
    const int half = ew >> 2;                 // column half of the tile this warp owns
    uint32_t *T = (uint32_t *)(epi_T + (ew >= 0 && ew < EPI_WARPS ? ew : 0) * EPI_T_FLOATS);   // packed split operands
    uint16_t *Bh = (uint16_t *)T, *Bl = Bh + EPI_BOX_ROWS * EPI_BOX_COLS;      // or the hi and lo boxes
    bool flow_first = true;                   // dataflow: no tile completed by this CTA yet
    // Epilogue: the next layer from tile w's accumulator, its FP64 partials and, in
    // the dataflow schedule, the tile's completion flag.
    auto epilogue_tile = [&](const TileWork &w) {
        const InstDesc &d = rc.inst[w.inst];
        const int np = d.np;
        const size_t mat = (size_t)np * np;
        const float *__restrict__ old;
        float *__restrict__ outf;
        uint16_t *__restrict__ o1;   // hi
        uint16_t *__restrict__ o2;   // lo
        const CUtensorMap *smap;     // store maps of hi, lo
        if (!w.resp) {
            old = xmaster(d, w.n, w.rec != 0);
            outf = xmaster(d, w.n + 1, w.rec != 0);
            const int so = xslot_of(d, w.n + 1);
            o1 = d.xop + (size_t)so * 2 * mat;
            o2 = o1 + mat;
            smap = d.xmap + (size_t)so * MAPS_PER_SLOT + 3;
        } else {
            const int yout = w.ybuf ^ 1;
            old = d.yf[w.ybuf];
            outf = d.yf[yout];
            o1 = d.yop + (size_t)yout * 2 * mat;
            o2 = o1 + mat;
            smap = d.ymap + (size_t)yout * MAPS_PER_SLOT + 3;
        }
        const float unscale = product_unscale<PREC>(w.resp != 0);
        const int rw0 = w.bi * C::TILE_M + (int)rank * 128 + quarter * 32;  // first row of this warp
        const int r = rw0 + lane;
        const int nreal = d.n;
        const float cf = w.cf;
        // Accelerated layer (a != 1) in terms of the product P of the stored
        // centred operands Y = X - I/2 (true Y = Y + cI): with T = aY + (1 - a/2) I
        // (X^2 branch) or T = aY + (a/2) I (2X - X^2 branch),
        //   X_{n+1} = ka (P + 2cY) + kb (Y + cI) + kc I,
        // ka = +-a^2, kb = a (2 - a), kc = (1 - a/2)^2 or a (1 - a/4); the
        // response / adjoint stream takes ka P + (kb + 2c ka) X1.
        const bool accel = (w.alpha != 1.0f);
        const float al = w.alpha;
        const float ka = w.flip ? -al * al : al * al;
        const float kb = al * (2.0f - al);
        const float kc = w.flip ? al * (1.0f - 0.25f * al) : (1.0f - 0.5f * al) * (1.0f - 0.5f * al);
        const float kx1 = fmaf(2.0f * cf, ka, kb);
        // ||Y||_F^2 of the next operands equals ||X||_F^2 off the diagonal (y = x
        // there); the diagonal difference y^2 - x^2 is accumulated apart (exact squares).
        FF ft = {0.f, 0.f}, fq = {0.f, 0.f}, fp = {0.f, 0.f}, fw = {0.f, 0.f};
        // With narrow tiles a pass of its own (flow_record) does the sums.
        constexpr bool NARROW = BN < 256;
        const bool stats = !w.resp && !NARROW;
        // The chunks this warp finishes form one range [j0, j1): chunks entirely
        // below the diagonal come first, chunks past np last.
        const int col0 = w.bj * BN + half * (BN / 2);   // this warp's first column
        int j0 = 0, j1 = (rw0 < np) ? BN / 2 / EPI_CHUNK : 0;
        while (j1 > 0 && col0 + (j1 - 1) * EPI_CHUNK >= np) --j1;
        while (j0 < j1 && col0 + j0 * EPI_CHUNK + EPI_CHUNK - 1 < rw0) ++j0;
        // The previous layer's (r, c) values -- (c, r) by symmetry, coalesced across
        // the warp, evict-first -- are loaded one chunk ahead, so that their latency
        // overlaps the current chunk's arithmetic and stores (the first chunk's, the
        // wait for the products).
        float xnx[EPI_CHUNK];
        if (j0 < j1) {
            const int cb0 = col0 + j0 * EPI_CHUNK;
#pragma unroll
            for (int jj = 0; jj < EPI_CHUNK; ++jj) xnx[jj] = __ldcs(old + (size_t)(cb0 + jj) * np + r);
        }
        int ok = 1;
        if (lane == 0) ok = mbar_wait(&tl.tfull[acc], acc_phase, abort, p.timeout_ns, p.err) ? 1 : 0;
        ok = warp_waited(ok);
        tc_fence_after();
        if (ok) {
#pragma unroll 1
            for (int j = j0; j < j1; ++j) {
                const int c0 = half * (BN / 2) + j * EPI_CHUNK;   // column offset in the tile
                const int cb = w.bj * BN + c0;
                float xov[EPI_CHUNK];
#pragma unroll
                for (int jj = 0; jj < EPI_CHUNK; ++jj) xov[jj] = xnx[jj];
                if (j + 1 < j1) {
#pragma unroll
                    for (int jj = 0; jj < EPI_CHUNK; ++jj)
                        xnx[jj] = __ldcs(old + (size_t)(cb + EPI_CHUNK + jj) * np + r);
                }
                float v[EPI_CHUNK];
                tmem_ld16(tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * BN + c0, v);
                // Each element's next split operands are computed once, stored to the
                // mirror (c, r) and staged packed (hi | lo << 16) for the direct (r, c)
                // stores below.  The FP32 master gets the mirror and the diagonal only.
                const bool upper = (cb > rw0 + 31);     // every element has r < c
                // Strictly upper chunks write their direct (r, c) operands as two boxes of
                // tensor stores; the diagonal ones through the transpose buffer, once the
                // previous chunk's boxes have left it.
                if (!upper) {
                    if (lane == 0) bulk_wait_read();
                    __syncwarp();
                }
                uint32_t hp[EPI_CHUNK / 2], lp[EPI_CHUNK / 2];   // (r, c), (r, c + 1) packed
                float x[EPI_CHUNK];
                if (upper) {
                    if (!w.resp && !accel) {   // a plain square
                        const float twoc = 2.0f * cf;
#pragma unroll
                        for (int jj = 0; jj < EPI_CHUNK; ++jj) {
                            const float xo = xov[jj];
                            const float t = fmaf(twoc, xo, v[jj] * unscale);
                            x[jj] = w.flip ? xo - t : t + xo;   // 2X - X^2 or X^2
                        }
                    } else if (!w.resp) {
                        const float twoc = 2.0f * cf;
#pragma unroll
                        for (int jj = 0; jj < EPI_CHUNK; ++jj)
                            x[jj] = fmaf(ka, fmaf(twoc, xov[jj], v[jj] * unscale), kb * xov[jj]);
                    } else if (!accel) {
                        // Response / adjoint stream: P = Y X1 + X1 Y; with X = Y + (1/2 + c) I
                        // the chain needs X X1 + X1 X = P + (1 + 2c) X1, negated for 2X - X^2.
                        const float kx = w.flip ? 1.0f - 2.0f * cf : 1.0f + 2.0f * cf;
                        const float sg = w.flip ? -unscale : unscale;
#pragma unroll
                        for (int jj = 0; jj < EPI_CHUNK; ++jj) x[jj] = fmaf(kx, xov[jj], v[jj] * sg);
                    } else {
#pragma unroll
                        for (int jj = 0; jj < EPI_CHUNK; ++jj) x[jj] = fmaf(kx1, xov[jj], ka * (v[jj] * unscale));
                    }
                    if (stats) {
#pragma unroll
                        for (int jj = 0; jj < EPI_CHUNK; ++jj) ff_add_sq1(fq, x[jj]);   // weight 2 / 2
                    }
                    // Mirror (c, r): the FP32 master one column per store; the operands two
                    // rows packed per lane, exchanged with the neighbour so that the even
                    // lane stores rows (r, r + 1) of column c and the odd one rows
                    // (r - 1, r) of column c + 1.
                    float *mf = outf + (size_t)cb * np + r;
#pragma unroll
                    for (int jj = 0; jj < EPI_CHUNK; ++jj) {
                        __stcs(mf, x[jj]);   // streaming stores: keep L2 for the operands
                        mf += np;
                    }
                    const int odd = lane & 1;
                    const uint32_t sel = odd ? 0x3276u : 0x5410u;
                    size_t m = (size_t)(cb + odd) * np + (r - odd);
#pragma unroll
                    for (int k = 0; k < EPI_CHUNK / 2; ++k) {
                        if (!w.resp) split2_pair<PREC, X_SHIFT>(x[2 * k], x[2 * k + 1], hp[k], lp[k]);
                        else split2_pair<PREC, Y_SHIFT>(x[2 * k], x[2 * k + 1], hp[k], lp[k]);
                        const uint32_t hn = __shfl_xor_sync(0xffffffffu, hp[k], 1);
                        const uint32_t ln = __shfl_xor_sync(0xffffffffu, lp[k], 1);
                        __stcs((uint32_t *)(o1 + m), __byte_perm(hp[k], hn, sel));
                        __stcs((uint32_t *)(o2 + m), __byte_perm(lp[k], ln, sel));
                        m += 2 * (size_t)np;
                    }
                } else {
                    // A chunk on the diagonal: selects instead of branches, and the lane's
                    // diagonal element (at most one, column jd) apart.
                    const int jd = r - cb;
                    const bool dreal = r < nreal;
                    if (!w.resp) {
                        // P = Y^2 for the stored operands Y = X - I/2; the true input is
                        // X + cI, so X^2 = P + 2cY + cI + X - I/4 (c^2 is below FP32 here).
                        const float twoc = 2.0f * cf;
                        const float cd = dreal ? (w.flip ? -cf : cf) : 0.0f, qd = dreal ? 0.25f : 0.0f;
                        const float hd = dreal ? 0.5f : 0.0f, kcd = dreal ? kc : 0.0f, cfd = dreal ? cf : 0.0f;
#pragma unroll
                        for (int jj = 0; jj < EPI_CHUNK; ++jj) {
                            const bool dg = jj == jd;
                            const float P = v[jj] * unscale;            // raw product
                            const float xo = xov[jj];
                            const float yo = dg ? xo - hd : xo;
                            if (accel) {
                                x[jj] = fmaf(ka, fmaf(twoc, yo, P), fmaf(kb, dg ? yo + cfd : yo, dg ? kcd : 0.0f));
                            } else {
                                const float t = (dg ? P - qd : P) + fmaf(twoc, yo, dg ? cd : 0.0f);
                                x[jj] = w.flip ? xo - t : t + xo;   // 2X - X^2 or X^2
                            }
                        }
                    } else {
                        const float kx = accel ? kx1 : w.flip ? 1.0f - 2.0f * cf : 1.0f + 2.0f * cf;
                        const float sg = accel ? ka : w.flip ? -1.0f : 1.0f;
#pragma unroll
                        for (int jj = 0; jj < EPI_CHUNK; ++jj) x[jj] = fmaf(kx, xov[jj], sg * (v[jj] * unscale));
                    }
                    if (!w.resp) {
                        float xd = 0.0f, Pd = 0.0f;
#pragma unroll
                        for (int jj = 0; jj < EPI_CHUNK; ++jj) {
                            if (!NARROW) ff_add_sq(fq, jj >= jd ? x[jj] : 0.0f, jj == jd ? 0.5f : 1.0f);
                            if (jj == jd) {
                                xd = x[jj];
                                Pd = v[jj] * unscale;
                            }
                        }
                        if (NARROW) {
                            if (jd >= 0 && jd < EPI_CHUNK) __stcg(d.pdiag[(w.n + 1) & 1] + r, Pd);
                        } else if (jd >= 0 && jd < EPI_CHUNK) {
                            ff_add(ft, xd);
                            if (dreal) {
                                ff_add(fp, Pd);
                                ff_add_sq(fw, xd - 0.5f, 1.0f);
                                ff_add_sq(fw, xd, -1.0f);
                            }
                        }
                    }
                    // mirror (c, r), consecutive r across the warp, and the diagonal of the
                    // FP32 master: streaming stores, keep L2 for the operands
                    size_t m = (size_t)cb * np + r;
#pragma unroll
                    for (int k = 0; k < EPI_CHUNK / 2; ++k) {
                        const int j0k = 2 * k, j1k = 2 * k + 1;
                        const float h = (dreal && !w.resp) ? 0.5f : 0.0f;   // next operands: Y = X - I/2
                        const float y0 = j0k == jd ? x[j0k] - h : x[j0k], y1 = j1k == jd ? x[j1k] - h : x[j1k];
                        if (!w.resp) split2_pair<PREC, X_SHIFT>(y0, y1, hp[k], lp[k]);
                        else split2_pair<PREC, Y_SHIFT>(y0, y1, hp[k], lp[k]);
                        if (j0k >= jd) __stcs(outf + m, x[j0k]);
                        if (j0k > jd) {
                            __stcs(o1 + m, (uint16_t)hp[k]);
                            __stcs(o2 + m, (uint16_t)lp[k]);
                        }
                        m += np;
                        if (j1k >= jd) __stcs(outf + m, x[j1k]);
                        if (j1k > jd) {
                            __stcs(o1 + m, (uint16_t)(hp[k] >> 16));
                            __stcs(o2 + m, (uint16_t)(lp[k] >> 16));
                        }
                        m += np;
                        T[lane * (EPI_CHUNK + 1) + j0k] = __byte_perm(hp[k], lp[k], 0x5410);
                        T[lane * (EPI_CHUNK + 1) + j1k] = __byte_perm(hp[k], lp[k], 0x7632);
                    }
                }
                if (upper) {
                    // The chunk's 32 x 16 boxes of hi and lo, row-major, to global memory
                    // by the tensor store unit (the operands need both triangles: TMA
                    // loads rows).
                    if (lane == 0) bulk_wait_read();   // the previous boxes have left the buffer
                    __syncwarp();
                    uint4 *bh = (uint4 *)(Bh + lane * EPI_BOX_COLS), *bl = (uint4 *)(Bl + lane * EPI_BOX_COLS);
                    bh[0] = make_uint4(hp[0], hp[1], hp[2], hp[3]);
                    bh[1] = make_uint4(hp[4], hp[5], hp[6], hp[7]);
                    bl[0] = make_uint4(lp[0], lp[1], lp[2], lp[3]);
                    bl[1] = make_uint4(lp[4], lp[5], lp[6], lp[7]);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_2d(smap, Bh, cb, rw0);
                        tma_store_2d(smap + 1, Bl, cb, rw0);
                        bulk_commit();
                    }
                } else {
                    __syncwarp();
                    // direct (r, c) split-operand stores through the transpose buffer: eight
                    // lanes a row, two columns each, on and above the diagonal
                    const int hl = lane >> 3, cl = 2 * (lane & 7);
#pragma unroll
                    for (int it = 0; it < 8; ++it) {
                        const int ii = 4 * it + hl;
                        const int rr = rw0 + ii, cc = cb + cl;
                        const uint32_t u0 = T[ii * (EPI_CHUNK + 1) + cl], u1 = T[ii * (EPI_CHUNK + 1) + cl + 1];
                        const size_t md = (size_t)rr * np + cc;
                        if (rr <= cc) {
                            __stcs((uint32_t *)(o1 + md), __byte_perm(u0, u1, 0x5410));
                            __stcs((uint32_t *)(o2 + md), __byte_perm(u0, u1, 0x7632));
                        } else if (rr == cc + 1) {
                            __stcs(o1 + md + 1, (uint16_t)u1);
                            __stcs(o2 + md + 1, (uint16_t)(u1 >> 16));
                        }
                    }
                    __syncwarp();
                }
            }
        }
        // Release the accumulator: every lane's loads have completed
        // (tcgen05.wait::ld); one arrival per warp on the MMA side's barrier.
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
            if (CG == 2) mbar_arrive_cluster(lead_tempty0 + acc * 8u);
            else mbar_arrive(&tl.tempty[acc]);
        }
        if (++acc == 2) {
            acc = 0;
            acc_phase ^= 1u;
        }
        if (stats) {
            write_record(tl.red, d.part[(w.n + 1) % 3] + w.tile * CG + (int)rank, ft, fq, fw, fp, ew, lane);
            asm volatile("bar.sync 1, %0;" ::"n"(EPI_WARPS * 32) : "memory");   // the buffer is free again
        }
        if (SCHED != RUN_ROUNDS) {
            // This warp's stores (generic proxy, and its tensor stores once complete)
            // reach the TMA reads (async proxy) of any CTA that sees its completion.
            asm volatile("fence.proxy.async.global;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
                bulk_wait_all();
                asm volatile("fence.proxy.async.global;" ::: "memory");
                __threadfence();
                // test_hook: CTA 0's first epilogue warp withholds its first completion (a
                // CTA that never finishes; the other CTAs' waits must run out).
                if (!(p.test_hook == 1 && blockIdx.x == 0 && ew == 0 && w.n == 0 && flow_first)) {
                    if (SCHED == RUN_BATCH) {
                        atomicAdd(&d.ctl->flow_done, 1u);
                    } else {
                        if (SCHED == RUN_FLOW) atomicAdd(p.tile_done + w.tile, 1u);
                        atomicAdd(p.layer_done, 1u);
                    }
                }
            }
            flow_first = false;
        }
    };

    // A list of `total` tiles (largest instances first) is dealt to the pairs in a snake
    // order, forward in even waves and backward in odd ones, which evens out the pairs'
    // shares of large and small tiles; each pair then takes its share smallest first, so
    // that the epilogues of its small tiles overlap the MMAs of the large ones after them.
    const auto round_tile = [&](int k) {
        return k * nclusters + ((k & 1) ? nclusters - 1 - cluster_id : cluster_id);
    };
    const auto round_count = [&](int total) {
        int nk = 0;
        while (round_tile(nk) < total) ++nk;
        return nk;
    };

    if constexpr (SCHED == RUN_BATCH) {
        // ------------------ dataflow schedule of a batch (density mode) ------------------
        const int nk = round_count(rc.prefix[p.B]);
        const auto tile_of = [&](int g, int r) {
            TileWork w;
            map_tile(rc, p.B, rc.inst, g, w.inst, w.job, w.tile);
            const TileWork f = describe_flow(rc, w.tile, p.tiles[rc.inst[w.inst].tile_off + w.tile], r);
            w.bi = f.bi;
            w.bj = f.bj;
            w.resp = w.ybuf = w.flip = w.rec = 0;
            w.xslot = xslot_of(rc.inst[w.inst], r);
            w.n = r;
            w.cf = 0.0f;
            w.alpha = 1.0f;
            return w;
        };
        bool any = nk > 0;
        if (warp == 0) {
            if (lane == 0)
                for (int r = 0; any && !*abort; ++r) {
                    any = false;
                    for (int k = nk - 1; k >= 0 && !*abort; --k) {
                        const TileWork w = tile_of(round_tile(k), r);
                        const int go = flow_wait_instance(p, rc.inst[w.inst].ctl, r, abort);
                        if (go < 0) tc_abort<CG>(rc, peer_abort);
                        if (go <= 0) continue;
                        any = true;
                        asm volatile("fence.proxy.async.global;" ::: "memory");
                        produce_tile(w);
                    }
                }
        } else if (warp == 1) {
            if (leader)
                for (int r = 0; any; ++r) {
                    any = false;
                    for (int k = nk - 1; k >= 0; --k) {
                        const TileWork w = tile_of(round_tile(k), r);
                        int go = 0;
                        if (lane == 0) go = flow_wait_instance(p, rc.inst[w.inst].ctl, r, abort);
                        go = warp_waited(go);
                        if (go < 0) tc_abort<CG>(rc, peer_abort);
                        if (go > 0) {
                            any = true;
                            if (!mma_tile(w)) go = -1;
                        }
                        if (go < 0) {
                            any = false;
                            break;
                        }
                    }
                }
        } else if (warp < 2 + EPI_WARPS) {
            // One thread waits for a list entry's decision and one barrier hands it to the
            // eight warps, so that they take the tile or leave together: epilogue_tile has
            // barriers of its own, and warps that each looked for themselves could part
            // where a decision and the launch's end meet.  Two entries by parity: one is
            // written again only after the next one's barrier, which its readers precede.
            unsigned int e = 0;
            for (int r = 0; any; ++r) {
                any = false;
                for (int k = nk - 1; k >= 0; --k) {
                    TileWork w = tile_of(round_tile(k), r);
                    TcSmemTail::FlowEntry &fe = tl.entry[e++ & 1];
                    if (ew == 0 && lane == 0) {
                        const InstCtl *ctl = rc.inst[w.inst].ctl;
                        fe.go = flow_wait_instance(p, ctl, r, abort);
                        fe.flip = __ldcg(&ctl->flow_flip);
                        fe.cf = __ldcg(&ctl->flow_cf);
                        fe.alpha = __ldcg(&ctl->flow_alpha);
                    }
                    asm volatile("bar.sync 1, %0;" ::"n"(EPI_WARPS * 32) : "memory");
                    const int go = fe.go;
                    if (go < 0) {
                        tc_abort<CG>(rc, peer_abort);
                        any = false;
                        break;
                    }
                    if (go == 0) continue;
                    any = true;
                    w.flip = fe.flip;
                    w.cf = fe.cf;
                    w.alpha = fe.alpha;
                    epilogue_tile(w);
                }
            }
        } else {
            flow_owner<CG>(rc, p, lane, abort);
        }
    } else if constexpr (SCHED == RUN_FLOW || SCHED == RUN_WAVE) {
        // ------------- dataflow schedule (one instance, density mode) -------------
        // No grid barrier between layers.  The producer and the MMA thread run on into
        // the next layer as soon as their own tiles are done (the producer waits per
        // K block for the tiles that wrote it); only the epilogue needs the layer's
        // sign and offset, so the epilogue warps alone wait for every tile of the
        // previous layer, reduce its partials and take the decision.  When the stop
        // rule fires they halt the CTA: loads and MMAs issued ahead are drained at
        // teardown.  Each tile's arithmetic, and so X and D, is that of the barrier
        // schedule bit for bit.
        const int ntl = rc.inst[0].ntiles;
        const int2 *tiles = p.tiles + rc.inst[0].tile_off;
        // When every pair has a few tiles in every layer (fewer than four), layer r's
        // round-robin starts at a rotated position, so that the pairs holding one
        // tile fewer change from layer to layer and the remainder tiles spread evenly
        // over the chain (a tile's arithmetic does not depend on the pair that
        // computes it).  With more tiles per pair the imbalance is small and the fixed
        // assignment keeps more of the operand panels in L2.
        const bool rotate = (ntl >= nclusters && ntl < 4 * nclusters);
        const auto first_tile = [&](int r) {
            return rotate ? (int)(((long long)cluster_id + (long long)r * (ntl % nclusters)) % nclusters) : cluster_id;
        };
        if (cluster_id >= ntl) {
            // no tiles here: only the epilogue warps take part (in the decisions)
        } else if (warp == 0) {
            if (lane == 0)
                for (int r = 0; !*abort; ++r)
                    for (int g = first_tile(r); g < ntl && !*abort; g += nclusters) produce_tile(describe_flow(rc, g, tiles[g], r));
        } else if (warp == 1) {
            if (leader) {
                bool ok = true;
                for (int r = 0; ok; ++r)
                    for (int g = first_tile(r); ok && g < ntl; g += nclusters)
                        ok = mma_tile(describe_flow(rc, g, tiles[g], r));
            }
        } else if (warp < 2 + EPI_WARPS) {
            for (int r = 0;; ++r) {
                const int g0 = first_tile(r);
                int2 bt = make_int2(0, 0);
                if (g0 < ntl) bt = tiles[g0];   // ahead of the wait
                if (!flow_decide<(BN < 256)>(rc, tl.red, tl.flow_sums, p, r, ew, lane, (unsigned int)(EPI_WARPS * CG * ntl), abort)) {
                    tc_abort<CG>(rc, peer_abort);   // stop rule or error: halt this CTA and its peer
                    break;
                }
                for (int g = g0; g < ntl; g += nclusters) {
                    if (g != g0) bt = tiles[g];
                    TileWork w = describe_flow(rc, g, bt, r);
                    w.flip = rc.choice[0] == SP2_CHOICE_FLIP;
                    w.cf = (float)rc.coff[0];
                    w.alpha = rc.alpha[0];
                    epilogue_tile(w);
                }
            }
        }
    } else {
        // --------- barrier schedule (responses, adjoints, layer application) ---------
        unsigned int target = 0;
        bool first = true;
        while (true) {
            if (!first) {
                __syncthreads();
                if (threadIdx.x == 0) {
                    const bool withhold = (p.test_hook == 1 && blockIdx.x == 0 && target == 0);
                    target += gridDim.x;
                    if (!grid_barrier(p.barrier, target, p.err, p.timeout_ns, withhold)) rc.abort = 1;
                }
                __syncthreads();
                if (rc.abort) break;
            }
            first = false;
            // Narrow tiles: the records of the layer just finished, one per CTA, and a
            // second barrier before they are summed.
            if (BN < 256 && rc.phase == 0 && rc.active[0] && rc.ran[0]) {
                if ((int)blockIdx.x < p.units && warp >= 2 && warp < 2 + EPI_WARPS)
                    flow_record(tl.red, rc.inst[0], p.tiles + rc.inst[0].unit_off, blockIdx.x, rc.layer[0] + 1, ew, lane);
                __syncthreads();
                if (threadIdx.x == 0) {
                    target += gridDim.x;
                    if (!grid_barrier(p.barrier, target, p.err, p.timeout_ns)) rc.abort = 1;
                }
                __syncthreads();
                if (rc.abort) break;
            }
            // The epilogue transpose buffers are idle here: use them for the sums.
            reduce_round_partials(rc, p, (double *)epi_T);
            if (p.mode == MODE_ADJOINT) {
                if (threadIdx.x == 0) decide_round(rc, p, (const double *)epi_T);
            } else {
                decide_round_parallel(rc, p, (const double *)epi_T, (int *)((double *)epi_T + 4 * MAX_BATCH));
            }
            if (threadIdx.x == 0) {
                // Make the previous round's global writes (other CTAs' epilogues,
                // generic proxy) visible to this CTA's TMA reads (async proxy).
                asm volatile("fence.proxy.async.global;" ::: "memory");
            }
            __syncthreads();
            if (rc.abort || rc.total == 0) break;

            const int nk = round_count(rc.total);
            if (warp == 0) {
                if (lane == 0)
                    for (int k = nk - 1; k >= 0 && !*abort; --k) produce_tile(describe(rc, p, round_tile(k)));
            } else if (warp == 1) {
                if (leader)
                    for (int k = nk - 1; k >= 0; --k)
                        if (!mma_tile(describe(rc, p, round_tile(k)))) break;
            } else if (warp < 2 + EPI_WARPS) {
                for (int k = nk - 1; k >= 0; --k) epilogue_tile(describe(rc, p, round_tile(k)));
                // This warp's tensor stores are complete; order this round's
                // generic-proxy stores before the async-proxy (TMA) reads of the next
                // round, on any SM.
                if (lane == 0) bulk_wait_all();
                __syncwarp();
                asm volatile("fence.proxy.async.global;" ::: "memory");
                __threadfence();
            }
        }
    }

    // ------------------------------ teardown ------------------------------
    // Tensor stores still reading this CTA's shared memory finish before it is released.
    if (warp >= 2 && warp < 2 + EPI_WARPS && lane == 0) bulk_wait_all();
    // After an abort: MMAs this launch issued complete before tensor memory and the
    // stages are released (the commit covers every earlier MMA of the issuing thread).
    if (warp == 1 && leader && __any_sync(0xffffffffu, *abort)) {
        umma_commit<CG>(&tl.drain);
        const unsigned long long t0 = global_ns();
        while (!mbar_try_wait(&tl.drain, 0u) && global_ns() - t0 < p.timeout_ns) {
        }
    }
    if (CG == 1 && warp == 0 && lane == 0 && rc.abort) {
        // Let loads still in flight land before the CTA exits: bounded waits on the
        // barriers that count them.
        for (int s = 0; s < C::STAGES; ++s) {
            if (pend[s]) {
                const unsigned long long t0 = global_ns();
                while (!mbar_try_wait(&tl.full[s], (uint32_t)(pend[s] - 1)) && global_ns() - t0 < p.timeout_ns) {
                }
            }
        }
    }
    __syncthreads();
    if (CG == 2) {
        cluster_sync_all();   // both CTAs' producers have stopped issuing copies
        if (threadIdx.x == 0 && leader) {
            // Copies of either CTA land on the even CTA's full barriers, which count
            // both CTAs' bytes of a stage (equal shares).  Every ring stage in
            // [consumed, max(issued)) may still have copies in flight: arm the barrier
            // for the odd CTA's share if only the odd CTA issued that stage, retire the
            // odd CTA's share if only this CTA did, then wait (bounded) for the phase.
            unsigned int odd_issued;
            const uint32_t odd_addr = cluster_addr(&tl.issued, 1);
            asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(odd_issued) : "r"(odd_addr) : "memory");
            const unsigned int own = tl.issued, done = tl.consumed;
            const unsigned int top = own > odd_issued ? own : odd_issued;
            for (unsigned int i = done; i < top; ++i) {
                const uint32_t slot = i % C::STAGES, ph = (i / C::STAGES) & 1u;
                if (i >= own) mbar_expect_tx(&tl.full[slot], C::STAGE_BYTES);
                else if (i >= odd_issued)
                    asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(
                                     smem_u32(&tl.full[slot])),
                                 "r"(C::STAGE_BYTES)
                                 : "memory");
                const unsigned long long t0 = global_ns();
                while (!mbar_try_wait(&tl.full[slot], ph) && global_ns() - t0 < p.timeout_ns) {
                }
            }
        }
        __syncthreads();
        cluster_sync_all();  // neither CTA leaves while its peer may still signal it
    }
    if (warp == 1) {
        tc_fence_after();
        if (CG == 2)
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::TMEM_COLS)
                         : "memory");
        else
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::TMEM_COLS)
                         : "memory");
    }
}

template <int CG, int BN, int SCHED>
const void *tc_kernel_of(int precision) {
    return (precision == SP2_BF16_SPLIT) ? (const void *)k_tc_persistent<SP2_BF16_SPLIT, CG, BN, SCHED>
                                         : (const void *)k_tc_persistent<SP2_FP16_SPLIT, CG, BN, SCHED>;
}
// The tile shapes: 256 x 256 and 128 x 256 with every schedule, 256 x 128 and 128 x 64
// for a lone instance.
const void *tc_kernel_ptr(int precision, int cg, int bn, int sched) {
    if (sched == RUN_BATCH)
        return cg == 2 ? tc_kernel_of<2, 256, RUN_BATCH>(precision) : tc_kernel_of<1, 256, RUN_BATCH>(precision);
    if (sched == RUN_ROUNDS) {
        if (cg == 2)
            return bn == 128 ? tc_kernel_of<2, 128, RUN_ROUNDS>(precision) : tc_kernel_of<2, 256, RUN_ROUNDS>(precision);
        return bn == 64 ? tc_kernel_of<1, 64, RUN_ROUNDS>(precision) : tc_kernel_of<1, 256, RUN_ROUNDS>(precision);
    }
    if (sched == RUN_WAVE) {
        if (cg == 2) return bn == 128 ? tc_kernel_of<2, 128, RUN_WAVE>(precision) : tc_kernel_of<2, 256, RUN_WAVE>(precision);
        return bn == 64 ? tc_kernel_of<1, 64, RUN_WAVE>(precision) : tc_kernel_of<1, 256, RUN_WAVE>(precision);
    }
    return cg == 2 ? tc_kernel_of<2, 256, RUN_FLOW>(precision) : tc_kernel_of<1, 256, RUN_FLOW>(precision);
}

}  // namespace

static_assert(SMEM_BYTES <= 232448, "dynamic shared memory above the 227 KB a CTA can hold");

// Number of CTAs of a co-resident persistent grid for the given tile shape
// (0 when the configuration cannot be launched on this device).
int tc_grid_size(int cta_group, int bn, int sm_count) {
    const void *fn = nullptr;
    for (int prec : {SP2_FP16_SPLIT, SP2_BF16_SPLIT})
        for (int sched : {RUN_ROUNDS, RUN_FLOW, RUN_BATCH, RUN_WAVE}) {
            fn = tc_kernel_ptr(prec, cta_group, bn, sched);
            if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES) != cudaSuccess) {
                cudaGetLastError();
                return 0;
            }
        }
    fn = tc_kernel_ptr(SP2_FP16_SPLIT, cta_group, bn, RUN_WAVE);
    if (cta_group == 1) {
        int b = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, fn, TC_THREADS, SMEM_BYTES) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        return b >= 1 ? sm_count : 0;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(sm_count);
    cfg.blockDim = dim3(TC_THREADS);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, fn, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if (nclusters * 2 > sm_count) nclusters = sm_count / 2;
    return nclusters * 2;
}

cudaError_t launch_tc_persistent(const RunParams &p, int cta_group, int bn, int grid, cudaStream_t s) {
    void *args[] = {(void *)&p};
    if (cta_group == 1) {
        // Cooperative launch (co-residency of the whole grid), through the
        // attribute form so that it can also be captured in a CUDA graph.
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(TC_THREADS);
        cfg.dynamicSmemBytes = SMEM_BYTES;
        cfg.stream = s;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelExC(&cfg, tc_kernel_ptr(p.precision, 1, bn, p.dataflow), args);
    }
    // CTA pairs: a cluster launch of exactly as many pairs as the device holds
    // at once (cudaOccupancyMaxActiveClusters, one CTA per SM), so on an idle GPU
    // every pair is resident for the grid barrier.  Without the cooperative
    // attribute (which the profiler cannot replay together with clusters) that
    // residency is not promised by the API: if concurrent work delays a pair,
    // the barrier's time limit ends the call with SP2_ERR_TIMEOUT.
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(TC_THREADS);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, tc_kernel_ptr(p.precision, 2, bn, p.dataflow), args);
}

}  // namespace sp2i
