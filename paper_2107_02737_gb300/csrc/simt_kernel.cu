// simt_kernel.cu -- the FP32 CUDA-core SP2 chain (the plain-precision comparator).
//
// One cooperative persistent launch runs every layer: per round each CTA takes
// upper-triangle T x T tiles (bi <= bj; T = 32, 64 or 128 by the launch's work) of
// X_{n+1} = X_n^2 or 2 X_n - X_n^2 (or the accelerated layer), computes the tile's product with FP32 FMAs on the
// centred operand X - I/2 (the B operand is rows of X because X is symmetric),
// writes the tile and its mirror, and records FP64 partials of
// Tr X_{n+1} and ||X_{n+1}||_F^2.  A grid barrier ends the round; every CTA then
// takes the same layer decision from the same partials (no host round trip).
#include "device_common.cuh"

namespace sp2i {

namespace {

// Tile side T with 128 threads as 8 (rows) x 16 (columns): a thread owns TM x TN
// elements, rows in groups of four 32 apart, columns in groups of CW 16 CW apart.
// What bounds the inner loop is shared-memory reads: a warp's read of one float per
// lane costs a cycle of the SM's port, TM + TN of them per TM x TN FMAs (and those
// TM TN / 4 cycles of the four FMA pipes).  16 x 8 elements per thread (24 cycles
// against 32) left room that 8 x 8 (16 against 16) did not, packed FMAs free the issue
// slots for it, and fragments read one k ahead hide its latency with one or two warps
// per scheduler: N = 3000 from 651 to 539 us per layer (58 to 70 % of the FP32 peak at
// 1.92 GHz over the executed tiles).
template <int T>
struct SimtCfg {
    static constexpr int BK = (T == 128) ? 8 : 16;      // K elements per staged block
    static constexpr int TM = T / 8, TN = T / 16;       // 16 x 8, 8 x 4, 4 x 2
    static constexpr int CW = TN < 4 ? TN : 4;          // adjacent columns per thread
    static constexpr int LDS = T + 4;                   // padded smem row (floats), keeps 16-byte alignment
    static constexpr int KPT = BK * T / SIMT_THREADS;   // K elements of one row a thread stages: 8, 8, 4
    static constexpr int FLOATS = 2 * 2 * BK * LDS;     // A and B, double-buffered
    static constexpr int LEAVES = T * T / 64;           // 4 x 16 blocks of the tile (tile_blocks)
};

template <int T>
struct SimtSmem {
    float stage[SimtCfg<T>::FLOATS];
    FF leaf[SimtCfg<T>::LEAVES];   // ||X||_F^2 of the tile's 4 x 16 blocks
    FF leaf_t[T / 4];              // Tr X of a diagonal tile's 4 x 4 blocks
};

// Two FP32 FMAs in one instruction (each rounded as a scalar FMA): acc = a b + acc.
__device__ __forceinline__ void ffma2(unsigned long long &acc, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

// acc = Y^2 over the tile for the centred operand Y = X - I/2 (I on the n real
// diagonal entries): Y has the eigenvalues of X shifted into [-1/2, 1/2], so the
// FP32 sums run over smaller terms; the epilogue adds X - I/4 back.  Every element is
// one chain of FMAs over increasing k, whatever T is.
template <int T>
__device__ __forceinline__ void simt_tile_mma(const float *X, int np, int n, int r0, int c0, float *stage,
                                              unsigned long long (&acc)[SimtCfg<T>::TM / 2][SimtCfg<T>::TN]) {
    using C = SimtCfg<T>;
    constexpr int BK = C::BK;
    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    // Staging: consecutive threads take consecutive rows, so the transposed stores
    // are free of bank conflicts.
    const int lrow = tid % T, lk = (tid / T) * C::KPT;
    const float *Ap = X + (size_t)(r0 + lrow) * np + lk;
    const float *Bp = X + (size_t)(c0 + lrow) * np + lk;
    float *const sA = stage, *const sB = stage + 2 * BK * C::LDS;
#pragma unroll
    for (int i = 0; i < C::TM / 2; ++i)
#pragma unroll
        for (int j = 0; j < C::TN; ++j) acc[i][j] = 0ull;

    float4 ra[C::KPT / 4], rb[C::KPT / 4];
    auto fetch = [&](int kt) {
#pragma unroll
        for (int q = 0; q < C::KPT / 4; ++q) {
            ra[q] = *(const float4 *)(Ap + (size_t)kt * BK + 4 * q);
            rb[q] = *(const float4 *)(Bp + (size_t)kt * BK + 4 * q);
        }
    };
    auto stash = [&](int buf, int kt) {
        float *a = sA + (buf * BK + lk) * C::LDS + lrow, *b = sB + (buf * BK + lk) * C::LDS + lrow;
        const int ka = r0 + lrow - kt * BK - lk, kb = c0 + lrow - kt * BK - lk;   // the diagonal's place, if in reach
        const float ha = (r0 + lrow < n) ? 0.5f : 0.0f, hb = (c0 + lrow < n) ? 0.5f : 0.0f;
#pragma unroll
        for (int q = 0; q < C::KPT / 4; ++q) {
            const float va[4] = {ra[q].x, ra[q].y, ra[q].z, ra[q].w};
            const float vb[4] = {rb[q].x, rb[q].y, rb[q].z, rb[q].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int k = 4 * q + e;
                a[k * C::LDS] = (k == ka) ? va[e] - ha : va[e];
                b[k * C::LDS] = (k == kb) ? vb[e] - hb : vb[e];
            }
        }
    };
    fetch(0);
    stash(0, 0);
    __syncthreads();
    const int nk = np / BK;
#pragma unroll 1
    for (int kt = 0; kt < nk; ++kt) {
        const int buf = kt & 1;
        if (kt + 1 < nk) fetch(kt + 1);
        const float *a0 = sA + buf * BK * C::LDS + ty * 4;
        const float *b0 = sB + buf * BK * C::LDS + tx * C::CW;
        // Fragments of the next k are read while this k's FMAs issue.
        ulonglong2 a[2][C::TM / 4];
        float b[2][C::TN];
        auto load = [&](int k, int u) {
#pragma unroll
            for (int g = 0; g < C::TM / 4; ++g) a[u][g] = *(const ulonglong2 *)(a0 + k * C::LDS + g * 32);
#pragma unroll
            for (int h = 0; h < C::TN / C::CW; ++h) {
                if constexpr (C::CW == 4) {
                    const float4 v = *(const float4 *)(b0 + k * C::LDS + h * 64);
                    b[u][4 * h] = v.x;
                    b[u][4 * h + 1] = v.y;
                    b[u][4 * h + 2] = v.z;
                    b[u][4 * h + 3] = v.w;
                } else {
                    const float2 v = *(const float2 *)(b0 + k * C::LDS);
                    b[u][0] = v.x;
                    b[u][1] = v.y;
                }
            }
        };
        load(0, 0);
#pragma unroll
        for (int k = 0; k < BK; ++k) {
            if (k + 1 < BK) load(k + 1, (k + 1) & 1);
#pragma unroll
            for (int j = 0; j < C::TN; ++j) {
                const unsigned long long bj = pack2(b[k & 1][j], b[k & 1][j]);
#pragma unroll
                for (int g = 0; g < C::TM / 4; ++g) {
                    ffma2(acc[2 * g][j], a[k & 1][g].x, bj);
                    ffma2(acc[2 * g + 1][j], a[k & 1][g].y, bj);
                }
            }
        }
        if (kt + 1 < nk) {
            stash(buf ^ 1, kt + 1);
            __syncthreads();
        }
    }
    __syncthreads();
}

// Place of a 4 x 16 block in the tree of a tile's sums: bit 0 its column half of a 32 x 32
// block, bits 1..3 its row there, then the 32 x 32 block: column, row of a 64 x 64 one,
// and that one's column, row.
__device__ __forceinline__ int leaf_index(int row4, int col16) {
    return (col16 & 1) | ((row4 & 7) << 1) | ((col16 & 2) << 3) | ((row4 & 8) << 2) | ((col16 & 4) << 4) |
           ((row4 & 16) << 3);
}

// The whole CTA, after the tile has been stored: Tr X and ||X||_F^2 of its 4 x 16 blocks.  A
// thread adds 4 x 2 elements at a time as a compensated FP32 pair, a fixed tree makes a
// block's pair of eight of those, and everything above a block is FP64 (tile_sum).  (One
// chain over the up to 128 elements a thread computes made ||X||_F^2 2.7e-15 off at
// N = 3000; blocks of 64 leave 3e-16.)  The elements come back from L2 (5 to 10 thousand
// cycles a tile of side 128, of the K loop's 400 to 800), out of line and not unrolled:
// summed in the epilogue's registers, or unrolled there, they had the K loop, whose
// accumulators fill the register file, compiled worse (N = 3000: 555 to 595 us per layer
// instead of 539).
template <int T>
__device__ __noinline__ void tile_blocks(const float *X, int np, int r0, int c0, FF *leaf, FF *leaf_t) {
    constexpr int W = T / 4, UNITS = W * W;   // 4 x 4 units, whole warps of them
#pragma unroll 1
    for (int u = threadIdx.x; u < UNITS; u += SIMT_THREADS) {
        const int row4 = u / W, col4 = u % W, r = r0 + 4 * row4, c = c0 + 4 * col4;
        float x[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 v = r <= c ? __ldcg((const float4 *)(X + (size_t)(r + i) * np + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
            x[i][0] = v.x;
            x[i][1] = v.y;
            x[i][2] = v.z;
            x[i][3] = v.w;
        }
        FF e[2] = {{0.f, 0.f}, {0.f, 0.f}};
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int i = 0; i < 4; ++i)   // an element above the diagonal counts twice
                ff_add_sq(e[q / 2], x[i][q], (r < c || i < q) ? 2.0f : i == q ? 1.0f : 0.0f);
        ff_add_ff(e[0], e[1]);
#pragma unroll
        for (int o = 1; o < 4; o *= 2) {
            FF b;
            b.s = __shfl_down_sync(0xffffffffu, e[0].s, o);
            b.c = __shfl_down_sync(0xffffffffu, e[0].c, o);
            ff_add_ff(e[0], b);
        }
        if ((col4 & 3) == 0) leaf[leaf_index(row4, col4 >> 2)] = e[0];
        if (r == c) {
            FF t = {x[0][0], 0.f}, b = {x[2][2], 0.f};
            ff_add(t, x[1][1]);
            ff_add(b, x[3][3]);
            ff_add_ff(t, b);
            leaf_t[row4] = t;
        }
    }
}

// One warp: the FP64 sums of a tile's N blocks, in G groups of adjacent places, by a binary
// tree over the places; group g's is valid in lane g 32 / G (all of it below 32 blocks).
template <int N, int G>
__device__ __forceinline__ double tile_sum(const FF *leaf, int lane) {
    constexpr int PER = N > 32 ? N / 32 : 1;   // adjacent places of a lane
    double v[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) v[k] = ff_value(leaf[(lane % (N / PER)) * PER + k]);
#pragma unroll
    for (int w = 1; w < PER; w *= 2)
#pragma unroll
        for (int k = 0; k < PER; k += 2 * w) v[k] += v[k + w];
#pragma unroll
    for (int o = 1; o < N / PER / G; o *= 2) v[0] += __shfl_down_sync(0xffffffffu, v[0], o);
    return v[0];
}

// SP2 update of one tile and mirror store.
// X_{n+1} = k2 X^2 + k1 X + k0 I (I on the n real diagonal entries): the plain
// layer (1, 0, 0) or (-1, 2, 0); the accelerated one T^2 with T = aX + (1 - a) I,
// (a^2, 2a(1 - a), (1 - a)^2), or 2T - T^2 with T = aX, (-a^2, 2a, 0).  With
// X^2 = acc + X - I/4 (acc = Y^2 of the centred operands) this is
// k2 acc + (k2 + k1) X + (k0 - k2/4) I.
template <int T>
__device__ __forceinline__ void simt_tile_epilogue(const float *Xold, float *Xnew, int np, int n, int r0, int c0,
                                                   int flip, float alpha,
                                                   const unsigned long long (&acc)[SimtCfg<T>::TM / 2][SimtCfg<T>::TN]) {
    using C = SimtCfg<T>;
    const int tid = threadIdx.x;
    const float k2 = flip ? -alpha * alpha : alpha * alpha;
    const float kx = alpha * (2.0f - alpha);
    const float kd = flip ? 0.25f * alpha * alpha : (1.0f - alpha) * (1.0f - alpha) - 0.25f * alpha * alpha;
    const int tx = tid & 15, ty = tid >> 4;
#pragma unroll
    for (int g = 0; g < C::TM / 4; ++g) {
        const int rb = r0 + g * 32 + ty * 4;
#pragma unroll
        for (int h = 0; h < C::TN / C::CW; ++h) {
            const int cb = c0 + h * 64 + tx * C::CW;
            float v[4][C::CW];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = rb + i;
                float xo[C::CW];
                if constexpr (C::CW == 4) {
                    const float4 x = *(const float4 *)(Xold + (size_t)r * np + cb);
                    xo[0] = x.x;
                    xo[1] = x.y;
                    xo[2] = x.z;
                    xo[3] = x.w;
                } else {
                    const float2 x = *(const float2 *)(Xold + (size_t)r * np + cb);
                    xo[0] = x.x;
                    xo[1] = x.y;
                }
#pragma unroll
                for (int q = 0; q < C::CW; ++q) {
                    const float2 s2 = unpack2(acc[2 * g + (i >> 1)][h * C::CW + q]);
                    const bool dg = (r == cb + q) && (r < n);
                    v[i][q] = fmaf(k2, (i & 1) ? s2.y : s2.x, fmaf(kx, xo[q], dg ? kd : 0.0f));
                }
            }
            if (rb + 3 < cb) {   // strictly above the diagonal: vector stores, direct and mirrored
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float *p = Xnew + (size_t)(rb + i) * np + cb;
                    if constexpr (C::CW == 4) *(float4 *)p = make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
                    else *(float2 *)p = make_float2(v[i][0], v[i][1]);
                }
#pragma unroll
                for (int q = 0; q < C::CW; ++q)
                    *(float4 *)(Xnew + (size_t)(cb + q) * np + rb) = make_float4(v[0][q], v[1][q], v[2][q], v[3][q]);
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int q = 0; q < C::CW; ++q) {
                        const int r = rb + i, c = cb + q;
                        if (r > c) continue;
                        Xnew[(size_t)r * np + c] = v[i][q];
                        if (r < c) Xnew[(size_t)c * np + r] = v[i][q];
                    }
            }
        }
    }
}

// Tile (bi, bj) of layer n and its record.
template <int T>
__device__ __forceinline__ void simt_tile(const InstDesc &d, int n, int bi, int bj, int flip, float alpha,
                                          float *stage, FF *leaf_t, FF *leaf_q) {
    const float *X = d.xf[n & 1];
    unsigned long long acc[SimtCfg<T>::TM / 2][SimtCfg<T>::TN];
    simt_tile_mma<T>(X, d.np, d.n, bi * T, bj * T, stage, acc);
    float *Xn = d.xf[(n + 1) & 1];
    simt_tile_epilogue<T>(X, Xn, d.np, d.n, bi * T, bj * T, flip, alpha, acc);
    __syncthreads();
    tile_blocks<T>(Xn, d.np, bi * T, bj * T, leaf_q, leaf_t);
    // One warp per value, beside the next tile's staging (the blocks' buffer is written
    // again only after that tile's K loop and its barriers).
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int rec = simt_record<T>(bi, bj);
    constexpr int G = T == 128 ? 4 : 1;   // records of a tile, one per 32 / G lanes
    if (w == 0) {
        const double q = tile_sum<SimtCfg<T>::LEAVES, G>(leaf_q, lane);
        if (lane % (32 / G) == 0) simt_records(d, n + 1, 1)[rec + lane / (32 / G)] = q;
    } else if (w == 1) {
        // Only a diagonal tile has a trace; of its four quarters the first (lane 0) and the
        // last (summed in lane 16, and lane 24's to write).
        double t = 0.0;
        if (bi == bj) {
            t = tile_sum<T / 4, G == 4 ? 2 : 1>(leaf_t, lane);
            if (G == 4) {
                t = __shfl_sync(0xffffffffu, t, lane < 16 ? 0 : 16);
                if (lane == 8 || lane == 16) t = 0.0;
            }
        }
        if (lane % (32 / G) == 0) simt_records(d, n + 1, 0)[rec + lane / (32 / G)] = t;
    }
}

template <int T>
__global__ void __launch_bounds__(SIMT_THREADS, T == 128 ? 2 : 4) k_simt_persistent(const __grid_constant__ RunParams p) {
    __shared__ RoundCtl rc;
    __shared__ __align__(16) SimtSmem<T> sm;
    static_assert(sizeof(sm.stage) >= 4 * MAX_BATCH * sizeof(double), "round sums reuse the staging buffers");
    if (threadIdx.x == 0) round_ctl_init(rc, p, p.inst);
    __syncthreads();
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
        // The operand staging buffers are idle here: use them for the sums.
        double *sums = (double *)sm.stage;
        reduce_round_partials_block<(T == 32 ? 4 : 1)>(rc, p, sums);
        if (threadIdx.x == 0) decide_round(rc, p, sums);
        __syncthreads();
        if (rc.abort || rc.total == 0) break;
        for (int g = blockIdx.x; g < rc.total; g += gridDim.x) {
            int i, job, tile;
            map_tile(rc, p.B, p.inst, g, i, job, tile);
            const InstDesc &d = p.inst[i];
            const int2 bt = p.tiles[d.tile_off + tile];
            const int n = rc.layer[i], flip = rc.choice[i] == SP2_CHOICE_FLIP;
            const float alpha = rc.alpha[i];
            simt_tile<T>(d, n, bt.x, bt.y, flip, alpha, sm.stage, sm.leaf_t, sm.leaf);
        }
    }
}

const void *simt_kernel(int side) {
    return side == 128 ? (const void *)k_simt_persistent<128>
                       : side == 64 ? (const void *)k_simt_persistent<64> : (const void *)k_simt_persistent<32>;
}

}  // namespace

int simt_blocks_per_sm(int side) {
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, simt_kernel(side), SIMT_THREADS, 0) != cudaSuccess) return 0;
    return b;
}

cudaError_t launch_simt_persistent(const RunParams &p, int side, int grid, cudaStream_t s) {
    void *args[] = {(void *)&p};
    // Cooperative launch in the attribute form (also capturable in a CUDA graph).
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(SIMT_THREADS);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, simt_kernel(side), args);
}

}  // namespace sp2i
