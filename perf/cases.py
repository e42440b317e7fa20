"""Performance workloads of the library, with exact results for each.

Density matrices of gapped, symmetric, orthogonalised Hamiltonians, as one step of
a quantum-based molecular-dynamics run asks for them: single solves from the
smallest systems to the headline size, in each precision, the batched solve of many
replicas, the first-order response, the reverse-mode gradient, the refined FP64
result and the non-orthogonal route.  Every case goes through the Python entry
points that a user's program calls, without a workspace of its own unless the entry
point is a plan.

Hamiltonians are H = U diag(lam) U^T with lam uniform in [-1, -0.05] (occupied) and
[0.05, 1] (unoccupied), the spectrum of the plain workload of ``inputs.py``, and U a
product of sparse rotations, so that inputs of any size are made on the GPU in
milliseconds and the exact density matrix, response and gradient are known:
``dense`` rotates across all distances (a random dense H), ``banded`` only near the
diagonal (a tight-binding-like H whose entries decay within a few hundred columns).
"""
import math

import torch

import paper_2107_02737_gb300.sp2 as sp2

# Layers that a chain needs on these spectra (they vary by a few with the size): for work().
LAYERS = {"plain": 32, "accelerated": 22}


def listed():
    return [
        # The smallest call: one molecule cluster, just past one block of 128; latency only.
        {"name": "density_n130_fp16", "kind": "density", "n": 130, "precision": "fp16", "band": "dense", "gap": False},
        # The plain FP32 workload of the benchmark configurations (N = 256).
        {"name": "density_n256_fp32", "kind": "density", "n": 256, "precision": "fp32", "band": "dense", "gap": False},
        # 100 water molecules at 6 orbitals each: an everyday MD step.
        {"name": "density_n600_fp16", "kind": "density", "n": 600, "precision": "fp16", "band": "banded", "gap": False},
        # An odd size, BF16 split, with HOMO/LUMO estimates of the previous MD step (accelerated chain).
        {"name": "density_n1537_bf16_gap", "kind": "density", "n": 1537, "precision": "bf16", "band": "banded",
         "gap": True},
        # The two sizes of the split-precision benchmark configuration.
        {"name": "density_n4096_fp16", "kind": "density", "n": 4096, "precision": "fp16", "band": "banded",
         "gap": False},
        {"name": "density_n8192_fp16", "kind": "density", "n": 8192, "precision": "fp16", "band": "banded",
         "gap": False},
        # The FP32 CUDA-core chain beyond one tile, ragged.
        {"name": "density_n3000_fp32", "kind": "density", "n": 3000, "precision": "fp32", "band": "banded",
         "gap": False},
        # 64 replicas of mixed size in one plan that the program keeps (the batched configuration).
        {"name": "plan_64_bf16", "kind": "plan", "count": 64, "top": 2048, "precision": "bf16"},
        # Forward derivative at the size of the differentiation configuration.
        {"name": "response_n4096_fp16", "kind": "response", "n": 4096, "precision": "fp16", "band": "banded"},
        # Forward solve, then the gradient of a scalar loss through it: ragged, one training step.
        {"name": "gradient_n1000_fp16", "kind": "gradient", "n": 1000, "precision": "fp16", "band": "dense"},
        # The FP64 result: chain plus two refinement layers.
        {"name": "refined_n4096", "kind": "refined", "n": 4096, "precision": "fp16", "band": "banded"},
        # Non-orthogonal basis: two congruences around the refined solve.
        {"name": "nonorth_n1800", "kind": "nonorth", "n": 1800, "precision": "fp16", "band": "banded"},
    ]


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["density", "density", "density", "plan", "response", "gradient", "refined", "nonorth"])
    band = rng.choice(["dense", "banded"])
    if kind == "density":
        precision = rng.choice(["fp16", "fp16", "bf16", "fp32"])
        hi = {"fp16": 7800, "bf16": 6000, "fp32": 3000}[precision]
        return {"kind": kind, "n": _log_size(rng, 100, hi), "precision": precision, "band": band,
                "gap": rng.random() < 0.25}
    if kind == "plan":
        return {"kind": kind, "count": rng.randint(8, 64), "top": rng.choice([512, 1024, 1536, 2048]),
                "precision": rng.choice(["bf16", "fp16"])}
    if kind in ("response", "gradient"):
        return {"kind": kind, "n": _log_size(rng, 200, 4000), "precision": rng.choice(["fp16", "bf16"]), "band": band}
    return {"kind": kind, "n": _log_size(rng, 300, 4000 if kind == "refined" else 2500), "precision": "fp16",
            "band": band}


# ----------------------------------- inputs -----------------------------------
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _uniform(g, n, lo, hi):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


class _Rotations:
    """U: layers of rotations of the pairs (i, i + stride), i // stride even, then odd."""

    def __init__(self, n, band, g):
        reach = n if band == "dense" else min(n, 64)
        self.layers = []
        stride = 1
        while stride < reach:
            for odd in (0, 1):
                i = torch.arange(n - stride, device="cuda")
                i = i[(i // stride) % 2 == odd]
                if i.numel():
                    angle = _uniform(g, i.numel(), -1.0, 1.0) * (math.pi if band == "dense" else 0.6)
                    self.layers.append((i, i + stride, torch.cos(angle)[:, None], torch.sin(angle)[:, None]))
            stride *= 2

    def rows(self, a):
        """U a, in place."""
        for i, j, c, s in self.layers:
            x, y = a[i], a[j]
            a[i] = c * x - s * y
            a[j] = s * x + c * y
        return a

    def conjugate(self, d):
        """U diag(d) U^T, bit-symmetric."""
        a = self.rows(torch.diag(d))
        a = self.rows(a.t().contiguous())
        return (a + a.t()) * 0.5


def _spectrum(n, g):
    """(occupied states, eigenvalues ascending in two groups, rotations' order)."""
    n_occ = n // 2
    occ, virt = _uniform(g, n_occ, -1.0, -0.05), _uniform(g, n - n_occ, 0.05, 1.0)
    lam = torch.cat([occ, virt])
    return n_occ, lam[torch.randperm(n, generator=g, device="cuda")]


def _system(n, band, g):
    n_occ, lam = _spectrum(n, g)
    return n_occ, lam, _Rotations(n, band, g)


def _symmetric(n, g, sigma, reach=None):
    a = torch.randn(n, n, generator=g, device="cuda", dtype=torch.float64) * sigma
    if reach is not None:
        i = torch.arange(n, device="cuda")
        a = torch.where((i[:, None] - i[None, :]).abs() <= reach, a, torch.zeros((), device="cuda", dtype=a.dtype))
    return a.triu() + a.triu(1).t()


def _inverse_factor(n, g):
    """Z: unit lower triangular with a few decaying sub-diagonals, as an inverse Cholesky factor of an overlap."""
    z = torch.eye(n, device="cuda", dtype=torch.float64)
    for d in range(1, min(17, n)):
        i = torch.arange(n - d, device="cuda")
        z[i + d, i] = torch.randn(n - d, generator=g, device="cuda", dtype=torch.float64) * 0.05 * math.exp(-d / 4)
    return z


def _batch_sizes(case, g):
    steps = case["top"] // 128
    return [128 * (1 + int(k)) for k in torch.randint(steps, (case["count"],), generator=g, device="cuda").tolist()]


def _made(case, seed):
    """The inputs of a case, and what their exact results are made of."""
    g = _generator(seed)
    if case["kind"] == "plan":
        # The sizes belong to the case (a plan is made for its sizes); the matrices to the seed.
        sizes = _batch_sizes(case, _generator(case["count"] * 4099 + case["top"]))
        return {"systems": [_system(n, "dense", g) for n in sizes]}
    n = case["n"]
    n_occ, lam, rot = _system(n, case["band"], g)
    made = {"n_occ": n_occ, "lam": lam, "rot": rot, "H": rot.conjugate(lam)}
    if case["kind"] == "response":
        made["H1"] = _symmetric(n, g, 0.01, 64)
    elif case["kind"] == "gradient":
        made["G"] = _symmetric(n, g, 1.0)
    elif case["kind"] == "nonorth":
        made["Z"] = _inverse_factor(n, g)
        # H in the non-orthogonal basis: Z^T H Z is the orthogonal one, so H = Z^-T H_orth Z^-1.
        w = torch.linalg.solve_triangular(made["Z"], torch.eye(n, device="cuda", dtype=torch.float64), upper=False)
        h = w.t() @ made["H"] @ w
        made["H"] = (h + h.t()) * 0.5
    return made


def prepare(case, seed):
    made = _made(case, seed)
    if case["kind"] == "plan":
        Hs = [rot.conjugate(lam) for _, lam, rot in made["systems"]]
        occ = [n_occ for n_occ, _, _ in made["systems"]]
        return {"case": case, "plan": sp2.BatchPlan(Hs, occ, precision=case["precision"], autotune=False)}
    state = {"case": case, "n_occ": made["n_occ"]}
    for key in ("H", "H1", "G", "Z"):
        if key in made:
            state[key] = made[key]
    if case.get("gap"):
        # Estimates inside the gap, a little off its edges, as an MD step has them from the step before.
        state["gap"] = (float(made["lam"][made["lam"] < 0].max()) + 0.005, float(made["lam"][made["lam"] > 0].min()) - 0.005)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "plan":
        state["plan"].launch()
        return list(state["plan"].Ds)
    n_occ, precision = state["n_occ"], case["precision"]
    if kind == "density":
        D, res = sp2.density(state["H"], n_occ, precision=precision, gap=state.get("gap"))
        return {"D": D, "band_energy": res.band_energy}
    if kind == "response":
        D, D1, res = sp2.response(state["H"], state["H1"], n_occ, precision=precision)
        return {"D": D, "D1": D1, "band_energy": res.band_energy}
    if kind == "gradient":
        D, fwd = sp2.density(state["H"], n_occ, precision=precision)
        _, dH, _ = sp2.adjoint(state["H"], state["G"], n_occ, precision=precision, fwd=fwd)
        return {"D": D, "dH": dH}
    if kind == "refined":
        D, res = sp2.density_refined(state["H"], n_occ, refine_layers=2, precision=precision)
        return {"D": D, "band_energy": res.band_energy}
    D, res = sp2.density_nonorth(state["H"], state["Z"], n_occ, refine_layers=2, precision=precision)
    return {"D": D, "band_energy": res.band_energy}


# ------------------------------------ work ------------------------------------
def work(case):
    """Per layer one product of symmetric matrices (its upper half: N^3 flops); H read and D written once."""
    if case["kind"] == "plan":
        sizes = _batch_sizes(case, _generator(case["count"] * 4099 + case["top"]))
        return {"bytes": sum(12 * n * n for n in sizes), "flops": sum(LAYERS["plain"] * n ** 3 for n in sizes)}
    n = case["n"]
    layers = LAYERS["accelerated" if case.get("gap") else "plain"]
    if case["kind"] == "density":
        return {"bytes": 12 * n * n, "flops": layers * n ** 3}
    if case["kind"] == "response":  # the square, and X X1 + X1 X (upper half of two products)
        return {"bytes": 24 * n * n, "flops": layers * 3 * n ** 3}
    if case["kind"] == "gradient":  # forward twice (the gradient call replays it), and the reverse sweep
        return {"bytes": 36 * n * n, "flops": layers * 4 * n ** 3}
    if case["kind"] == "refined":
        return {"bytes": 16 * n * n, "flops": (layers + 2) * n ** 3}
    return {"bytes": 24 * n * n, "flops": (layers + 2 + 6) * n ** 3}


# ----------------------------------- exact ------------------------------------
def _derivative(lam, rot, M):
    """First-order change of theta(mu - H) for a symmetric change M of H."""
    n = lam.numel()
    u = rot.rows(torch.eye(n, device="cuda", dtype=torch.float64))
    f = (lam < 0).to(torch.float64)
    df, dl = f[:, None] - f[None, :], lam[:, None] - lam[None, :]
    k = torch.where(df != 0, df / torch.where(df != 0, dl, torch.ones_like(dl)), torch.zeros_like(dl))
    return u @ (k * (u.t() @ M @ u)) @ u.t()


def exact(case, seed):
    made = _made(case, seed)
    if case["kind"] == "plan":
        return [rot.conjugate((lam < 0).to(torch.float64)) for _, lam, rot in made["systems"]]
    lam, rot = made["lam"], made["rot"]
    occupied = (lam < 0).to(torch.float64)
    D = rot.conjugate(occupied)
    energy = float((lam * occupied).sum())
    if case["kind"] == "response":
        return {"D": D, "D1": _derivative(lam, rot, made["H1"]), "band_energy": energy}
    if case["kind"] == "gradient":
        return {"D": D, "dH": _derivative(lam, rot, made["G"])}
    if case["kind"] == "nonorth":
        D = made["Z"] @ D @ made["Z"].t()
    return {"D": D, "band_energy": energy}
