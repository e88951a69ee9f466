"""The work this library does for its users, as measurable cases.

A case is one call sequence a program makes with the public Python binding
(paper_1106_5990_gb300.amgd / .autograd) on one matrix, at one size:

  replay    a captured build replayed for new values of A on the same pattern
            (a time-dependent or nonlinear solve that rebuilds its strength
            graph every step): values in, strength CSR out
  oneshot   amgd.build() on a sparse CUDA tensor: handle, sweeps, distances and
            strength graph of a matrix that is seen once
  steps     the calls of the path one by one on a handle the program keeps:
            start vectors, sweeps, distances (a, r, LS), strength CSR
  smooth    sweeps alone on vectors of the caller's own (the 7 random + 1
            constant start and 40 Gauss-Seidel sweeps of the paper's section 5.2)
  train     one training step through autograd: the built-in loss on the
            distances and its gradient with respect to A's values and omega
  depth     distances and strength graph over the graph of A^2, on vectors that
            have been relaxed before
  coarsen   compatible-relaxation coarsening (Algorithm 1) from given distances
  interp    least-squares interpolation over a given coarse set (section 4.3)

Matrices are made on the GPU.  The pattern of a case depends on its sizes only
and the values on the seed, so outputs of two seeds have the same shapes.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1106_5990_gb300 import amgd, autograd

DEV = "cuda"
THETA = 0.5
DEPTH = 2           # search depth of the "depth" cases
GAMMA = 1.5         # size penalty of the "interp" cases
CR = dict(nu=5, theta=0.5, delta=0.6, tol=0.5, max_sets=12, omega=1.0)


def listed():
    def case(name, kind, matrix, n, K, storage, sweep, nu, omega, **more):
        return dict(name=name, kind=kind, matrix=matrix, n=n, K=K, storage=storage, sweep=sweep,
                    nu=nu, omega=omega, **more)
    return [
        # the smallest repeated build: a 64x64 five-point grid, everything in cache, bound by
        # launches and latency
        case("replay_p5_64_fp64", "replay", "p5", 64, 8, "fp64", "jacobi", 4, 2 / 3),
        # a build of the size most of the paper's experiments have, done once: 7-point, 128x128
        case("oneshot_a7_128_fp64", "oneshot", "a7", 128, 8, "fp64", "jacobi", 4, 2 / 3),
        # a matrix that arrives on the GPU, is analysed once and dropped: a graph Laplacian
        case("oneshot_graph_150k_fp32", "oneshot", "graph", 150000, 16, "fp32", "jacobi", 4, 2 / 3),
        # odd everything: 333x333 grid, K = 13, LS weights, a proper three-coloring, FP64
        case("steps_a7_333_k13_fp64", "steps", "a7", 333, 13, "fp64", "color3", 4, 1.0, weights=True),
        # the largest: 3D diffusion with jumping coefficients, K = 32, every output kept
        case("steps_jump_128_k32_fp32", "steps", "jump", 128, 32, "fp32", "jacobi", 6, 0.8),
        # the benchmark's workload as a program runs it: new values, one replay
        case("replay_a9_1024_fp32", "replay", "a9", 1024, 16, "fp32", "redblack", 8, 1.0),
        # a batch of graph Laplacians of uneven size in one handle, BF16 vectors
        case("replay_graphs_bf16", "replay", "graphs", 200000, 16, "bf16", "jacobi", 4, 2 / 3, nmat=6),
        # the paper's own recipe for test vectors, in FP64
        case("smooth_a7_400_fp64", "smooth", "a7", 400, 8, "fp64", "color3", 40, 1.0),
        # learning the entries of A: forward and reverse pass
        case("train_a5_512_fp32", "train", "a5", 512, 16, "fp32", "jacobi", 10, 2 / 3),
        # long-range strength: 25 entries per row
        case("depth2_a9_512_bf16", "depth", "a9", 512, 16, "bf16", "redblack", 8, 1.0),
        # the two steps of a multigrid setup that use the distances
        case("coarsen_a9_512", "coarsen", "a9", 512, 16, "fp64", "redblack", 4, 1.0),
        case("interp_a9_512", "interp", "a9", 512, 16, "fp64", "redblack", 4, 1.0, caliber=2),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    kind = rng.choice(["replay", "oneshot", "steps", "smooth", "train", "depth", "coarsen", "interp"])
    K = rng.choice([5, 8, 8, 12, 16, 16, 24, 32])
    storage = rng.choice(["fp64", "fp32", "bf16"])
    sweep = rng.choice(["jacobi", "redblack", "color3"])
    matrix = rng.choice(["p5", "a5", "a7", "a9"])
    n = log_int(48, 900)
    more = {}
    if kind in ("replay", "oneshot", "steps") and rng.random() < 0.4:
        matrix, sweep = rng.choice([("jump", "jacobi"), ("graph", "jacobi")] +
                                   ([("graphs", "jacobi")] if kind == "replay" else []))
        n = log_int(12, 110) if matrix == "jump" else log_int(3000, 250000)
        if matrix == "graphs":
            more["nmat"] = rng.randint(2, 5)
    if kind == "oneshot":
        sweep = "jacobi"
    if kind == "steps":
        more["weights"] = rng.random() < 0.3
    if kind == "smooth":
        storage, n = rng.choice(["fp64", "fp32"]), log_int(48, 600)
    if kind == "train":
        storage, sweep, n = rng.choice(["fp64", "fp32"]), "jacobi", log_int(48, 600)
    if kind == "depth":
        n = log_int(48, 512)
    if kind in ("coarsen", "interp"):
        storage, K, n = "fp64", rng.choice([8, 16]), log_int(48, 600)
        matrix, sweep = rng.choice([("a9", "redblack"), ("a7", "color3"), ("p5", "redblack")])
    if kind == "interp":
        more["caliber"] = rng.choice([1, 2, 2, 3])
    while _rows(dict(matrix=matrix, n=n, **more)) * K > 30_000_000:
        K = max(4, K // 2)
    return dict(kind=kind, matrix=matrix, n=n, K=K, storage=storage, sweep=sweep,
                nu=rng.choice([2, 4, 6, 10]), omega=1.0 if sweep != "jacobi" else 2 / 3, **more)


# ---------------------------------------------------------------------------
# matrices
# ---------------------------------------------------------------------------
def _rows(case):
    n = case["n"]
    if case["matrix"] == "jump":
        return n ** 3
    if case["matrix"] == "graphs":
        return sum(_graph_sizes(case))
    return n if case["matrix"] == "graph" else n * n


def _graph_sizes(case):
    # uneven sizes between n / 20 and n
    m = case["nmat"]
    return [max(64, int(case["n"] * (0.05 + 0.95 * (b + 0.5) / m))) for b in range(m)]


_WIDTH = {"p5": 5, "a5": 5, "a7": 7, "a9": 9, "jump": 7, "graph": 17, "graphs": 17}


def _stencil(case, g):
    """{(dx, dy): value}; the anisotropy and its angle come from the seed."""
    m = case["matrix"]
    u = torch.rand(2, generator=g).tolist()
    if m == "p5":
        s = 1.0 + u[0]
        return {(0, 0): 2 + 2 * s, (1, 0): -1.0, (-1, 0): -1.0, (0, 1): -s, (0, -1): -s}
    if m == "a5":
        e = 1e-2 * (1 + u[0])
        return {(0, 0): 2 + 2 * e, (1, 0): -1.0, (-1, 0): -1.0, (0, 1): -e, (0, -1): -e}
    eps, al = 1e-3 * (1 + u[0]), math.pi / 6 + 0.2 * (u[1] - 0.5)
    a = math.cos(al) ** 2 + eps * math.sin(al) ** 2
    b = (1 - eps) * math.sin(2 * al)
    c = math.sin(al) ** 2 + eps * math.cos(al) ** 2
    if m == "a7":
        h = b / 2
        return {(0, 0): 2 * a + 2 * c - b, (1, 0): -a + h, (-1, 0): -a + h, (0, 1): -c + h,
                (0, -1): -c + h, (1, 1): -h, (-1, -1): -h}
    return {(0, 0): 2 * a + 2 * c, (1, 0): -a, (-1, 0): -a, (0, 1): -c, (0, -1): -c,
            (1, 1): -b / 4, (-1, -1): -b / 4, (1, -1): b / 4, (-1, 1): b / 4}


def _csr(n, col, val, mask):
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(mask.sum(1), 0, out=rp[1:])
    return rp, col[mask].to(torch.int32), val[mask]


def _grid_offsets(N, offs):
    i = torch.arange(N * N, device=DEV)
    iy, ix = i // N, i % N
    jx = torch.stack([ix + dx for dx, _ in offs], 1)
    jy = torch.stack([iy + dy for _, dy in offs], 1)
    return jy * N + jx, (jx >= 0) & (jx < N) & (jy >= 0) & (jy < N)


def _graph(n, pattern, seed, shift):
    """Graph Laplacian: Poisson(8) targets per node made symmetric, lognormal weights."""
    gp = torch.Generator(DEV).manual_seed(pattern)
    gv = torch.Generator(DEV).manual_seed(seed)
    deg = torch.poisson(torch.full((n,), 8.0, device=DEV), generator=gp).long()
    src = torch.repeat_interleave(torch.arange(n, device=DEV), deg)
    dst = torch.randint(0, n - 1, (src.numel(),), generator=gp, device=DEV)
    dst = dst + (dst >= src)
    key = torch.unique(torch.minimum(src, dst) * n + torch.maximum(src, dst))
    lo, hi = key // n, key % n
    w = torch.exp(torch.randn(key.numel(), generator=gv, device=DEV, dtype=torch.float64))
    d = torch.zeros(n, dtype=torch.float64, device=DEV)
    d.index_add_(0, lo, w).index_add_(0, hi, w)
    diag = torch.arange(n, device=DEV)
    r, c = torch.cat([lo, hi, diag]), torch.cat([hi, lo, diag])
    v = torch.cat([-w, -w, d + shift])
    order = torch.argsort(r * n + c)
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(r, minlength=n), 0, out=rp[1:])
    return rp, c[order].to(torch.int32), v[order]


def _matrices(case, seed):
    """The case's matrices as (row_ptr, col, val) on the GPU, columns ascending."""
    m, N = case["matrix"], case["n"]
    if m == "graph":
        return [_graph(N, N, seed, 1e-6)]
    if m == "graphs":
        return [_graph(s, N + b, seed * 1000 + b, 1e-6) for b, s in enumerate(_graph_sizes(case))]
    if m == "jump":
        # cell-centred 7-point diffusion, kappa = exp(2z), harmonic face means
        g = torch.Generator(DEV).manual_seed(seed)
        n = N ** 3
        kappa = torch.exp(2 * torch.randn(n, generator=g, device=DEV, dtype=torch.float64))
        i = torch.arange(n, device=DEV)
        ix, iy, iz = i % N, (i // N) % N, i // (N * N)
        col, val, mask = [], [], []
        diag = torch.zeros(n, dtype=torch.float64, device=DEV)
        for dx, dy, dz in [(0, 0, -1), (0, -1, 0), (-1, 0, 0), (0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1)]:
            jx, jy, jz = ix + dx, iy + dy, iz + dz
            ok = (jx >= 0) & (jx < N) & (jy >= 0) & (jy < N) & (jz >= 0) & (jz < N)
            j = torch.where(ok, (jz * N + jy) * N + jx, 0)
            col.append(j)
            mask.append(ok)
            if dx == dy == dz == 0:
                val.append(diag)
                continue
            kf = torch.where(ok, 2 * kappa * kappa[j] / (kappa + kappa[j]), 2 * kappa)
            diag += kf
            val.append(-kf)
        return [_csr(n, torch.stack(col, 1), torch.stack(val, 1), torch.stack(mask, 1))]
    st = _stencil(case, torch.Generator().manual_seed(seed))
    offs = sorted(st, key=lambda t: (t[1], t[0]))
    col, mask = _grid_offsets(N, offs)
    val = torch.tensor([st[o] for o in offs], dtype=torch.float64, device=DEV).expand(N * N, len(offs))
    return [_csr(N * N, col, val, mask)]


def _joined(mats):
    """One block-diagonal CSR of a batch."""
    rps, cols, vals, ro, so = [torch.zeros(1, dtype=torch.int64, device=DEV)], [], [], 0, 0
    for rp, col, val in mats:
        rps.append(rp[1:] + so)
        cols.append(col + ro)
        vals.append(val)
        ro += rp.numel() - 1
        so += col.numel()
    return torch.cat(rps), torch.cat(cols), torch.cat(vals)


def _color(case):
    N = case["n"]
    if case["sweep"] == "jacobi":
        return None
    i = torch.arange(N * N, device=DEV)
    return ((i % N + i // N) % (2 if case["sweep"] == "redblack" else 3)).to(torch.int32)


def _weights(case):
    K = case["K"]
    return np.linspace(0.5, 1.5, K) if case.get("weights") else None


def _own_start(case, rows, seed):
    """K - 1 random vectors and the constant."""
    g = torch.Generator(DEV).manual_seed(seed + 77)
    X = 2 * torch.rand(rows, case["K"], generator=g, device=DEV, dtype=torch.float64) - 1
    X[:, -1] = 1.0
    return X.contiguous()


def _coarse(case, seed):
    """Every second grid line in both directions, and a fifth of the other points."""
    N = case["n"]
    g = torch.Generator(DEV).manual_seed(seed + 5)
    i = torch.arange(N * N, device=DEV)
    c = (i % N % 2 == 0) & (i // N % 2 == 0)
    return (c | (torch.rand(N * N, generator=g, device=DEV) < 0.2)).to(torch.uint8)


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind, K = case["kind"], case["K"]
    mats = _matrices(case, seed)
    if kind == "oneshot":
        rp, col, val = mats[0]
        n = rp.numel() - 1
        return dict(case=case, seed=seed, n=n, E=val.numel() - n,
                    A=torch.sparse_csr_tensor(rp, col, val, size=(n, n)))
    if len(mats) > 1:
        h = amgd.Handle(None, None, None, K, seed=seed,
                        batch=[tuple(t.cpu().numpy() for t in m) for m in mats])
    else:
        h = amgd.Handle(*mats[0], K=K, seed=seed)
    rp, col, val = _joined(mats)
    st = dict(case=case, seed=seed, h=h, val=val,
              sweep=amgd.AMGD_SWEEP_JACOBI if case["sweep"] == "jacobi" else amgd.AMGD_SWEEP_MCGS)
    h.set_precision(case["storage"])
    color = _color(case)
    if color is not None:
        h.set_coloring(color)
    if kind == "depth":
        h.set_search_depth(DEPTH)
    w = _weights(case)
    if w is not None:
        h.set_weights(w)
    if kind in ("replay", "steps", "depth"):
        st["s_rp"] = torch.zeros(h.n + 1, dtype=torch.int64, device=DEV)
        st["s_col"] = torch.zeros(max(h.E_p, 1), dtype=torch.int32, device=DEV)
    if kind in ("steps", "depth"):
        st["out"] = {k: torch.zeros(h.nnz_p, dtype=torch.float64, device=DEV) for k in ("a", "dist", "ls")}
    if kind == "replay":
        # a program that replays a build tunes its kernels once
        h.autotune(st["sweep"], case["omega"])
        h.graph_capture(seed, case["nu"], case["omega"], st["sweep"], THETA, st["s_rp"], st["s_col"])
    elif kind == "smooth":
        st["X"] = _own_start(case, h.n, seed)
        st["Y"] = torch.zeros_like(st["X"])
    elif kind == "train":
        h.autotune(st["sweep"], case["omega"])
        st["omega"] = torch.tensor(case["omega"], dtype=torch.float64, device=DEV, requires_grad=True)
        st["val"] = val.clone().requires_grad_(True)
    elif kind == "depth":
        h.relax(case["nu"], case["omega"], st["sweep"])
    elif kind == "coarsen":
        X = _relaxed(case, rp, col, val, _own_start(case, h.n, seed))
        st["ls"] = _fits(rp, col, val, X, None, rp, col)[1]
        st["C0"] = torch.zeros(h.n, dtype=torch.uint8, device=DEV)
        st["C"] = torch.zeros(h.n, dtype=torch.uint8, device=DEV)
        st["rho"] = np.zeros(CR["max_sets"] + 1)
    elif kind == "interp":
        h.set_vectors(_relaxed(case, rp, col, val, _own_start(case, h.n, seed)))
        st["C"] = _coarse(case, seed)
        cap = h.n * case["caliber"]
        st["p_rp"] = torch.zeros(h.n + 1, dtype=torch.int64, device=DEV)
        st["p_col"] = torch.zeros(cap, dtype=torch.int32, device=DEV)
        st["p_val"] = torch.zeros(cap, dtype=torch.float64, device=DEV)
        st["row_ls"] = torch.zeros(h.n, dtype=torch.float64, device=DEV)
    return st


def run(st):
    case, seed = st["case"], st["seed"]
    kind = case["kind"]
    if kind == "oneshot":
        a, dist, (s_rp, s_col) = amgd.build(st["A"], case["K"], seed=seed, nu=case["nu"],
                                            omega=case["omega"], theta=THETA,
                                            precision=case["storage"])
        # the number of strong edges depends on the values: padded to the pattern's
        return a, dist, s_rp, torch.nn.functional.pad(s_col, (0, st["E"] - s_col.numel()))
    h = st["h"]
    if kind == "replay":
        h.set_values_async(st["val"])
        h.graph_launch()
        return st["s_rp"], st["s_col"]
    if kind == "steps":
        h.init_vectors(seed)
        h.relax(case["nu"], case["omega"], st["sweep"])
        h.distances(THETA, out=st["out"])
        h.strength(st["s_rp"], st["s_col"])
        return st["out"]["a"], st["out"]["dist"], st["out"]["ls"], st["s_rp"], st["s_col"]
    if kind == "smooth":
        h.set_vectors(st["X"])
        h.relax(case["nu"], case["omega"], st["sweep"])
        return h.get_vectors(st["Y"])
    if kind == "train":
        loss = autograd.strength_loss(h, st["val"], st["omega"], seed, case["nu"], THETA)
        gv, gw = torch.autograd.grad(loss, (st["val"], st["omega"]))
        return loss.detach(), gv, gw
    if kind == "depth":
        h.distances(THETA, out=st["out"])
        h.strength(st["s_rp"], st["s_col"])
        return st["out"]["a"], st["out"]["dist"], st["out"]["ls"], st["s_rp"], st["s_col"]
    if kind == "coarsen":
        st["C"].copy_(st["C0"])
        stages = ctypes.c_int32()
        amgd.check(amgd.amgd_cr_coarsen(h.h, st["C"].data_ptr(), amgd.AMGD_MEM_DEVICE,
                                        st["ls"].data_ptr(), amgd.AMGD_MEM_DEVICE, st["sweep"],
                                        CR["omega"], CR["nu"], CR["theta"], CR["delta"], CR["tol"],
                                        CR["max_sets"], seed, st["rho"].ctypes.data,
                                        ctypes.byref(stages)), h.h)
        return st["C"], st["rho"], stages.value
    nnz = ctypes.c_int64()
    amgd.check(amgd.amgd_ls_interpolation(h.h, st["C"].data_ptr(), amgd.AMGD_MEM_DEVICE,
                                          case["caliber"], GAMMA, st["p_rp"].data_ptr(),
                                          st["p_col"].data_ptr(), st["p_val"].data_ptr(),
                                          st["p_col"].numel(), ctypes.byref(nnz),
                                          st["row_ls"].data_ptr(), amgd.AMGD_MEM_DEVICE), h.h)
    return st["p_rp"], st["p_col"], st["p_val"], st["row_ls"], nnz.value


def work(case):
    """Inputs read once, outputs written once; the fused multiply-adds of the path."""
    kind, n, K, nu = case["kind"], _rows(case), case["K"], case["nu"]
    nnz = n * _WIDTH[case["matrix"]]
    A = 12 * nnz + 8 * n
    S = 8 * n + 4 * nnz // 2
    if kind in ("replay", "oneshot", "steps"):
        outs = {"replay": 0, "oneshot": 16 * nnz, "steps": 24 * nnz}[kind]
        return dict(bytes=A + S + outs, flops=2 * nnz * K * (nu + 5))
    if kind == "smooth":
        return dict(bytes=A + 16 * n * K, flops=2 * nnz * K * nu)
    if kind == "train":
        return dict(bytes=A + 8 * nnz, flops=2 * nnz * K * (3 * nu + 15))
    if kind == "depth":
        wide = {"a9": 25, "a7": 19}.get(case["matrix"], 13) * n
        es = {"fp64": 8, "fp32": 4, "bf16": 2}[case["storage"]]
        return dict(bytes=A + es * n * K + 28 * wide + 8 * n, flops=2 * K * (nnz + 4 * wide))
    if kind == "coarsen":
        return dict(bytes=A + 8 * nnz + n, flops=2 * nnz * CR["nu"])
    return dict(bytes=A + 8 * n * K + 9 * n + 12 * n * case["caliber"], flops=2 * n * K * 40)


# ---------------------------------------------------------------------------
# the same results in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _start(n, K, seed, b):
    """X0 of matrix b: Philox4x64-10 at counter (i, k / 8, 0, 0), key (seed, b)."""
    X = np.empty((n, -(-K // 8) * 8))
    for blk in range(-(-K // 8)):
        before = ((blk << 64) - 1) % (1 << 256)      # the generator counts before it draws
        g = np.random.Philox(key=[seed, b], counter=[(before >> s) % (1 << 64) for s in (0, 64, 128, 192)])
        m = g.random_raw(4 * n).view(np.uint32).reshape(n, 8).astype(np.float64)
        X[:, 8 * blk:8 * blk + 8] = (2 * m + 1) * 2.0 ** -32 - 1
    return torch.from_numpy(X[:, :K].copy()).to(DEV)


def _spmm(rp, col, val, X):
    """A X, differentiable in val and X."""
    row = torch.repeat_interleave(torch.arange(rp.numel() - 1, device=DEV), rp.diff())
    return torch.zeros_like(X).index_add(0, row, val[:, None] * X[col.long()])


def _diag(rp, col, val):
    row = torch.repeat_interleave(torch.arange(rp.numel() - 1, device=DEV), rp.diff())
    return val[col == row]


def _relaxed(case, rp, col, val, X, omega=None):
    """nu weighted-Jacobi sweeps, or Gauss-Seidel over the colors: a row takes the new values
    of smaller colors and the sweep's start values of all others."""
    omega = case["omega"] if omega is None else omega
    c = (omega / _diag(rp, col, val))[:, None]
    color = _color(case)
    if color is None:
        for _ in range(case["nu"]):
            X = X - c * _spmm(rp, col, val, X)
        return X
    color = color[:, None]
    A = torch.sparse_csr_tensor(rp, col.long(), val, size=(rp.numel() - 1,) * 2)
    for _ in range(case["nu"]):
        new = X
        for k in range(int(color.max()) + 1):
            new = torch.where(color == k, X - c * (A @ torch.where(color < k, new, X)), new)
        X = new
    return X


def _fits(rp, col, val, X, w, prp, pcol):
    """(a, LS) per slot of the pattern (prp, pcol): 0 and NaN on the diagonal."""
    Y = X - _spmm(rp, col, val, X) / _diag(rp, col, val)[:, None]
    w = 1.0 if w is None else torch.as_tensor(w, device=DEV)
    row = torch.repeat_interleave(torch.arange(prp.numel() - 1, device=DEV), prp.diff())
    pcol = pcol.long()
    y, x = Y[row], X[pcol]
    a = (w * x * y).sum(1) / (w * x * x).sum(1)
    ls = (w * (y - a[:, None] * x).square()).sum(1)
    # a row of A with a single off-diagonal fits it exactly
    single = (rp.diff() == 2)[row]
    if bool(single.any()):
        r0 = torch.repeat_interleave(torch.arange(rp.numel() - 1, device=DEV), rp.diff())
        off = r0 != col
        v1 = torch.zeros(rp.numel() - 1, dtype=val.dtype, device=DEV).index_put((r0[off],), val[off].detach())
        j1 = torch.zeros_like(rp[1:]).index_put((r0[off],), col[off].long())
        hit = single & (pcol == j1[row])
        a = torch.where(hit, (-v1 / _diag(rp, col, val))[row], a)
        ls = torch.where(hit, torch.zeros_like(ls), ls)
    eye = row == pcol
    return torch.where(eye, torch.zeros_like(a), a), torch.where(eye, torch.full_like(ls, math.nan), ls)


def _strong(prp, pcol, ls):
    row = torch.repeat_interleave(torch.arange(prp.numel() - 1, device=DEV), prp.diff())
    l = torch.where(torch.isnan(ls), torch.full_like(ls, math.inf), ls)
    m = torch.full((prp.numel() - 1,), math.inf, dtype=l.dtype, device=DEV).scatter_reduce(0, row, l, "amin")
    return (row != pcol) & ((l == 0) | (THETA * l < m[row]))


def _pattern2(case):
    """The graph of A^2 of a grid stencil, columns ascending."""
    st = _stencil(case, torch.Generator().manual_seed(0))
    N = case["n"]
    one = [o for o in st if st[o] != 0.0]
    offs = sorted({(a + c, b + d) for a, b in one for c, d in one}, key=lambda t: (t[1], t[0]))
    col, mask = _grid_offsets(N, offs)
    # a two-step walk has to stay on the grid, which on a convex stencil it can
    rp, c, _ = _csr(N * N, col, col.double(), mask)
    return rp, c


def _cr_rho(case, rp, col, val, ls, seed):
    """rho of every stage of Algorithm 1 (max norm), by plain F-relaxation, thresholds and
    rounds of local maxima in the order (lambda, key, smaller index)."""
    n = rp.numel() - 1
    row = torch.repeat_interleave(torch.arange(n, device=DEV), rp.diff())
    cl = col.long()
    color = _color(case)
    d = _diag(rp, col, val)
    coarse = torch.zeros(n, dtype=torch.bool, device=DEV)
    rho = np.zeros(CR["max_sets"] + 1)
    for stage in range(CR["max_sets"] + 1):
        u = (~coarse).double()
        for _ in range(CR["nu"]):
            new = u
            for k in range(int(color.max()) + 1):
                hat = torch.where(color < k, new, u)
                s = torch.zeros_like(u).index_add(0, row, val * hat[cl])
                new = torch.where((color == k) & ~coarse, u - CR["omega"] / d * s, new)
            u = new
        norm = float(u.abs().max())
        rho[stage] = 0.0 if bool(coarse.all()) else norm ** (1.0 / CR["nu"])
        if not rho[stage] > CR["delta"] or stage >= CR["max_sets"]:
            break
        cand = ~coarse & (u.abs() / norm > CR["tol"])
        ff = ~coarse[row] & ~coarse[cl] & (row != cl)
        l = torch.where(ff, ls, torch.full_like(ls, math.inf))
        m = torch.full((n,), math.inf, dtype=ls.dtype, device=DEV).scatter_reduce(0, row, l, "amin")
        strong = ff & ((l == 0) | (CR["theta"] * l < m[row]))
        lam = torch.zeros(n, dtype=torch.int64, device=DEV).index_add(
            0, cl, (strong & cand[row] & cand[cl]).long())
        before = [(1 << 64) - 1, stage - 1, 1, 0] if stage else [(1 << 64) - 1, (1 << 64) - 1, 0, 0]
        raw = np.random.Philox(key=[seed, 0], counter=before).random_raw(4 * n)[::4]
        order = np.lexsort((np.arange(n)[::-1], raw, lam.cpu().numpy()))      # ascending priority
        pri = torch.empty(n, dtype=torch.int64, device=DEV)
        pri[torch.from_numpy(order.copy()).to(DEV)] = torch.arange(n, device=DEV)
        e = strong & cand[row] & cand[cl]
        a, b = torch.cat([row[e], cl[e]]), torch.cat([cl[e], row[e]])
        left = cand.clone()
        while bool(left.any()):
            live = left[a] & left[b]
            best = torch.full((n,), -1, dtype=torch.int64, device=DEV).scatter_reduce(0, a[live], pri[b[live]], "amax")
            take = left & (pri > best)
            coarse |= take
            left &= ~take
            left[b[take[a]]] = False
    return rho


def _interp(case, rp, col, val, X, coarse):
    """(P's values and LS per row): every subset of at most `caliber` coarse neighbours, fitted
    by normal equations; sizes compete with the penalty."""
    import itertools
    n, dev = rp.numel() - 1, DEV
    Y = X - _spmm(rp, col, val, X) / _diag(rp, col, val)[:, None]
    row = torch.repeat_interleave(torch.arange(n, device=dev), rp.diff())
    cand = (coarse[col.long()] == 1) & (coarse[row] == 0)
    cnt = torch.zeros(n, dtype=torch.int64, device=dev).index_add(0, row, cand.long())
    ptr = torch.cumsum(cnt, 0) - cnt
    cols = col.long()[cand]
    out_ls = torch.zeros(n, dtype=torch.float64, device=dev)
    wts = torch.zeros(n, case["caliber"], dtype=torch.float64, device=dev)
    size = torch.zeros(n, dtype=torch.int64, device=dev)
    out_ls[:] = torch.where(coarse == 1, 0.0, Y.square().sum(1))
    size[coarse == 1] = 1
    wts[coarse == 1, 0] = 1.0
    for m in range(1, int(cnt.max()) + 1):
        i = torch.nonzero((cnt == m) & (coarse == 0)).flatten()
        if not i.numel():
            continue
        B, y = X[cols[ptr[i][:, None] + torch.arange(m, device=dev)]], Y[i]       # rows, m, K
        syy = y.square().sum(1)
        cur, cur_size = torch.ones_like(syy), torch.zeros_like(i)
        for s in range(1, min(case["caliber"], m) + 1):
            sets = torch.tensor(list(itertools.combinations(range(m), s)), device=dev)
            W = B[:, sets]                                                          # rows, sets, s, K
            G = W @ W.transpose(-1, -2)
            p = torch.linalg.solve_ex(G, W @ y[:, None, :, None])[0]
            ls = (y[:, None] - (p * W).sum(2)).square().sum(-1)
            ls = torch.where(torch.isfinite(ls), ls, torch.full_like(ls, math.inf))
            best, k = ls.min(1)
            win = (syy > 0) & (best / syy < cur ** (GAMMA * (s - cur_size)))
            cur = torch.where(win, best / syy, cur)
            cur_size = torch.where(win, s, cur_size)
            out_ls[i[win]] = best[win]
            size[i[win]] = s
            wts[i[win], :] = 0
            wts[i[win], :s] = p[torch.arange(len(i), device=dev), k].squeeze(-1)[win]
    pv = wts[torch.arange(case["caliber"], device=dev)[None, :] < size[:, None]]
    return torch.nn.functional.pad(pv, (0, n * case["caliber"] - pv.numel())), out_ls


def exact(case, seed):
    kind, K = case["kind"], case["K"]
    if kind == "replay":
        return None                                          # row pointer and columns only
    mats = _matrices(case, seed)
    rp, col, val = _joined(mats)
    n = rp.numel() - 1
    w = _weights(case)
    if kind == "smooth":
        return _relaxed(case, rp, col, val, _own_start(case, n, seed))
    if kind == "coarsen":
        X = _relaxed(case, rp, col, val, _own_start(case, n, seed))
        return None, _cr_rho(case, rp, col, val, _fits(rp, col, val, X, None, rp, col)[1], seed), None
    if kind == "interp":
        X = _relaxed(case, rp, col, val, _own_start(case, n, seed))
        pv, ls = _interp(case, rp, col, val, X, _coarse(case, seed))
        return None, None, pv, ls, None
    X = _start(n, K, seed, 0)
    if kind == "train":
        val = val.clone().requires_grad_(True)
        omega = torch.tensor(case["omega"], dtype=torch.float64, device=DEV, requires_grad=True)
        X = _relaxed(case, rp, col, val, X, omega)
        ls = _fits(rp, col, val, X, None, rp, col)[1]
        kept = _strong(rp, col, ls.detach()) & (ls.detach() > 0)
        loss = (1 / ls[kept]).square().sum()
        return (loss.detach(), *torch.autograd.grad(loss, (val, omega)))
    X = _relaxed(case, rp, col, val, X)
    prp, pcol = _pattern2(case) if kind == "depth" else (rp, col)
    a, ls = _fits(rp, col, val, X, w, prp, pcol)
    dist = 1 / ls
    if kind == "oneshot":
        return a, dist, None, None
    return a, dist, ls, None, None
