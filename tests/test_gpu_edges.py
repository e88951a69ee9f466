"""The kernels' dispatch edges on the GPU against the oracle.

Sweeps keep the rounding order of the definition on every route (the row's own
CSR entries or the sliced copy of the matrix that repeated sweeps read), so
FP64 vectors are compared bit for bit with the oracle and FP32/BF16 vectors bit
for bit between the two routes.  Distances are held to the parity rules of
parity.py; strength patterns, interpolation and everything a handle built from
device memory returns are compared exactly."""
import ctypes
import math

import numpy as np
import pytest

import oracle
from paper_1106_5990_gb300 import inputs
from test_gpu_adjoint import rel, run_gpu, x0
from test_gpu_parity import arrow, compare_fp64, gpu_build

pytestmark = pytest.mark.gpu
amgd = pytest.importorskip("paper_1106_5990_gb300.amgd")
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1106_5990_gb300 import _build
    _build.build()


# slices of 32 rows and their remainders; 2 to 9 entries in a slice's width;
# rows sorted by length within windows (uneven rows); one row far too long for a
# slice (the sweeps stay on the CSR)
SWEEPS = {
    "lap1d_31": lambda: inputs.lap1d(31),
    "lap1d_33": lambda: inputs.lap1d(33),
    "poisson5_37": lambda: inputs.poisson2d_5pt(37),
    "aniso7_33": lambda: inputs.aniso2d_7pt(33, 0.1, -math.pi / 4),
    "aniso9_66": lambda: inputs.aniso2d_9pt(66, 1e-3, math.pi / 6),
    "graph_4129": lambda: inputs.graph_laplacian(4129, 8.0, 4),
    "arrow_3001": lambda: arrow(3001),
}


def on_sliced_copy(h, sweep=amgd.AMGD_SWEEP_JACOBI):
    """A captured build makes the sliced copy (if the matrix has one): the handle's sweeps
    read it from there on.  The vectors stay."""
    s_rp = torch.empty(h.n + 1, dtype=torch.int64, device="cuda")
    s_col = torch.empty(max(h.E_p, 1), dtype=torch.int32, device="cuda")
    h.graph_capture(1, 1, 1.0, sweep, 0.5, s_rp, s_col)


@pytest.mark.parametrize("name", [*SWEEPS, "hub_3001"])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("K", [1, 5, 8, 32, 64])
@pytest.mark.parametrize("sweep", ["jacobi", "mcgs"])
def test_sweeps_on_the_sliced_copy(name, prec, K, sweep):
    """Against the CSR (one short call of a fresh handle) and, in FP64, the oracle; then
    with new values."""
    rp, col, val = hub(3001, (300,), 2) if name == "hub_3001" else SWEEPS[name]()
    n = len(rp) - 1
    color = inputs.greedy_coloring(rp, col) if sweep == "mcgs" else None
    mode, omode = (amgd.AMGD_SWEEP_MCGS, oracle.SWEEP_MCGS) if color is not None else (amgd.AMGD_SWEEP_JACOBI, 0)
    val2 = val * np.random.default_rng(8).uniform(1, 1.01, len(val))

    def handle(v):
        h = amgd.Handle(rp, col, v, K, 7)
        h.set_precision(prec)
        if color is not None:
            h.set_coloring(color)
        h.init_vectors(7)
        return h

    for v, update in ((val, False), (val2, True)):
        with handle(v) as h:
            h.relax(3, 0.9, mode)
            want = h.get_vectors()
        with handle(val) as h:
            on_sliced_copy(h, mode)
            if update:
                h.set_values(v)
            h.relax(1, 0.9, mode)
            h.relax(2, 0.9, mode)
            assert np.array_equal(h.get_vectors(), want)
        if prec == "fp64":
            assert np.array_equal(want, oracle.relax(rp, col, v, oracle.tv_init(n, K, 7), 3, 0.9, omode, color))


def test_a_copy_for_one_arithmetic_type():
    """A row of 300 entries in a small graph: the mixed sweeps read the copy, FP64 the CSR."""
    rp, col, val = hub(3001, (300,), 2)
    with amgd.Handle(rp, col, val, 8, 7) as h, amgd.Handle(rp, col, val, 8, 7) as fresh:
        for prec in ("fp64", "fp32", "bf16", "fp64", "fp32"):
            for k in (h, fresh):
                k.set_precision(prec)
                k.init_vectors(7)
            on_sliced_copy(h)
            h.set_values(val)
            h.relax(3, 0.9)
            fresh.relax(3, 0.9)
            assert np.array_equal(h.get_vectors(), fresh.get_vectors()), prec


def test_the_copy_is_built_when_it_has_paid():
    """A handle that is swept a few times allocates nothing for it; one whose sweeps go on
    gets the copy (11 MB of entries)."""
    rp, col, val = inputs.poisson2d_5pt(512)
    with amgd.Handle(rp, col, val, 8, 7) as h:
        h.relax(2, 0.7)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        h.relax(2, 0.7)
        h.relax(2, 0.7)
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] == free
        for _ in range(100):
            h.relax(4, 0.7)
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] <= free - (8 << 20)
        X = oracle.relax(rp, col, val, oracle.tv_init(len(rp) - 1, 8, 7), 406, 0.7)
        assert np.array_equal(h.get_vectors(), X)


def test_a_saved_line_for_the_csr_gives_the_copy_back(tmp_path):
    """A handle that has the copy and loads a line that says CSR: value updates need not
    keep the copy current any more."""
    import re
    rp, col, val = inputs.poisson2d_5pt(512)
    cache = tmp_path / "tune.txt"
    with amgd.Handle(rp, col, val, 8, 7) as h:
        h.autotune(amgd.AMGD_SWEEP_JACOBI, 0.7, str(cache))
    cache.write_text(re.sub(r";relax=(\d+),(\d+),(\d+),\d+(.*);sliced=[01]", r";relax=\1,\2,\3,0\4;sliced=0", cache.read_text()))
    with amgd.Handle(rp, col, val, 8, 7) as h:
        h.relax(400, 0.7)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        h.autotune(amgd.AMGD_SWEEP_JACOBI, 0.7, str(cache))
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] >= free + (8 << 20)
        h.set_values(2 * val)
        h.relax(3, 0.7)
        X = oracle.relax(rp, col, val, oracle.tv_init(len(rp) - 1, 8, 7), 403, 0.7)
        assert np.array_equal(h.get_vectors(), X)
    assert len(cache.read_text().splitlines()) == 1


def test_the_copy_is_built_beside_a_capture():
    """Another stream is captured in global mode while the handle's sweeps build the copy."""
    rp, col, val = SWEEPS["aniso9_66"]()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    x = torch.zeros(8, device="cuda")
    with amgd.Handle(rp, col, val, 8, 7) as h:   # every kernel is loaded
        h.relax(400, 0.7)
        h.relax(400, 0.7)
        want = h.get_vectors()
    with amgd.Handle(rp, col, val, 8, 7) as h:
        h.set_stream(s2)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s1, capture_error_mode="global"):
            x.add_(1)
            h.relax(400, 0.7)
            h.relax(400, 0.7)
            x.add_(1)
        s2.synchronize()
        assert np.array_equal(h.get_vectors(), want)
        g.replay()
        torch.cuda.synchronize()
        assert (x == 2).all()
        h.set_stream(None)


@pytest.mark.parametrize("name", list(SWEEPS))
@pytest.mark.parametrize("K", [1, 5, 8, 32, 64])
@pytest.mark.parametrize("sweep", ["jacobi", "mcgs"])
def test_repeated_sweeps_and_new_values(name, K, sweep):
    rp, col, val = SWEEPS[name]()
    n = len(rp) - 1
    color = inputs.greedy_coloring(rp, col) if sweep == "mcgs" else None
    mode, omode = (amgd.AMGD_SWEEP_MCGS, oracle.SWEEP_MCGS) if color is not None else (amgd.AMGD_SWEEP_JACOBI, 0)
    rng = np.random.default_rng(8)
    val2, val3, val4 = (val * (1 + 0.01 * rng.random(len(val))) for _ in range(3))
    with amgd.Handle(rp, col, val, K, 7) as h:
        if color is not None:
            h.set_coloring(color)
        X = oracle.tv_init(n, K, 7)
        for v, nu in ((None, 1), (None, 2), (val2, 2)):
            if v is not None:
                h.set_values(v)
            X = oracle.relax(rp, col, val if v is None else v, X, nu, 0.9, omode, color)
            h.relax(nu, 0.9, mode)
            assert np.array_equal(h.get_vectors(), X), nu
        h.set_values_async(torch.from_numpy(val3).cuda())
        h.relax(1, 0.9, mode)
        h.sync()
        X = oracle.relax(rp, col, val3, X, 1, 0.9, omode, color)
        assert np.array_equal(h.get_vectors(), X)
        # back to the CSR kernels, whose value copies the updates left out of date
        G, NV, U, _ = h.kernel_shape(amgd.AMGD_KERNEL_RELAX)
        try:
            h.set_kernel_shape(amgd.AMGD_KERNEL_RELAX, G, NV, U, 1)
        except amgd.AmgdError:
            return                               # this shape's stage exceeds the shared memory
        h.relax(1, 0.9, mode)
        X = oracle.relax(rp, col, val3, X, 1, 0.9, omode, color)
        assert np.array_equal(h.get_vectors(), X)
        h.set_values(val4)
        h.relax(1, 0.9, mode)
        X = oracle.relax(rp, col, val4, X, 1, 0.9, omode, color)
        assert np.array_equal(h.get_vectors(), X)


@pytest.mark.parametrize("built", [False, True])
@pytest.mark.parametrize("sweep", ["jacobi", "mcgs"])
def test_sweeps_in_a_graph_of_the_callers(built, sweep):
    """Sweeps that the caller's own capture records neither allocate nor wait, and the
    graph follows value updates, whichever copy of the matrix the handle's sweeps read."""
    rp, col, val = SWEEPS["aniso9_66"]()
    n, K = len(rp) - 1, 8
    color = inputs.greedy_coloring(rp, col) if sweep == "mcgs" else None
    mode, omode = (amgd.AMGD_SWEEP_MCGS, oracle.SWEEP_MCGS) if color is not None else (amgd.AMGD_SWEEP_JACOBI, 0)
    s = torch.cuda.Stream()
    with amgd.Handle(rp, col, val, K, 7) as h:
        if color is not None:
            h.set_coloring(color)
        h.set_stream(s)
        X = oracle.tv_init(n, K, 7)

        def eager(v):
            h.relax(2, 0.9, mode)
            return oracle.relax(rp, col, v, X, 2, 0.9, omode, color)

        X = eager(val)
        if built:
            X = eager(val)
            val = val * 1.25
            h.set_values(val)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            h.relax(2, 0.9, mode)
        assert np.array_equal(h.get_vectors(), X)        # recorded, not run
        for scale in (1.0, 1.5, 0.75):
            h.set_values(val * scale)
            with torch.cuda.stream(s):
                g.replay()
            s.synchronize()
            X = oracle.relax(rp, col, val * scale, X, 2, 0.9, omode, color)
            assert np.array_equal(h.get_vectors(), X), scale
            X = eager(val * scale)
            assert np.array_equal(h.get_vectors(), X), scale
        h.set_stream(None)


@pytest.mark.parametrize("built", [False, True])
@pytest.mark.parametrize("sweep", ["jacobi", "mcgs"])
def test_value_updates_in_a_graph_of_the_callers(built, sweep):
    """A recorded update reaches the sweeps of later calls, whether the sliced copy is there
    when it is recorded, is asked for afterwards or is given up with its coloring."""
    rp, col, val = SWEEPS["aniso9_66"]()
    n, K = len(rp) - 1, 8
    color = inputs.greedy_coloring(rp, col)
    mode, omode = (amgd.AMGD_SWEEP_MCGS, oracle.SWEEP_MCGS) if sweep == "mcgs" else (amgd.AMGD_SWEEP_JACOBI, 0)
    s = torch.cuda.Stream()
    buf = torch.from_numpy(val).cuda()
    with amgd.Handle(rp, col, val, K, 7) as h:
        h.set_coloring(color)
        h.set_stream(s)
        X = oracle.tv_init(n, K, 7)

        def eager(v):
            h.relax(1, 0.9, mode)
            return oracle.relax(rp, col, v, X, 1, 0.9, omode, color)

        h.set_values_async(buf)
        h.sync()
        X = eager(val)
        if built:
            on_sliced_copy(h, mode)
            X = eager(val)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            h.set_values_async(buf)
        h.sync()
        if not built:
            on_sliced_copy(h, mode)
        for _ in range(2):
            X = eager(val)
            assert np.array_equal(h.get_vectors(), X)    # recorded, not run
        for scale in (1.5, 0.75):
            v = val.copy()
            v[col != np.repeat(np.arange(n), np.diff(rp))] *= scale
            buf.copy_(torch.from_numpy(v))
            torch.cuda.synchronize()
            with torch.cuda.stream(s):
                g.replay()
            s.synchronize()
            for _ in range(2):
                X = eager(v)
                assert np.array_equal(h.get_vectors(), X), scale
            h.set_coloring((len(np.bincount(color)) - 1 - color).astype(np.int32))
            h.set_coloring(color)
        h.set_stream(None)


@pytest.mark.filterwarnings("ignore:DEBUG")
@pytest.mark.parametrize("warmed", ["sliced", "staged"])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_reverse_pass_in_a_graph_of_the_callers(warmed, prec, tmp_path):
    """A training step that the caller records recomputes its sweeps on the CSR, which the
    handle never frees, allocates nothing there, and follows value updates."""
    rp, col, val = SWEEPS["aniso9_66"]()
    K, nu, rng = 8, 4, np.random.default_rng(4)
    s = torch.cuda.Stream()
    vb = torch.zeros(len(val), dtype=torch.float64, device="cuda")

    def step(h):
        h.init_vectors(7)
        h.relax(nu, 0.6)
        amgd.check(amgd.amgd_distances(h.h, 0.5, None, None, None, amgd.AMGD_MEM_DEVICE), h.h)
        amgd.check(amgd.amgd_backward(h.h, None, amgd.AMGD_MEM_DEVICE, vb.data_ptr(), None, None), h.h)

    def handle(v):
        h = amgd.Handle(rp, col, v, K, 7)
        h.set_precision(prec)
        h.set_checkpointing(2)
        return h

    with handle(val) as h:
        h.set_stream(s)
        G, NV, U, _ = h.kernel_shape(amgd.AMGD_KERNEL_RELAX)
        if warmed == "staged":                   # the buffers exist, the sliced copy does not
            h.set_kernel_shape(amgd.AMGD_KERNEL_RELAX, G, NV, U, 1)
            step(h)
            h.set_kernel_shape(amgd.AMGD_KERNEL_RELAX, G, NV, U, 0)
        else:
            on_sliced_copy(h)
            step(h)
        s.synchronize()
        g = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(g, stream=s):
            step(h)
        g.debug_dump(str(tmp_path / "graph.dot"))
        kernels = (tmp_path / "graph.dot").read_text()
        assert "k_relax" in kernels and "k_relax_sell" not in kernels
        for _ in range(2):
            v = val * (1 + 0.3 * rng.random(len(val)))
            h.set_values(v)
            vb.zero_()
            torch.cuda.synchronize()
            with torch.cuda.stream(s):
                g.replay()
            s.synchronize()
            got = vb.cpu().numpy()
            with handle(v) as h2:
                step(h2)
                torch.cuda.synchronize()
            assert np.any(got) and np.array_equal(got, vb.cpu().numpy())
        h.set_stream(None)


@pytest.mark.parametrize("name", ["poisson5_37", "aniso9_66", "graph_4129", "arrow_3001"])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("K", [4, 16, 64])
def test_jacobi_sweeps_of_a_colored_handle(name, prec, K):
    """Jacobi sweeps run over all rows at once; the sliced copy is padded where a color
    ends (color sizes off the slices of 32 rows; rows in order and sorted by length)."""
    rp, col, val = SWEEPS[name]()
    n = len(rp) - 1
    color = inputs.greedy_coloring(rp, col)
    assert all(k % 32 for k in np.bincount(color))
    s_rp = torch.empty(n + 1, dtype=torch.int64, device="cuda")
    s_col = torch.empty(len(col), dtype=torch.int32, device="cuda")
    want = None
    if prec == "fp64":
        want = oracle.relax(rp, col, val, oracle.tv_init(n, K, 7), 3, 0.8)
    for colored in (False, True):
        with amgd.Handle(rp, col, val, K, 7) as h:
            h.set_precision(prec)
            if colored:
                h.set_coloring(color)
            h.init_vectors(7)
            if colored:
                on_sliced_copy(h)
            for nu in (1, 1, 1) if colored else (3,):
                h.relax(nu, 0.8)
                if colored:
                    h.set_values(val)
            got = [h.get_vectors()]
            if colored:
                h.relax(1, 0.8, amgd.AMGD_SWEEP_MCGS)
                h.graph_capture(7, 3, 0.8, amgd.AMGD_SWEEP_JACOBI, 0.5, s_rp, s_col)
                h.graph_launch()
                got.append(h.get_vectors())
                h.autotune(amgd.AMGD_SWEEP_JACOBI, 0.8)
                h.init_vectors(7)
                h.relax(3, 0.8)
                got.append(h.get_vectors())
        want = got[0] if want is None else want
        for g in got:
            assert np.array_equal(g, want)


@pytest.mark.parametrize("name", ["aniso9_66", "graph_4129", "lap1d_33"])
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("K", [3, 16, 64])
def test_both_sweep_routes_round_alike(name, prec, K):
    rp, col, val = SWEEPS[name]()
    color = inputs.greedy_coloring(rp, col)
    out = []
    for parts in ((3,), (1, 2)):                 # the second call of a handle reads the sliced copy
        with amgd.Handle(rp, col, val, K, 7) as h:
            h.set_precision(prec)
            h.set_coloring(color)
            h.init_vectors(7)
            for nu in parts:
                h.relax(nu, 1.1, amgd.AMGD_SWEEP_MCGS)
            out.append(h.get_vectors())
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("name", ["aniso9_66", "graph_4129", "arrow_3001"])
@pytest.mark.parametrize("K", [8, 32])
def test_tuned_handles_and_saved_lines(name, K, tmp_path):
    """A tuned handle, then handles that load its line as it is, with the sliced copy
    asked for, without the field (lines of before) and with the chunked kernel."""
    import re
    rp, col, val = SWEEPS[name]()
    color = inputs.greedy_coloring(rp, col)
    want = oracle.relax(rp, col, val, oracle.tv_init(len(rp) - 1, K, 7), 3, 1.0, oracle.SWEEP_MCGS, color)
    val2 = val * 1.5
    want2 = oracle.relax(rp, col, val2, want, 1, 1.0, oracle.SWEEP_MCGS, color)
    cache = tmp_path / "tune.txt"

    def run():
        with amgd.Handle(rp, col, val, K, 7) as h:
            h.set_coloring(color)
            h.autotune(amgd.AMGD_SWEEP_MCGS, 1.0, str(cache))
            for _ in range(3):
                h.relax(1, 1.0, amgd.AMGD_SWEEP_MCGS)
            assert np.array_equal(h.get_vectors(), want)
            h.set_values(val2)
            h.relax(1, 1.0, amgd.AMGD_SWEEP_MCGS)
            assert np.array_equal(h.get_vectors(), want2)

    run()
    line = cache.read_text()
    assert re.search(r";sliced=[01];", line)
    for pattern, text in ((r"$^", ""), (r";sliced=[01]", ";sliced=1"), (r";sliced=[01]", ""),
                          (r";relax=(\d+),(\d+),(\d+),\d+(.*);sliced=[01]", r";relax=\1,\2,\3,3\4;sliced=0")):
        cache.write_text(re.sub(pattern, text, line))
        run()
        assert len(cache.read_text().splitlines()) == 1          # served from the file


@pytest.mark.parametrize("K", [2, 13, 33, 64])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("name", ["lap1d_31", "graph_4129", "arrow_3001"])
def test_distances_with_zero_columns(name, K, weighted):
    """Few and many rows, rows longer than a batch; some vectors' rows are zero
    (S_xx = 0: a = 0, LS = S_yy).  LS in extended precision from the oracle's target:
    the oracle's unfused products alone err by up to 1.2e-12 of an LS of 1e-8 S_yy."""
    rp, col, val = SWEEPS[name]()
    n = len(rp) - 1
    w = np.random.default_rng(1).uniform(0.5, 2.0, K) if weighted else None
    X = oracle.tv_init(n, K, 5)
    X[::7] = 0.0
    got = gpu_build(rp, col, val, K, 5, 0, 1.0, 0.5, w=w, X0=X)
    Y = oracle.target(rp, col, val, X)
    a, ls = oracle.edge_ls(rp, col, val, X, Y, w)
    rows = np.repeat(np.arange(n), np.diff(rp))
    fit = (rows != col) & (np.diff(rp)[rows] != 2)          # one off-diagonal: LS = 0 exactly
    x, y = X[col[fit]].astype(np.longdouble), Y[rows[fit]].astype(np.longdouble)
    wl = np.ones(K, np.longdouble) if w is None else w.astype(np.longdouble)
    xx = (wl * x * x).sum(1)
    q = (wl * x * y).sum(1) / np.where(xx == 0, 1, xx)
    ls[fit] = (wl * (y - q[:, None] * x) ** 2).sum(1)
    want = dict(X=X, Y=Y, a=a, ls=ls, flag=oracle.threshold(rp, col, ls, 0.5)[0])
    compare_fp64(rp, col, val, got, want, 0.5, w)


def hub(n, lengths, seed):
    """A graph of some eleven entries a row, a row of each length first, and last a row
    with row 0 as its one neighbour."""
    rng = np.random.default_rng(seed)
    adj = [set(rng.integers(0, n, 3).tolist()) | {i} for i in range(n)]
    for i, m in enumerate(lengths):
        adj[i] |= set(rng.choice(n, m, replace=False).tolist())
    for i in range(n):
        for j in list(adj[i]):
            adj[j].add(i)
    for i, m in enumerate(lengths):              # rows of just these lengths; columns stay symmetric enough
        keep = sorted(adj[i] - {i}, key=lambda j: rng.random())[:m - 1]
        adj[i] = set(keep) | {i}
    adj[n - 1] = {0, n - 1}
    rp = np.concatenate([[0], np.cumsum([len(a) for a in adj])]).astype(np.int64)
    col = np.concatenate([sorted(a) for a in adj]).astype(np.int32)
    rows = np.repeat(np.arange(n), np.diff(rp))
    val = -rng.uniform(0.5, 1.5, len(col))
    val[rows == col] = 1.5 * np.diff(rp)
    return rp, col, val


def dense(n, seed):
    rng = np.random.default_rng(seed)
    val = -rng.uniform(0.5, 1.5, (n, n)) + 2 * n * np.eye(n)
    return (np.arange(n + 1) * n).astype(np.int64), np.tile(np.arange(n, dtype=np.int32), n), val.ravel()


@pytest.mark.parametrize("K", [1, 7, 16, 32, 64])
@pytest.mark.parametrize("prec,summation", [("fp64", "plain"), ("fp32", "compensated"), ("fp32", "plain"),
                                            ("bf16", "compensated")])
@pytest.mark.parametrize("form", ["colored", "weighted", "plain target", "depth 2"])
def test_long_rows_round_alike(K, prec, summation, form):
    """Rows of 64 to 600 entries, fitted by blocks of their own, and the same rows in a
    handle whose other rows are so long that these are not: the same bits."""
    if form == "depth 2":
        m, extra = hub(6000, (300,), 2), dense(1500, 3)
    else:
        m, extra = hub(700, (64, 65, 66, 257, 513, 600), 2), dense(600, 3)
    N = len(m[0]) - 1
    X = np.random.default_rng(4).uniform(-1, 1, (N + len(extra[0]) - 1, K))
    X[5::90] = 0.0
    out = []
    for mats in ([m], [m, extra]):
        n = sum(len(t[0]) - 1 for t in mats)
        with amgd.Handle(None, None, None, K, 1, batch=mats) as h:
            h.set_precision(prec)
            h.set_summation(summation)
            if form == "colored":
                h.set_coloring((np.arange(n) % 3).astype(np.int32))
            elif form == "weighted":
                h.set_weights(np.linspace(0.5, 1.5, K))
            elif form == "plain target":
                h.set_target(1)
            else:
                h.set_search_depth(2)
            h.set_vectors(X[:n])
            d = h.distances(0.5)
            rp, col = h.strength()
            if form == "depth 2":
                last = int(h.distance_pattern()[0][N])
            else:
                last = len(m[1])
            out.append([d["a"][:last], d["ls"][:last], rp[:N + 1], col[:rp[N]]])
    for a, b in zip(*out):
        assert np.array_equal(a, b, equal_nan=True)


def circulant(n, m, seed):
    """m entries in every row, the diagonal first among the column offsets."""
    rng = np.random.default_rng(seed)
    off = np.concatenate([[0], rng.choice(np.arange(1, n), m - 1, replace=False)])
    col = np.sort((np.arange(n)[:, None] + off) % n, 1).astype(np.int32)
    val = -rng.uniform(0.5, 1.5, (n, m))
    val[col == np.arange(n)[:, None]] = 1.5 * m
    return (np.arange(n + 1) * m).astype(np.int64), col.ravel(), val.ravel()


@pytest.mark.parametrize("K", [1, 7, 16, 32, 64])
@pytest.mark.parametrize("prec,summation", [("fp64", "plain"), ("fp32", "compensated"), ("fp32", "plain"),
                                            ("bf16", "compensated"), ("bf16", "plain")])
@pytest.mark.parametrize("n,m", [(97, 2), (301, 6), (301, 40), (700, 63), (301, 200)])
@pytest.mark.parametrize("form", ["colored", "weighted", "plain target"])
def test_shares_of_a_row_round_alike(n, m, prec, summation, K, form):
    """Two to thirty-two lane groups per row in a small handle; one, or a block per row of
    200 entries, in a large one: the same bits."""
    M, extra = circulant(n, m, 2), inputs.lap1d(40001)
    X = np.random.default_rng(4).uniform(-1, 1, (n + 40001, K))
    X[5::90] = 0.0
    out = []
    for mats in ([M], [M, extra]):
        rows = sum(len(t[0]) - 1 for t in mats)
        with amgd.Handle(None, None, None, K, 1, batch=mats) as h:
            h.set_precision(prec)
            h.set_summation(summation)
            if form == "colored":
                h.set_coloring((np.arange(rows) % 3).astype(np.int32))
            elif form == "weighted":
                h.set_weights(np.linspace(0.5, 1.5, K))
            else:
                h.set_target(1)
            h.set_vectors(X[:rows])
            d = h.distances(0.5)
            rp, col = h.strength()
            out.append([d["a"][:n * m], d["ls"][:n * m], rp[:n + 1], col[:rp[n]]])
    for a, b in zip(*out):
        assert np.array_equal(a, b, equal_nan=True)


@pytest.mark.parametrize("K", [1, 7, 16, 32, 64])
@pytest.mark.parametrize("prec,summation", [("fp64", "plain"), ("fp32", "compensated"), ("fp32", "plain"),
                                            ("bf16", "compensated")])
@pytest.mark.parametrize("form", ["colored", "depth 2"])
@pytest.mark.parametrize("rows", [4129, 40003])
def test_sorted_rows_round_alike(rows, prec, summation, K, form):
    """A graph whose rows are fitted in the order of their lengths, and the same graph in a
    handle of rows so even that they are fitted as they come."""
    side = 500 if rows < 10000 else 700
    M, extra = inputs.graph_laplacian(rows, 4.0, 4), inputs.poisson2d_5pt(side)
    X = np.random.default_rng(4).uniform(-1, 1, (rows + side * side, K))
    if form == "depth 2":
        if rows > 10000 or K > 16:
            pytest.skip("one size of the wider pattern")
        M = inputs.graph_laplacian(rows, 1.5, 4)
    out = []
    for mats in ([M], [M, extra]):
        n = sum(len(t[0]) - 1 for t in mats)
        with amgd.Handle(None, None, None, K, 1, batch=mats) as h:
            h.set_precision(prec)
            h.set_summation(summation)
            if form == "colored":
                h.set_coloring((np.arange(n) % 3).astype(np.int32))
            else:
                h.set_search_depth(2)
            h.set_vectors(X[:n])
            d = h.distances(0.5)
            rp, col = h.strength()
            last = int(h.distance_pattern()[0][rows])
            out.append([d["a"][:last], d["ls"][:last], rp[:rows + 1], col[:rp[rows]]])
    for a, b in zip(*out):
        assert np.array_equal(a, b, equal_nan=True)


def test_reciprocals_of_the_fp32_range():
    """dist = 1 / LS of the FP32 path over the type's whole range: equal to the
    FP64 quotient of the exported LS to one unit of its last place."""
    rp, col, val = inputs.graph_laplacian(4129, 8.0, 4)
    n = len(rp) - 1
    rng = np.random.default_rng(2)
    X = rng.standard_normal((n, 4)) * 10.0 ** rng.uniform(-19, 18, (n, 1))
    X[::50] = 0.0
    with amgd.Handle(rp, col, val, 4, 1) as h:
        h.set_precision("fp32")
        h.set_target(1)
        h.set_vectors(X)
        d = h.distances(0.5)
    ls, dist = d["ls"], d["dist"]
    assert np.array_equal(np.isnan(ls), np.isnan(dist))
    ok = ~np.isnan(ls)
    assert (ls[ok] == 0).any() and (ls[ok] > 1e30).any() and ((ls[ok] > 0) & (ls[ok] < 1e-30)).any()
    with np.errstate(divide="ignore"):
        want = 1.0 / ls[ok]
    inf = np.isinf(want)
    assert np.array_equal(dist[ok][inf], want[inf])
    assert np.all(np.abs(dist[ok][~inf] - want[~inf]) <= np.spacing(want[~inf]))


@pytest.mark.parametrize("n", [32767, 32768, 32769, 2048 * 1024, 2048 * 1024 + 1])
def test_strength_at_the_compaction_edges(n):
    rp, col, val = inputs.lap1d(n)
    with amgd.Handle(rp, col, val, 2, 3) as h:
        h.relax(1, 0.7)
        ls = h.distances(0.5, want=("ls",))["ls"]
        s_rp, s_col = h.strength()
    flag = oracle.threshold(rp, col, ls, 0.5)[0]
    w_rp, w_col = oracle.strength_csr(rp, col, flag)
    assert np.array_equal(s_rp, w_rp) and np.array_equal(s_col, w_col)


def shuffled(rp, col, val, seed):
    """The same rows with their entries in random order."""
    rng = np.random.default_rng(seed)
    rows = np.repeat(np.arange(len(rp) - 1), np.diff(rp))
    o = np.lexsort((rng.random(len(col)), rows))
    return rp, col[o], val[o]


def device(m):
    return [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in m]


@pytest.mark.parametrize("name,order", [("aniso9_66", "sorted"), ("graph_4129", "shuffled"), ("arrow_3001", "shuffled"),
                                        ("lap1d_31", "sorted")])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_create_from_device_memory(name, order, prec):
    m = SWEEPS[name]()
    if order == "shuffled":
        m = shuffled(*m, 3)                      # arrow: a row of 3001 entries out of order
    color = inputs.greedy_coloring(m[0], m[1])
    out = []
    for mat in (m, device(m)):
        with amgd.Handle(*mat, 8, 4) as h:
            h.set_precision(prec)
            h.init_vectors(4)
            h.relax(1, 0.8)
            h.set_coloring(color)                # reads the pattern on the host
            h.relax(2, 1.0, amgd.AMGD_SWEEP_MCGS)
            d = h.distances(0.5)
            s = h.strength()
            h.set_search_depth(2)
            d2 = h.distances(0.5, want=("ls",))
            out.append([h.get_vectors(), d["a"], d["ls"], d["dist"], s[0], s[1], d2["ls"]])
    for a, b in zip(*out):
        assert np.array_equal(a, b, equal_nan=True)


@pytest.mark.parametrize("prec", ["fp64", "bf16"])
def test_batch_create_from_device_memory(prec):
    mats = [inputs.graph_laplacian(k, 8.0, 4, b) for b, k in enumerate((700, 33, 1100))]
    dev = [device(m) for m in mats]
    L, hs = amgd.lib(), []
    ns = np.array([len(m[0]) - 1 for m in mats], np.int64)
    for group, ptr, mem in ((mats, lambda x: x.ctypes.data, amgd.AMGD_MEM_HOST),
                            (dev, lambda x: x.data_ptr(), amgd.AMGD_MEM_DEVICE)):
        arr = [(ctypes.c_void_p * 3)(*[ptr(m[k]) for m in group]) for k in range(3)]
        h = amgd.Handle(batch=mats, row_ptr=None, col=None, val=None, K=16, seed=6)
        if mem == amgd.AMGD_MEM_DEVICE:
            h.close()
            h.h = ctypes.c_void_p()
            amgd.check(L.amgd_create_batch(3, *arr, ns.ctypes.data, 16, 6, mem, ctypes.byref(h.h)))
        h.set_precision(prec)
        h.init_vectors(6)
        h.relax(3, 0.7)
        hs.append((h.distances(0.5)["ls"], h.get_vectors(), *h.strength()))
        h.close()
    for a, b in zip(*hs):
        assert np.array_equal(a, b, equal_nan=True)


def _bad(kind):
    rp, col, val = (x.copy() for x in (arrow(2001) if kind == "duplicate_long" else inputs.aniso2d_9pt(40, 1e-3, 0.3)))
    i = 0 if kind == "duplicate_long" else 700
    a, b = int(rp[i]), int(rp[i + 1])
    d = a + int(np.nonzero(col[a:b] == i)[0][0])
    if kind == "row_ptr":
        rp[i] = rp[i + 1] + 3
    elif kind == "row_ptr_start":
        rp[0] = 1
    elif kind == "row_ptr_past_the_end":
        rp[i] = rp[-1] + 5
    elif kind == "column_high":
        col[b - 1] = len(rp) - 1
    elif kind == "column_negative":
        col[a] = -1
    elif kind.startswith("duplicate"):
        col[a + 1 if d != a + 1 else a + 2] = col[b - 1]
    elif kind == "nan":
        val[a] = np.nan
    elif kind == "inf":
        val[b - 1] = np.inf
    elif kind == "zero_diagonal":
        val[d] = 0.0
    elif kind == "no_diagonal":
        j = np.setdiff1d(np.arange(len(rp) - 1), col[a:b])[0]
        col[d] = j
    return rp, col, val


@pytest.mark.parametrize("kind", ["row_ptr", "row_ptr_start", "row_ptr_past_the_end", "column_high", "column_negative",
                                  "duplicate", "duplicate_long", "nan", "inf", "zero_diagonal", "no_diagonal"])
def test_create_refuses_alike_from_host_and_device(kind):
    m = _bad(kind)
    codes = []
    for mat in (m, device(m)):
        with pytest.raises(amgd.AmgdError) as e:
            amgd.Handle(*mat, 4, 1)
        codes.append(e.value.status)
    assert codes[0] == codes[1]


def test_a_batch_names_its_first_fault():
    mats = [_bad("zero_diagonal"), _bad("row_ptr_start")]
    dev = [device(m) for m in mats]
    ns = np.array([len(m[0]) - 1 for m in mats], np.int64)
    codes = []
    for group, ptr, mem in ((mats, lambda x: x.ctypes.data, amgd.AMGD_MEM_HOST),
                            (dev, lambda x: x.data_ptr(), amgd.AMGD_MEM_DEVICE)):
        arr = [(ctypes.c_void_p * 2)(*[ptr(m[k]) for m in group]) for k in range(3)]
        h = ctypes.c_void_p()
        codes.append(amgd.lib().amgd_create_batch(2, *arr, ns.ctypes.data, 4, 1, mem, ctypes.byref(h)))
    assert codes[0] == codes[1] != 0


@pytest.mark.parametrize("K", [2, 3, 4, 6, 17, 64])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16"])
def test_interpolation_of_every_candidate_count(K, prec):
    """Unit weights, 0 to 8 and more candidates in a row; K below, at and off the
    four components that a load takes."""
    rp, col, val = inputs.random_csr(700, 2.5, 21, symmetric_pattern=True)
    n = len(rp) - 1
    coarse = (np.random.default_rng(3).random(n) < 0.45).astype(np.uint8)
    X = oracle.relax(rp, col, val, oracle.tv_init(n, K, 2), 2, 0.7)
    if prec != "fp64":
        X = torch.from_numpy(X).to(torch.bfloat16 if prec == "bf16" else torch.float32).to(torch.float64).numpy()
    prp, pcol = oracle.distance_graph(rp, col, 2)
    rows = np.repeat(np.arange(n), np.diff(prp))
    m = np.bincount(rows[coarse[pcol] == 1], minlength=n)[coarse == 0]
    assert set(range(9)) <= set(m.tolist())
    Y = oracle.target(rp, col, val, X)
    for caliber in (1, 3):
        with amgd.Handle(rp, col, val, K, 2) as h:
            h.set_precision(prec)
            h.set_search_depth(2)
            h.set_vectors(X)
            got = h.ls_interpolation(coarse, caliber, 1.5)
        for g, w_ in zip(got, oracle.ls_interp(X, Y, prp, pcol, coarse, caliber, 1.5)):
            assert np.array_equal(g, w_)


@pytest.mark.parametrize("K", [6, 8, 13])
def test_interpolation_with_tiny_diagonals(K):
    """1 / a_ii overflows: infinite targets and LS in the components that there are."""
    rp, col, val = inputs.random_csr(700, 2.5, 21, symmetric_pattern=True)
    n = len(rp) - 1
    val[np.nonzero(np.repeat(np.arange(n), np.diff(rp)) == col)[0][5::40]] = 1e-310
    coarse = (np.random.default_rng(3).random(n) < 0.45).astype(np.uint8)
    X = oracle.tv_init(n, K, 2)
    want = oracle.ls_interp(X, oracle.target(rp, col, val, X), rp, col, coarse, 2, 1.5)
    assert np.isinf(want[3]).any() and not np.isnan(want[3]).any()
    with amgd.Handle(rp, col, val, K, 2) as h:
        got = h.ls_interpolation(coarse, 2, 1.5)
    for g, w_ in zip(got, want):
        assert np.array_equal(g, w_)


@pytest.mark.parametrize("K", [4, 8, 16, 32, 64])
@pytest.mark.parametrize("pattern", ["symmetric", "general"])
@pytest.mark.parametrize("weighted", [False, True])
def test_reverse_pass_of_every_row_width(K, pattern, weighted):
    """1 to 32 lanes per row, the row's entries shared among them.  FP64 storage:
    1e-11 of the oracle's gradient.  FP32 and BF16 storage without sweeps, from
    start vectors that are exact in the type: the fits alone, in 48 bits or more
    (2^-48 over sums of a few thousand terms: 1e-10)."""
    mat = inputs.random_csr(300, 6.0, 9, symmetric_pattern=pattern == "symmetric")
    w = np.random.default_rng(1).uniform(0.5, 2.0, K) if weighted else None
    lsb = np.random.default_rng(5).standard_normal(len(mat[1]))
    for prec, nu, tol in (("fp64", 3, 1e-11), ("fp32", 0, 1e-10), ("bf16", 0, 1e-10)):
        g = run_gpu(mat, K, 7, nu, 0.6, 0.5, 2, prec=prec, w=w, ls_bar=lsb)
        X0 = g["X0"]                             # the draws rounded to the type (its own tests pin them)
        if prec == "fp64":
            assert np.array_equal(X0, x0(mat, K, 7))
        o = oracle.adjoint_jacobi(*mat, X0, nu, 0.6, 0.5, w, 0, ls_bar=lsb)
        assert rel(g["val_bar"], o["val_bar"]) <= tol, prec
