"""Kernels that may be launched while the one before them still runs: long
chains in which each call reads what the call before it wrote, and the buffers
come round again, must give the bits of the same chain with a synchronisation
after every call; also under graph capture and after the geometry is
rewritten."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2506_20994_gb300 as ax  # noqa: E402
from paper_2506_20994_gb300 import synth  # noqa: E402

from _cases import GKEYS, operator_case  # noqa: E402


def _t(a, dt=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda").to(dt)


def _scale(c, dt=torch.float64):
    """Operands scaled so that repeated applies stay in range."""
    d = {k: _t(c[k], dt) for k in ("u", "dx", "dxt", "h1") + GKEYS}
    d["h1"] = d["h1"] * float(0.3 * np.linalg.norm(c["u"]) / np.linalg.norm(c["w"]))
    return d


def _same(step, bufs, n=24):
    """step(out, in, k) over three buffers in turn, with and without waits."""
    ref = [b.clone() for b in bufs]
    for k in range(n):
        step(ref[(k + 1) % 3], ref[k % 3], k)
        torch.cuda.synchronize()
    for _ in range(3):
        got = [b.clone() for b in bufs]
        torch.cuda.synchronize()
        for k in range(n):
            step(got[(k + 1) % 3], got[k % 3], k)
        torch.cuda.synchronize()
        for a, b in zip(got, ref):
            assert torch.equal(a, b)


@pytest.mark.parametrize("dims,lx", [((1, 1, 1), 8), ((5, 3, 2), 6), ((8, 8, 8), 8),
                                     ((9, 9, 8), 10), ((17, 13, 11), 6)])
def test_handle_raw_and_gather_scatter_chains(dims, lx):
    c = operator_case(dims, lx, seed=600 + lx)
    d = _scale(c)
    G = [d[k] for k in GKEYS]
    op = ax.Operator(lx, d["dx"], d["dxt"], d["h1"], *G)
    gs = ax.GatherScatter(ax.box_numbering(*dims, lx))
    bufs = [d["u"].clone(), torch.zeros_like(d["u"]), torch.zeros_like(d["u"])]
    _same(lambda w, u, k: op.apply(w, u), bufs)
    _same(lambda w, u, k: ax.ax_helm(w, u, d["dx"], d["dxt"], d["h1"], *G, lx), bufs)

    def mixed(w, u, k):
        if k % 2:
            op.apply(w, u)
        else:
            ax.ax_helm(w, u, d["dx"], d["dxt"], d["h1"], *G, lx)
        gs.sum(w)
        if k % 5 == 4:
            w.mul_(0.5)  # a kernel of another library in between
    _same(mixed, bufs)


def test_rewritten_geometry_and_capture():
    lx = 8
    c = operator_case((6, 5, 4), lx, seed=611)
    d = _scale(c)
    op = ax.Operator(lx, d["dx"], d["dxt"], d["h1"], *[d[k] for k in GKEYS])
    h = [d["h1"], (d["h1"] * 1.25).contiguous()]
    bufs = [d["u"].clone(), torch.zeros_like(d["u"]), torch.zeros_like(d["u"])]

    def step(w, u, k):
        if k % 3 == 0:
            op.set_h1(h[(k // 3) % 2])
        op.apply(w, u)
    _same(step, bufs)
    # a captured chain, replayed after the geometry changed outside the graph
    a, b = torch.empty_like(d["u"]), torch.empty_like(d["u"])
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        op.set_h1(h[0])
        op.apply(a, d["u"])
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            for _ in range(4):
                op.apply(a, d["u"])
                op.apply(b, a)
        for q in (0, 1, 0):
            op.set_h1(h[q])
            g.replay()
            s.synchronize()
            got = b.clone()
            op.apply(a, d["u"])
            s.synchronize()
            op.apply(b, a)
            s.synchronize()
            assert torch.equal(got, b)


def test_solvers_repeat_bitwise():
    P = ax.Poisson(synth.box_vertices(9, 8, 7, seed=4), 8)
    P.set_check_every(8)
    b = P.rhs(synth.poisson_source)
    x0, n0 = P.cg(b, tol=1e-9)[:2]
    r = P.residual(b, x0).reshape(-1)
    cm = P.gs.inverse_multiplicity()
    bb = b.reshape(-1)
    assert float((cm * r * r).sum()) <= (1.5e-9) ** 2 * float((cm * bb * bb).sum())
    for _ in range(4):
        x, n = P.cg(b, tol=1e-9)[:2]
        assert n == n0 and torch.equal(x, x0)


@pytest.mark.parametrize("dims,lx", [((1, 1, 1), 8), ((8, 8, 8), 8), ((6, 5, 4), 5),
                                     ((9, 8, 7), 6), ((5, 4, 3), 7), ((16, 16, 4), 3)])
def test_reduced_precision_chains(dims, lx):
    """fp32, bf16 and trilinear applies and the fp32 gather-scatter, at orders
    of the persistent kernels and of the k-loop ones."""
    c = operator_case(dims, lx, seed=620 + lx)
    f, h = torch.float32, torch.bfloat16
    d, e = _scale(c, f), _scale(c, h)
    dx, dxt = _t(c["dx"], f), _t(c["dxt"], f)
    G, Gh = [d[k] for k in GKEYS], [e[k] for k in GKEYS]
    gs = ax.GatherScatter(ax.box_numbering(*dims, lx))
    bufs = [d["u"].clone(), torch.zeros_like(d["u"]), torch.zeros_like(d["u"])]

    def step32(w, u, k):
        ax.ax_helm_f32(w, u, dx, dxt, d["h1"], *G, lx)
        if k % 3 == 2:
            gs.sum(w)
    _same(step32, bufs)

    def step16(w, u, k):
        ax.ax_helm_bf16(w, u.to(h), dx, dxt, e["h1"], *Gh, lx)
    _same(step16, bufs)
    cor = _t(ax.box_corners(c["vertices"])).reshape(-1)
    xi, wq = (_t(a) for a in ax.gll(lx))
    _same(lambda w, u, k: ax.ax_helm_trilinear_f32(w, u, dx, dxt, d["h1"], cor, xi, wq, lx), bufs)


@pytest.mark.parametrize("lx", [2, 3, 4, 5, 7, 9, 13])
def test_k_loop_and_six_matrix_chains(lx):
    c = operator_case((5, 4, 3), lx, seed=640 + lx)
    d = _scale(c)
    G = [d[k] for k in GKEYS]
    bufs = [d["u"].clone(), torch.zeros_like(d["u"]), torch.zeros_like(d["u"])]
    dx, dxt, dy, dyt = d["dx"], d["dxt"], d["dx"].clone(), d["dxt"].clone()

    def step(w, u, k):
        if k % 2:
            ax.ax_helm(w, u, dx, dxt, d["h1"], *G, lx)
        else:
            ax.ax_helm_xyz(w, u, dx, dy, dx, dxt, dyt, dxt, d["h1"], *G, lx)
    _same(step, bufs)


def test_mixed_solves_and_training_repeat_bitwise():
    P = ax.Poisson(synth.box_vertices(7, 6, 5, seed=4), 8, h1=ax.fourier_coefficient(3))
    P.set_check_every(4)
    b = P.rhs(synth.poisson_source)
    M = ax.Mlp(512, 32, arch=ax.AX_MLP_SYM,
               params=ax.mlp_init_params(512, 32, seed=1, arch=ax.AX_MLP_SYM, scale=1.0))
    runs = [lambda: P.mpcg(b, mode=ax.AX_PREC_F32, tol=1e-9)[0],
            lambda: P.mpcg(b, mode=ax.AX_PREC_BF16, tol=1e-9, inner_tol=1e-2)[0],
            lambda: P.fcg(b, M, tol=1e-9)[0], lambda: P.mpfcg(b, M, tol=1e-9)[0]]
    for run in runs:
        x0 = run()
        assert bool(torch.isfinite(x0).all())
        for _ in range(3):
            assert torch.equal(run(), x0)
    R, E = ax.iterate_pairs(P, b, iterates=(2, 8, 32))
    got = []
    for _ in range(3):
        N = ax.Mlp(512, 32, arch=ax.AX_MLP_SYM,
                   params=ax.mlp_init_params(512, 32, seed=1, arch=ax.AX_MLP_SYM))
        ax.train_energy(P, N, R, E, epochs=4)
        got.append(N.get_params())
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])


def test_rewrite_then_capture_then_eager_apply():
    """An apply that is only recorded between the rewrite of the geometry and
    the apply that follows it on the stream."""
    lx = 8
    c = operator_case((9, 8, 7), lx, seed=613)
    d = _scale(c)
    op = ax.Operator(lx, d["dx"], d["dxt"], d["h1"], *[d[k] for k in GKEYS])
    h = [d["h1"], (d["h1"] * 1.25).contiguous()]
    ref = []
    for q in (0, 1):
        op.set_h1(h[q])
        torch.cuda.synchronize()
        ref.append(torch.empty_like(d["u"]))
        op.apply(ref[q], d["u"])
        torch.cuda.synchronize()
    w, a = torch.empty_like(d["u"]), torch.empty_like(d["u"])
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        for k in range(20):
            op.set_h1(h[k % 2])
            g = torch.cuda.CUDAGraph()
            g.capture_begin(capture_error_mode="relaxed")  # (the context manager synchronises)
            op.apply(a, d["u"])
            g.capture_end()
            op.apply(w, d["u"])
            s.synchronize()
            assert torch.equal(w, ref[k % 2])
            g.replay()
            s.synchronize()
            assert torch.equal(a, ref[k % 2])


def test_one_handle_on_two_streams_and_threads():
    """Applies of one handle from two host threads, each on its own stream,
    between rewrites of its geometry that both wait for."""
    import threading
    lx = 8
    c = operator_case((6, 5, 4), lx, seed=614)
    d = _scale(c)
    op = ax.Operator(lx, d["dx"], d["dxt"], d["h1"], *[d[k] for k in GKEYS])
    gate, errors = threading.Barrier(2, timeout=60), []

    def work(t):
        try:
            s = torch.cuda.Stream()
            u = (d["u"] * (1.0 + t)).contiguous()
            a, b = torch.empty_like(u), torch.empty_like(u)
            torch.cuda.synchronize()
            with torch.cuda.stream(s):
                for k in range(10):
                    gate.wait()
                    if k % 2 == t:  # this thread rewrites, both wait for it
                        op.set_h1((d["h1"] * (1.0 + 0.1 * k)).contiguous())
                        s.synchronize()
                    gate.wait()
                    op.apply(a, u)
                    op.apply(b, a)
                    got = b.clone()
                    s.synchronize()
                    op.apply(a, u)
                    s.synchronize()
                    op.apply(b, a)
                    s.synchronize()
                    if not torch.equal(got, b):
                        errors.append((t, k))
        except Exception as e:  # noqa: BLE001
            errors.append(e)
            gate.abort()
    th = [threading.Thread(target=work, args=(t,)) for t in (0, 1)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not errors


def test_chains_that_fork_and_join_under_capture():
    """A recorded chain whose links come from another stream's event, a copy
    and a memset as well as from the kernel in front."""
    lx = 8
    c = operator_case((6, 5, 4), lx, seed=615)
    d = _scale(c)
    op = ax.Operator(lx, d["dx"], d["dxt"], d["h1"], *[d[k] for k in GKEYS])
    u = d["u"]
    a, b, x, y = (torch.zeros_like(u) for _ in range(4))

    def chain(s, t):
        with torch.cuda.stream(s):
            op.apply(a, u)
        t.wait_stream(s)
        with torch.cuda.stream(t):  # first on t: its link is the event
            op.apply(b, a)
            x.copy_(b)
            op.apply(y, x)
        with torch.cuda.stream(s):
            x2 = a * 2.0
            s.wait_stream(t)  # two links: the kernel on s and the event of t
            op.apply(a, y)
            a.add_(x2)
            b.zero_()
            op.apply(x, a)
            return x
    s, t = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    ref = chain(s, t)
    torch.cuda.synchronize()
    ref = ref.clone()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        chain(s, t)
    for _ in range(5):
        x.zero_()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(x, ref)


@pytest.mark.parametrize("lx", [6, 7, 8])
def test_chains_of_elements_in_fp64_units(lx):
    """Every element outside the double-float window (recomputed with fp64
    units), with the mass term, in vectors that start between two sectors, so
    that neighbouring elements share one."""
    c = operator_case((9, 8, 7), lx, seed=650 + lx)
    d = _scale(c)
    G = [d[k] for k in GKEYS]
    op = ax.Operator(lx, d["dx"], d["dxt"], d["h1"], *G)
    h2 = torch.full_like(d["u"], 0.1)
    op.set_h2(h2, torch.ones_like(h2))
    n = d["u"].numel()
    raw = [torch.zeros(n + 1, dtype=torch.float64, device="cuda") for _ in range(3)]
    raw[0][1:] = d["u"].reshape(-1) * 1e-60

    def step(w, u, k):
        op.apply(w[1:], u[1:])
    _same(step, raw)

    def step_raw(w, u, k):
        ax.ax_helm(w[1:].view(d["u"].shape), u[1:].view(d["u"].shape), d["dx"], d["dxt"], d["h1"],
                   *G, lx)
    _same(step_raw, raw)


@pytest.mark.parametrize("lx", [3, 4, 5, 7, 8, 13])
def test_matrices_written_by_the_kernel_in_front(lx):
    """The 1-D matrices rewritten between two applies by a library kernel
    chained in front of the second (a gather-scatter that doubles every entry
    it pairs up)."""
    c = operator_case((9, 8, 7) if lx < 9 else (3, 3, 2), lx, seed=660 + lx)
    f = torch.float32
    d = _scale(c, f)
    G = [d[k] for k in GKEYS]
    ids = np.arange(lx * lx) // 2  # pairs of neighbouring entries share an id
    gs = ax.GatherScatter(ids)
    dx0, dxt0 = _t(c["dx"], f).reshape(-1), _t(c["dxt"], f).reshape(-1)

    def chain(wait):
        dx, dxt, out = dx0.clone(), dxt0.clone(), []
        torch.cuda.synchronize()
        for _ in range(6):
            w = torch.empty_like(d["u"])
            ax.ax_helm_f32(w, d["u"], dx, dxt, d["h1"], *G, lx)
            if wait:
                torch.cuda.synchronize()
            gs.sum(dx)
            if wait:
                torch.cuda.synchronize()
            gs.sum(dxt)
            if wait:
                torch.cuda.synchronize()
            out.append(w)
        torch.cuda.synchronize()
        return out
    ref = chain(True)
    assert not torch.equal(ref[0], ref[1])
    for _ in range(5):
        for a, b in zip(chain(False), ref):
            assert torch.equal(a, b)


@pytest.mark.parametrize("dims,lx", [((11, 11, 11), 7), ((12, 20, 10), 5), ((20, 20, 1), 13),
                                     ((20, 20, 1), 9), ((10, 10, 3), 11)])
def test_chains_of_grids_that_fill_part_of_a_wave(dims, lx):
    """Grids of two and more blocks per SM that are less than one full wave:
    their blocks are held to an even share of each SM."""
    c = operator_case(dims, lx, seed=670 + lx)
    d = _scale(c)
    G = [d[k] for k in GKEYS]
    bufs = [d["u"].clone(), torch.zeros_like(d["u"]), torch.zeros_like(d["u"])]
    _same(lambda w, u, k: ax.ax_helm(w, u, d["dx"], d["dxt"], d["h1"], *G, lx), bufs, n=9)
    _same(lambda w, u, k: ax.ax_helm_xyz(w, u, d["dx"], d["dx"], d["dx"], d["dxt"], d["dxt"],
                                         d["dxt"], d["h1"], *G, lx), bufs, n=6)
    f = torch.float32
    e = _scale(c, f)
    Gf = [e[k] for k in GKEYS]
    buf32 = [e["u"].clone(), torch.zeros_like(e["u"]), torch.zeros_like(e["u"])]
    _same(lambda w, u, k: ax.ax_helm_f32(w, u, e["dx"], e["dxt"], e["h1"], *Gf, lx), buf32, n=9)
    cor = _t(ax.box_corners(c["vertices"])).reshape(-1)
    xi, wq = (_t(a) for a in ax.gll(lx))
    _same(lambda w, u, k: ax.ax_helm_trilinear_f32(w, u, e["dx"], e["dxt"], e["h1"], cor, xi, wq, lx),
          buf32, n=9)
    w = torch.empty_like(d["u"])
    ax.ax_helm(w, d["u"], d["dx"], d["dxt"], d["h1"], *G, lx)
    ref = c["w"] * float(d["h1"].max() / _t(c["h1"]).max())  # linear in h1
    assert float((w - _t(ref)).norm()) <= 1e-12 * float(_t(ref).norm())
