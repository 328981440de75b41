"""The library's host side under a fake runtime over host memory, no GPU.

Allocations that fail half-way through a group: the call returns AX_ENOMEM, the
next one allocates whatever is missing instead of using it, nothing is freed
twice and nothing is left when the handles are gone.  Solves whose kernels
never report: they return AX_ELAUNCH, waiting the way the process asked for."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fake") / "libfake_cuda.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", so, os.path.join(HERE, "fake_cuda.c")],
                   check=True)
    return so


@pytest.mark.parametrize("what", ["loss_grad", "precondition", "mpcg", "mpcg_modes", "mpfcg",
                                  "train_energy"])
def test_failed_allocation_is_made_up_for(fake, what):
    env = dict(os.environ, LD_PRELOAD=fake, PYTHONPATH=os.path.dirname(HERE))
    r = subprocess.run([sys.executable, os.path.abspath(__file__), fake, what], env=env,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


def test_training_holds_no_more_than_its_workspace(fake):
    """Energy training leaves nothing in the problem's handle, and past the 64
    places of 608 partial sums its workspace grows by 16 bytes a pair."""
    test_failed_allocation_is_made_up_for(fake, "held")


def test_wait_for_a_stream_that_fails_or_runs_dry(fake):
    """The convergence test's values never come: AX_ELAUNCH from every solver
    once the stream is idle or reports an error; and a process that asked for
    blocking synchronisation gets it instead of polling."""
    test_failed_allocation_is_made_up_for(fake, "wait")


# ------------------------------------------------ in the process with the fake
def _program(fake, what):
    import paper_2506_20994_gb300 as ax
    from paper_2506_20994_gb300 import _lib, synth
    F, L = ctypes.CDLL(fake), _lib.lib()
    lx, keep = 6, []
    a = lambda x: (keep.append(np.ascontiguousarray(x)), keep[-1].ctypes.data)[1]
    geo = ax.box_geometry(synth.box_vertices(2, 2, 1, seed=1), lx)
    dx, dxt = ax.dmat(lx)
    nel, n = 4, 4 * lx ** 3
    one, b = a(np.ones(n)), a(np.zeros(n))
    out, X = a(np.zeros(4 * n)), a(np.zeros(9 * lx ** 3, np.float32))
    glob = a(ax.box_numbering(2, 2, 1, lx))
    geom = [a(geo[k]) for k in ("g11", "g22", "g33", "g12", "g13", "g23")]
    par = ax.mlp_init_params(lx ** 3, 16, seed=1, arch=ax.AX_MLP_SYM)
    params, num = a(par), ctypes.c_double()
    ref = lambda c: ctypes.addressof(c)

    def ok(rc):
        assert rc == 0, rc

    def handles():
        gs, P, M = ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
        ok(L.ax_gs_setup(ref(gs), glob, n, None))
        ok(L.ax_poisson_create(ref(P), lx, nel, a(dx), a(dxt), one, *geom, one, gs, None))
        ok(L.ax_mlp_create_ex(ref(M), lx ** 3, 16, ax.AX_MLP_SYM))
        ok(L.ax_mlp_set_params(M, params, par.size, None))
        return gs, P, M

    if what == "held":
        F.fake_bytes.restype = ctypes.c_longlong
        gs, P, M = handles()
        own = F.fake_bytes()
        held = {}
        for K in (1, 64, 1000):
            ok(L.ax_mlp_train_energy(P, M, out, out, K, 1, 1e-3, ref(num), None))
            held[K] = F.fake_bytes() - own
        assert held[1000] - held[64] == 16 * (1000 - 64), held
        ok(L.ax_mlp_destroy(M))
        ok(L.ax_mlp_create_ex(ref(M), lx ** 3, 16, ax.AX_MLP_SYM))
        assert F.fake_bytes() == own, (F.fake_bytes(), own)
        return

    if what == "wait":
        gs, P, M = handles()
        solves = [lambda: L.ax_cg_solve(P, out, b, 1e-8, 9, None, None, None),
                  lambda: L.ax_fcg_solve(P, M, out, b, 1e-8, 9, None, None, None, None)]
        for solve in solves:
            for result in (0, 700):  # idle; an earlier kernel's fault, as reported
                for flags in (0, 1, 2):  # automatic, spin, yield
                    F.fake_stream(result, flags)
                    assert solve() == _lib.AX_ELAUNCH
                    assert F.fake_queries() == 1
            F.fake_stream(0, 4)  # blocking: asked only once it has waited
            assert solve() == _lib.AX_ELAUNCH
            assert F.fake_queries() == 0 and F.fake_syncs() >= 1
        return

    def session(call, fail):
        """All handles made, `call` with its `fail`-th allocation failing (0:
        none), called again; returns the allocations held then."""
        gs, P, M = handles()
        F.fake_fail_in(fail)
        rc = call(P, M)
        hit = fail > 0 and F.fake_pending() == 0
        F.fake_fail_in(0)
        assert rc == (_lib.AX_ENOMEM if hit else 0), (fail, rc)
        if hit:
            ok(call(P, M))
        held = F.fake_live()
        ok(call(P, M))
        assert F.fake_live() == held
        L.ax_mlp_destroy(M)
        L.ax_poisson_destroy(P)
        L.ax_gs_free(gs)
        assert F.fake_live() == 0 and F.fake_bad_frees() == 0, (fail, F.fake_live(), F.fake_bad_frees())
        return hit, held

    def mpcg(P, mode):
        return L.ax_mpcg_solve(P, mode, out, b, 1e-8, 1e-4, 4, 9, None, None, None, None)

    def modes(P, M):
        return mpcg(P, ax.AX_PREC_F32) or mpcg(P, ax.AX_PREC_BF16) or mpcg(P, ax.AX_PREC_F32)

    call = {
        "loss_grad": lambda P, M: (L.ax_mlp_loss_grad(M, X, X, 3, ref(num), None, None)
                                   or L.ax_mlp_loss_grad(M, X, X, 9, ref(num), None, None)),
        "precondition": lambda P, M: L.ax_precondition(P, M, out, b, None),
        "mpcg": lambda P, M: mpcg(P, ax.AX_PREC_F32),
        "mpcg_modes": modes,
        "mpfcg": lambda P, M: L.ax_mpfcg_solve(P, M, ax.AX_PREC_BF16, out, b, 1e-8, 1e-4, 4, 9,
                                               None, None, None, None, None),
        "train_energy": lambda P, M: L.ax_mlp_train_energy(P, M, out, out, 2, 1, 1e-3, ref(num),
                                                           None),
    }[what]
    _, held = session(call, 0)
    fail, hit = 1, True
    while hit:
        hit, now = session(call, fail)
        assert now == held, (fail, now, held)
        fail += 1
    assert fail > 2  # at least one allocation was made to fail


if __name__ == "__main__":
    _program(sys.argv[1], sys.argv[2])
