"""The solvers on both sides of the mesh size from which the gather-scatter is
launched without overlap, and the flexible loop's wide loads with and without
a scalar remainder: the residual is formed anew with the library's operator."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2506_20994_gb300 as ax  # noqa: E402
from paper_2506_20994_gb300 import synth  # noqa: E402

TOL = 1e-7


def _solve_and_check(dims, lx, solve):
    P = ax.Poisson(synth.box_vertices(*dims), lx)
    b = P.rhs(synth.poisson_source)
    x, relres = solve(P, b)
    Ax = torch.empty_like(b)
    P.apply(Ax, x)
    m = P.d["mask"].reshape(b.shape)
    r, s = (m * (b - Ax)).norm(), (m * b).norm()
    # the returned figure weighs shared points by 1/copies (1 to 8 of them), so
    # the plain norms' ratio is within a factor sqrt(8) of it
    assert relres <= TOL
    assert float(r / s) <= 8 ** 0.5 * TOL * 1.01


# 512000 and 563200 points: below and above the line for fp32 vectors
@pytest.mark.parametrize("mode", [ax.AX_PREC_F32, ax.AX_PREC_BF16])
@pytest.mark.parametrize("dims", [(10, 10, 10), (11, 10, 10)])
def test_refinement_around_the_size_line(dims, mode):
    def solve(P, b):
        q = P.mpcg(b, mode=mode, tol=TOL)
        return q[0], q[-2]
    _solve_and_check(dims, 8, solve)


# 2^24 points and one element layer less: the fp64 line
@pytest.mark.parametrize("dims", [(32, 32, 31), (32, 32, 32)])
def test_cg_around_the_size_line(dims):
    def solve(P, b):
        q = P.cg(b, tol=TOL)
        return q[0], q[-2]
    _solve_and_check(dims, 8, solve)


# an even and an odd number of points (lx odd: the last one by itself)
@pytest.mark.parametrize("dims,lx", [((3, 3, 3), 5), ((3, 3, 3), 6), ((1, 1, 1), 7)])
def test_flexible_loop_points_odd_and_even(dims, lx):
    def solve(P, b):
        q = P.fcg(b, None, tol=TOL)
        return q[0], q[2]
    _solve_and_check(dims, lx, solve)


@pytest.mark.parametrize("lx", [6, 8, 10, 12])
@pytest.mark.parametrize("flexible", [False, True], ids=["cg", "fcg"])
def test_solution_belongs_to_the_residual(lx, flexible):
    """x where it is updated by the update kernel (lx 6, 10) and by the next
    step's apply (lx 8, 12): after any number of steps, tested at every one of
    them or at the last, ||b - A x|| is the recurrence's residual norm.  The two
    differ by rounding: some hundred operations of 2^-53 on terms of ||b||'s
    size."""
    P = ax.Poisson(synth.box_vertices(4, 3, 3, seed=lx), lx, h1=ax.fourier_coefficient(2))
    b = P.rhs(synth.poisson_source)
    c = P.gs.inverse_multiplicity()
    norm = lambda v: float((c * v.reshape(-1) * v.reshape(-1)).sum()) ** 0.5
    for steps in (1, 2, 7, 24):
        for every in (1, 5, 1000):
            P.set_check_every(every)
            f = P.fcg if flexible else P.cg
            r = f(b, None, tol=0.0, maxit=steps, raise_on_error=False) if flexible else f(
                b, tol=0.0, maxit=steps, raise_on_error=False)
            assert r[1] == steps
            assert abs(norm(P.residual(b, r[0])) / norm(b) - r[2]) <= 1e-12 + 1e-10 * r[2]


# both sides of the lines of the other operators: fp32 data at 2^18 points (lx
# 8 and 10), the flexible fp32 loop at 2^19 (lx 12), and orders without a line
@pytest.mark.parametrize("dims,lx,mode", [((7, 8, 8), 8, ax.AX_PREC_F32), ((8, 8, 8), 8, ax.AX_PREC_F32),
                                          ((6, 6, 7), 10, ax.AX_PREC_F32), ((7, 7, 6), 10, ax.AX_PREC_F32),
                                          ((7, 7, 6), 10, ax.AX_PREC_BF16), ((14, 14, 14), 6, ax.AX_PREC_F32),
                                          ((13, 12, 12), 7, ax.AX_PREC_F32)])
def test_refinement_around_the_other_lines(dims, lx, mode):
    def solve(P, b):
        q = P.mpcg(b, mode=mode, tol=TOL, inner_tol=1e-2 if mode == ax.AX_PREC_BF16 else 1e-4)
        return q[0], q[-2]
    _solve_and_check(dims, lx, solve)


@pytest.mark.parametrize("dims", [(6, 7, 7), (7, 7, 7)])
def test_flexible_refinement_around_the_line(dims):
    def solve(P, b):
        q = P.mpfcg(b, None, tol=TOL)
        return q[0], q[3]
    _solve_and_check(dims, 12, solve)
