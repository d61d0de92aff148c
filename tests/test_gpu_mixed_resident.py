"""Mixed-precision solves in one launch: what is not a number never passes for a solution, and guesses are used."""
import pytest

torch = pytest.importorskip("torch")

from workloads import box_basin, random_vector  # noqa: E402

pytestmark = pytest.mark.gpu

import paper_1207_0486_gb300 as pm  # noqa: E402

KERNELS = [pm.KERNEL_STREAM, pm.KERNEL_AUTO]
MIXED = [pm.FP32_REFINE, pm.BF16_REFINE]


@pytest.mark.parametrize("kernel", KERNELS)
@pytest.mark.parametrize("precision", MIXED)
def test_no_iteration_on_a_right_hand_side_that_is_not_a_number(precision, kernel):
    """max_iter = 0 reports the first residual: not a number is not converged."""
    op = pm.assemble_operator(box_basin())
    rhs = torch.from_numpy(random_vector(op.n, 5)).cuda()
    rhs[17] = float("nan")
    for which, prec in ((pm.OP_VEL_U2, pm.PREC_IC0), (pm.OP_PRESSURE, pm.PREC_LINE), (pm.OP_MASS, pm.PREC_JACOBI)):
        st = op.solve(which, rhs, torch.zeros_like(rhs), pm.Options(max_iter=0, prec=prec, precision=precision, kernel=kernel),
                      allow_not_converged=True)
        assert st.status == pm.PM_NOT_CONVERGED and st.iters == 0
    op.close()


@pytest.mark.parametrize("kernel", KERNELS)
@pytest.mark.parametrize("precision", MIXED)
def test_last_iteration_that_overflows(precision, kernel):
    """A basin 1e-20 deep: the mass matrix's entries are near 1e-23, so from b of 1e17 the one allowed iteration of plain
    CG takes a step beyond FP32's range, with every sum inside it. x is infinite and the true residual not a
    number: not converged."""
    op = pm.assemble_operator(box_basin(eps=1e-20))
    rhs = torch.from_numpy(1e17 * random_vector(op.n, 6)).cuda()
    x = torch.zeros_like(rhs)
    st = op.solve(pm.OP_MASS, rhs, x, pm.Options(max_iter=1, prec=pm.PREC_NONE, precision=precision, kernel=kernel),
                  allow_not_converged=True)
    assert st.iters == 1 and not bool(torch.isfinite(x).all())
    assert st.status == pm.PM_NOT_CONVERGED
    op.close()


@pytest.mark.parametrize("shape", [(40, 40, 12), (14, 15, 16)])   # 19,200 rows: the grid; 3,360: one cluster
@pytest.mark.parametrize("precision", [pm.FP64, *MIXED])
@pytest.mark.parametrize("which,prec", [(pm.OP_PRESSURE, pm.PREC_IC0), (pm.OP_PRESSURE, pm.PREC_LINE),
                                        (pm.OP_PRESSURE, pm.PREC_JACOBI), (pm.OP_VEL_U3, pm.PREC_LINE)])
def test_from_a_guess_that_has_not_converged(shape, precision, which, prec):
    """Against the stream of kernels, from zero and from a random guess. Both solutions have a true residual of rtol, so
    their difference has one of at most the two; an outer step or a restart ends where a residual passes its target,
    which rounding can move by one step."""
    op = pm.assemble_operator(box_basin(nh=shape[0], nhy=shape[1], nz=shape[2]))
    b, guess = (torch.from_numpy(random_vector(op.n, seed)).cuda() for seed in (51, 52))
    rtol = 1e-8
    for from_guess in (False, True):
        xs, outer = [], []
        for kernel in KERNELS:
            xs.append(guess.clone() if from_guess else torch.zeros_like(b))
            st = op.solve(which, b, xs[-1], pm.Options(rtol=rtol, prec=prec, precision=precision, x0_is_guess=from_guess,
                                                       inner_rtol=1e-2, kernel=kernel))
            assert st.status == pm.PM_OK and st.rel_residual_true <= rtol and st.iters > 0
            outer.append(st.outer_iters)
        assert abs(outer[0] - outer[1]) <= 1
        rr, _, _ = op.residual(which, torch.zeros_like(b), xs[0] - xs[1], torch.empty_like(b))
        assert rr ** 0.5 <= 2 * 1.05 * rtol * float(b.norm())
    op.close()
