"""Mixed-precision solves in one launch: what is not a number never passes for a solution."""
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
