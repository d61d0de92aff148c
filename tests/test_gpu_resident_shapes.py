"""Resident solves of basins with fewer columns than blocks, or hardly more: every block takes its share of the rows."""
import time

import pytest

torch = pytest.importorskip("torch")

from workloads import box_basin, random_vector  # noqa: E402

pytestmark = pytest.mark.gpu

import paper_1207_0486_gb300 as pm  # noqa: E402


def rhs_of(op, seed):
    return torch.from_numpy(random_vector(op.n, seed)).cuda()


@pytest.mark.parametrize("shape", [(2, 2, 9001), (3, 5, 2003), (12, 13, 333), (2, 3, 2734)])   # the last: a cluster's size + 20
@pytest.mark.parametrize("precision", [pm.FP64, pm.FP32_REFINE])
@pytest.mark.parametrize("prec", [pm.PREC_JACOBI, pm.PREC_IC0, pm.PREC_NONE])
def test_few_tall_columns(shape, precision, prec):
    """Mass solves to a true residual of rtol: two of them differ by at most the two residuals."""
    nh, ny, nz = shape
    op = pm.assemble_operator(box_basin(nh=nh, nhy=ny, nz=nz))
    b = rhs_of(op, 31)
    rtol = 1e-9
    xs = []
    for kernel in (pm.KERNEL_STREAM, pm.KERNEL_AUTO):
        xs.append(torch.zeros_like(b))
        st = op.solve(pm.OP_MASS, b, xs[-1], pm.Options(rtol=rtol, prec=prec, precision=precision, kernel=kernel))
        assert st.status == pm.PM_OK and st.rel_residual_true <= rtol
    if precision == pm.FP64 and prec != pm.PREC_IC0:
        xs.append(torch.zeros_like(b))
        op.solve_noalloc(pm.OP_MASS, b, xs[-1], pm.Options(rtol=rtol, prec=prec))
    for x in xs[1:]:
        rr, _, _ = op.residual(pm.OP_MASS, torch.zeros_like(b), xs[0] - x, torch.empty_like(b))
        assert rr ** 0.5 <= 2 * 1.05 * rtol * float(b.norm())
    op.close()


def test_few_tall_columns_use_every_block():
    """16 columns of 20,000 levels by the diagonal: no slower than the stream of kernels, which spreads rows over all SMs
    (whole columns in 16 blocks took 2.4 times as long)."""
    op = pm.assemble_operator(box_basin(nh=4, nz=20000))
    b = rhs_of(op, 32)
    x = torch.zeros_like(b)

    def seconds(solve, kernel):
        o = pm.Options(rtol=1e-15, prec=pm.PREC_JACOBI, kernel=kernel, max_iter=60)
        best = 1e9
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            assert solve(pm.OP_VEL_U1, b, x, o, allow_not_converged=True).iters == 60
            best = min(best, time.perf_counter() - t0)
        return best

    stream = seconds(op.solve, pm.KERNEL_STREAM)
    assert seconds(op.solve, pm.KERNEL_AUTO) <= 1.2 * stream
    assert seconds(op.solve_noalloc, pm.KERNEL_AUTO) <= 1.2 * stream
    op.close()
