"""A resident solve's bounded wait that runs out."""
import pytest

torch = pytest.importorskip("torch")

from workloads import box_basin, random_vector  # noqa: E402

pytestmark = pytest.mark.gpu

import paper_1207_0486_gb300 as pm  # noqa: E402


def test_a_result_reported_after_a_wait_ran_out_is_a_timeout():
    """One block gives up at the last barrier, rank 0 passes it and reports its result: the solve has timed out all
    the same. Solves before and after it are alike."""
    op = pm.assemble_operator(box_basin(nh=40, nz=12))   # 19,200 rows: the grid
    b = torch.from_numpy(random_vector(op.n, 3)).cuda()
    xs = []
    for k in range(2):
        for solve in (op.solve, op.solve_noalloc):
            x = torch.zeros_like(b)
            assert solve(pm.OP_MASS, b, x, pm.Options(rtol=1e-9, prec=pm.PREC_JACOBI)).status == pm.PM_OK
            xs.append(x)
        if k == 0:
            assert pm.debug_barrier_timeout() == pm.PM_TIMEOUT
    assert torch.equal(xs[0], xs[2]) and torch.equal(xs[1], xs[3])
    op.close()
