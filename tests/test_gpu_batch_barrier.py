"""The persistent kernel's grid barrier: blocks that wait must not slow down the blocks that share their SM."""
import time

import pytest

torch = pytest.importorskip("torch")

from workloads import box_basin, random_vector  # noqa: E402

pytestmark = pytest.mark.gpu

import paper_1207_0486_gb300 as pm  # noqa: E402


def test_waiting_blocks_leave_the_ic0_phases_their_cache():
    """One system of 2,048 rows in a server that fills the GPU: a few blocks work, the others of their SMs wait. An iteration
    has 22 barriers with IC0 and 5 with the line preconditioner; it takes 5 times as long, and took 6.8 times while every
    poll of a waiting block dropped its SM's L1."""
    op = pm.assemble_operator(box_basin())
    b = torch.from_numpy(random_vector(op.n, 61)).cuda()
    best = {}
    for prec in (pm.PREC_LINE, pm.PREC_IC0):
        srv = pm.Server(slots=1, nz_cap=8, tile_cols=64, block=128,
                        opts=pm.Options(rtol=1e-300, prec=prec, max_iter=10 ** 8, inner_rtol=1e-30))
        x = torch.zeros_like(b)
        work = torch.empty(srv.workspace_bytes(op), dtype=torch.uint8, device="cuda")
        srv.admit(op, pm.OP_MASS if prec == pm.PREC_IC0 else pm.OP_PRESSURE, b, x, work)
        srv.run(1)
        best[prec] = 1e9
        for _ in range(4):
            t0 = time.perf_counter()
            assert srv.run(16) == 1
            best[prec] = min(best[prec], time.perf_counter() - t0)
        srv.close()
    op.close()
    assert best[pm.PREC_IC0] <= 5.9 * best[pm.PREC_LINE], best


@pytest.mark.parametrize("precision", [pm.FP64, pm.FP32_REFINE])
def test_ic0_batches_on_either_side_of_one_block_per_sm(precision):
    """Few tiles (a block has its SM to itself) and many (blocks share one): every solution is the system's own, bit for
    bit."""
    shapes = [(25, 12), (60, 20), (48, 16)]
    ops = [pm.assemble_operator(box_basin(nh=nh, nz=nz)) for nh, nz in shapes]
    o = pm.Options(rtol=1e-8, prec=pm.PREC_IC0, precision=precision, inner_rtol=1e-2)
    which = [pm.OP_MASS, pm.OP_VEL_U1, pm.OP_VEL_U3]
    alone = {}
    for count in (1, 3, 40):
        so = [ops[i % 3] for i in range(count)]
        sw = [which[i % 3] for i in range(count)]
        bs = [torch.from_numpy(random_vector(op.n, 70 + i % 3)).cuda() for i, op in enumerate(so)]
        bt = pm.Batch(so, sw, o)
        xs = [torch.zeros_like(b) for b in bs]
        for k, st in enumerate(bt.solve(bs, xs)):
            assert st.status == pm.PM_OK
            if k % 3 not in alone:
                alone[k % 3] = (xs[k].clone(), st.iters)
            assert torch.equal(xs[k], alone[k % 3][0]) and st.iters == alone[k % 3][1], (count, k)
        bt.close()
    for op in ops:
        op.close()
