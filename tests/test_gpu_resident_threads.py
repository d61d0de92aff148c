"""Line solves of different operators from different host threads: each launch asks for its own block's tile of
shared memory, between none and more than the 48 KB that need no permission."""
import threading

import pytest

torch = pytest.importorskip("torch")

from workloads import box_basin, random_vector  # noqa: E402

pytestmark = pytest.mark.gpu

import paper_1207_0486_gb300 as pm  # noqa: E402

# rows, dynamic shared memory of a block (FP64): 2.4k, 2.3 KB (cluster); 84k, 4.6 KB; 0.41M, 22 KB; 0.91M, 49 KB
BOXES = [(17, 8), (46, 40), (101, 40), (151, 40)]


@pytest.mark.parametrize("precision", [pm.FP64, pm.FP32_REFINE])
def test_line_solves_of_different_sizes_from_different_threads(precision):
    """Every call runs its two iterations and leaves bit for bit what it leaves alone."""
    ops = [pm.assemble_operator(box_basin(nh=nh, nz=nz)) for nh, nz in BOXES for _ in range(2)]
    rhs = [torch.from_numpy(random_vector(op.n, 71 + i)).cuda() for i, op in enumerate(ops)]
    o = pm.Options(rtol=1e-14, prec=pm.PREC_LINE, precision=precision, max_iter=2, inner_rtol=1e-10)

    def solve(i, x, stream=None):
        return ops[i].solve(pm.OP_PRESSURE, rhs[i], x, o, stream=stream, allow_not_converged=True)

    alone = [torch.zeros_like(b) for b in rhs]
    for i, x in enumerate(alone):
        assert solve(i, x).iters == 2
    torch.cuda.synchronize()
    bad = []

    def work(i):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            x = torch.zeros_like(rhs[i])
            for k in range(150):
                try:
                    solve(i, x, s)
                except pm.PMError as e:
                    bad.append((ops[i].n, k, str(e)))
                    return
            s.synchronize()
            if not torch.equal(x, alone[i]):
                bad.append((ops[i].n, "differs"))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(ops))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad
    for op in ops:
        op.close()
