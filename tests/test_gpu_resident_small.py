"""The smallest resident solves: one block up to 400 rows (IC0 1,024), one cluster of blocks above."""
import time

import pytest

torch = pytest.importorskip("torch")

from workloads import box_basin, random_vector  # noqa: E402

pytestmark = pytest.mark.gpu

import paper_1207_0486_gb300 as pm  # noqa: E402

# rows: 8, 99, 400, 405 (Jacobi, line: the last one block, the first cluster), 512, 1,024, 1,029 (the same for IC0)
SHAPES = [(2, 2, 2), (3, 3, 11), (5, 5, 16), (9, 9, 5), (8, 8, 8), (8, 16, 8), (7, 7, 21)]


def rhs_of(op, seed):
    return torch.from_numpy(random_vector(op.n, seed)).cuda()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("precision", [pm.FP64, pm.FP32_REFINE, pm.BF16_REFINE])
@pytest.mark.parametrize("prec", [pm.PREC_JACOBI, pm.PREC_NONE, pm.PREC_IC0, pm.PREC_LINE])
def test_small_solves_match_the_stream(shape, precision, prec):
    """From zero and from a guess, velocity, mass and pressure, to a true residual of rtol: two solutions differ by at
    most the two residuals."""
    nh, ny, nz = shape
    op = pm.assemble_operator(box_basin(nh=nh, nhy=ny, nz=nz))
    b, guess = rhs_of(op, 41), rhs_of(op, 42)
    rtol = 1e-8
    for which in (pm.OP_VEL_U2, pm.OP_MASS, pm.OP_PRESSURE):
        if prec == pm.PREC_NONE and which == pm.OP_PRESSURE:
            continue
        for from_guess in (False, True):
            o = pm.Options(rtol=rtol, prec=prec, precision=precision, x0_is_guess=from_guess, inner_rtol=1e-2)
            xs = []
            for kernel in (pm.KERNEL_STREAM, pm.KERNEL_AUTO):
                xs.append(guess.clone() if from_guess else torch.full_like(b, float("nan")))
                o.kernel = kernel
                st = op.solve(which, b, xs[-1], o)
                assert st.status == pm.PM_OK and st.rel_residual_true <= rtol
            if precision == pm.FP64 and prec in (pm.PREC_JACOBI, pm.PREC_NONE):
                xs.append(guess.clone() if from_guess else torch.full_like(b, float("nan")))
                assert op.solve_noalloc(which, b, xs[-1], o).status == pm.PM_OK
            for x in xs[1:]:
                rr, _, _ = op.residual(which, torch.zeros_like(b), xs[0] - x, torch.empty_like(b))
                assert rr ** 0.5 <= 2 * 1.05 * rtol * float(b.norm())
    op.close()


@pytest.mark.parametrize("precision", [pm.FP64, pm.FP32_REFINE])
def test_one_block_ends_as_the_others_do(precision):
    """A zero and a non-finite right-hand side, no iteration allowed, too few allowed: 72 rows in one block."""
    op = pm.assemble_operator(box_basin(nh=3, nhy=3, nz=8))
    b = rhs_of(op, 43)
    for prec in (pm.PREC_JACOBI, pm.PREC_IC0, pm.PREC_LINE):
        o = pm.Options(rtol=1e-8, prec=prec, precision=precision, inner_rtol=1e-2)
        x = torch.ones_like(b)
        st = op.solve(pm.OP_PRESSURE, torch.zeros_like(b), x, o)
        assert st.status == pm.PM_OK and st.iters == 0 and float(x.abs().max()) == 0.0
        bad = b.clone()
        bad[5] = float("inf")
        with pytest.raises(pm.PMError):
            op.solve(pm.OP_PRESSURE, bad, x, o)
        for cap in (0, 2):
            o.max_iter = cap
            st = op.solve(pm.OP_PRESSURE, b, torch.zeros_like(b), o, allow_not_converged=True)
            assert st.status == pm.PM_NOT_CONVERGED and st.iters == cap
    op.close()


def test_an_iteration_of_one_block_is_cheaper_than_a_clusters():
    """IC0 pressure in FP64, 512 rows against 2,048: by 16 blocks an iteration of either costs its barriers alike (ratio
    0.93), one block's is a third cheaper."""
    us = []
    for nh in (8, 16):
        op = pm.assemble_operator(box_basin(nh=nh))
        b = rhs_of(op, 44)
        best = 1e9
        for _ in range(20):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            st = op.solve(pm.OP_PRESSURE, b, torch.zeros_like(b), pm.Options(rtol=1e-10, prec=pm.PREC_IC0))
            best = min(best, (time.perf_counter() - t0) / st.iters)
        us.append(best * 1e6)
        op.close()
    assert us[0] <= 0.85 * us[1], us
