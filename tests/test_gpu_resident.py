"""The resident solve (one launch per solve) at the sizes where its teams and tiles can go wrong: fewer
columns than blocks, columns that do not divide among the blocks, odd level counts, empty colours, either side
of the line between the cluster and the grid, columns too tall for the shared-memory tile."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import ell_to_csr  # noqa: E402
from workloads import box_basin, ocean_basin, random_vector  # noqa: E402

pytestmark = pytest.mark.gpu

import paper_1207_0486_gb300 as pm  # noqa: E402

SYSTEMS = [(pm.OP_VEL_U1, pm.PREC_IC0), (pm.OP_VEL_U3, pm.PREC_LINE), (pm.OP_MASS, pm.PREC_IC0),
           (pm.OP_MASS, pm.PREC_NONE), (pm.OP_PRESSURE, pm.PREC_IC0), (pm.OP_PRESSURE, pm.PREC_LINE),
           (pm.OP_PRESSURE, pm.PREC_JACOBI)]


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


@pytest.mark.parametrize("shape", [(2, 2, 2), (3, 2, 5), (5, 4, 3), (4, 17, 9), (9, 8, 16)])
@pytest.mark.parametrize("precision", [pm.FP64, pm.FP32_REFINE, pm.BF16_REFINE])
@pytest.mark.parametrize("which,prec", SYSTEMS)
def test_small_systems_against_a_dense_solve(shape, precision, which, prec):
    """Against numpy's dense solution of the stored operator. A residual of rtol ||b|| moves the solution by
    at most cond(A) rtol ||x||; the dense solve itself is good to cond(A) n u."""
    nh, ny, nz = shape
    op = pm.assemble_operator(box_basin(nh=nh, nhy=ny, nz=nz))
    vals, nbr, _ = op.export(which)
    A = ell_to_csr(vals, nbr, op.nz).toarray()
    b = random_vector(op.n, 5 + which)
    m = None
    if which == pm.OP_PRESSURE:   # zero-mean multiplier: b without its m part, x with m'x = 0
        vm, _, _ = op.export(pm.OP_MASS)
        m = vm.sum(axis=0)
        b = b - (b.sum() / m.sum()) * m
        K = np.block([[A, m[:, None]], [m[None, :], np.zeros((1, 1))]])
        ref = np.linalg.solve(K, np.append(b, 0.0))[:-1]
        ev = np.linalg.eigvalsh(A)
        cond = ev[-1] / ev[1]
    else:
        ref = np.linalg.solve(A, b)
        cond = np.linalg.cond(A)
    x = torch.zeros(op.n, dtype=torch.float64, device="cuda")
    rtol = 1e-10
    st = op.solve(which, dev(b), x, pm.Options(rtol=rtol, prec=prec, precision=precision, max_restarts=8))
    assert st.status == pm.PM_OK and st.rel_residual_true <= max(rtol, st.rel_residual_floor)
    err = np.linalg.norm(x.cpu().numpy() - ref) / np.linalg.norm(ref)
    # the pressure's relative change is measured against ||x|| >= ||b|| / lambda_max
    assert err <= cond * (max(rtol, st.rel_residual_floor) + op.n * 2.0 ** -52), (err, cond)
    if m is not None:
        assert abs(m @ x.cpu().numpy()) <= 1e-11 * np.abs(ref).max() * m.sum()
    op.close()


@pytest.mark.parametrize("basin", ["below", "above", "odd", "ocean", "tall"])
@pytest.mark.parametrize("which,prec", [s for s in SYSTEMS if s != (pm.OP_PRESSURE, pm.PREC_IC0)])
@pytest.mark.parametrize("guess", [False, True])
def test_resident_matches_stream(basin, which, prec, guess):
    """The same recurrence either way: iteration counts within two (2 % above 100 iterations), the true
    residual at rtol, and solutions that differ by what two residuals of rtol can: e = A^-1 (r1 - r2), measured
    by the residual of the difference."""
    b = {"below": lambda: box_basin(nh=31, nhy=33, nz=8),        # 8,184 rows: the cluster
         "above": lambda: box_basin(nh=37, nhy=37, nz=12),       # 16,428 rows: the grid
         "odd": lambda: box_basin(nh=61, nhy=47, nz=13),
         "ocean": lambda: ocean_basin(nx=96, ny=80, nz=17, dx=5e4),
         "tall": lambda: box_basin(nh=3, nhy=3, nz=199)}[basin]()
    op = pm.assemble_operator(b)
    rhs = dev(random_vector(op.n, 9))
    x0 = dev(random_vector(op.n, 10)) if guess else torch.zeros(op.n, dtype=torch.float64, device="cuda")
    rtol = 1e-9
    xs, st = [], []
    for kernel in (pm.KERNEL_STREAM, pm.KERNEL_RESIDENT):
        x = x0.clone()
        st.append(op.solve(which, rhs, x, pm.Options(rtol=rtol, prec=prec, kernel=kernel, x0_is_guess=guess)))
        xs.append(x)
    assert st[0].status == st[1].status == pm.PM_OK
    for s in st:
        assert s.rel_residual_true <= max(rtol, s.rel_residual_floor)
    if st[0].outer_iters == st[1].outer_iters:
        assert abs(st[0].iters - st[1].iters) <= max(2 * (1 + st[0].outer_iters), 0.02 * st[0].iters)
    r = torch.empty_like(rhs)
    d = xs[0] - xs[1]
    rr, _, _ = op.residual(which, torch.zeros_like(rhs), d, r)
    bb = float(rhs.norm())
    assert rr ** 0.5 <= sum(max(rtol, s.rel_residual_floor) for s in st) * 1.05 * bb
    op.close()


@pytest.mark.parametrize("precision", [pm.FP64, pm.FP32_REFINE])
def test_limits_and_empty_work(precision):
    """No iteration allowed, a cap, a zero right-hand side, a guess that already solves the system."""
    op = pm.assemble_operator(box_basin(nh=40, nz=12))   # 19,200 rows: the grid
    rhs = dev(random_vector(op.n, 3))
    x = torch.zeros_like(rhs)
    o = dict(prec=pm.PREC_IC0, precision=precision, rtol=1e-9)
    st = op.solve(pm.OP_VEL_U2, rhs, x, pm.Options(max_iter=0, **o), allow_not_converged=True)
    assert st.status == pm.PM_NOT_CONVERGED and st.iters == 0 and float(x.abs().max()) == 0.0
    st = op.solve(pm.OP_VEL_U2, rhs, x, pm.Options(max_iter=7, **o), allow_not_converged=True)
    assert st.status == pm.PM_NOT_CONVERGED and st.iters == 7 and st.rel_residual_true < 1.0
    st = op.solve(pm.OP_VEL_U2, rhs, x, pm.Options(**o))
    full = st.iters
    st = op.solve(pm.OP_VEL_U2, rhs, x, pm.Options(x0_is_guess=True, **{**o, "rtol": 1e-8}))
    assert st.iters == 0 and full > 0 and st.rel_residual_true <= 1e-8
    st = op.solve(pm.OP_VEL_U2, torch.zeros_like(rhs), x, pm.Options(**o))
    assert st.status == pm.PM_OK and st.iters == 0 and float(x.abs().max()) == 0.0
    bad = rhs.clone()
    bad[5000] = float("nan")
    with pytest.raises(pm.PMError) as e:
        op.solve(pm.OP_VEL_U2, bad, x, pm.Options(**o))
    assert e.value.status == pm.PM_BREAKDOWN
    st = op.solve(pm.OP_VEL_U2, rhs, x, pm.Options(**o))
    assert st.iters == full
    op.close()


def test_two_threads_on_their_own_streams():
    """Different operators may be solved from different host threads: the launches of two grids and of a cluster
    next to a grid leave each other room, and every solution is bit for bit the one of a solve alone."""
    import threading
    ops = [pm.assemble_operator(box_basin(nh=s, nz=12)) for s in (20, 60, 70)]
    rhs = [dev(random_vector(op.n, 21 + i)) for i, op in enumerate(ops)]
    o = pm.Options(rtol=1e-9, prec=pm.PREC_IC0)
    alone = []
    for op, b in zip(ops, rhs):
        x = torch.zeros_like(b)
        op.solve(pm.OP_VEL_U1, b, x, o)
        alone.append(x)
    torch.cuda.synchronize()
    bad = []

    def work(i):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(10):
                x = torch.zeros_like(rhs[i])
                try:
                    ops[i].solve(pm.OP_VEL_U1, rhs[i], x, o, stream=s)
                except pm.PMError as e:
                    bad.append((i, str(e)))
                    return
                if not torch.equal(x, alone[i]):
                    bad.append((i, "differs"))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad
    for op in ops:
        op.close()


@pytest.mark.parametrize("shape", [(21, 19, 32), (21, 19, 8), (23, 17, 31), (9, 11, 47), (5, 7, 210)])
@pytest.mark.parametrize("precision", [pm.FP32_REFINE, pm.BF16_REFINE])
@pytest.mark.parametrize("which,prec", SYSTEMS)
def test_mixed_stream_matches_resident(shape, precision, which, prec):
    """The mixed-precision stream of kernels: four rows per thread where the levels are a multiple of four, the line
    kernel at 32 levels, others, and tall columns, against the resident solve. Both end
    at a true residual of rtol (or the FP64 floor), so their difference has at most the two residuals' sum. Iteration counts are not compared: an FP32
    recurrence of thousands of iterations depends on its rounding (the Jacobi pressure system of 31 levels takes 3808 or
    4388 iterations on the stream path and 3730 to 4388 resident under changes of 1e-7 in b)."""
    nh, ny, nz = shape
    op = pm.assemble_operator(box_basin(nh=nh, nhy=ny, nz=nz))
    rhs = dev(random_vector(op.n, 40 + which))
    rtol = 1e-9
    xs, st = [], []
    for kernel in (pm.KERNEL_STREAM, pm.KERNEL_AUTO):
        x = torch.zeros_like(rhs)
        st.append(op.solve(which, rhs, x, pm.Options(rtol=rtol, prec=prec, precision=precision, inner_rtol=1e-2,
                                                     kernel=kernel)))
        xs.append(x)
    for s in st:
        assert s.status == pm.PM_OK and s.rel_residual_true <= max(rtol, s.rel_residual_floor)
    r = torch.empty_like(rhs)
    rr, _, _ = op.residual(which, torch.zeros_like(rhs), xs[0] - xs[1], r)
    assert rr ** 0.5 <= sum(max(rtol, s.rel_residual_floor) for s in st) * 1.05 * float(rhs.norm())
    op.close()
