"""Live kernel times of solves that run in one launch, and the benchmark's roofline of a step made of them."""
import pytest

N = 79_936          # rows of a 64 x 64 x 32 basin
STREAM = {k: (0.0, 0) for k in range(5)}


def test_roofline_of_a_step_of_resident_solves():
    import bench
    r = bench.roofline_of({**STREAM, 5: (30.0, 8)}, N, 2, 31.0, 6791.0, "measured", 2070.0, solve_bytes=6e9)
    assert r["kernel"] == "k_resident" and r["bound"] == "hbm" and list(r["classes"]) == ["k_resident"]
    assert r["achieved"] == round(6e9 / 30e-3 / 1e9, 1)
    assert r["classes"]["k_resident"]["launches_per_step"] == 4
    assert abs(r["kernel_share_of_step"] - 30.0 / 31.0) < 1e-3


def test_roofline_of_resident_solves_beside_streamed_ones():
    import bench
    spmv = 100 * N * (15 * 8 + 8 + 8)
    r = bench.roofline_of({**STREAM, 0: (10.0, 100), 5: (30.0, 2)}, N, 1, 45.0, 6791.0, "measured", 2070.0,
                          solve_bytes=spmv + 3e9)
    assert r["kernel"] == "k_resident" and set(r["classes"]) == {"k_cg_spmv", "k_resident"}
    assert r["achieved"] == round(3e9 / 30e-3 / 1e9, 1)


def test_roofline_of_a_step_without_work():
    import bench
    r = bench.roofline_of({**STREAM, 5: (0.0, 0)}, N, 1, 1.0, 6791.0, "measured")
    assert r["kernel"] is None and r["classes"] == {}


@pytest.mark.gpu
def test_a_resident_solve_is_timed():
    torch = pytest.importorskip("torch")
    import paper_1207_0486_gb300 as pm
    from paper_1207_0486_gb300 import api
    from workloads import box_basin, random_vector
    op = pm.assemble_operator(box_basin())
    b = torch.from_numpy(random_vector(op.n, 8)).cuda()
    stream = (api.KT_SPMV, api.KT_UPDATE, api.KT_PUPDATE, api.KT_IC0, api.KT_LINE)
    for precision in (pm.FP64, pm.FP32_REFINE, pm.BF16_REFINE):
        for kernel, resident in ((pm.KERNEL_AUTO, True), (pm.KERNEL_STREAM, False)):
            api.kernel_timing(True)
            for _ in range(3):
                op.solve(pm.OP_VEL_U1, b, torch.zeros_like(b), pm.Options(rtol=1e-8, prec=pm.PREC_IC0, precision=precision,
                                                                          kernel=kernel, inner_rtol=1e-2))
            got = {k: api.kernel_timing_get(k) for k in (*stream, api.KT_RESIDENT)}
            api.kernel_timing(False)
            ms, launches = got[api.KT_RESIDENT]
            assert launches == (3 if resident else 0) and (ms > 0.0) == resident
            assert (sum(got[k][1] for k in stream) == 0) == resident
    op.close()
