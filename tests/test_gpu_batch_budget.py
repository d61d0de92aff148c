"""Which of the batched kernel's two register budgets a launch takes, and that it changes no result."""
import pytest

torch = pytest.importorskip("torch")

from workloads import box_basin, random_vector  # noqa: E402

pytestmark = pytest.mark.gpu

import paper_1207_0486_gb300 as pm  # noqa: E402

BOXES = [(48, 8), (70, 20), (90, 31), (110, 16), (135, 40), (160, 24)]


@pytest.fixture(scope="module")
def ops():
    made = [pm.assemble_operator(box_basin(nh=nh, nz=nz)) for nh, nz in BOXES]
    yield made
    for op in made:
        op.close()


def entries(ops, systems):
    return [ops[i % 6] for i in range(systems)], [(pm.OP_PRESSURE, pm.OP_VEL_U1, pm.OP_VEL_U3)[i // 6 % 3] for i in range(systems)]


@pytest.mark.parametrize("precision,systems,per_sm", [
    (pm.FP64, 6, 2), (pm.FP64, 12, 3), (pm.FP64, 24, 3),                          # 469, 938, 1,876 tiles
    (pm.FP32_REFINE, 6, 2), (pm.FP32_REFINE, 13, 2), (pm.FP32_REFINE, 24, 3),     # 469, 947, 1,876 tiles
    (pm.BF16_REFINE, 13, 2), (pm.BF16_REFINE, 24, 3)])
def test_budget_follows_the_tiles(ops, precision, systems, per_sm):
    """All systems iterating: two blocks per SM where a block has a tile or a few, three where they are many."""
    so, sw = entries(ops, systems)
    bt = pm.Batch(so, sw, pm.Options(rtol=1e-8, prec=pm.PREC_LINE, precision=precision, inner_rtol=1e-4))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    i = bt.info()
    bt.close()
    if sms == 152:
        assert i["grid"] == per_sm * sms, i


@pytest.mark.parametrize("precision,systems,per_sm", [
    (pm.FP64, 5, 3), (pm.FP64, 12, 2), (pm.FP64, 24, 2),                          # 319, 938, 1,876 tiles
    (pm.FP32_REFINE, 5, 3), (pm.FP32_REFINE, 24, 2), (pm.BF16_REFINE, 60, 2)])    # 319, 1,876, 4,690 tiles
def test_budget_of_mass_systems(ops, precision, systems, per_sm):
    """Mass systems alone gain more from two blocks per SM: a batch takes them wherever the busiest block ends sooner."""
    bt = pm.Batch([ops[i % 6] for i in range(systems)], [pm.OP_MASS] * systems,
                  pm.Options(rtol=1e-8, prec=pm.PREC_LINE, precision=precision, inner_rtol=1e-4))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    i = bt.info()
    bt.close()
    if sms == 152:
        assert i["grid"] == (per_sm * sms if per_sm == 2 else min(per_sm * sms, i["tiles"])), i


@pytest.mark.parametrize("precision", [pm.FP64, pm.FP32_REFINE, pm.BF16_REFINE])
def test_solutions_do_not_depend_on_the_budget(ops, precision):
    """Twenty-four systems that end at very different iterations, so that the launches pass from three blocks per SM to
    two: every solution is bit for bit the one of a batch of that system alone."""
    so, sw = entries(ops, 24)
    o = pm.Options(rtol=1e-8, prec=pm.PREC_LINE, precision=precision, inner_rtol=1e-4, max_iter=20000)
    bs = [torch.from_numpy(random_vector(op.n, 400 + i)).cuda() for i, op in enumerate(so)]
    xs = [torch.zeros_like(b) for b in bs]
    bt = pm.Batch(so, sw, o)
    st = bt.solve(bs, xs)
    iters = [s.iters for s in st]
    assert max(iters) > 64 + min(iters)
    for i in (0, 1, 5, 8, 17, 23):
        one = pm.Batch([so[i]], [sw[i]], o)
        x = torch.zeros_like(bs[i])
        s1 = one.solve([bs[i]], [x])
        assert s1[0].iters == iters[i] and torch.equal(x, xs[i]), i
        one.close()
    again = [torch.zeros_like(b) for b in bs]   # both captured launches, replayed
    assert [s.iters for s in bt.solve(bs, again)] == iters
    assert all(torch.equal(a, b) for a, b in zip(xs, again))
    bt.close()
