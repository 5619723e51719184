"""The intermediates of a ragged batch's two lanes of length classes: one is enough where the device
has no room for the second, or where no recording uses it (in place, FST_GRAPHS=0)."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1611_04950_gb300 import fst as F  # noqa: E402
from paper_1611_04950_gb300 import workloads  # noqa: E402

PARAMS = [(n, 0.1, 1e-6) for n in (200001, 180000, 150001, 140000, 135001, 133000, 50001, 40000, 9001)]


def _batch():
    return [workloads.gaussian(1, n, seed=n)[0].float().cuda() for n, _, _ in PARAMS]


def test_no_room_for_the_second_lane():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ps = F.PlanSet(PARAMS)
    ys = _batch()
    ref = [o.clone() for o in ps.project(ys)]
    outs = [torch.empty_like(y) for y in ys]
    # the first call of a signature allocates two descriptor arrays, partials and coefficients,
    # then the two intermediates
    F.fst_test_alloc_fail(1, after=5)
    try:
        for _ in range(3):                       # direct, recorded, replayed
            for o in outs:
                o.zero_()
            ps.project(ys, outs)
            assert all(torch.equal(o, r) for o, r in zip(outs, ref))
    finally:
        F.fst_test_alloc_fail(0)
    ps.close()


@pytest.mark.parametrize("inplace,graphs", [(True, "1"), (False, "0")])
def test_one_intermediate_where_one_is_used(monkeypatch, inplace, graphs):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    monkeypatch.setenv("FST_GRAPHS", graphs)
    params = PARAMS[6:] + [(200000 + i, 0.1, 1e-1) for i in range(32)]
    ps = F.PlanSet(params)
    ys = [workloads.gaussian(1, n, seed=n)[0].float().cuda() for n, _, _ in params]
    outs = ys if inplace else [torch.empty_like(y) for y in ys]
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ps.project(ys, outs)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    inter = 32 * (8 << 19)                       # the longest class: 32 slots of 2^19 complex samples
    assert used < inter + inter // 2, used
    ps.close()
