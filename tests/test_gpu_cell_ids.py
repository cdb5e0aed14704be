"""Cell ids of the split calls: frames whose ids leave no bit to mark a cell's
creator (their inserts add every contribution in the second pass), and inserts so
large that a warp's tile, and its range of ids, is a wider one.  Against the
persistent launch or the ordinary insert; fixed point exactly, FP32 within the
summation bound (n + 1) 2^-24 each."""
import pytest
import torch

from paper_1902_05942_gb300 import pps
from paper_1902_05942_gb300.configs import FilterConfig
from test_gpu_launch_shapes import _built, _vertices  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu

EYE = (0.5, 3.0, -12.0)


def _cfg(log2_slots, **kw):
    return FilterConfig(log2_slots=log2_slots, max_probes=64, voxel_scale=4.0, pixel_angle=0.01, **kw)


def _flat(n, seed, size=0.2):
    v = _vertices(n, seed)
    for k in ("px", "py", "pz"):
        v[k] = (v[k] * size).contiguous()
    for k, x in (("nx", 0.0), ("ny", 0.0), ("nz", 1.0)):
        v[k] = torch.full_like(v[k], x)
    return v


def _frame(tab, parts, blend):
    tab.build(EYE, 3)
    ids = [torch.empty(v["px"].numel(), dtype=torch.int32, device="cuda") for v in parts]
    for v, i in zip(parts, ids):
        tab.insert(v, i)
    if blend:
        tab.blend(0.25)
    return [(tab.query(v, i), tab.query(v)) for v, i in zip(parts, ids)], ids


def _compare(a, b, fixed):
    for c in ("count", "status"):
        assert torch.equal(a[c], b[c])
    for c in "rgb":
        if fixed:
            assert torch.equal(a[c], b[c])
        else:
            bound = 2 * (b["count"].float() + 1) * 2.0 ** -24 * b[c].abs() + 1e-7
            assert bool(((a[c] - b[c]).abs() <= bound).all())


@pytest.mark.parametrize("fixed", [False, True])
@pytest.mark.parametrize("kw", [dict(), dict(hist_mode=1, log2_hist_slots=17),
                                dict(hist_mode=1, log2_hist_slots=17, hist_migrate=True),
                                dict(normal_in_home_hash=False, normal_search=2)])
@pytest.mark.parametrize("batch", [2, 4])
def test_ids_that_leave_no_bit(fixed, kw, batch):
    parts = [_flat(n, 3 + n) for n in (5003, 1, 255, 1030)]
    res = []
    for wide in (False, True):
        tab = pps.Table(_cfg(15, accum_fixed=fixed, **kw))
        tab.tune(batch)
        pps.pps_selftest_wide_ids(tab.handle, wide)
        for _ in range(2):  # and over the last frame's slots
            out, ids = _frame(tab, parts, "hist_mode" in kw)
        st = tab.stats()
        assert st["overflow_vertices"] == 0 and st["occupied_slots"] == st["frame_cells"]
        res.append((out, st))
        tab.close()
    for k in ("frame_cells", "occupied_slots", "vertices", "hist_occupied"):
        assert res[0][1][k] == res[1][1][k]
    for (a, a2), (b, b2) in zip(res[0][0], res[1][0]):
        _compare(a, b, fixed)
        _compare(a2, b2, fixed)


@pytest.mark.parametrize("n", [(1 << 24) - 1, (1 << 24) + 1025])
@pytest.mark.parametrize("fixed", [False, True])
def test_inserts_with_wider_tiles(n, fixed):
    first, v = _flat(777, 1, 1.0), _flat(n, 2, 1.0)
    tab, ref = (pps.Table(_cfg(22, accum_fixed=fixed)) for _ in range(2))
    for _ in range(2):
        out, ids = _frame(tab, [first, v, first], False)
    assert tab.stats()["overflow_vertices"] == 0
    assert tab.stats()["frame_cells"] == tab.stats()["occupied_slots"]
    both = {k: torch.cat([first[k], v[k], first[k]]) for k in v}
    ids = torch.cat([torch.arange(777), torch.arange(n), torch.arange(777)]).to(torch.int32).cuda()
    want = ref.filter(both, EYE, 3, ids=ids)
    assert ref.stats()["frame_cells"] == tab.stats()["frame_cells"]
    for (a, b), at in zip(out, (0, 777, 777 + n)):
        part = {k: t[at:at + a["r"].numel()] for k, t in want.items()}
        _compare(a, part, fixed)
        _compare(b, part, fixed)
    tab.build(EYE, 4)
    assert tab.stats()["occupied_slots"] == 0
    for t in (tab, ref):
        t.close()
