"""Frames that outgrow a table's cell arrays while the last frame's cells are
still in its slots: tables with a migrating history or the search for similar
normals, and frames left open by the split calls.  The slots are emptied by the
records of the old arrays, so that comes before the new ones.  Against a table
large enough from the start, fixed point, exactly."""
import dataclasses

import pytest
import torch

from paper_1902_05942_gb300 import pps
from test_gpu_migration import CAM, _built, _cfg, _cloud, _dev  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu

KEYS = ("r", "g", "b", "count", "status")


def _pair(**kw):
    # 2^12 slots: room for 19 tiles of 256 vertices at first; 2^16: for 6,000 vertices and more
    cfg = _cfg(accum_fixed=True, max_probes=64, **kw)
    return [pps.Table(dataclasses.replace(cfg, log2_slots=k)) for k in (12, 16)]


@pytest.mark.parametrize("kw", [
    dict(),
    dict(hist_mode=0, log2_hist_slots=0, hist_migrate=False, normal_in_home_hash=False, normal_search=2)])
@pytest.mark.parametrize("sizes", [(100, 6000), (1, 5000, 100, 20000)])
def test_a_frame_that_outgrows_the_cell_arrays(kw, sizes):
    small, large = _pair(**kw)
    blend = "hist_mode" not in kw
    for f, n in enumerate(sizes):
        v = _dev(_cloud(n, 5 + f))
        cam = (CAM[0] + f, CAM[1], CAM[2] - 3 * f)
        a, b = (t.filter(v, cam, f, blend=blend, alpha=0.25) for t in (small, large))
        sa, sb = small.stats(), large.stats()
        assert sa["overflow_vertices"] == sb["overflow_vertices"] == 0
        for k in ("frame_cells", "occupied_slots", "hist_occupied", "vertices"):
            assert sa[k] == sb[k], (f, k)
        for k in KEYS:
            assert torch.equal(a[k], b[k]), (f, k)
    small.close()
    large.close()


@pytest.mark.parametrize("kw", [dict(), dict(hist_migrate=False)])
def test_a_filter_call_that_outgrows_an_open_frame(kw):
    small, large = _pair(**kw)
    first, then = _dev(_cloud(200, 1)), _dev(_cloud(7000, 2))
    for t in (small, large):
        t.build(CAM, 0)
        t.insert(first)
    a, b = (t.filter(then, CAM, 1, blend=True, alpha=0.25) for t in (small, large))
    assert small.stats()["overflow_vertices"] == 0
    for k in KEYS:
        assert torch.equal(a[k], b[k]), k
    assert small.stats()["frame_cells"] == large.stats()["frame_cells"]
    small.close()
    large.close()
