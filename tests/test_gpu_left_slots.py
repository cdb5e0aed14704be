"""Launches that leave their frame in the slots (they empty the whole table
before they fill it) and launches that count on empty ones, on one table in any
order: batches that share it, replayed graphs, which the host does not see, and
the split calls between them.  Against one table per call, fixed point, exactly."""
import pytest
import torch

from paper_1902_05942_gb300 import pps
from paper_1902_05942_gb300.configs import FilterConfig
from test_gpu_launch_shapes import _built, _vertices  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu

KEYS = ("r", "g", "b", "count", "status")


def _cfg(log2_slots):
    return FilterConfig(log2_slots=log2_slots, max_probes=64, voxel_scale=4.0, pixel_angle=0.01,
                        accum_fixed=True)


def _cam(frame):
    return (0.5 * frame, 3.0, -12.0)


def _views(large, *small):
    """A view, and others of its first vertices (they look for cells it has)."""
    v = _vertices(large, 3)
    return [v] + [{k: t[:n].clone() for k, t in v.items()} for n in small]


def _reference(log2_slots, v, frame):
    t = pps.Table(_cfg(log2_slots))
    out = t.filter(v, _cam(frame), frame)
    torch.cuda.synchronize()
    t.close()
    return out


def _same(out, ref, what):
    for k in KEYS:
        assert torch.equal(out[k], ref[k]), (what, k)


# the larger view sweeps its table, the smaller empties its own slots; from 2^20 vertices on a
# launch of its own
@pytest.mark.parametrize("log2_slots,large,small", [(16, 30_000, 300), (21, (1 << 20) + 5, 300),
                                                    (24, 1 << 21, (1 << 20) + 1)])
def test_batches_that_share_a_table(log2_slots, large, small):
    tab = pps.Table(_cfg(log2_slots))
    vs = _views(large, small, 1)
    outs = [pps.empty_output(v["px"].numel()) for v in vs]
    batches = [pps.Batch([(tab, v, o)]) for v, o in zip(vs, outs)]
    refs = [_reference(log2_slots, v, 7) for v in vs]
    for f, i in enumerate((0, 1, 0, 2, 1, 1, 0, 0, 1)):
        batches[i].run([_cam(7)], 7)
        _same(outs[i], refs[i], (f, i))
    for b in batches:
        b.close()
    # afterwards, on its own
    for f, i in enumerate((1, 0, 1)):
        _same(tab.filter(vs[i], _cam(7), 7), refs[i], ("filter", f))
    tab.close()


def test_replayed_graphs_in_any_order():
    tab = pps.Table(_cfg(16))
    vs = _views(30_000, 300)
    outs = [pps.empty_output(v["px"].numel()) for v in vs]
    refs = [_reference(16, v, 7) for v in vs]
    for v, o in zip(vs, outs):  # the tables' arrays are made by the first call of a size
        tab.filter(v, _cam(7), 7, out=o)
    graphs = []
    for v, o in zip(vs, outs):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            tab.filter(v, _cam(7), 7, out=o)
        graphs.append(g)

    def replay(i):
        for k in KEYS:
            outs[i][k].zero_()
        graphs[i].replay()
        _same(outs[i], refs[i], ("replay", i))

    def split(i):
        tab.build(_cam(7), 7)
        tab.insert(vs[i])
        _same(tab.query(vs[i]), refs[i], ("split", i))
        tab.build(_cam(7), 7)  # leaves the frame empty
        assert tab.stats()["occupied_slots"] == 0

    for i in (0, 1, 0, 0, 1, 1):
        replay(i)
    for i, j in ((0, 1), (0, 0), (1, 0), (1, 1)):
        replay(i)
        _same(tab.filter(vs[j], _cam(7), 7), refs[j], ("filter", i, j))
        replay(j)
        replay(i)
        split(j)
        tab.filter(vs[1], _cam(7), 7)
    tab.close()


def test_occupancy_is_counted_in_the_slots():
    """Between frames too: a replayed insert, of which the host knows nothing,
    shows in the statistics and the dump; what a launch left behind does not."""
    tab = pps.Table(_cfg(16))
    large, v = _views(30_000, 300)
    tab.build(_cam(7), 7)
    tab.insert(v)
    cells = tab.stats()["occupied_slots"]
    assert cells == tab.stats()["frame_cells"] > 0
    graph = torch.cuda.CUDAGraph()
    tab.build(_cam(7), 7)
    with torch.cuda.graph(graph):
        tab.insert(v)
    tab.filter(v, _cam(7), 7)  # empties its own slots
    assert tab.stats()["occupied_slots"] == 0 and not tab.dump()[0].any()
    graph.replay()
    assert tab.stats()["occupied_slots"] == cells and (tab.dump()[0] != 0).sum() == cells
    tab.filter(large, _cam(7), 7)  # empties the table first and leaves its own cells
    assert tab.stats()["occupied_slots"] == 0 and not tab.dump()[0].any()
    tab.filter(v, _cam(7), 7)
    assert tab.stats()["occupied_slots"] == 0 and not tab.dump()[0].any()
    tab.close()
