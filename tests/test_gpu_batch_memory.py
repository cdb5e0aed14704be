"""What a batch reserves, and batches whose tables move their arrays: a table
has room for the cell ids of its view's tiles, no more, and a batch finds the
arrays that a larger call on the same table has made since."""
import pytest
import torch

from paper_1902_05942_gb300 import pps
from test_gpu_launch_shapes import _built, _vertices  # noqa: F401 (fixture)
from test_gpu_left_slots import KEYS, _cam, _cfg, _reference, _views

pytestmark = pytest.mark.gpu


def _flat(v, scale=1.0):
    """The vertices with one normal (fewer cells than slots), in a smaller place."""
    v = {k: (t * scale if k in ("px", "py", "pz") else t).contiguous() for k, t in v.items()}
    for k, x in (("nx", 0.0), ("ny", 0.0), ("nz", 1.0)):
        v[k] = torch.full_like(v[k], x)
    return v


def test_a_view_reserves_the_ids_of_its_own_tiles():
    """2.6 M vertices: 1.375 ids each in tiles of 256, which a table of 2^21 slots
    has from the start (2^22 cells); the launch's stash takes 4 bytes a vertex."""
    n = 2_600_000
    v, out = _flat(_vertices(n, 1)), pps.empty_output(n)
    tab = pps.Table(_cfg(21))
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    batch = pps.Batch([(tab, v, out)])
    assert before - torch.cuda.mem_get_info()[0] <= 4 * n + (32 << 20)
    batch.run([_cam(7)], 7)
    ref = _reference(21, v, 7)
    for k in KEYS:
        assert torch.equal(out[k], ref[k]), k
    batch.close()
    tab.close()


@pytest.mark.parametrize("sizes", [(200, 30_000), (5000, (1 << 20) + 9), ((1 << 20) + 9, 3_500_000)])
def test_batches_after_a_larger_call_on_their_table(sizes):
    small, large = sizes
    log2_slots = 12 if small == 200 else 21  # the larger view outgrows its cell arrays
    tab = pps.Table(_cfg(log2_slots))
    vs = [_flat(v, 0.02 if log2_slots == 12 else 1.0) for v in _views(large, small)[::-1]]
    outs = [pps.empty_output(v["px"].numel()) for v in vs]
    refs = [_reference(log2_slots, v, 7) for v in vs]
    first = pps.Batch([(tab, vs[0], outs[0])])
    first.run([_cam(7)], 7)
    second = pps.Batch([(tab, vs[1], outs[1])])
    for i in (0, 1, 0, 1, 1, 0):
        (first, second)[i].run([_cam(7)], 7)
        torch.cuda.synchronize()
        for k in KEYS:
            assert torch.equal(outs[i][k], refs[i][k]), (i, k)
    assert tab.stats()["overflow_vertices"] == 0
    first.close()
    second.close()
    tab.close()
