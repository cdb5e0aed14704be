"""The order of a cell's additions on tables with a half-precision history,
where it is a visible difference: one cell holds A = 3 (1 + 2^-11) and twice
t = 0.75 * 2^-23, at opposite ends of a stream of many tiles.  In FP32 A + t is A
(t is below half an ulp, 2^-23), and t + t before A makes A + 2^-22.  The averages
are 1 + 2^-11, half-way between two halves and rounded to the even one, 1, and
1 + 2^-11 + 2^-23, which becomes 1 + 2^-10.  Plain and temporal frames on tables
of up to 2^23 slots add from the end of the stream, all others from its start."""
import pytest
import torch

from paper_1902_05942_gb300 import pps, scene
from paper_1902_05942_gb300.configs import FilterConfig

pytestmark = pytest.mark.gpu

N = 2_600_001  # 1,270 tiles, far more than there are CTAs


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1902_05942_gb300 import build
    build.build()
    torch.cuda.set_device(0)
    yield


def _stream(backwards, variants):
    g = torch.Generator(device="cuda").manual_seed(3)
    p = torch.rand((3, N), generator=g, device="cuda") * 40 - 20
    nz = torch.ones(N, device="cuda")
    c = torch.rand((3, N), generator=g, device="cuda")
    small, large = ((N - 1, N - 5000), 0) if backwards else ((0, 5000), N - 1)
    for j in (*small, large):
        p[:, j] = torch.tensor([500.0, 1.0, 1.0])
        c[:, j] = 0.75 * 2.0 ** -23 if j != large else 3 * (1 + 2.0 ** -11)
    v = dict(zip(scene.STREAMS, [*p, 0 * nz, 0 * nz, nz, *c]))
    v = {k: t.contiguous() for k, t in v.items()}
    if variants:
        v["extra"] = torch.zeros(N, dtype=torch.int32, device="cuda")
    return v, (*small, large)


@pytest.mark.parametrize("log2_slots,kind,backwards", [
    (21, "plain", True), (23, "plain", True), (24, "plain", False), (21, "variants", False),
    (21, "neighbors", False), (21, "evict", False), (21, "migrate", False), (21, "split", False),
    (21, "batch", False)])
def test_sums_of_a_half_precision_history_keep_their_order(log2_slots, kind, backwards):
    v, mine = _stream(backwards, kind == "variants")
    cfg = FilterConfig(log2_slots=log2_slots, max_probes=64, voxel_scale=4.0, pixel_angle=0.01,
                       jitter=False, hist_mode=2, log2_hist_slots=23, hist_evict=kind == "evict",
                       hist_migrate=kind == "migrate",
                       fallback="neighbors" if kind == "neighbors" else "none")
    tab = pps.Table(cfg)
    eye = (0.0, 0.0, 0.0)
    out = pps.empty_output(N)
    if kind == "batch":
        b = pps.Batch([(tab, v, out)], blend=True, alpha=0.2)
        b.run([eye], 0)
        torch.cuda.synchronize()
        b.close()
    elif kind == "split":
        ids = torch.empty(N, dtype=torch.int32, device="cuda")
        tab.build(eye, 0)
        tab.insert(v, ids)
        tab.blend(0.2)
        tab.query(v, ids, out)
    else:
        tab.filter(v, eye, 0, blend=True, alpha=0.2, out=out)
    st = tab.stats()
    assert st["overflow_vertices"] == 0 and st["device_error"] == 0
    for j in mine:
        assert int(out["count"][j]) == 3
        assert [float(out[c][j]) for c in "rgb"] == [1 + 2.0 ** -10] * 3
    tab.close()
