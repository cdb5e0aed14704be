"""Launches that overlap or are chosen by size: batches whose views are filtered
partly by launches of their own (2^20 vertices and more) and partly by the shared
one, against one call per view; and the learned fallback's evaluation, which
starts beside the end of the listing, called, repeated and replayed from a
captured graph.  Fixed point and the same network, so results are compared
exactly."""
import numpy as np
import pytest
import torch

from mlp_cases import random_weights
from paper_1902_05942_gb300 import pps, scene
from paper_1902_05942_gb300.configs import FilterConfig

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1902_05942_gb300 import build
    build.build()
    torch.cuda.set_device(0)
    yield


def _vertices(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    p = torch.rand((3, n), generator=g, device="cuda") * 40 - 20
    q = torch.nn.functional.normalize(torch.randn((3, n), generator=g, device="cuda"), dim=0)
    c = torch.rand((3, n), generator=g, device="cuda")
    return {k: t.contiguous() for k, t in zip(scene.STREAMS, [*p, *q, *c])}


@pytest.mark.parametrize("sizes", [(1 << 20,), ((1 << 20) - 1, 1 << 20), (5, (1 << 20) + 77, 1, 4097),
                                   (1 << 20, 1 << 20, 300)])
@pytest.mark.parametrize("hist", [0, 1])
def test_batch_of_own_and_shared_launches(sizes, hist):
    def cfg(n):
        # the large views sweep their table, the small ones empty slots
        return FilterConfig(log2_slots=21 if n > 5000 else 16, max_probes=64, voxel_scale=4.0,
                            pixel_angle=0.01, accum_fixed=True, hist_mode=hist, log2_hist_slots=22)
    cams = [(0.5 * i, 3.0, -12.0) for i in range(len(sizes))]
    vs = [_vertices(n, 7 + i) for i, n in enumerate(sizes)]
    one = [pps.Table(cfg(n)) for n in sizes]
    many = [pps.Table(cfg(n)) for n in sizes]
    outs = [pps.empty_output(n) for n in sizes]
    batch = pps.Batch([(many[i], vs[i], outs[i]) for i in range(len(sizes))], blend=bool(hist), alpha=0.2)
    for f in range(3):
        batch.run(cams, f)
        for i, n in enumerate(sizes):
            ref = one[i].filter(vs[i], cams[i], f, blend=bool(hist), alpha=0.2)
            for k in ("r", "g", "b", "count", "status"):
                assert torch.equal(outs[i][k], ref[k]), (f, i, k)
            a, b = one[i].stats(), many[i].stats()
            assert a["device_error"] == b["device_error"] == 0 and b["vertices"] == n
            for k in ("frame_cells", "overflow_vertices", "hist_overflow"):
                assert a[k] == b[k]
    batch.close()
    for t in one + many:
        t.close()


@pytest.mark.parametrize("n", [1, 127, 1025, 40_000, 300_001])
def test_fallback_inference_repeated_and_captured(n):
    v = _vertices(n, 3)
    g = torch.Generator(device="cuda").manual_seed(11)
    net = pps.MLP(pps.mlp_params(), init=random_weights(5))
    base = pps.empty_output(n)
    for k in "rgb":
        base[k].copy_(torch.rand(n, generator=g, device="cuda"))
    base["count"].copy_(torch.randint(1, 9, (n,), generator=g, device="cuda", dtype=torch.int32))
    base["status"].copy_(torch.randint(0, 3, (n,), generator=g, device="cuda").to(torch.uint8))
    ref = net.forward(v)
    low = (base["count"] < 4) & (base["status"] != 2)

    def check(o):
        torch.cuda.synchronize()
        for k in "rgb":
            assert torch.equal(o[k], torch.where(low, ref[k], base[k]))
        assert torch.equal(o["status"], torch.where(low, torch.full_like(o["status"], 3), base["status"]))

    out = {k: t.clone() for k, t in base.items()}
    net.infer(v, out)
    check(out)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        net.infer(v, out)
    for _ in range(3):
        for k, t in base.items():
            out[k].copy_(t)
        graph.replay()
        check(out)
    # one after the other with nothing between: the second finds the same list
    for k, t in base.items():
        out[k].copy_(t)
    for _ in range(5):
        net.infer(v, out)
    check(out)
    net.close()
