"""Keys of inputs at the ends of FP32's range, with the jitter on: zeros of either
sign, subnormals, values near the largest, infinities and NaN in positions and
normals.  One rounding per operation, like the oracle, bit for bit."""
import numpy as np
import pytest
import torch

from oracle import pps_oracle as O
from paper_1902_05942_gb300 import pps, scene
from paper_1902_05942_gb300.configs import FilterConfig

pytestmark = pytest.mark.gpu

SPECIAL = np.array([0.0, -0.0, 1.0, -1.0, np.nan, np.inf, -np.inf, 1e-45, -1e-45, 2.0 ** -126, -3e-39,
                    3.4e38, -3.4e38, 0.9999999, -0.9999999, 1e-7, 0.9921875], dtype=np.float32)


def _inputs(kind, n):
    rng = np.random.default_rng(11)
    if kind == "special":
        return SPECIAL[rng.integers(0, SPECIAL.size, (6, n))]
    if kind == "bits":
        return rng.integers(0, 1 << 32, (6, n), dtype=np.uint32).view(np.float32)
    a = rng.standard_normal((6, n)) * 10.0 ** rng.integers(-40, 39, (6, n))
    return np.clip(a, -3.4e38, 3.4e38).astype(np.float32)


@pytest.mark.parametrize("kind", ["special", "bits", "wide"])
@pytest.mark.parametrize("lod", [(-24, 24), (-125, 126)])
def test_keys_at_the_ends_of_the_range(kind, lod):
    from paper_1902_05942_gb300 import build
    build.build()
    torch.cuda.set_device(0)
    a = _inputs(kind, 400_000)
    cfg = FilterConfig(log2_slots=12, max_probes=8, voxel_scale=4.0, pixel_angle=0.0013,
                       lod_min=lod[0], lod_max=lod[1])
    kw = cfg.oracle_kwargs()
    kw["log2_slots"] = 32  # the full home hash
    v = {k: torch.from_numpy(np.ascontiguousarray(x)).cuda() for k, x in zip(scene.STREAMS, [*a, *a[:3]])}
    for cam in ((0.0, 0.0, 0.0), (1.5, -2.25, 1e6)):
        tab = pps.Table(cfg)
        tab.build(cam, 9)
        h, f = tab.keys(v)
        with np.errstate(all="ignore"):
            want = O.vertex_keys(O.KeyParams(**kw), cam, 9, *a)
        assert np.array_equal(h.cpu().numpy().view(np.uint32), want.home)
        assert np.array_equal(f.cpu().numpy().view(np.uint32), want.fp)
        tab.close()
