"""What pps_get_tuning says: the values in effect, and nothing about an insert of
key and probe warps, which the library does not have."""
import pytest
import torch

from paper_1902_05942_gb300 import pps
from test_gpu_left_slots import _cfg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log2_slots", [16, 24])
def test_fields(log2_slots):
    from paper_1902_05942_gb300 import build
    build.build()
    torch.cuda.set_device(0)
    tab = pps.Table(_cfg(log2_slots))
    assert pps.pps_get_tuning(tab.handle) == dict(batch=2, insert=0, key_warps=0, block=512, merge=2)
    tab.tune(batch=4, insert=2, key_warps=12, block=256, merge=1)
    assert pps.pps_get_tuning(tab.handle) == dict(batch=4, insert=2, key_warps=12, block=256, merge=1)
    tab.close()
