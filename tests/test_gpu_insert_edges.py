"""The insert at the edges of its tiles, rows and queue, against the oracle:
vertex counts around the widths of a row (32), a step (64) and a tile (64 to
256); tables that are swept whole and tables emptied slot by slot, in turn on
one table and followed by the split calls; probe limits of one and two on a
crowded table.  Fixed point, so every count and value is compared exactly."""
import numpy as np
import pytest
import torch

from oracle import pps_oracle as O
from paper_1902_05942_gb300 import pps
from test_gpu_parity import _audit_overflow, _check_frame, _dev, _gen, _np, _oracle, _rgb, _small

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stream():
    from paper_1902_05942_gb300 import build
    build.build()
    torch.cuda.set_device(0)
    spec, _ = _small(width=96, height=96, bounces=3)
    return spec, _gen(spec)


@pytest.mark.parametrize("batch,merge", [(2, 2), (4, 2), (2, 1), (2, 3)])
def test_counts_around_rows_steps_and_tiles(stream, batch, merge):
    spec, v = stream
    _, cfg = _small(width=96, height=96, accum_fixed=True, log2_slots=14, max_probes=64)
    tab = pps.Table(cfg)
    tab.tune(batch, merge=merge)
    # 2,048 vertices and more sweep this table, fewer empty their slots
    for i, n in enumerate((1, 31, 32, 33, 63, 65, 127, 129, 255, 2047, 257, 2048, 300, 6001, 1, 64)):
        d = _dev(v, n)
        out = tab.filter(d, spec.view.eye, i)
        fr = _oracle(cfg, spec.view.eye, i, _np(v, n))
        _check_frame(out, fr, fixed=True)
        st = tab.stats()
        assert st["occupied_slots"] == 0 and st["frame_cells"] == fr.tuples.shape[0]
    # the split calls after a swept frame and after one emptied slot by slot
    for i, n in ((40, 6001), (41, 129)):
        tab.filter(_dev(v, n), spec.view.eye, i)
        d = _dev(v, 777)
        tab.build(spec.view.eye, i)
        slots = torch.empty(777, dtype=torch.int32, device="cuda")
        tab.insert(d, slots)
        fr = _oracle(cfg, spec.view.eye, i, _np(v, 777))
        _check_frame(tab.query(d, slots), fr, fixed=True)
        _check_frame(tab.query(d), fr, fixed=True)
        fp, _ = tab.dump()
        assert np.count_nonzero(fp) == fr.tuples.shape[0] == tab.stats()["occupied_slots"]
    tab.close()


@pytest.mark.parametrize("max_probes", [1, 2, 7])
def test_crowded_table(stream, max_probes):
    """Many more keys than the probe limit lets in: overflow is all or none per
    key, the other vertices are exact, and nothing is left behind."""
    spec, v = stream
    _, cfg = _small(width=96, height=96, accum_fixed=True, log2_slots=12, max_probes=max_probes)
    n = 9000
    tab = pps.Table(cfg)
    for f in range(2):
        d = _dev(v, n)
        out = tab.filter(d, spec.view.eye, f)
        vn = _np(v, n)
        ovf = _audit_overflow(out, vn, _oracle(cfg, spec.view.eye, f, vn))
        assert ovf.any()
        keep = np.nonzero(~ovf)[0]
        fr = _oracle(cfg, spec.view.eye, f, {k: a[keep] for k, a in vn.items()},
                     ids=keep.astype(np.uint32))
        assert np.array_equal(out["count"].cpu().numpy().astype(np.int64)[keep], fr.count)
        assert np.array_equal(_rgb(out)[keep], fr.mean_fixed)
        st = tab.stats()
        assert st["overflow_vertices"] == ovf.sum() and st["frame_cells"] == fr.tuples.shape[0]
    tab.close()


@pytest.mark.parametrize("hist_mode", [1, 2])
def test_blend_with_a_crowded_history(stream, hist_mode):
    """A history that fills up, with windows many entries long, some claimed in
    this frame: every cell finds its own entry again.  The oracle blends the
    fixed-point averages in FP64: FP32 blends stay within 8 u per frame of it;
    a half-precision store may round such a value to the neighbouring half, one
    step (2^-10 relatively, 2^-24 among subnormals) per frame."""
    spec, v = stream
    n = 2500
    _, cfg = _small(width=96, height=96, accum_fixed=True, log2_slots=13, max_probes=256,
                    hist_mode=hist_mode, log2_hist_slots=12)
    tab = pps.Table(cfg)
    hist = O.History.empty()
    vn = _np(v, n)
    for f in range(2):
        out = tab.filter(_dev(v, n), spec.view.eye, f, blend=True, alpha=-1.0)
        fr = _oracle(cfg, spec.view.eye, f, vn)
        c_new = np.zeros((fr.tuples.shape[0], 3))
        c_new[fr.cell] = fr.mean_fixed
        hist, val, cnt = O.blend(hist, fr, -1.0, fp16=hist_mode == 2, c_new=c_new)
        assert np.array_equal(out["count"].cpu().numpy().astype(np.int64), cnt)
        err = np.abs(_rgb(out).astype(np.float64) - val)
        if hist_mode == 1:
            assert np.all(err <= 8 * 2.0 ** -24 * (f + 1) * np.abs(val))
        else:
            assert np.all(err <= (f + 1) * (2.0 ** -10 * np.abs(val) + 2.0 ** -24))
        # every distinct key has its entry, or found its window full (which, in
        # the table's last free entries, only keys new in this frame do: they
        # take this frame's average, as without history)
        st = tab.stats()
        assert st["hist_occupied"] + st["hist_overflow"] == hist.tuples.shape[0]
    tab.close()
