"""Grains and view offsets of the image front end written to page-locked memory by the run's last kernel, or
copied by the fetch, at the sizes where the way changes (16,384 grains, 1,024 views)."""
import numpy as np
import pytest

from paper_1311_5334_gb300 import synth

pytestmark = pytest.mark.gpu


def spikes(width, height, n):
    """One frame with n isolated dark pixels, in raster order."""
    raw = np.full((1, height, width), 220, np.uint8)
    slots = np.stack(np.meshgrid(np.arange(0, height, 2), np.arange(0, width, 2), indexing="ij"), -1).reshape(-1, 2)[:n]
    assert len(slots) == n
    raw[0, slots[:, 0], slots[:, 1]] = 5 + np.arange(n) % 100
    gain = np.full((height, width), 128, np.uint8)
    return synth.Frames(raw=raw, gain=gain, thr=np.full((height, width), 20, np.uint8), width=width)


def want_of(oracle_mod, f):
    g = oracle_mod.frames_filter(f.raw, f.gain, f.thr)
    return oracle_mod.frames_grains(g, synth.GRAIN_THRESHOLD, synth.PITCH_NUM, synth.PITCH_DEN)[:2]


@pytest.mark.parametrize("width,height,views,n", [(512, 256, 1, 16383), (512, 256, 1, 16384), (512, 260, 1, 16385),
                                                  (512, 64, 2, 8192), (16, 8, 1023, 5), (16, 8, 1024, 16),
                                                  (16, 8, 1025, 5), (16, 8, 1024, 17)])
def test_limits_of_published_grains(oracle_mod, width, height, views, n):
    from paper_1311_5334_gb300 import et

    f = spikes(width, height, n)
    wx, wp = want_of(oracle_mod, f)
    assert len(wx) == n
    fp = et.make_frame_params(width, height, 1, synth.PITCH_NUM, synth.PITCH_DEN, synth.GRAIN_THRESHOLD, row_pitch=width)
    with et.Context(0) as ctx, et.Frames(ctx, fp, f.gain, f.thr) as fr:
        fr.run(np.tile(f.raw.reshape(-1), views))
        xyz, pulse, voff = fr.fetch()
    assert np.array_equal(xyz, np.tile(wx, (views, 1))) and np.array_equal(pulse, np.tile(wp, views))
    assert np.array_equal(voff, np.arange(views + 1) * n)
