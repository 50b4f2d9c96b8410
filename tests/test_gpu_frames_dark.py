"""Stacks of which most voxels pass the threshold: those no brighter in the frame before are ruled out before
the test, over all depths (pieces of 8 frames and whole stacks), at saturation, where unequal raw values have
equal pulses, and in tiles crowded all the same.  The number of candidates counts all that pass."""
import numpy as np
import pytest

from paper_1311_5334_gb300 import synth

pytestmark = pytest.mark.gpu

SHAPES = [(1, 40, 64), (9, 33, 300), (17, 200, 16), (40, 70, 270)]


def stack(kind, shape, rng):
    d, h, w = shape
    z = np.arange(d)[:, None, None]
    if kind == "dark":
        raw = np.zeros(shape)
    elif kind == "darker":
        raw = np.broadcast_to(120 - 3 * z, shape)
    elif kind == "brighter":
        raw = np.broadcast_to(3 * z, shape)
    elif kind == "waves":
        raw = 60 + 50 * np.sin(z / 2.5) + rng.integers(0, 3, (1, h, w))
    else:
        raw = rng.integers(0, 256, shape)
    return np.clip(raw, 0, 255).astype(np.uint8)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind", ["dark", "darker", "brighter", "waves", "noise"])
@pytest.mark.parametrize("gains", ["flat", "saturated", "mixed"])
def test_dark_stacks_equal_the_oracle(oracle_mod, shape, kind, gains):
    from paper_1311_5334_gb300 import et

    d, h, w = shape
    rng = np.random.default_rng([d, w, len(kind)])
    pitch = (w + 15) // 16 * 16
    raw = np.full((d, h, pitch), 255, np.uint8)
    raw[:, :, :w] = stack(kind, shape, rng)
    gain, thr = {"flat": (np.full((h, w), 128), np.full((h, w), 20)),
                 "saturated": (np.full((h, w), 255), np.full((h, w), 3)),
                 "mixed": (rng.integers(0, 256, (h, w)), rng.integers(0, 90, (h, w)))}[gains]
    f = synth.Frames(raw=raw, gain=gain.astype(np.uint8), thr=thr.astype(np.uint8), width=w)
    filtered = oracle_mod.frames_filter(f.raw, f.gain, f.thr)
    wx, wp, _ = oracle_mod.frames_grains(filtered, 25, synth.PITCH_NUM, synth.PITCH_DEN)
    fp = et.make_frame_params(w, h, d, synth.PITCH_NUM, synth.PITCH_DEN, 25, row_pitch=pitch)
    with et.Context(0) as ctx, et.Frames(ctx, fp, f.gain, f.thr) as fr:
        fr.run(np.concatenate([raw.reshape(-1)] * 2))
        xyz, pulse, voff = fr.fetch()
        st = fr.stats()
    assert np.array_equal(xyz, np.concatenate([wx, wx])) and np.array_equal(pulse, np.concatenate([wp, wp]))
    assert list(voff) == [0, len(wx), 2 * len(wx)]
    assert st["n_candidates"] == 2 * int((filtered > 25).sum())
