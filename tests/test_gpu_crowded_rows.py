"""Raster order where image rows hold many grains: up to 768 (96 in runs of more than 2^19 grains) are ranked
along their chain, rows with more by buckets, in one handle's runs in any order, with few grains (published)
and many (copied)."""
import numpy as np
import pytest

from paper_1311_5334_gb300 import synth

pytestmark = pytest.mark.gpu


def spikes(width, rows, depth=3, height=24, seed=0):
    """Isolated dark pixels of distinct depth: rows[k] of them in every other row, in random columns."""
    rng = np.random.default_rng([seed, width])
    raw = np.full((depth, height, width), 220, np.uint8)
    for z in range(0, depth, 2):
        for y in range(0, height, 2):
            n = rows[(y // 2) % len(rows)]
            x = 2 * rng.choice(width // 2, n, replace=False)
            raw[z, y, x] = rng.integers(5, 120, n)
    gain = np.full((height, width), 128, np.uint8)
    return synth.Frames(raw=raw, gain=gain, thr=np.full((height, width), 20, np.uint8), width=width)


def want_of(oracle_mod, f):
    g = oracle_mod.frames_filter(f.raw, f.gain, f.thr)
    return oracle_mod.frames_grains(g, synth.GRAIN_THRESHOLD, synth.PITCH_NUM, synth.PITCH_DEN)[:2]


@pytest.mark.parametrize("width,kinds", [
    (1600, [(768,), (769,), (96,), (3, 768, 769, 800)]),
    (4096, [(2048, 0, 1), (1,), (768, 2048), (2048,)]),
])
def test_rows_equal_the_oracle(oracle_mod, width, kinds):
    from paper_1311_5334_gb300 import et

    views = [spikes(width, rows, seed=k) for k, rows in enumerate(kinds)]
    want = [want_of(oracle_mod, f) for f in views]
    d, h, _ = views[0].raw.shape
    fp = et.make_frame_params(width, h, d, synth.PITCH_NUM, synth.PITCH_DEN, synth.GRAIN_THRESHOLD, row_pitch=width)
    with et.Context(0) as ctx, et.Frames(ctx, fp, views[0].gain, views[0].thr) as fr:
        for k in [0, 1, 2, 3, 1, 0, 3, 2]:
            fr.run(views[k].raw)
            for _ in range(2):
                xyz, pulse, voff = fr.fetch()
                assert np.array_equal(xyz, want[k][0]) and np.array_equal(pulse, want[k][1])
                assert list(voff) == [0, len(want[k][0])]
            crowded = max(kinds[k]) > 768
            assert fr.stats()["kernel_launches"] == (7 if crowded else 4)
        fr.run(np.concatenate([f.raw.reshape(-1) for f in views]))
        xyz, pulse, voff = fr.fetch()
    assert np.array_equal(xyz, np.concatenate([w[0] for w in want]))
    assert np.array_equal(pulse, np.concatenate([w[1] for w in want]))
    assert list(voff) == [0, *np.cumsum([len(w[0]) for w in want])]


@pytest.mark.parametrize("per_row", [256, 257])
def test_many_grains(oracle_mod, per_row):
    """2,048 rows: 2^19 grains or a few more, above the first guess of the grain buffers."""
    from paper_1311_5334_gb300 import et

    f = spikes(1536, (per_row,), height=2048)
    wx, wp = want_of(oracle_mod, f)
    d, h, w = f.raw.shape
    fp = et.make_frame_params(w, h, d, synth.PITCH_NUM, synth.PITCH_DEN, synth.GRAIN_THRESHOLD, row_pitch=w)
    with et.Context(0) as ctx, et.Frames(ctx, fp, f.gain, f.thr) as fr:
        for _ in range(2):
            fr.run(f.raw)
            xyz, pulse, _ = fr.fetch()
            assert len(wx) == 2048 * per_row and fr.stats()["kernel_launches"] == (7 if per_row > 256 else 4)
            assert np.array_equal(xyz, wx) and np.array_equal(pulse, wp)
