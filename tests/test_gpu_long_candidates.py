"""Candidates of more than 32 grains, read 128 at a time by the association: at the edges of the steps, on
lines that share grains, so that candidates wait for one another, and in windows of a few candidates."""
import numpy as np
import pytest

from paper_1311_5334_gb300 import synth

pytestmark = pytest.mark.gpu

EXT = (60000, 60000, 2000)
GAP = 200


def grid(lengths, seed):
    """Lines along x of the given numbers of grains, and as many along y that share grains with them."""
    rng = np.random.default_rng(seed)
    pts = set()
    for k, n in enumerate(lengths):
        y = 400 + GAP * 5 * k
        for j in range(n):
            pts.add((400 + GAP * j, y, 1000))
            pts.add((y, 400 + GAP * j, 1000))
    a = np.array(sorted(pts), dtype=np.int32)
    return np.ascontiguousarray(a[rng.permutation(len(a))])


@pytest.mark.parametrize("lengths", [(32, 33), (127, 128, 129), (255, 256, 257), (64, 96, 200), (40,) * 12])
@pytest.mark.parametrize("window", [0, 7])
def test_shared_lines_equal_the_oracle(oracle_mod, lengths, window):
    from paper_1311_5334_gb300 import et

    p = synth.params(EXT, seed_min=GAP, seed_max=2 * GAP + 1, min_hits=9)
    xyz = grid(lengths, len(lengths))
    with oracle_mod.Oracle(xyz, EXT, p["seed_min"], p["seed_max"], p["tube_r"], p["min_hits"]) as o:
        want = o.find_tracks().as_tuples()
    assert len(want) >= 2 * len(lengths) - 2 and max(t[2] for t in want) >= max(lengths)
    with et.Context(0) as ctx, et.Batch(ctx, p) as b:
        b.set_tuning(assoc_window=window)
        b.load(xyz, [0, len(xyz)])
        b.find()
        tracks, members, _ = b.fetch()
    assert et.track_tuples(tracks, members) == want
