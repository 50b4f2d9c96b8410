"""Members of a track in ascending order where they are sorted by a network in a warp (65 to 512) or from a
bitmap (more), by one block for one track or several tracks a block, in views whose caller indices need one
or two bitmaps."""
import numpy as np
import pytest

from paper_1311_5334_gb300 import synth

pytestmark = pytest.mark.gpu

GAP = 200


def line(n, y, z=1000):
    return np.stack([100 + GAP * np.arange(n), np.full(n, y), np.full(n, z)], 1)


def shuffled(parts, seed):
    """The grains in random order, and the new indices of each part's, ascending."""
    order = np.random.default_rng(seed).permutation(sum(len(a) for a in parts))
    xyz = np.ascontiguousarray(np.concatenate(parts).astype(np.int32)[order])
    where = np.empty(len(order), dtype=np.int64)
    where[order] = np.arange(len(order))
    out, o = [], 0
    for a in parts:
        out.append(tuple(sorted(int(i) for i in where[o:o + len(a)])))
        o += len(a)
    return xyz, out


def found(et, xyz, offs, ext):
    p = synth.params(ext, seed_min=GAP, seed_max=2 * GAP + 1)
    with et.Context(0) as ctx, et.Batch(ctx, p) as b:
        b.load(xyz, offs)
        b.find()
        tracks, members, voff = b.fetch()
    return et.track_tuples(tracks, members), voff


@pytest.mark.parametrize("sizes", [(63, 64, 65, 66), (127, 128, 129), (255, 256, 257), (511, 512, 513, 1023)])
def test_sizes_of_the_network(sizes):
    from paper_1311_5334_gb300 import et

    xyz, want = shuffled([line(n, 500 + 1500 * k) for k, n in enumerate(sizes)], sum(sizes))
    got, _ = found(et, xyz, [0, len(xyz)], (210000, 8000, 2000))
    assert sorted((t[2], t[3]) for t in got) == sorted((n, w) for n, w in zip(sizes, want))


@pytest.mark.parametrize("views,n", [(1, 513), (40, 520), (200, 600)])
def test_long_tracks_of_many_views(views, n):
    from paper_1311_5334_gb300 import et

    parts = [shuffled([line(n, 500), line(30, 1500)], k) for k in range(views)]
    got, voff = found(et, np.concatenate([p[0] for p in parts]), np.arange(views + 1) * (n + 30), (130000, 2000, 2000))
    assert list(voff) == [2 * k for k in range(views + 1)]
    for k, (_, want) in enumerate(parts):
        assert [t[3] for t in got[2 * k:2 * k + 2]] == want


@pytest.mark.parametrize("side", [10, 102])
def test_indices_of_large_views(side):
    """A lattice of grains too far apart to pair (1,000, or 1,061,208: two bitmaps) around two long lines."""
    from paper_1311_5334_gb300 import et

    a = 5000 + 10000 * np.arange(side)
    fog = np.stack(np.meshgrid(a, a, a, indexing="ij"), -1).reshape(-1, 3)
    e = 10000 * side + 121000
    xyz, want = shuffled([line(600, 500), line(700, 3000, 2000), fog], side)
    got, _ = found(et, xyz, [0, len(xyz)], (e, e, e))
    assert sorted(t[3] for t in got) == sorted(want[:2])
