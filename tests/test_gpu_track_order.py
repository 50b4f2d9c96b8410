"""Members of a track in ascending order and tracks in acceptance order, at the
sizes where the way they are sorted changes: members by rank inside a warp (up
to 512 of a track) or from a bitmap (more), tracks in one block (up to 4,096
possible) or by the general sort."""
import numpy as np
import pytest

from paper_1311_5334_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(8, 31, 32, 33), (511, 512, 513), (64, 1500)])
def test_members_of_long_lines_ascend(oracle_mod, sizes):
    from paper_1311_5334_gb300 import et

    ext = (320000, 30000, 5000)   # lines along x, far apart in y
    lines = [np.stack([200 + 200 * np.arange(k), np.full(k, 3000 + 5000 * i), np.full(k, 2500)], 1)
             for i, k in enumerate(sizes)]
    xyz = np.concatenate(lines).astype(np.int32)
    xyz = np.ascontiguousarray(xyz[np.random.default_rng(len(xyz)).permutation(len(xyz))])
    p = synth.params(ext)
    with oracle_mod.Oracle(xyz, ext, p["seed_min"], p["seed_max"], p["tube_r"], p["min_hits"]) as o:
        want = o.find_tracks().as_tuples()
    assert sorted(t[2] for t in want) == sorted(sizes)
    with et.Context(0) as ctx:
        view = ctx.view(xyz, p)
        view.find()
        assert et.track_tuples(*view.fetch()) == want
        view.close()


@pytest.mark.parametrize("views,fog", [(1, 300), (3, 0), (5, 2000), (9, 4000)])
def test_tracks_of_batches_in_order(oracle_mod, views, fog):
    """views x fog crosses 4,096 x min_hits grains; one view of a batch is empty."""
    from paper_1311_5334_gb300 import et

    vs = [synth.make_view([5, k], n_fog=fog + 37 * k, n_through=max(2, fog // 60)) for k in range(views)]
    p = synth.params(vs[0].extent)
    xyz = [v.xyz for v in vs]
    if views > 1:
        xyz[1] = xyz[1][:0]
    offs = np.concatenate([[0], np.cumsum([len(x) for x in xyz])])
    with et.Context(0) as ctx:
        b = et.Batch(ctx, p)
        b.load(np.concatenate(xyz), offs)
        b.find()
        tracks, members, voff = b.fetch()
        b.close()
    for k, x in enumerate(xyz):
        got = et.track_tuples(tracks[voff[k]:voff[k + 1]], members)
        if len(x) == 0:
            assert got == []
            continue
        with oracle_mod.Oracle(x, vs[0].extent, p["seed_min"], p["seed_max"], p["tube_r"], p["min_hits"]) as o:
            assert got == o.find_tracks().as_tuples()
