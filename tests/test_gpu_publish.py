"""Results written to page-locked memory by the run's last kernel, or copied by
the fetch, at the sizes where the way changes (1,024 views, 1,024 tracks, 16,384
members), and the memory's next owner after a batch that was never fetched."""
import numpy as np
import pytest

from paper_1311_5334_gb300 import synth

pytestmark = pytest.mark.gpu

EXT = (40000, 3000, 3000)


def line(n):
    return np.stack([100 + 700 * np.arange(n), np.full(n, 1500), np.full(n, 1500)], 1).astype(np.int32)


@pytest.mark.parametrize("views,grains", [(1024, 9), (1025, 9), (1024, 16), (1023, 17)])
def test_limits_of_published_results(oracle_mod, views, grains):
    """One line of `grains` grains in every view: one track of all of them."""
    from paper_1311_5334_gb300 import et

    p = synth.params(EXT)
    xyz = line(grains)
    with oracle_mod.Oracle(xyz, EXT, p["seed_min"], p["seed_max"], p["tube_r"], p["min_hits"]) as o:
        want = o.find_tracks().as_tuples()
    assert len(want) == 1 and want[0][2] == grains
    with et.Context(0) as ctx, et.Batch(ctx, p) as b:
        b.load(np.tile(xyz, (views, 1)), np.arange(views + 1) * grains)
        b.find()
        tracks, members, voff = b.fetch()
    assert list(voff) == list(range(views + 1))
    for k in range(views):
        assert et.track_tuples(tracks[k:k + 1], members) == want


def test_batch_dropped_in_flight(oracle_mod):
    pytest.importorskip("torch")
    from paper_1311_5334_gb300 import et

    big = synth.make_view([6, 1], n_fog=20000, n_through=200)
    p = synth.params(big.extent)
    small = synth.make_view([6, 2], n_fog=300, n_through=5)
    with oracle_mod.Oracle(small.xyz, small.extent, p["seed_min"], p["seed_max"], p["tube_r"], p["min_hits"]) as o:
        want = o.find_tracks().as_tuples()
    with et.Context(0, use_torch_allocator=True) as ctx:
        for _ in range(5):
            b = et.Batch(ctx, p)
            b.load(big.xyz, [0, len(big.xyz)])
            b.find()
            b.load(small.xyz, [0, len(small.xyz)])   # the run above is dropped
            b.close()
            b = et.Batch(ctx, p)
            b.load(small.xyz, [0, len(small.xyz)])
            b.find()
            tracks, members, _ = b.fetch()
            b.close()
            assert et.track_tuples(tracks, members) == want
