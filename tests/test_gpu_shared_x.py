"""Canonical order of grains that share their x: ranked among themselves up to
a limit (64 others), by the full sort beyond it, alone and in a batch, with
duplicates reported either way; and scans of the cell counts around the sizes
where one block does them."""
import numpy as np
import pytest

from paper_1311_5334_gb300 import synth

pytestmark = pytest.mark.gpu


def planes(seed, group, extent, n_planes=12):
    """Grains on a few planes of constant x, `group` on each, in random order,
    with a track of twelve grains in one of the planes."""
    rng = np.random.default_rng([seed, group])
    xs = rng.choice(extent[0], n_planes, replace=False)
    out = []
    for x in xs:
        yz = set()
        while len(yz) < group:
            yz.add((int(rng.integers(0, extent[1])), int(rng.integers(0, extent[2]))))
        out += [(int(x), y, z) for y, z in yz]
    y0 = int(rng.integers(0, extent[1] - 5000))
    keep = [g for g in out if g[0] != xs[0]] + [g for g in out if g[0] == xs[0]][:max(0, group - 12)]
    line = {(int(xs[0]), y0 + 400 * k, 2500) for k in range(12)}
    a = np.array(sorted(set(keep) | line), dtype=np.int32)
    return np.ascontiguousarray(a[rng.permutation(len(a))])


def want_of(oracle_mod, xyz, p):
    with oracle_mod.Oracle(xyz, p["extent"], p["seed_min"], p["seed_max"], p["tube_r"], p["min_hits"]) as o:
        return o.find_tracks().as_tuples()


@pytest.mark.parametrize("group", [13, 64, 65, 66, 300])
def test_grains_on_planes_equal_the_oracle(oracle_mod, group):
    from paper_1311_5334_gb300 import et

    p = synth.params((30000, 30000, 5000))
    views = [planes(k, g, p["extent"]) for k, g in enumerate((group, 13, group))]
    offs = np.concatenate([[0], np.cumsum([len(v) for v in views])])
    with et.Context(0) as ctx:
        b = et.Batch(ctx, p)
        for graph in (False, True, True):
            b.load(np.concatenate(views), offs)
            b.find(use_graph=graph)
            tracks, members, voff = b.fetch()
            for k, v in enumerate(views):
                assert et.track_tuples(tracks[voff[k]:voff[k + 1]], members) == want_of(oracle_mod, v, p)
        b.close()
        dup = views[0].copy()
        dup[-1] = dup[0]
        v = ctx.view(dup, p)
        v.find()
        with pytest.raises(et.EtError) as e:
            v.fetch()
        assert e.value.status == et.DUPLICATE_GRAIN
        v.close()


@pytest.mark.parametrize("cells", [(1, 1, 1), (32, 16, 16), (33, 16, 16), (40, 30, 20)])
def test_cell_tables_around_the_one_block_scan(oracle_mod, cells):
    """2 x 8,192 and 2 x 8,448 cells lie on either side of the limit of 16,384."""
    from paper_1311_5334_gb300 import et

    v = synth.make_view(23, n_fog=1500, n_through=15)
    p = synth.params(v.extent)
    with et.Context(0) as ctx:
        b = et.Batch(ctx, p)
        b.set_tuning(cell=[-(-e // c) for e, c in zip(v.extent, cells)])
        b.load(v.xyz, [0, v.n])
        b.find()
        tracks, members, _ = b.fetch()
        assert et.track_tuples(tracks, members) == want_of(oracle_mod, v.xyz, p)
        b.close()
