"""One crowded view in a batch of many nearly empty ones: the automatic cells follow the crowded view only
as far as the batch's one cell table and the device memory allow."""
import numpy as np
import pytest

from paper_1311_5334_gb300 import synth

pytestmark = pytest.mark.gpu


def mixed(n_small, place):
    big = synth.make_view([12, n_small], n_fog=10000, n_through=100)
    p = synth.params(big.extent)
    small = np.array([[100, 100, 100], [20000, 9000, 300]], dtype=np.int32)
    views = [small] * n_small
    views.insert(place, big.xyz)
    offs = np.concatenate([[0], np.cumsum([len(v) for v in views])])
    return big, p, np.concatenate(views), offs


def check(oracle_mod, et, ctx, big, p, xyz, offs, place):
    with oracle_mod.Oracle(big.xyz, p["extent"], p["seed_min"], p["seed_max"], p["tube_r"], p["min_hits"]) as o:
        want = o.find_tracks().as_tuples()
    with et.Batch(ctx, p) as b:
        b.load(xyz, offs)
        b.find()
        tracks, members, voff = b.fetch()
    assert len(want) > 20 and et.track_tuples(tracks, members) == want
    assert (tracks["view"] == place).all()
    assert (voff[:place + 1] == 0).all() and (voff[place + 1:] == len(want)).all()


@pytest.mark.parametrize("n_small,place", [(300, 7), (60000, 30000)])
def test_crowded_view_among_small_ones(oracle_mod, n_small, place):
    from paper_1311_5334_gb300 import et

    big, p, xyz, offs = mixed(n_small, place)
    with et.Context(0) as ctx:
        check(oracle_mod, et, ctx, big, p, xyz, offs, place)


def test_small_cell_table_where_memory_is_short(oracle_mod):
    """An allocator that refuses single requests above 256 MB: the dense view's cells would take 1.9 GB for
    this batch, the mean density's a few."""
    torch = pytest.importorskip("torch")
    from paper_1311_5334_gb300 import et

    big, p, xyz, offs = mixed(2000, 2000)
    refused = []

    def alloc(nbytes, _):
        if nbytes > 256 << 20:
            refused.append(nbytes)
            return None
        return torch.cuda.caching_allocator_alloc(int(nbytes), 0)

    hooks = (et.ALLOC_FN(alloc), et.FREE_FN(lambda ptr, _: torch.cuda.caching_allocator_delete(ptr)))
    with et.Context(0) as ctx:
        et._check(et.lib().et_ctx_set_allocator(ctx._h, hooks[0], hooks[1], None))
        check(oracle_mod, et, ctx, big, p, xyz, offs, 2000)
    assert len(refused) == 1
