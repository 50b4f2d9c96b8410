"""Calls that fail on the host leave their handle in a defined state: what was there before is not mixed with
what did not come, and the next good call works."""
import numpy as np
import pytest

from paper_1311_5334_gb300 import synth

pytestmark = pytest.mark.gpu

EXT = (3000, 3000, 3000)


def want_of(oracle_mod, xyz, p):
    with oracle_mod.Oracle(xyz, p["extent"], p["seed_min"], p["seed_max"], p["tube_r"], p["min_hits"]) as o:
        return o.find_tracks().as_tuples()


def line(n):
    return np.stack([100 + 200 * np.arange(n), np.full(n, 1500), np.full(n, 1500)], 1).astype(np.int32)


def test_failed_load_leaves_nothing_to_fetch(oracle_mod):
    """400 views on cells of 16 units (6.6 M cells a view) pass the limit of the cell table."""
    from paper_1311_5334_gb300 import et

    p = synth.params(EXT, seed_min=100, seed_max=900)
    xyz = line(12)
    want = want_of(oracle_mod, xyz, p)
    assert len(want) == 1
    with et.Context(0) as ctx, et.Batch(ctx, p) as b:
        b.set_tuning(cell=(16, 16, 16), row_lists=1)
        for _ in range(2):
            b.load(xyz, [0, 12])
            b.find()
            tracks, members, _ = b.fetch()
            assert et.track_tuples(tracks, members) == want
            with pytest.raises(et.EtError) as e:
                b.load(np.tile(xyz, (400, 1)), np.arange(401) * 12)
            assert e.value.status == et.INVALID_ARG
            for call in (b.fetch, b.sync, b.find):
                with pytest.raises(et.EtError) as e:
                    call()
                assert e.value.status == et.NOT_READY
