"""A batch that met grains crowded on shared x: the run is repeated with the full sort, later loads take it
from the start, and views that do not crowd get the short sort back."""
import numpy as np
import pytest

from paper_1311_5334_gb300 import synth
from tests.test_gpu_shared_x import planes, want_of

pytestmark = pytest.mark.gpu

EXT = (30000, 30000, 5000)


@pytest.mark.parametrize("group", [65, 66])
def test_streams_with_crowded_views(oracle_mod, group):
    """Captured from the first run on, so that a captured short sort meets the crowd and is run again."""
    from paper_1311_5334_gb300 import et

    p = synth.params(EXT)
    plain = synth.make_view(61, n_fog=700, n_through=10).xyz
    crowd = planes(3, group, EXT)
    want = {id(x): want_of(oracle_mod, x, p) for x in (plain, crowd)}
    with et.Context(0) as ctx, et.Batch(ctx, p) as b:
        for x in [crowd, crowd] + [plain] * 10 + [crowd, plain, crowd, crowd] + [plain] * 9:
            b.load(x, [0, len(x)])
            b.find(use_graph=True)
            tracks, members, _ = b.fetch()
            assert et.track_tuples(tracks, members) == want[id(x)]
            b.find(use_graph=True)
            tracks, members, _ = b.fetch()
            assert et.track_tuples(tracks, members) == want[id(x)]


def test_short_sort_comes_back():
    """The stage that holds the sort takes 51 us for this view, 81 with the full sort."""
    from paper_1311_5334_gb300 import et

    v = synth.dense()
    p = synth.params(v.extent)
    crowd = planes(5, 300, EXT)

    def sort_ms(b, x, n):
        out = []
        for _ in range(n):
            b.load(x, [0, len(x)])
            b.find()
            b.fetch()
            out.append(b.stats()["stage_ms"]["cells"])
        return out

    with et.Context(0) as ctx, et.Batch(ctx, p) as b:
        b.set_profiling()
        before = np.median(sort_ms(b, v.xyz, 20)[5:])
        sort_ms(b, crowd, 3)
        after = np.median(sort_ms(b, v.xyz, 30)[15:])
    assert after < 1.4 * before, (before, after)
