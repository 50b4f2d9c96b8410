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


class Memory:
    """Allocation hooks through PyTorch's allocator that can be told to refuse."""

    def __init__(self, et, ctx):
        import torch

        self.refuse = False

        def alloc(nbytes, _):
            return None if self.refuse else torch.cuda.caching_allocator_alloc(int(nbytes), 0)

        self.hooks = (et.ALLOC_FN(alloc), et.FREE_FN(lambda ptr, _: torch.cuda.caching_allocator_delete(ptr)))
        et._check(et.lib().et_ctx_set_allocator(ctx._h, self.hooks[0], self.hooks[1], None))


@pytest.mark.parametrize("graph", [False, True])
def test_run_after_growing_the_buffers_failed(oracle_mod, graph):
    """More candidates than the first buffers hold, and no memory for larger ones: neither a fetch nor another
    run uses buffers that were given back."""
    pytest.importorskip("torch")
    from paper_1311_5334_gb300 import et

    v = synth.make_view(51, n_fog=6000, n_through=40)
    p = synth.params(v.extent, min_hits=2)
    want = want_of(oracle_mod, v.xyz, p)
    with et.Context(0) as ctx:
        mem = Memory(et, ctx)
        with et.Batch(ctx, p) as b:
            b.load(v.xyz, [0, v.n])
            mem.refuse = True
            b.find(use_graph=graph)
            for call in (b.fetch, b.fetch, lambda: b.find(use_graph=graph), lambda: b.find(use_graph=graph)):
                with pytest.raises(et.EtError) as e:
                    call()
                assert e.value.status == et.OOM
            mem.refuse = False
            b.find(use_graph=graph)
            tracks, members, _ = b.fetch()
            assert b.stats()["n_candidates"] > 65536
    assert et.track_tuples(tracks, members) == want


def test_run_after_a_failed_autotune(oracle_mod):
    """No memory for a trial's cell table: the tuning of before is kept and laid out again."""
    pytest.importorskip("torch")
    from paper_1311_5334_gb300 import et

    v = synth.make_view(52, n_fog=3000, n_through=30)
    p = synth.params(v.extent)
    want = want_of(oracle_mod, v.xyz, p)
    with et.Context(0) as ctx:
        mem = Memory(et, ctx)
        with et.Batch(ctx, p) as b:
            b.set_tuning(cell=(2000, 4000, 4000), row_lists=1)   # a table smaller than any trial's
            b.load(v.xyz, [0, v.n])
            mem.refuse = True
            with pytest.raises(et.EtError) as e:
                b.autotune()
            assert e.value.status == et.OOM
            with pytest.raises(et.EtError) as e:
                b.find()
            assert e.value.status == et.OOM
            mem.refuse = False
            b.find()
            tracks, members, _ = b.fetch()
            assert b.stats()["cell"] == (2000, 4000, 4000)
    assert et.track_tuples(tracks, members) == want


def stack(seed):
    return synth.random_blobs((5, 40, 64), n=30, seed=seed)


def frames_of(et, ctx, f):
    d, h, pitch = f.raw.shape
    fp = et.make_frame_params(f.width, h, d, synth.PITCH_NUM, synth.PITCH_DEN, synth.GRAIN_THRESHOLD, row_pitch=pitch)
    return et.Frames(ctx, fp, f.gain, f.thr)


def frames_want(oracle_mod, f):
    g = oracle_mod.frames_filter(f.raw, f.gain, f.thr)
    return oracle_mod.frames_grains(g, synth.GRAIN_THRESHOLD, synth.PITCH_NUM, synth.PITCH_DEN)


def test_failed_frames_run_leaves_nothing_to_fetch(oracle_mod):
    """No memory for the upload of three stacks after a run of one."""
    pytest.importorskip("torch")
    from paper_1311_5334_gb300 import et

    f = stack(81)
    wx, wp, _ = frames_want(oracle_mod, f)
    with et.Context(0) as ctx:
        mem = Memory(et, ctx)
        with frames_of(et, ctx, f) as fr, et.Batch(ctx, synth.params(synth.FRAME_EXTENT)) as b:
            for _ in range(2):
                fr.run(f.raw, n_views=1)
                xyz, pulse, voff = fr.fetch()
                assert np.array_equal(xyz, wx) and np.array_equal(pulse, wp) and list(voff) == [0, len(wx)]
                mem.refuse = True
                with pytest.raises(et.EtError) as e:
                    fr.run(np.tile(f.raw.reshape(-1), 3), n_views=3)
                assert e.value.status == et.OOM
                for call in (fr.fetch, lambda: fr.to_batch(b)):
                    with pytest.raises(et.EtError) as e:
                        call()
                    assert e.value.status == et.NOT_READY
                mem.refuse = False


def test_frames_run_after_failed_grain_buffers(oracle_mod):
    """Rows of 40 stacks need larger buffers than those of one, and there is no memory: the next runs, larger or
    smaller, use no buffers that were given back."""
    torch = pytest.importorskip("torch")
    from paper_1311_5334_gb300 import et

    f = stack(82)
    wx, wp, _ = frames_want(oracle_mod, f)
    one = torch.from_numpy(f.raw.reshape(-1).copy()).cuda()
    many = one.repeat(40)
    with et.Context(0) as ctx:
        mem = Memory(et, ctx)
        with frames_of(et, ctx, f) as fr:
            fr.run(one, n_views=1)
            fr.fetch()
            mem.refuse = True
            for raw, n in ((many, 40), (one, 1), (many, 40), (one, 1)):
                with pytest.raises(et.EtError) as e:
                    fr.run(raw, n_views=n)
                assert e.value.status == et.OOM
                with pytest.raises(et.EtError) as e:
                    fr.fetch()
                assert e.value.status == et.NOT_READY
            mem.refuse = False
            for raw, n in ((one, 1), (many, 40)):
                fr.run(raw, n_views=n)
                xyz, pulse, voff = fr.fetch()
                assert np.array_equal(xyz, np.tile(wx, (n, 1))) and np.array_equal(pulse, np.tile(wp, n))
                assert list(voff) == [k * len(wx) for k in range(n + 1)]
