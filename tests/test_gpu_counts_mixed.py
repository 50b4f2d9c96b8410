"""The allocation-free counts on pair lists that mix countable pairs with ones
that get -1, at any position: the lists are short enough for 4 pairs per warp,
in between, and long enough for 32, and end inside a warp's share."""
import numpy as np
import pytest

from paper_1311_5334_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 5, 1003, 150001, 400003])
def test_mixed_pairs_equal_the_oracle(oracle_mod, count):
    import torch
    from paper_1311_5334_gb300 import et

    v = synth.make_view(17, n_fog=1500, n_through=15)
    p = synth.params(v.extent)
    o = oracle_mod.Oracle(v.xyz, v.extent, p["seed_min"], p["seed_max"], p["tube_r"], p["min_hits"])
    try:
        lo, hi = o.seeds()
        base = np.stack([lo, hi], 1).astype(np.int64)
        want_base = np.asarray(o.count_pairs(base[:, 0], base[:, 1]))
    finally:
        o.close()
    rng = np.random.default_rng(count)
    pick = rng.integers(0, len(base), count)
    pairs, want = base[pick], want_base[pick].astype(np.int64)
    swap = rng.random(count) < 0.5                       # a pair has no direction
    pairs = np.where(swap[:, None], pairs[:, ::-1], pairs)
    bad = rng.random(count) < 0.4
    kind = rng.integers(0, 3, count)
    far = np.argsort(v.xyz[:, 0])
    pairs[bad & (kind == 0), 1] = pairs[bad & (kind == 0), 0]            # equal indices
    pairs[bad & (kind == 1), 0] = v.n                                     # outside the view
    pairs[bad & (kind == 2)] = (far[0], far[-1])                          # seed_max or more apart
    want[bad] = -1
    d_xyz = torch.from_numpy(v.xyz).cuda()
    d_pairs = torch.from_numpy(np.ascontiguousarray(pairs, dtype=np.int32)).cuda()
    outs = [torch.full((count,), -7, dtype=torch.int32, device="cuda") for _ in range(2)]
    for out in outs:                                     # back to back, no wait between
        et.tube_count_noalloc(d_xyz, p, d_pairs, out)
    torch.cuda.synchronize()
    for out in outs:
        assert np.array_equal(out.cpu().numpy(), want)
