"""The allocation-free counts of tiny views with lists of pairs around the numbers where a warp's first share
is the whole work (32 pairs for each of four blocks of eight warps an SM) and where shares are taken on."""
import numpy as np
import pytest

from paper_1311_5334_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grains", [2, 120])
def test_pair_lists_around_one_share_a_warp(oracle_mod, grains):
    import torch
    from paper_1311_5334_gb300 import et

    v = synth.make_view(19, n_fog=max(2, grains - 40), n_through=0 if grains == 2 else 1)
    xyz = v.xyz[:grains]
    p = synth.params(v.extent)
    with oracle_mod.Oracle(xyz, v.extent, p["seed_min"], p["seed_max"], p["tube_r"], p["min_hits"]) as o:
        i, j = np.meshgrid(np.arange(len(xyz)), np.arange(len(xyz)), indexing="ij")
        near = (i != j) & (np.abs(xyz[i] - xyz[j]) < p["seed_max"]).all(-1)
        table = np.full(i.shape, -1, dtype=np.int64)
        if near.any():
            table[near] = o.count_pairs(i[near], j[near])
    with et.Context(0) as ctx:
        warps = ctx.info()["sm_count"] * 4 * 8
    d_xyz = torch.from_numpy(np.ascontiguousarray(xyz)).cuda()
    rng = np.random.default_rng(grains)
    for count in [n + k for n in (4 * warps, 8 * warps, 32 * warps, 64 * warps) for k in (-1, 0, 1)]:
        pairs = rng.integers(0, len(xyz), (count, 2)).astype(np.int32)
        out = torch.full((count,), -7, dtype=torch.int32, device="cuda")
        et.tube_count_noalloc(d_xyz, p, torch.from_numpy(pairs).cuda(), out)
        assert np.array_equal(out.cpu().numpy(), table[pairs[:, 0], pairs[:, 1]])


@pytest.mark.parametrize("extent", [(1 << 20, 2, 3), (3, 1 << 20, 2), (2, 3, 1 << 20), (1 << 20, 1, 1), (700000, 40, 300000)])
def test_long_thin_views(oracle_mod, extent):
    """Extents of which the cell list with rows along x, or the one along y, has most of its cells."""
    import torch
    from paper_1311_5334_gb300 import et

    rng = np.random.default_rng(sum(extent))
    xyz = np.unique(rng.integers(0, extent, (3000, 3)), axis=0).astype(np.int32)
    xyz = np.ascontiguousarray(xyz[rng.permutation(len(xyz))])
    p = synth.params(extent, seed_min=0, seed_max=1000, tube_r=3)
    order = np.lexsort(xyz.T)
    i = rng.integers(0, len(xyz) - 4, 5000)
    pairs = np.stack([order[i], order[i + rng.integers(1, 4, 5000)]], 1).astype(np.int32)
    good = (np.abs(xyz[pairs[:, 0]] - xyz[pairs[:, 1]]) < p["seed_max"]).all(1)
    want = np.full(len(pairs), -1, dtype=np.int64)
    with oracle_mod.Oracle(xyz, extent, p["seed_min"], p["seed_max"], p["tube_r"], p["min_hits"]) as o:
        want[good] = o.count_pairs(pairs[good, 0].astype(np.int64), pairs[good, 1].astype(np.int64))
    out = torch.full((len(pairs),), -7, dtype=torch.int32, device="cuda")
    et.tube_count_noalloc(torch.from_numpy(xyz).cuda(), p, torch.from_numpy(pairs).cuda(), out)
    assert np.array_equal(out.cpu().numpy(), want)


def test_cells_by_the_number_of_pairs(oracle_mod):
    """The same pairs of a large view, first by few in a call, on coarse cells, then by many."""
    import torch
    from paper_1311_5334_gb300 import et

    v = synth.make_view(29, n_fog=40000, n_through=200)
    p = synth.params(v.extent)
    order = np.lexsort((v.xyz[:, 2] // 1500, v.xyz[:, 1] // 1500, v.xyz[:, 0] // 1500))
    rng = np.random.default_rng(29)
    i = rng.integers(0, v.n - 20, 100000)
    pairs = np.stack([order[i], order[i + rng.integers(1, 20, len(i))]], 1)
    near = (np.abs(v.xyz[pairs[:, 0]] - v.xyz[pairs[:, 1]]) < p["seed_max"]).all(1)
    want = np.full(len(pairs), -1, dtype=np.int64)
    with oracle_mod.Oracle(v.xyz, v.extent, p["seed_min"], p["seed_max"], p["tube_r"], p["min_hits"]) as o:
        want[near] = o.count_pairs(pairs[near, 0], pairs[near, 1])
    d_xyz, d_pairs = (torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda() for a in (v.xyz, pairs))
    for count in (1, 100, 8192, 8194, 40000, len(pairs)):
        out = torch.full((count,), -7, dtype=torch.int32, device="cuda")
        et.tube_count_noalloc(d_xyz, p, d_pairs[:count].contiguous(), out)
        assert np.array_equal(out.cpu().numpy(), want[:count])
