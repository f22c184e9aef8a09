"""Both hit-index kernels (by fine bins up to 8,192 bins, by bins and sub-bins above or where shared
memory asks for it) against the bin rule in numpy FP32: bin counts at the edge between them, empty,
tiny and the largest slabs, many hits in one fine bin, hits beyond the extents and NaN."""
from types import SimpleNamespace

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

LO, HI = -29.0, 31.0


@pytest.fixture(scope="module")
def kf():
    import __graft_entry__ as ge
    ge.build_library()
    import paper_1906_02253_gb300 as k
    k.load_library()
    return k


def _floor_index(a, n):
    f = np.floor(a)
    return np.clip(np.where(f >= 0, np.minimum(f, 1e8), -1), 0, n - 1).astype(np.int64)  # NaN: bin 0


def _reference(hits, n_phi, n_2nd):
    with np.errstate(invalid="ignore", over="ignore"):
        turn = hits[:, 0] + np.float32(np.pi)
        pb = _floor_index(turn * np.float32(n_phi / (2 * np.pi)), n_phi)
        fine = _floor_index(turn * np.float32(n_phi * 8 / (2 * np.pi)), n_phi * 8)
        vb = _floor_index((hits[:, 1] - np.float32(LO)) * np.float32(n_2nd / (HI - LO)), n_2nd)
    b, sub = pb * n_2nd + vb, np.clip(fine - pb * 8, 0, 7)
    order = np.lexsort((np.arange(len(b)), sub, b))
    counts = np.bincount(b, minlength=n_phi * n_2nd)
    per_sub = np.bincount(b * 8 + sub, minlength=n_phi * n_2nd * 8).reshape(-1, 8).cumsum(1)
    return order, np.concatenate([[0], counts.cumsum()]), per_sub


@pytest.mark.parametrize("n_phi,n_2nd", [(1, 1), (3, 5), (64, 32), (256, 32), (1024, 8), (257, 32), (128, 128)])
@pytest.mark.parametrize("slabs", [(0, 1, 5, 0), (1000, 33, 20000), (20704, 3), (20706, 3), (32768, 3)])  # (20,706 at 64 x 32 bins: two blocks of the fine kernel no longer fit an SM)
def test_routes_match_the_bin_rule(kf, n_phi, n_2nd, slabs):
    surf = [SimpleNamespace(type=0, r_or_z=4.0 + i, lo=LO, hi=HI, x_over_x0=0.0, n_phi=n_phi, n_2nd=n_2nd)
            for i in range(len(slabs))]
    geom = kf.Geometry(SimpleNamespace(surfaces=surf, bz=3.8, sigma_rphi=0.01, sigma_2nd=0.1, prior=(1.0,) * 5))
    rng = np.random.default_rng(n_phi * 100 + n_2nd + sum(slabs))
    n = sum(slabs)
    hits = np.stack([rng.uniform(-np.pi, np.pi, n), rng.uniform(LO - 1, HI + 1, n)], 1).astype(np.float32)
    hits[::7, 0] = hits[3 % n, 0]                     # many hits in few fine bins
    hits[::14] = hits[0]
    hits[1::50, 0] = np.float32(np.pi)
    hits[2::50, 0] = -np.float32(np.pi)
    hits[min(4, n - 1), 0] = np.nan
    offs = np.concatenate([[0], np.cumsum(slabs)]).astype(np.int32)
    d_hits, d_offs = torch.from_numpy(hits).cuda(), torch.from_numpy(offs).cuda()
    # the largest slabs with the most bins exceed shared memory on either route
    if n_phi * n_2nd * 4 + 5 * max(slabs) > 220000:
        pytest.skip("beyond the kernels' shared memory")
    ix = kf.build_hit_index(geom, d_hits, d_offs, 1, max(slabs))
    bin_off, ids, sub = ix.bin_off.cpu().numpy(), ix.sorted_ids.cpu().numpy(), ix.sub_off.cpu().numpy().astype(np.uint16)
    out, rec = ix.sorted_hits.cpu().numpy(), ix.sorted_rec
    for s in range(len(slabs)):
        a, b = offs[s], offs[s + 1]
        order, off, per_sub = _reference(hits[a:b], n_phi, n_2nd)
        assert np.array_equal(ids[a:b], a + order)
        assert np.array_equal(bin_off[s], a + off)
        assert np.array_equal(sub[s], per_sub)
        assert np.array_equal(out[a:b], hits[a:b][order], equal_nan=True)
    assert np.array_equal(rec.view(torch.int32)[:, 3].cpu().numpy(), ids)
    assert np.array_equal(rec[:, 2].cpu().numpy(), out[:, 1], equal_nan=True)
    # a slab above the bound is left empty and reported; the optional outputs may be absent
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    if max(slabs) > 40:
        ix2 = kf.HitIndex(geom, 1, n)
        ix2.c.sorted_rec = ix2.c.sub_off = None
        kf.build_hit_index(geom, d_hits, d_offs, 1, 40, index=ix2, status=status)
        assert status.item() == 1
        for s in range(len(slabs)):
            a = offs[s]
            got = ix2.bin_off[s].cpu().numpy()
            assert np.array_equal(got, np.full_like(got, a) if slabs[s] > 40 else a + _reference(hits[a:offs[s + 1]], n_phi, n_2nd)[1])
