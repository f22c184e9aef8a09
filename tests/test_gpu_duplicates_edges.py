"""Duplicate removal counts shared hits through the hits' users, or through the lists where a hit has
many: hits with fewer and with more users than twice a list's entries, lists with hits at or above
n_hits (which the inverted index leaves out but the lists share), the same hit twice in a list, empty
lists, equal chi2 and directions at the cut, against a pass over all pairs."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,lmax,n_hits,top", [(1, 1, 1, 1), (40, 4, 12, 12), (400, 17, 300, 300), (400, 31, 200, 260),
                                               (129, 5, 0, 9), (600, 9, 250, 270), (500, 6, 9, 11)])
def test_all_pairs(n, lmax, n_hits, top):
    import __graft_entry__ as ge
    ge.build_library()
    import paper_1906_02253_gb300 as kf
    rng = np.random.default_rng(n + lmax + top)
    base = rng.integers(-1, top, (max(1, n // 3), lmax))
    lists = base[rng.integers(0, len(base), n)]
    swap = rng.random((n, lmax)) < 0.3
    lists = np.where(swap, rng.integers(-1, top, (n, lmax)), lists).astype(np.int32)
    if n > 5:
        lists[5] = -1
        lists[4, : lmax // 2 + 1] = lists[4, 0]
    nhits = (lists >= 0).sum(1).astype(np.int32)
    chi2 = rng.integers(0, 4, n).astype(np.float32)
    state = np.zeros((6, n), np.float32)
    state[4], state[5] = rng.choice([0.0, 0.01, 0.0625], n), rng.choice([1.0, 1.03125, 1.125], n)
    event = rng.integers(0, 2, n).astype(np.int32)
    want = np.ones(n, np.int32)
    for j in range(n):
        own = (lists[j] >= 0).sum()
        for i in range(n):
            # (a candidate is found through a hit of the index)
            met = np.isin(lists[j][(lists[j] >= 0) & (lists[j] < n_hits)], lists[i]).any()
            better = nhits[i] > nhits[j] if nhits[i] != nhits[j] else (chi2[i] < chi2[j] if chi2[i] != chi2[j] else i < j)
            if i == j or not met or event[i] != event[j] or not better:
                continue
            if not (abs(state[4, i] - state[4, j]) < np.float32(0.02) and abs(state[5, i] - state[5, j]) < np.float32(0.05)):
                continue
            if 2 * np.isin(lists[j][lists[j] >= 0], lists[i]).sum() > own:
                want[j] = 0
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    keep = kf.remove_duplicates(t(lists.T), t(nhits), t(chi2), t(state), t(event), n_hits, dphi=0.02, dtheta=0.05)
    assert np.array_equal(keep.cpu().numpy(), want)
