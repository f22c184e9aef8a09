"""The finder's selection of a seed's best children: the plain instances rank them by counting, the
instances with options by a tournament. Region steering with each region's list holding every
barrel layer in order selects an option instance without changing which surface is next, so both
must find the same tracks, here with windows wide enough that the children of a seed go far beyond
its slots, with more slots than candidates kept, and in two passes; and a first pass that has more
slots than candidates kept must give what one pass gives."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kf():
    import __graft_entry__ as ge
    ge.build_library()
    import paper_1906_02253_gb300 as k
    k.load_library()
    return k


@pytest.fixture(scope="module")
def event(kf):
    wl = synth.workload("find", n_events=1, tracks_lo=1500, tracks_hi=1500, noise_frac=1.0, seed=41)
    b = synth.generate(wl)
    g = kf.Geometry(wl)
    dev = kf.to_device_event_batch(b)
    return wl, g, dev, kf.build_hit_index(g, dev["hits"], dev["slab_offsets"], 1, dev["max_slab_hits"])


@pytest.mark.parametrize("chi2_cut", [30.0, 3000.0])
@pytest.mark.parametrize("k_max,capacity,adaptive", [(1, 0, 0), (1, 6, 0), (2, 0, 0), (3, 0, 0), (4, 0, 2), (5, 0, 0), (5, 8, 2),
                                                     (6, 0, 4), (6, 16, 0), (7, 0, 0), (8, 0, 2), (11, 0, 4), (16, 0, 0)])
def test_counting_and_tournament_agree(kf, event, chi2_cut, k_max, capacity, adaptive):
    wl, g, dev, ix = event
    layers = list(range(len(wl.surfaces)))
    steer = dict(c_barrel=0.4, c_endcap=3.0, lists=[layers] * 5)

    def find(tables):
        prm = kf.find_params(chi2_cut, k_max, 1, wl.lmax, k_capacity=capacity, adaptive_capacity=adaptive,
                             steering_tables=tables)
        return kf.find_tracks(g, ix, dev["hits"], dev["hit_surface"], dev["seed_hits"], dev["seed_event"], prm)

    a, b = find(None), find(steer)
    assert torch.equal(a["status"], b["status"])
    same = (a["hits"] == b["hits"]).all(0)
    # the two instances are compiled apart: a tie within rounding may fall the other way
    assert same.float().mean().item() >= 0.999
    assert torch.allclose(a["chi2"][same], b["chi2"][same], rtol=1e-3, atol=1e-3)
    assert np.isfinite(a["chi2"].cpu().numpy()).all()


@pytest.mark.parametrize("chi2_cut", [10.0, 30.0, 300.0, 3000.0])
@pytest.mark.parametrize("k_max,capacity,first", [(1, 4, 2), (1, 16, 8), (2, 8, 4), (3, 8, 4), (5, 8, 5), (5, 8, 6), (7, 16, 8)])
def test_first_pass_with_more_slots_than_candidates_kept(kf, event, chi2_cut, k_max, capacity, first):
    """A lane of such a pass may see more passing hits than the k_max its list holds without its seed's
    children outnumbering the slots: only those of the list may become children."""
    wl, g, dev, ix = event

    def find(adaptive):
        prm = kf.find_params(chi2_cut, k_max, 1, wl.lmax, k_capacity=capacity, adaptive_capacity=adaptive)
        return kf.find_tracks(g, ix, dev["hits"], dev["hit_surface"], dev["seed_hits"], dev["seed_event"], prm)

    one, two = find(0), find(first)
    for k in ("hits", "nhits", "status", "chi2", "state", "cov"):
        assert torch.equal(one[k].view(torch.int32), two[k].view(torch.int32)), k
