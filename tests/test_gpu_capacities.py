"""The finder's compiled candidate capacities (1, 2, 4, 6, 8, 16 slots) are kernels of their own, and the
capacity is a choice of schedule: for the same k_max every one of them, and every pair of passes that
adaptive capacity makes of them, gives the same bits, with and without each option and the network."""
import os
from dataclasses import replace

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

MATERIAL, FIELD = dict(eloss=0.0363), dict(field_z2=-4e-6, field_r2=-1e-6)


@pytest.fixture(scope="module")
def kf():
    import __graft_entry__ as ge
    ge.build_library()
    import paper_1906_02253_gb300 as k
    k.load_library()
    return k


@pytest.mark.parametrize("name,option", [("hi_occ", "plain"), ("hi_occ", "steering"), ("hi_occ", "material"), ("hi_occ", "field"),
                                         ("hi_occ", "all"), ("duplicates", "plain")])  # (many of the last one's seeds curl)
@pytest.mark.parametrize("top_n,margin", [(0, 0.0), (1, 0.0), (2, 0.7)])
def test_every_capacity_gives_the_same_bits(kf, name, option, top_n, margin):
    wl = synth.workload(name, n_events=3, tracks_lo=4000, tracks_hi=4000)
    if option in ("material", "all"):
        wl = replace(wl, material=synth.material_map(wl.surfaces), **MATERIAL)
    if option in ("field", "all"):
        wl = replace(wl, **FIELD)
    dev = kf.to_device_event_batch(synth.generate(wl))
    g = kf.Geometry(wl)
    ix = kf.build_hit_index(g, dev["hits"], dev["slab_offsets"], 3, dev["max_slab_hits"])
    steer = synth.steering_tables(wl, 0.4, 1.8, endcap_barrels=3) if option in ("steering", "all") else None
    net = None
    if top_n:
        z = np.load(os.path.join(os.path.dirname(kf.__file__), "data", "mlp_hi_occ.npz"))
        net = kf.mlp_buffer(z["weights"], z["mean"], z["sd"])
    sizes = [1, 2, 4, 6, 8, 16]
    for k_max in sizes:
        want = None
        for capacity in (c for c in sizes if c >= max(k_max, top_n)):
            for first in [0] + [c for c in sizes if max(top_n, 1) <= c < capacity]:
                prm = kf.find_params(wl.chi2_cut, k_max, wl.max_miss, wl.lmax, k_capacity=capacity, adaptive_capacity=first,
                                     steering_tables=steer, mlp=net, top_n=top_n, score_margin=margin)
                out = kf.find_tracks(g, ix, dev["hits"], dev["hit_surface"], dev["seed_hits"], dev["seed_event"], prm)
                got = {k: out[k].view(torch.int32).clone() for k in ("hits", "nhits", "status", "chi2", "state", "cov")}
                want = want or got
                for k in got:
                    assert torch.equal(got[k], want[k]), (k_max, capacity, first, k)
