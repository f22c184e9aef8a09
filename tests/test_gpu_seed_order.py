"""Finding with the seeds taken in the library's own order (by direction in geometries with disks, curling
seeds first in the others; a workspace of the full size) gives bit for bit what it gives with the
seeds in index order (a workspace without the order's 4 bytes per seed), at the edges of the ordering kernel's blocks, with failed and removed seeds, in one pass and
two, plain, learned and with options."""
import ctypes
import os

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
def batch(kf):
    wl = synth.workload("field", n_events=2, tracks_lo=2300, tracks_hi=2300, seed=17)
    b = synth.generate(wl)
    return wl, kf.to_device_event_batch(b)


@pytest.fixture(scope="module")
def barrel(kf):
    """Barrel seeds, the odd ones of hits of different particles, which curl."""
    wl = synth.workload("find", n_events=2, tracks_lo=2300, tracks_hi=2300, seed=18)
    dev = kf.to_device_event_batch(synth.generate(wl))
    dev["seed_hits"][1, 1::2] = dev["seed_hits"][1, 1::2].roll(1)
    return wl, dev


def _up(v):
    return (v + 255) // 256 * 256


def _all_written(out, n_hits):
    """Every seed has outputs: nothing of the -7 that the buffers held, no hit id outside the hits."""
    assert ((out["status"] >= 0) & (out["status"] <= 2)).all()
    assert (out["nhits"] >= 0).all()
    assert ((out["hits"] >= -1) & (out["hits"] < n_hits)).all()
    bad = out["status"] != 0
    assert (out["hits"][:, bad] == -1).all() and (out["nhits"][bad] == 0).all()
    assert out["chi2"][bad].isnan().all() and out["state"][:, bad].isnan().all() and out["cov"][:, bad].isnan().all()


@pytest.mark.parametrize("option", ["disks", "barrel", "barrel_static"])
def test_a_seed_whose_fit_gives_no_chi2_fails(kf, batch, barrel, option):
    """A NaN coordinate of a seed's second or third barrel hit leaves its circle as it is and makes the
    chi2 NaN: the seed fails, and its outputs say so."""
    wl, dev = batch if option == "disks" else barrel
    g = kf.Geometry(wl)
    hits = dev["hits"].clone()
    ids = dev["seed_hits"].long()
    on_barrel = (dev["hit_surface"][ids[1]] < 17) & (dev["hit_surface"][ids[2]] < 17)
    some = torch.nonzero(on_barrel).squeeze(1)[5:2000:20]
    hits[ids[1, some[0::2]], 1] = float("nan")
    hits[ids[2, some[1::2]], 1] = float("nan")
    ix = kf.build_hit_index(g, hits, dev["slab_offsets"], 2, dev["max_slab_hits"])
    n = ids.shape[1]
    out = dict(hits=torch.full((wl.lmax, n), -7, dtype=torch.int32, device="cuda"))
    for k in ("nhits", "status"):
        out[k] = torch.full((n,), -7, dtype=torch.int32, device="cuda")
    out["chi2"] = torch.full((n,), -7.0, device="cuda")
    out["state"], out["cov"] = torch.full((6, n), -7.0, device="cuda"), torch.full((21, n), -7.0, device="cuda")
    prm = kf.find_params(wl.chi2_cut, wl.k_max, wl.max_miss, wl.lmax)
    if option == "barrel_static":
        P = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
        rc = kf.load_library().kf_find_tracks_static(
            g.ref, ctypes.byref(ix.c), P(hits), P(dev["hit_surface"]), P(dev["seed_hits"]), P(dev["seed_event"]), n,
            ctypes.byref(prm), P(out["hits"]), P(out["nhits"]), P(out["chi2"]), P(out["state"]), P(out["cov"]), P(out["status"]),
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == kf.KF_OK
    else:
        kf.find_tracks(g, ix, hits, dev["hit_surface"], dev["seed_hits"], dev["seed_event"], prm, out=out)
    _all_written(out, hits.shape[0])
    assert len(some) > 50 and (out["status"][some] == 1).all()
    state, _ = kf.seed_states(g, hits, dev["hit_surface"], dev["seed_hits"], dev["seed_event"], 2)
    assert torch.equal(state[27] < 0, out["status"] != 0) and not state[27].isnan().any()


@pytest.mark.parametrize("n", [1, 2, 127, 128, 129, 2047, 2048, 2049, 4600])
@pytest.mark.parametrize("option", ["plain", "two_passes", "learned", "field", "barrel", "barrel_all_kept", "barrel_few_curl",
                                    "barrel_steered"])
def test_order_changes_no_result(kf, batch, barrel, n, option):
    wl, dev = barrel if option.startswith("barrel") else batch
    from dataclasses import replace
    g = kf.Geometry(wl if option == "field" else replace(wl, field_z2=0.0, field_r2=0.0))
    ix = kf.build_hit_index(g, dev["hits"], dev["slab_offsets"], 2, dev["max_slab_hits"])
    some = torch.linspace(0, dev["seed_hits"].shape[1] - 1, n).long().cuda()
    if option == "barrel_few_curl":  # below the share from which they go first
        some[10:] = some[10:] // 2 * 2
    seeds, event = dev["seed_hits"][:, some].contiguous(), dev["seed_event"][some].contiguous()
    keep = torch.ones(n, dtype=torch.int32, device="cuda")
    if n > 10:
        seeds[1, 3] = -1          # failed: no such hit
        seeds[:, 5] = seeds[0, 5]  # failed: one hit three times
        event[7] = 9              # failed: no such event
        keep[::6] = 0             # removed by cleaning
    if option == "barrel_all_kept":
        keep = None
    net = None
    if option == "learned":
        z = np.load(os.path.join(os.path.dirname(kf.__file__), "data", "mlp_hi_occ.npz"))
        net = kf.mlp_buffer(z["weights"], z["mean"], z["sd"])
    layers = list(range(len(wl.surfaces)))
    steer = dict(c_barrel=0.4, c_endcap=3.0, lists=[layers] * 5) if option == "barrel_steered" else None
    if steer:  # failed seeds without removed ones, and a failed seed whose third hit is the missing one
        keep = None
        if n > 10:
            seeds[2, 9] = -1
    prm = kf.find_params(wl.chi2_cut, wl.k_max, wl.max_miss, wl.lmax, seed_keep=keep, steering_tables=steer, mlp=net, top_n=2 if net is not None else 0,
                         score_margin=0.7 if net is not None else 0.0, adaptive_capacity=2 if option == "two_passes" else 0)
    full = kf.find_workspace_size(n, prm)
    room = torch.empty(full, dtype=torch.uint8, device="cuda")
    P = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    outs = []
    for size in (full, full - _up(4 * n)):
        out = dict(hits=torch.full((wl.lmax, n), -7, dtype=torch.int32, device="cuda"))
        for k in ("nhits", "status"):
            out[k] = torch.full((n,), -7, dtype=torch.int32, device="cuda")
        out["chi2"] = torch.full((n,), -7.0, device="cuda")
        out["state"], out["cov"] = torch.full((6, n), -7.0, device="cuda"), torch.full((21, n), -7.0, device="cuda")
        rc = kf.load_library().kf_find_tracks(
            g.ref, ctypes.byref(ix.c), P(dev["hits"]), P(dev["hit_surface"]), P(seeds), P(event), n, ctypes.byref(prm),
            P(out["hits"]), P(out["nhits"]), P(out["chi2"]), P(out["state"]), P(out["cov"]), P(out["status"]), P(room), size,
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == kf.KF_OK
        outs.append({k: v.clone() for k, v in out.items()})
    a, b = outs
    for k in a:
        assert torch.equal(a[k].view(torch.int32), b[k].view(torch.int32)), k
    _all_written(a, dev["hits"].shape[0])
    keep = torch.ones(n, dtype=torch.int32, device="cuda") if keep is None else keep
    want = torch.where(keep == 0, 2, 0)
    if n > 10:
        for i in (3, 5, 7):
            want[i] = 1 if keep[i] else 2
    if option.startswith("barrel"):  # seeds of hits of different particles may fail as well
        assert torch.equal(a["status"] == 2, keep == 0)
    else:
        assert torch.equal(a["status"], want.to(torch.int32))
    # a smaller one is refused
    rc = kf.load_library().kf_find_tracks(
        g.ref, ctypes.byref(ix.c), P(dev["hits"]), P(dev["hit_surface"]), P(seeds), P(event), n, ctypes.byref(prm), P(out["hits"]),
        P(out["nhits"]), P(out["chi2"]), P(out["state"]), P(out["cov"]), P(out["status"]), P(room), full - _up(4 * n) - 256,
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == kf.KF_ERR_ARG
