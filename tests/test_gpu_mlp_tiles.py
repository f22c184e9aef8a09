"""The network kernels at the edges of their tiles and groups (128 samples a tile, four groups a block
in the forward pass, two in the loss gradient, one block per SM) against the network in FP64: single
rows, a tile less and more than full, every group of every block with a tile and one row more, and
gradient buffers at addresses that 16-byte reductions cannot take."""
import os

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kf():
    import __graft_entry__ as ge
    ge.build_library()
    import paper_1906_02253_gb300 as k
    k.load_library()
    return k


def _inputs(kf, n, seed):
    z = np.load(os.path.join(os.path.dirname(kf.__file__), "data", "mlp_hi_occ.npz"))
    g = torch.Generator(device="cuda").manual_seed(seed)
    mean, sd = torch.from_numpy(z["mean"]).cuda(), torch.from_numpy(z["sd"]).cuda()
    rows = (mean + sd * torch.randn(n, 14, generator=g, device="cuda")).contiguous()
    return kf.mlp_buffer(z["weights"], z["mean"], z["sd"]), rows, (torch.rand(n, generator=g, device="cuda") < 0.4).float()


def _net(params, rows):
    f = params.double()
    W = [f[:896].reshape(64, 14), f[896:960], f[960:5056].reshape(64, 64), f[5056:5120], f[5120:5184], f[5184]]
    x = (rows.double() - f[5185:5199]) / f[5199:5213]
    h1 = torch.relu(x @ W[0].T + W[1])
    h2 = torch.relu(h1 @ W[2].T + W[3])
    # the same on absolute values: every product and sum errs by a few roundings of its terms
    a1 = x.abs() @ W[0].abs().T + W[1].abs()
    a2 = a1 @ W[2].abs().T + W[3].abs()
    return W, x, h1, h2, h2 @ W[4] + W[5], a1, a2, a2 @ W[4].abs() + W[5].abs()


SIZES = [1, 2, 127, 128, 129, 19456, 38913, 77825, 100003]  # 152 SMs: 152, 304 and 608 tiles, and one row more


@pytest.mark.parametrize("n", SIZES)
def test_forward_at_tile_edges(kf, n):
    params, rows, _ = _inputs(kf, n, n)
    out = torch.full((n + 64,), 7.0, device="cuda")
    kf.mlp_forward(params, rows, out=out)
    _, _, _, _, z, _, _, bound = _net(params, rows)
    # at most 64 + 64 + 14 FP32 additions deep, each within 2^-24 of its terms' absolute values
    assert ((out[:n].double() - z).abs() <= 142 * 2.0 ** -24 * bound).all()
    assert (out[n:] == 7.0).all()


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_gradient_at_tile_edges(kf, n, shift):
    params, rows, labels = _inputs(kf, n, n + 1)
    room = torch.full((kf.MLP_PARAMS + 8,), 7.0, device="cuda")
    loss, grad = kf.mlp_loss_grad(params, rows, labels, grad=room[shift:shift + kf.MLP_PARAMS])
    W, x, h1, h2, z, a1, a2, _ = _net(params, rows)
    y = labels.double()
    g = torch.sigmoid(z) - y
    e2 = g[:, None] * W[4] * (h2 > 0)
    e1 = (e2 @ W[2]) * (h1 > 0)
    want = torch.cat([(e1.T @ x).reshape(-1), e1.sum(0), (e2.T @ h1).reshape(-1), e2.sum(0), h2.T @ g, g.sum()[None]]) / n
    ae2 = W[4].abs().expand(n, 64)
    ae1 = ae2 @ W[2].abs()
    size = torch.cat([(ae1.T @ x.abs()).reshape(-1), ae1.sum(0), (ae2.T @ a1).reshape(-1), ae2.sum(0), a2.sum(0),
                      torch.tensor([float(n)], dtype=torch.float64, device="cuda")]) / n
    # chains of 142 (layers), 64 (back through W2) and, per tile and block, 128 additions; a unit within
    # rounding of zero may be masked the other way, which moves its terms by that rounding
    assert ((grad.double() - want).abs() <= 2.0 ** -15 * size).all()
    assert abs(loss.item() - (torch.nn.functional.softplus(z) - z * y).mean().item()) <= 1e-5
    assert (room[:shift] == 7.0).all() and (room[shift + kf.MLP_PARAMS:] == 7.0).all()


# (a block's only tile; the first tiles of its two groups; a later one of the first)
@pytest.mark.parametrize("n,tile", [(128, 0), (40000, 0), (40000, 200), (100003, 0), (100003, 200), (100003, 450)])
def test_a_wait_that_gives_up_adds_nothing_of_its_block(kf, n, tile):
    """The loss says so (NaN), and the gradient is that of the other blocks' tiles (block b takes the
    tiles b, b + blocks, ...), none of the failed block's partial sums."""
    params, rows, labels = _inputs(kf, n, n + 2)
    blocks = min((n + 127) // 128, torch.cuda.get_device_properties(0).multi_processor_count)
    loss, grad = kf.mlp_wait_probe(params, rows, labels, tile)
    assert loss.isnan().all()
    other = (torch.arange(n, device="cuda") // 128) % blocks != tile % blocks
    W, x, h1, h2, z, _, _, _ = _net(params, rows[other])
    g = torch.sigmoid(z) - labels[other].double()
    e2 = g[:, None] * W[4] * (h2 > 0)
    e1 = (e2 @ W[2]) * (h1 > 0)
    want = torch.cat([(e1.T @ x).reshape(-1), e1.sum(0), (e2.T @ h1).reshape(-1), e2.sum(0), h2.T @ g, g.sum()[None]]) / n
    # FP32 sums: about 1e-6 of the gradient's norm; one block's share is 1 / 152 of it
    assert (grad.double() - want).norm() <= 2e-5 * want.norm() if other.any() else not grad.any()
    # the call without a failure is whole again
    loss, grad = kf.mlp_loss_grad(params, rows, labels)
    assert loss.isfinite().all() and grad.isfinite().all()


@pytest.mark.parametrize("n", [1, 127, 129, 20000])
@pytest.mark.parametrize("mean,sd", [(1e38, 0.1), (-1e38, 0.1), (1e5, 1e-35), (3.0, 1e-44)])
def test_rows_past_the_end_leave_no_trace(kf, n, mean, sd):
    """A constant feature at a mean far beyond its spread is zero in every row, whatever the normaliser
    would make of a row of zeros."""
    params, rows, labels = _inputs(kf, n, n + 3)
    params[5185 + 3], params[5199 + 3] = mean, sd
    rows[:, 3] = mean
    loss, grad = kf.mlp_loss_grad(params, rows, labels)
    out = kf.mlp_forward(params, rows)
    params[5185 + 3], params[5199 + 3] = 0.0, 1.0
    rows[:, 3] = 0.0
    want_loss, want = kf.mlp_loss_grad(params, rows, labels)
    # the same inputs but for the quotient's last bit; the blocks' sums are added in any order
    assert grad.isfinite().all() and (grad - want).norm() <= 1e-5 * want.norm()
    assert abs(loss.item() - want_loss.item()) <= 1e-5 * want_loss.item()
    want = kf.mlp_forward(params, rows)
    assert (out - want).abs().max() <= 1e-5 * want.abs().max().clamp(min=1.0)
