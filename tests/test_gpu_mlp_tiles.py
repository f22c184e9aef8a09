"""The network kernels at the edges of their tiles and groups (128 samples a tile, four groups a block
in the forward pass, two in the loss gradient, one block per SM) against the network in FP64: single
rows, a tile less and more than full, every group of every block with a tile and one row more, and
gradient buffers at addresses that 16-byte reductions cannot take; the precision of the six-product
split, and the standardised inputs against the quotient."""
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
    err = (out[:n].double() - z).abs()
    assert (err <= 142 * 2.0 ** -24 * bound).all()
    # the six products' precision: measured 1.9e-7 of the largest logit at most over these sizes; a two-part
    # split gives 1.1e-5
    print(f"{n} rows: largest error {(err.max() / z.abs().max()).item():.2e} of the largest logit")
    assert err.max() <= 1e-6 * z.abs().max()
    assert (out[n:] == 7.0).all()


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_gradient_at_tile_edges(kf, n, shift):
    params, rows, labels = _inputs(kf, n, n + 1)
    # One row of every tile (the last row among them) counts: the others' labels are what the network says,
    # so that their errors vanish and a counted row that is lost, or taken twice, shows.
    p = torch.sigmoid(_net(params, rows)[4])
    tile = torch.arange(0, n, 128, device="cuda")
    counted = (tile + (37 * tile) // 128 % 128).clamp(max=n - 1)
    soft = p.float()
    soft[counted] = 1.0 - (p[counted] > 0.5).float()
    labels = soft
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
    # chains of 142 (layers), 64 (back through W2) and, per tile and block, 128 additions: 334 roundings
    assert ((grad.double() - want).abs() <= 2.0 ** -15 * size).all()
    err = ((grad.double() - want).norm() / want.norm()).item()
    print(f"{n} rows: gradient error {err:.2e} of its norm")
    assert err <= 334 * 2.0 ** -24
    one = lambda i: torch.cat([torch.outer(e1[i], x[i]).reshape(-1), e1[i], torch.outer(e2[i], h1[i]).reshape(-1), e2[i],  # noqa: E731
                               h2[i] * g[i], g[i][None]]).norm() / n
    assert min(one(int(i)) for i in counted[-3:]) > 8 * 334 * 2.0 ** -24 * want.norm()  # (a lost row would show)
    want_loss = (torch.nn.functional.softplus(z) - z * y).mean().item()
    assert abs(loss.item() - want_loss) <= 2e-6 * want_loss
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


def test_gradient_precision(kf):
    """A minibatch's gradient: measured 1.6e-7 of its norm (5.2e-7 with the largest product first)."""
    params, rows, labels = _inputs(kf, 4096, 5)
    loss, grad = kf.mlp_loss_grad(params, rows, labels)
    W, x, h1, h2, z, _, _, _ = _net(params, rows)
    g = torch.sigmoid(z) - labels.double()
    e2 = g[:, None] * W[4] * (h2 > 0)
    e1 = (e2 @ W[2]) * (h1 > 0)
    want = torch.cat([(e1.T @ x).reshape(-1), e1.sum(0), (e2.T @ h1).reshape(-1), e2.sum(0), h2.T @ g, g.sum()[None]]) / 4096
    err = ((grad.double() - want).norm() / want.norm()).item()
    print(f"gradient error {err:.2e} of its norm")
    assert err <= 1e-6


@pytest.mark.parametrize("outside", [0.0, 1.5 * 2.0 ** -101, 1.5 * 2.0 ** 100])
def test_standardised_inputs_are_the_quotient(kf, outside):
    """A network that passes one input through unchanged shows the standardised inputs: the reciprocal
    form (every sd within [2^-100, 2^100]) and the division (one sd outside) both give the bits of
    (x - mean) / sd, over mantissas and exponents of either, sd at the range's ends and one ulp inside."""
    g = torch.Generator(device="cuda").manual_seed(7)
    n = 20000
    for rep in range(6):
        sd = (1 + torch.rand(14, generator=g, device="cuda")) * 2.0 ** torch.randint(-40, 40, (14,), generator=g, device="cuda")
        if rep == 1:  # mantissas of ones
            sd = torch.nextafter(2.0 ** torch.randint(-40, 40, (14,), generator=g, device="cuda").float(), torch.zeros((), device="cuda"))
        if rep == 2:
            sd[0], sd[1] = 2.0 ** 100, 2.0 ** -100
            sd[2] = float(np.nextafter(np.float32(2.0 ** 100), np.float32(0)))
            sd[3] = float(np.nextafter(np.float32(2.0 ** -100), np.float32(1)))
        if outside:
            sd[5] = outside
        # quotients of either sign within [2^-12, 2^12], a mean among the features' own sizes
        rows = (torch.randn(n, 14, generator=g, device="cuda") * 2.0 ** torch.randint(-8, 9, (n, 14), generator=g, device="cuda")) * sd
        mean = rows[0] * 0.5 if rep else torch.zeros(14, device="cuda")
        for k in (0, 1, 2, 3, 5, 8, 13):
            p = torch.zeros(kf.MLP_BUFFER, device="cuda")
            p[:896].view(64, 14)[0, k], p[:896].view(64, 14)[1, k] = 1.0, -1.0
            p[960:5056].view(64, 64)[:] = torch.eye(64, device="cuda")
            p[5120], p[5121] = 1.0, -1.0
            p[5185:5199], p[5199:5213] = mean, sd
            got, want = kf.mlp_forward(p, rows), (rows[:, k] - mean[k]) / sd[k]
            assert torch.equal(got, want), (rep, k, (got != want).sum().item(), (got - want).abs().max().item())
