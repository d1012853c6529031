"""The proposal network's fused forward, backward and update kernels at the
edges of their work split -- one row tile, tile counts on both sides of each
share of the output tiles (one wave of CTAs), more tiles than SMs -- and with
inputs and outputs at 4-byte alignment, against FP64 autograd: outputs within
1e-2 of their largest, each gradient within 2e-2 of its norm (BF16 operands),
and rows beyond n untouched.  The loss against the FP64 mean of the terms at
the network's own outputs (the forward entry's): FP32 terms and sums over at
most 2^10 of them in a row, so within 2^-13 of the terms' mean magnitude."""
import numpy as np
import pytest
import torch

from paper_1904_06680_gb300 import npp, proposal

pytestmark = pytest.mark.gpu
H, I, O = 256, proposal.N_IN, 2 * proposal.N_THETA
SIZES = [H * I, H, H * H, H, O * H, O]


def _params(seed):
    rng = np.random.default_rng(seed)
    parts = [rng.standard_normal((H, I)) * np.sqrt(2.0 / I), 0.2 * rng.standard_normal(H),
             rng.standard_normal((H, H)) * np.sqrt(2.0 / H), 0.2 * rng.standard_normal(H),
             rng.standard_normal((O, H)) * 0.5 / np.sqrt(H), 0.2 * rng.standard_normal(O)]
    return np.concatenate([p.ravel() for p in parts]).astype(np.float32)


def _shifted(t, shift):
    """the same values at an address `shift` floats past an allocation's start"""
    buf = torch.full((t.numel() + shift + 4,), float("nan"), device="cuda")
    buf[shift:shift + t.numel()] = t.reshape(-1)
    return buf, buf[shift:shift + t.numel()].view(t.shape)


def _exact(v, x):
    W1, b1, W2, b2, W3, b3 = torch.split(v, SIZES)
    h = torch.relu(x @ W1.reshape(H, I).T + b1)
    h = torch.relu(h @ W2.reshape(H, H).T + b2)
    y = h @ W3.reshape(O, H).T + b3
    return y[:, :O // 2], y[:, O // 2:].clamp(-3.0, 1.0)


def _inputs(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand(n, I, generator=g, device="cuda")
    x[:, 64:] = 2 * x[:, 64:] - 1
    return x, 1.3 * torch.randn(n, O // 2, generator=g, device="cuda")


@pytest.mark.parametrize("batch,n,shift", [(128, 1, 0), (128, 128, 1), (384, 129, 2), (1024, 300, 0), (4864, 4863, 0),
                                           (4992, 4992, 1), (9856, 9731, 0), (20096, 20096, 0)])
def test_forward(batch, n, shift):
    vec = _params(batch)
    net = proposal.ProposalNet(batch=batch)
    net.set_params(vec)
    _, x = _shifted(_inputs(n, n)[0], shift)
    mbuf, mean = _shifted(torch.zeros(n, O // 2, device="cuda"), shift)
    sbuf, std = _shifted(torch.zeros(n, O // 2, device="cuda"), shift)
    npp.npp_proposal_forward(net.P, x, n, mean, std)
    mu, ls = _exact(torch.from_numpy(vec).cuda().double(), x.double())
    scale = torch.maximum(mu.abs().max(), ls.abs().max())
    assert float((mean.double() - mu).abs().max()) <= 1e-2 * float(scale)
    assert float((std.double().log() - ls).abs().max()) <= 1e-2 * float(scale)
    for buf in (mbuf, sbuf):
        assert bool(torch.isnan(buf[:shift]).all()) and bool(torch.isnan(buf[shift + n * (O // 2):]).all())
    net.close()


@pytest.mark.parametrize("batch,shift", [(128, 0), (384, 1), (4864, 0), (4992, 0), (9856, 1), (20096, 0)])
def test_gradients(batch, shift):
    vec = _params(batch + 1)
    net = proposal.ProposalNet(batch=batch)
    net.set_params(vec)
    x0, t0 = _inputs(batch, batch)
    _, x = _shifted(x0, shift)
    _, theta = _shifted(t0, shift)
    loss = torch.zeros(1, device="cuda")
    npp.npp_proposal_train_step(net.P, x, theta, 0.0, loss)
    got = torch.from_numpy(net.grads()).cuda().double()
    np.testing.assert_array_equal(net.params(), vec)
    v = torch.from_numpy(vec).cuda().double().requires_grad_(True)
    mu, ls = _exact(v, x.double())
    g, = torch.autograd.grad((ls + 0.5 * (theta.double() - mu) ** 2 * torch.exp(-2 * ls)).mean(), v)
    mean, std = torch.zeros(batch, O // 2, device="cuda"), torch.zeros(batch, O // 2, device="cuda")
    npp.npp_proposal_forward(net.P, x, batch, mean, std)
    own = std.double().log(), 0.5 * ((theta.double() - mean.double()) / std.double()) ** 2
    terms = own[0].abs() + own[1]
    assert abs(float(loss) - float((own[0] + own[1]).mean())) <= 2.0 ** -13 * float(terms.mean())
    for a, b in zip(torch.split(got, SIZES), torch.split(g, SIZES)):
        assert float((a - b).norm()) <= 2e-2 * float(b.norm())
    net.close()
