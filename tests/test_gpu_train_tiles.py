"""asd_mlp_loss_grad at the edges of its 64-sample tiles and input padding, against FP64
back-propagation, and the weights of a view that is not 16-byte aligned."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def asd():
    from paper_2308_07487_gb300 import asd as m
    return m


def _params(asd, n_in, depth, seed):
    P = asd.lib.asd_mlp_param_count(n_in, depth)
    return (0.25 * synth.rng(seed).normal(size=P)).astype(np.float32)


def _rounded(p, n_in, depth):
    """The parameters that the kernel sees: BF16 weights, FP32 biases."""
    out = p.astype(np.float64)
    for name, part in omlp.unpack(np.arange(len(p)), n_in, depth).items():
        if name[0] == "W":
            i = part.astype(np.int64).ravel()
            out[i] = torch.from_numpy(p[i]).bfloat16().double().numpy()
    return out


@pytest.mark.parametrize("depth", [2, 3])
@pytest.mark.parametrize("n_in", [3, 6, 12, 18, 21, 24])
@pytest.mark.parametrize("n", [1, 63, 64, 65, 20000])
def test_gradient(asd, depth, n_in, n):
    g = synth.rng(7)
    x = g.normal(size=(n, n_in)).astype(np.float32)
    y = synth.random_unit(n, 8)
    p = _params(asd, n_in, depth, 9)
    net = asd.Mlp(n_in, params=p, depth=depth)
    net.grad.fill_(1.0)      # the call adds to what is there
    net.loss.fill_(2.0)
    net.loss_grad(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda())
    torch.cuda.synchronize()
    w = _rounded(p, n_in, depth)
    loss, grad = omlp.nll(w, x, y, n_in, depth), omlp.grad(w, x, y, n_in, depth)
    got = net.grad.cpu().numpy().astype(np.float64) - 1.0
    scale = np.linalg.norm(grad)
    # FP32 sums of n terms, and the 1.0 that was there
    assert np.linalg.norm(got - grad) <= 3e-6 * scale + 1e-6 * np.sqrt(len(grad))
    assert abs(net.loss.item() - 2.0 - loss) <= 1e-6 * abs(loss) + 1e-6


def test_unaligned_weights(asd):
    n_in, depth, n = 12, 3, 500
    p = _params(asd, n_in, depth, 3)
    x = torch.from_numpy(synth.rng(4).normal(size=(n, n_in)).astype(np.float32)).cuda()
    y = torch.from_numpy(synth.random_unit(n, 5)).cuda()
    a = asd.Mlp(n_in, params=p, depth=depth)
    a.loss_grad(x, y)
    b = asd.Mlp(n_in, params=p, depth=depth)
    moved = torch.empty(b.wb.numel() + 1, dtype=torch.bfloat16, device="cuda")
    moved[1:] = b.wb
    shift = moved.data_ptr() + 2 - b.wb.data_ptr()
    for f in ("W1", "W2", "Wm", "W3"):
        setattr(b.c, f, getattr(b.c, f) + shift)
    b.loss_grad(x, y)
    torch.cuda.synchronize()
    torch.testing.assert_close(a.grad, b.grad, rtol=1e-4, atol=1e-3)
    assert abs(a.loss.item() - b.loss.item()) < 1e-9 * abs(a.loss.item())
