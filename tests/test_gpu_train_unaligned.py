"""asd_mlp_loss_grad with weight matrices that start off a 16-byte boundary, one at a time and
all together, against FP64 back-propagation.  A call with other weights of the same shape, on
every SM, goes before each one, so that shared memory left over from it is of no help."""
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


def _params(n_in, depth, seed):
    """BF16-representable weights and FP32 biases."""
    p = (0.25 * synth.rng(seed).normal(size=omlp.n_params(n_in, depth))).astype(np.float32)
    return torch.from_numpy(p).bfloat16().float().numpy()


def _xy(n, n_in, seed):
    return (synth.rng(seed).normal(size=(n, n_in)).astype(np.float32),
            synth.random_unit(n, seed + 1))


@pytest.mark.parametrize("depth", [2, 3])
@pytest.mark.parametrize("n_in", [6, 12, 18, 24])
@pytest.mark.parametrize("which", ["W1", "W2", "Wm", "W3", "all"])
def test_shifted_weights(asd, depth, n_in, which):
    if which == "Wm" and depth == 2:
        pytest.skip("two layers have no third matrix")
    n = 500
    other = asd.Mlp(n_in, params=_params(n_in, depth, 30), depth=depth)
    ox, oy = _xy(64 * 4 * torch.cuda.get_device_properties(0).multi_processor_count, n_in, 31)
    other.loss_grad(torch.from_numpy(ox).cuda(), torch.from_numpy(oy).cuda())

    p = _params(n_in, depth, 40)
    x, y = _xy(n, n_in, 41)
    net = asd.Mlp(n_in, params=p, depth=depth)
    moved = torch.empty(net.wb.numel() + 1, dtype=torch.bfloat16, device="cuda")
    moved[1:] = net.wb
    shift = moved.data_ptr() + 2 - net.wb.data_ptr()
    for f in ("W1", "W2", "W3") + (("Wm",) if depth == 3 else ()):
        if which in (f, "all"):
            setattr(net.c, f, getattr(net.c, f) + shift)
            assert getattr(net.c, f) % 16 != 0
    net.loss_grad(torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda())
    assert asd.sync_status() == 0
    loss, grad = omlp.nll(p, x, y, n_in, depth), omlp.grad(p, x, y, n_in, depth)
    # FP32 sums of 500 terms (the bounds that aligned weights are held to)
    got = net.grad.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - grad) <= 3e-6 * np.linalg.norm(grad)
    assert abs(net.loss.item() - loss) <= 1e-6 * abs(loss) + 1e-6
