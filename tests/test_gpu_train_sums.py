"""asd_mlp_loss_grad sums each 64-sample tile by itself before it joins its block's sums: a
block's later tiles keep their small terms beside a large one of its first tile."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth", [2, 3])
@pytest.mark.parametrize("n_in", [6, 12, 24])
def test_small_terms_after_a_large_one(depth, n_in):
    """Every sample has the same input, and the fourth output's weights are zero, so each
    gradient entry but that output's is linear in y.  Sample 0 has y = y0; the samples of
    every tile k * (number of SMs), k = 1 .. 64, have 2^-25 y0, exactly 2^-25 of its terms and
    below half a unit in the last place of them; all others have y = 0.  Blocks take tiles a
    multiple of the number of SMs apart, so block 0 meets the large term and small ones.
    Together the small terms are 64 * 64 * 2^-25 = 2^-13 of the large one; a tile's 64 are
    2^-19 of it, added with an error of at most 2^-24 of it per tile and per block sum: 2^-17
    leaves room for 128 additions, and a sum that drops the small terms is off by at least
    half of them, 2^-14."""
    from paper_2308_07487_gb300 import asd
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 64 * (64 * sms + 1)
    p = (0.25 * synth.rng(50).normal(size=omlp.n_params(n_in, depth))).astype(np.float32)
    idx = omlp.unpack(np.arange(len(p)), n_in, depth)
    last = np.concatenate([idx["W3"][3], idx["b3"][3:]]).astype(np.int64)
    p[last[:-1]] = 0.0
    x = torch.from_numpy(synth.rng(51).normal(size=n_in).astype(np.float32)).cuda().repeat(n, 1)
    y0 = torch.from_numpy(synth.random_unit(1, 52)[0]).cuda()
    grads = []
    for small in (False, True):
        y = torch.zeros((n // 64, 64, 3), device="cuda")
        y[0, 0] = y0
        if small:
            y[sms::sms] = y0 * 2.0 ** -25
        net = asd.Mlp(n_in, params=p, depth=depth)
        net.loss_grad(x, y.reshape(n, 3))
        assert asd.sync_status() == 0
        grads.append(np.delete(net.grad.cpu().numpy().astype(np.float64), last))
    big, both = grads
    assert np.count_nonzero(big) > 0.99 * len(big)
    assert (np.abs(both - big * (1 + 2.0 ** -13)) <= 2.0 ** -17 * np.abs(big)).all()
