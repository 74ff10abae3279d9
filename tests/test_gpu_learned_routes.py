"""The learned proposal's kernel takes one or two sites per thread and the first layer's rows
padded to 12, 20 or 24 inputs.  With the caller's uniforms, copies of a system on either side of
the line between one and two sites (an odd number of sites per colour, so that a thread has only
one) must give the same spins bit for bit, and each colour's update is restated in FP64."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import dynamics, mlp as omlp
from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu

N, HALF, T = 99, 50, 0.8   # 50 and 49 sites per colour


def _system(z):
    """z random neighbours of the other colour per site, some absent."""
    g = synth.rng(z)
    first = np.arange(N) < HALF
    nbr = np.where(first[:, None], HALF + g.integers(0, N - HALF, size=(N, z)),
                   g.integers(0, HALF, size=(N, z))).astype(np.int32)
    nbr[g.random((N, z)) < 0.1] = -1
    J = np.where(nbr >= 0, g.normal(size=(N, z)), 0).astype(np.float32)
    return dataclasses.replace(synth.open_chain(N), nbr=nbr, J=J, Hz=0.2,
                               colors=[np.arange(HALF, dtype=np.int32),
                                       np.arange(HALF, N, dtype=np.int32)])


def _copies(lat, k):
    o = (np.arange(k) * N)[:, None, None]
    return dataclasses.replace(
        lat, nbr=np.where(lat.nbr >= 0, lat.nbr + o, -1).reshape(k * N, -1).astype(np.int32),
        J=np.tile(lat.J, (k, 1)), coords=np.tile(lat.coords, (k, 1)), pos=np.tile(lat.pos, (k, 1)),
        colors=[(c + o[:, :, 0]).reshape(-1).astype(np.int32) for c in lat.colors])


def _update(Y, lat, sites, u, p, depth):
    """FP64 move of `sites` of Y [N][3]: new spins, and which of them are decided clearly."""
    z = lat.nbr.shape[1]
    x = np.where(lat.nbr[sites][..., None] >= 0, Y[lat.nbr[sites]], 0.0).reshape(len(sites), 3 * z)
    mu, kappa, (_, _, o, vn) = omlp.forward(p, x, 3 * z, depth)
    h = dynamics.local_field(Y[None], lat.nbr, lat.J, lat.Hz)[0, sites]
    old = Y[sites]
    new = dynamics.around(mu, dynamics.vmf_w(kappa, u[:, 0]), 2 * np.pi * u[:, 1])
    la = -((new - old) * h).sum(-1) / T + kappa * ((old - new) * mu).sum(-1)
    pr = np.exp(np.minimum(la, 0.0))
    # (a small output vector, the switch of the frame at 0.9 and a near-even decision magnify
    # the FP32 forward pass's rounding)
    clear = (vn > 0.05) & (np.abs(np.abs(mu[:, 2]) - 0.9) > 1e-3) & (np.abs(u[:, 2] - pr) > 2e-3)
    return np.where((u[:, 2] < pr)[:, None], new, old), clear


@pytest.mark.parametrize("depth", [2, 3])
@pytest.mark.parametrize("z", [1, 2, 4, 5, 6, 7, 8])
def test_one_and_two_sites_per_thread(z, depth):
    from paper_2308_07487_gb300 import asd
    lat = _system(z)
    p = torch.from_numpy((0.3 * synth.rng(70).normal(size=omlp.n_params(3 * z, depth))).astype(
        np.float32)).bfloat16().float().numpy()
    spins = synth.random_unit(N, 71)
    u = synth.rng(72).random((1, 1, N, 4)).astype(np.float32)
    line = 256 * torch.cuda.get_device_properties(0).multi_processor_count   # sites per colour
    out = []
    for k in (1, line // HALF - 2, line // HALF + 2 | 1):   # the last: odd, 49 k sites odd too
        sp = torch.from_numpy(np.tile(spins, (k, 1))[None]).cuda()
        un = torch.from_numpy(np.tile(u, (1, 1, k, 1))).cuda()
        st = asd.System(_copies(lat, k)).thermalize(sp, T, 1, asd.ASD_LEARNED,
                                                    net=asd.Mlp(3 * z, params=p, depth=depth),
                                                    uniforms=un, stats=True)
        assert asd.sync_status() == 0
        assert st[0] == k * N
        out.append(sp.reshape(k, N, 3))
    for o in out[1:]:
        assert torch.equal(o, out[0].expand_as(o))
    got = out[0][0].cpu().numpy().astype(np.float64)
    Y = spins.astype(np.float64)
    for sites in lat.colors:
        new, clear = _update(Y, lat, sites, u[0, 0, sites].astype(np.float64), p, depth)
        assert clear.mean() > 0.8
        assert np.abs(got[sites] - new)[clear].max() < 1e-3
        assert (new[clear] != Y[sites][clear]).any()
        Y[sites] = got[sites]
