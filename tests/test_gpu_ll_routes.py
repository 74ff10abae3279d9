"""asd_ll_integrate chooses by size between one block per sample, a cooperative launch with
one, two or four sites per thread, and one launch per stage; every route does the same
arithmetic, so disjoint copies of one lattice must follow the same trajectory bit for bit
whichever route the copied system takes, and that trajectory is checked against FP64."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import dynamics
from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def asd():
    from paper_2308_07487_gb300 import asd as m
    return m


def _copies(lat, k):
    """k disjoint copies of a lattice as one system of k N sites."""
    N = lat.n_sites
    o = (np.arange(k) * N)[:, None, None]
    nbr = np.where(lat.nbr[None] >= 0, lat.nbr[None] + o, -1).reshape(k * N, -1).astype(np.int32)

    def rep(x):
        return None if x is None else np.tile(x, (k,) + (1,) * (x.ndim - 1))
    return dataclasses.replace(lat, coords=rep(lat.coords), nbr=nbr, J=rep(lat.J),
                               pos=rep(lat.pos), D=rep(lat.D),
                               colors=[np.arange(k * N, dtype=np.int32)])


def _run(asd, lat, s0, S, F, stride, alias=False):
    sysm = asd.System(lat)
    traj = torch.empty((lat.n_sites, S, F, 3), device="cuda")
    out = s0 if alias else torch.empty_like(s0)
    sysm.ll_integrate(s0, 0.02, F, stride, traj, spins_out=out)
    assert asd.sync_status() == 0
    return traj, out


LATS = {
    "square_z4": lambda: synth.hypercubic(10, 2, True),
    "cubic_dm_z6": lambda: synth.with_dm_anisotropy(synth.hypercubic(5, 3, False, pm_j=True,
                                                                     seed=3), 0.3, 0.2),
    "chain_z2": lambda: synth.open_chain(97),
}


@pytest.mark.parametrize("name", list(LATS))
@pytest.mark.parametrize("sites", [1024, 1025, 2048, 2049, 5000, 170000, 330000, 640000])
def test_routes_agree(asd, name, sites):
    lat = LATS[name]()
    N, F, stride, S = lat.n_sites, 7, 2, 2 if sites < 10000 else 1
    k = -(-sites // N)
    spins = synth.random_unit(S * N, 11).reshape(S, N, 3)
    ref, ref_out = _run(asd, lat, torch.from_numpy(spins).cuda(), S, F, stride)
    big = torch.from_numpy(np.tile(spins, (1, k, 1))).cuda()
    traj, out = _run(asd, _copies(lat, k), big, S, F, stride)
    traj = traj.reshape(k, N, S, F, 3)
    assert torch.equal(traj, ref[None].expand_as(traj))
    out = out.reshape(S, k, N, 3)
    assert torch.equal(out, ref_out[:, None].expand_as(out))
    r64 = dynamics.ll_rk4(spins.astype(np.float64), lat.nbr, lat.J, lat.Hz, 0.02, F, stride,
                          D=lat.D, A=lat.A)
    assert np.abs(ref.cpu().numpy() - r64).max() < 5e-6


@pytest.mark.parametrize("copies", [1, 30])
@pytest.mark.parametrize("F,stride", [(1, 1), (2, 5000), (4100, 1)])
def test_long_and_empty_runs(asd, copies, F, stride):
    """Runs are cut into launches of 4096 steps; the final state may overwrite the start."""
    lat = synth.hypercubic(9, 2, True)
    lat_k = _copies(lat, copies)
    spins = torch.from_numpy(np.tile(synth.random_unit(lat.n_sites, 5), (copies, 1))).cuda()
    traj, out = _run(asd, lat_k, spins.clone()[None], 1, F, stride)
    traj2, out2 = _run(asd, lat_k, spins.clone()[None], 1, F, stride, alias=True)
    assert torch.equal(out, out2) and torch.equal(traj, traj2)
    assert torch.equal(traj[:, 0, 0], spins)
    if stride == 1:
        assert torch.equal(traj[:, 0, -1], out[0])
    norm = out.double().norm(dim=-1)
    assert (norm - 1).abs().max() < 1e-3
    one = traj.reshape(copies, -1, F, 3)
    assert torch.equal(one, one[:1].expand_as(one))
