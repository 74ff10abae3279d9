"""asd_thermalize at the sizes where its rules for a route change: many samples of a few sites, one
sweep or several of more sites than the device takes at once, many bonds, one colour.  Each is
compared, sample by sample, with a call of few samples (the caller's uniforms)."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu


def _random_bonds(N, z, dm):
    """Two colours; every site has z neighbours of the other colour."""
    g = synth.rng(z)
    half = N // 2
    other = np.where(np.arange(N) < half, half, 0)[:, None]
    nbr = (other + g.integers(0, half, size=(N, z))).astype(np.int32)
    nbr[g.random((N, z)) < 0.1] = -1
    D = (0.2 * g.normal(size=(N, z, 3))).astype(np.float32) if dm else None
    return dataclasses.replace(synth.open_chain(N), nbr=nbr,
                               J=g.normal(size=(N, z)).astype(np.float32), D=D,
                               colors=[np.arange(half, dtype=np.int32),
                                       np.arange(half, N, dtype=np.int32)])


def _one_colour(N):
    lat = synth.open_chain(N)
    return dataclasses.replace(lat, nbr=np.full((N, 2), -1, np.int32),
                               colors=[np.arange(N, dtype=np.int32), np.zeros(0, np.int32)])


# lattice, samples per SM (plus a ragged rest)
CASES = {
    "one_site": (lambda: synth.open_chain(1), 40),
    "five_sites": (lambda: synth.open_chain(5), 40),
    "warp_per_colour": (lambda: synth.open_chain(64), 40),
    "filled_small": (lambda: synth.hypercubic(16, 2, True), 9),
    "filled_2500": (lambda: synth.hypercubic(50, 2, True), 1),
    "filled_many": (lambda: synth.hypercubic(50, 2, True), 5),
    "bonds_9": (lambda: _random_bonds(200, 9, False), 9),
    "bonds_7_dm": (lambda: _random_bonds(200, 7, True), 9),
    "bonds_8": (lambda: _random_bonds(200, 8, False), 9),
    "one_colour": (lambda: _one_colour(300), 4),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("sweeps", [1, 3])
@pytest.mark.parametrize("proposal", ["cone", "heatbath"])
def test_rules(name, sweeps, proposal):
    from paper_2308_07487_gb300 import asd
    make, per_sm = CASES[name]
    lat = make()
    N, few = lat.n_sites, 7
    S = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + 3
    sysm = asd.System(lat)
    prop = asd.ASD_HEATBATH if proposal == "heatbath" else asd.ASD_METROPOLIS
    spins = torch.from_numpy(synth.random_unit(few * N, 11).reshape(few, N, 3)).cuda()
    u = torch.from_numpy(synth.rng(3).random((sweeps, few, N, 4)).astype(np.float32)).cuda()
    pick = torch.arange(S, device="cuda") * 3 % few
    ref, many = spins.clone(), spins[pick].contiguous()
    each = []
    for s in range(few):
        st = sysm.thermalize(ref[s], 0.7, sweeps, prop, cone=0.8,
                             uniforms=u[:, s].contiguous(), stats=True)
        assert st[0] == sweeps * N
        each.append(st[1])
    st = sysm.thermalize(many, 0.7, sweeps, prop, cone=0.8, uniforms=u[:, pick].contiguous(),
                         stats=True)
    assert asd.sync_status() == 0
    assert torch.equal(many, ref[pick])
    assert st[:2] == (sweeps * N * S, sum(each[int(p)] for p in pick.cpu()))
