"""asd_thermalize runs Metropolis and heat-bath sweeps in one block per sample, in one
cooperative launch, or with one launch per colour; every route does the same arithmetic.
With the caller's uniforms, copies of a lattice and finer colourings take other routes and
must give the same spins bit for bit; adaptive runs must agree on the cone and the counts."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def asd():
    from paper_2308_07487_gb300 import asd as m
    return m


def _copies(lat, k):
    """k disjoint copies of a lattice as one system, coloured like the original."""
    N = lat.n_sites
    o = (np.arange(k) * N)[:, None, None]
    nbr = np.where(lat.nbr[None] >= 0, lat.nbr[None] + o, -1).reshape(k * N, -1).astype(np.int32)

    def rep(x):
        return None if x is None else np.tile(x, (k,) + (1,) * (x.ndim - 1))
    colors = [(c[None] + np.arange(k)[:, None] * N).reshape(-1).astype(np.int32)
              for c in lat.colors]
    return dataclasses.replace(lat, coords=rep(lat.coords), nbr=nbr, J=rep(lat.J),
                               pos=rep(lat.pos), D=rep(lat.D), colors=colors)


LATS = {
    "square_z4": lambda: synth.hypercubic(10, 2, True),
    "glass_dm_z6": lambda: synth.with_dm_anisotropy(
        synth.hypercubic(5, 3, False, pm_j=True, seed=3), 0.3, 0.2),
    "chain_z2": lambda: synth.open_chain(97),
}


@pytest.mark.parametrize("name", list(LATS))
@pytest.mark.parametrize("proposal", ["metropolis", "cone", "heatbath"])
@pytest.mark.parametrize("sites", [4096, 5000, 40000, 400000])
def test_routes_agree(asd, name, proposal, sites):
    lat, sweeps, S = LATS[name](), 5, 2
    N = lat.n_sites
    k = -(-sites // N) if sites > 4096 else sites // N
    prop = asd.ASD_HEATBATH if proposal == "heatbath" else asd.ASD_METROPOLIS
    cone = 0.8 if proposal == "cone" else 0.0
    spins = synth.random_unit(S * N, 11).reshape(S, N, 3)
    u = synth.rng(3).random((sweeps, S, N, 4)).astype(np.float32)

    def run(lat, reps):
        sp = torch.from_numpy(np.tile(spins, (1, reps, 1))).cuda()
        un = torch.from_numpy(np.tile(u, (1, 1, reps, 1))).cuda()
        st = asd.System(lat).thermalize(sp, 0.7, sweeps, prop, cone=cone, uniforms=un, stats=True)
        assert asd.sync_status() == 0
        return sp.reshape(S, reps, N, 3), st
    ref, st = run(lat, 1)
    assert st[0] == sweeps * S * N and 0 < st[1] <= st[0]
    # more than 16 colours: one launch per colour
    fine = dataclasses.replace(lat, colors=[p.astype(np.int32) for c in lat.colors
                                            for p in np.array_split(c, 9)])
    got, st_fine = run(fine, 1)
    assert torch.equal(got, ref) and st_fine == st
    got, st_big = run(_copies(lat, k), k)
    assert torch.equal(got, ref.expand_as(got))
    assert st_big[:2] == (st[0] * k, st[1] * k)


@pytest.mark.parametrize("L,S", [(10, 1), (10, 3), (64, 1), (80, 2)])
def test_adaptive_cone(asd, L, S):
    """Adaptive runs: any route against one launch per colour (the same random numbers: the
    caller's), and a run cut in two calls against one."""
    lat = synth.hypercubic(L, 2, True)
    N, sweeps = lat.n_sites, 9
    spins = torch.from_numpy(synth.random_unit(S * N, 2).reshape(S, N, 3)).cuda()
    un = torch.from_numpy(synth.rng(4).random((sweeps, S, N, 4)).astype(np.float32)).cuda()
    fine = dataclasses.replace(lat, colors=[p.astype(np.int32) for c in lat.colors
                                            for p in np.array_split(c, 9)])
    out = []
    for la in (lat, fine):
        sp = spins.clone()
        st = asd.System(la).thermalize(sp, 0.4, sweeps, asd.ASD_METROPOLIS, adapt=True,
                                       uniforms=un, stats=True)
        out.append((sp, st))
    assert out[0][1] == out[1][1]
    assert torch.equal(out[0][0], out[1][0])
    sysm = asd.System(lat)
    a, b = spins.clone(), spins.clone()
    sysm.thermalize(a, 0.4, 8, asd.ASD_METROPOLIS, cone=0.5, seed=5, counter=3)
    for c in (0, 4):
        sysm.thermalize(b, 0.4, 4, asd.ASD_METROPOLIS, cone=0.5, seed=5, counter=3 + c)
    assert torch.equal(a, b)


def test_no_sweeps_and_long_runs(asd):
    """No sweeps leave the spins; a run longer than one launch equals two shorter ones."""
    for L in (8, 80):
        lat = synth.hypercubic(L, 2, True)
        sysm = asd.System(lat)
        spins = torch.from_numpy(synth.random_unit(lat.n_sites, 2)[None]).cuda()
        a = spins.clone()
        assert sysm.thermalize(a, 0.4, 0, asd.ASD_METROPOLIS, cone=0.3, stats=True)[:2] == (0, 0)
        assert torch.equal(a, spins)
        st = sysm.thermalize(a, 0.4, 5000, asd.ASD_HEATBATH, seed=1, stats=True)
        b = spins.clone()
        sysm.thermalize(b, 0.4, 3000, asd.ASD_HEATBATH, seed=1)
        sysm.thermalize(b, 0.4, 2000, asd.ASD_HEATBATH, seed=1, counter=3000)
        assert torch.equal(a, b) and st[0] == 5000 * lat.n_sites
