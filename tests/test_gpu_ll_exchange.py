"""The cooperative one-site-per-thread route of asd_ll_integrate exchanges stage inputs between
blocks as words that carry their stage number.  Which neighbours a block finds in its own
shared memory and which it waits for depends on the site numbering only, so a randomly
renumbered lattice (nearly every bond crosses blocks) must follow the same trajectory bit for
bit, with as many buffers as the call's work area holds (asd_ll_integrate_noalloc has fewer at
the large end), over several launches, and stay bitwise repeatable."""
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


def _renumbered(lat, p):
    """Site i becomes site p[i]; the order of its bonds stays."""
    def move(x):
        if x is None:
            return None
        y = np.empty_like(x)
        y[p] = x
        return y
    nbr = np.where(lat.nbr >= 0, p[lat.nbr], -1).astype(np.int32)
    return dataclasses.replace(lat, coords=move(lat.coords), nbr=move(nbr), J=move(lat.J),
                               pos=move(lat.pos), D=move(lat.D),
                               colors=[np.arange(lat.n_sites, dtype=np.int32)])


def _run(asd, lat, spins, S, F, stride, noalloc=False):
    sysm = asd.System(lat)
    s0 = torch.from_numpy(spins).cuda()
    traj = torch.empty((lat.n_sites, S, F, 3), device="cuda")
    out = torch.empty_like(s0)
    (sysm.ll_integrate_noalloc if noalloc else sysm.ll_integrate)(s0, 0.02, F, stride, traj,
                                                                   spins_out=out)
    assert asd.sync_status() == 0
    return traj, out


CASES = {
    "square_z4": (lambda: synth.hypercubic(75, 2, True), 2, 7, 2),
    "cubic_z6": (lambda: synth.hypercubic(18, 3, True), 1, 7, 2),
    "cubic_dm_z6": (lambda: synth.with_dm_anisotropy(
        synth.hypercubic(14, 3, False, pm_j=True, seed=3), 0.3, 0.2), 1, 7, 2),
    "chain_z2": (lambda: synth.open_chain(3001), 3, 9, 1),
    "cubic_large": (lambda: synth.hypercubic(53, 3, True), 1, 6, 3),
    "two_launches": (lambda: synth.hypercubic(47, 2, True), 1, 2, 4100),
}


@pytest.mark.parametrize("name", list(CASES))
def test_renumbered_sites_follow_the_same_trajectory(asd, name):
    make, S, F, stride = CASES[name]
    lat = make()
    N = lat.n_sites
    p = np.random.default_rng(8).permutation(N)
    spins = synth.random_unit(S * N, 11).reshape(S, N, 3)
    moved = np.empty_like(spins)
    moved[:, p] = spins
    traj, out = _run(asd, lat, spins, S, F, stride)
    lat_p = _renumbered(lat, p)
    tp = torch.from_numpy(p).cuda()
    for noalloc in (False, True, True):
        traj_p, out_p = _run(asd, lat_p, moved, S, F, stride, noalloc)
        assert torch.equal(traj_p[tp], traj)
        assert torch.equal(out_p[:, tp], out)
