"""asd_ll_integrate with any number of bonds per site (they are read in groups): tables of
random neighbours with empty slots and DM vectors, on the routes that exchange spins through
global memory, against the block route bit for bit and against FP64."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import dynamics
from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dm", [False, True])
@pytest.mark.parametrize("z", [1, 3, 5, 7, 8, 13, 26, 32])
@pytest.mark.parametrize("sites", [2500, 20000, 170000])
def test_any_number_of_bonds(z, dm, sites):
    from paper_2308_07487_gb300 import asd
    N, F, stride = 100, 5, 2
    k = -(-sites // N)
    g = synth.rng(z)
    nbr = g.integers(0, N, size=(N, z)).astype(np.int32)
    nbr[g.random((N, z)) < 0.15] = -1
    J = g.normal(size=(N, z)).astype(np.float32) / np.float32(z)
    D = (0.3 * g.normal(size=(N, z, 3)) / z).astype(np.float32) if dm else None
    lat = dataclasses.replace(synth.open_chain(N), nbr=nbr, J=J, D=D, A=0.2, Hz=0.1)
    o = (np.arange(k) * N)[:, None, None]
    big = dataclasses.replace(lat, nbr=np.where(nbr >= 0, nbr + o, -1).reshape(k * N, z).astype(np.int32),
                              J=np.tile(J, (k, 1)), D=None if D is None else np.tile(D, (k, 1, 1)),
                              coords=np.tile(lat.coords, (k, 1)), pos=np.tile(lat.pos, (k, 1)),
                              colors=[np.arange(k * N, dtype=np.int32)])
    s0 = synth.random_unit(N, 3)
    out = []
    for la, n in ((lat, 1), (big, k)):
        sp = torch.from_numpy(np.tile(s0, (n, 1))[None]).cuda()
        tr = torch.empty((n * N, 1, F, 3), device="cuda")
        asd.System(la).ll_integrate(sp, 0.05, F, stride, tr)
        assert asd.sync_status() == 0
        out.append(tr.reshape(n, N, F, 3))
    assert torch.equal(out[1], out[0].expand_as(out[1]))
    r64 = dynamics.ll_rk4(s0[None].astype(np.float64), nbr, J, 0.1, 0.05, F, stride, D=D, A=0.2)
    assert np.abs(out[0][0].cpu().numpy() - np.asarray(r64).reshape(N, F, 3)).max() < 5e-6
