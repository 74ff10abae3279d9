"""FP32 form at the edges of its tiles and stages: row ranges that start on and off 16-byte
boundaries and end inside a tile, K = 3 T0 below, at and above whole stages of 16, several
samples, centring and phase sums, against the FP64 oracle at the form's bar."""
import numpy as np
import pytest
import torch

import oracle
from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def asd():
    from paper_2308_07487_gb300 import asd as m
    return m


@pytest.mark.parametrize("rows", [None, (1, 2), (1, 130), (2, 131), (3, 259), (4, 128), (127, 343)])
@pytest.mark.parametrize("T0,S,center", [(1, 1, False), (5, 2, True), (16, 1, False), (17, 3, True)])
def test_tiles(asd, rows, T0, S, center):
    lat = synth.hypercubic(7, 3, False, jitter=0.1, seed=3)
    n_t, w, nb = 3, 0.5, 12
    F = T0 + n_t - 1
    tr = synth.traj_precess(lat.n_sites, F, seed=5, S=S)
    q = np.array([[0.0, 0, 0], [0.3, 0.2, 0.1], [1.0, -0.4, 2.0]])
    plan = asd.CorrPlan.for_lattice(lat, F, T0, n_t, w, nb, precision="fp32", S=S, center=center,
                                    q=q, phase_sine=True)
    C = torch.zeros((n_t, nb), dtype=torch.float64, device="cuda")
    Sq = torch.zeros((n_t, len(q), 2), dtype=torch.float64, device="cuda")
    d = torch.from_numpy(np.ascontiguousarray(tr)).cuda()
    plan.run(d, C, Sq, rows=rows)
    assert asd.sync_status() == 0
    plan.close()
    ref = oracle.pair_corr(tr, T0, list(range(n_t)), oracle.Geometry.of_lattice(lat), w, nb, q=q,
                           rows=rows, center=center)
    assert oracle.rounding_ratio(C.cpu().numpy(), ref).max() <= 1e-6
    got = Sq.cpu().numpy()
    assert oracle.phase_error(got[..., 0], ref, "cos").max() <= 1e-5
    assert oracle.phase_error(got[..., 1], ref, "sin").max() <= 1e-5
