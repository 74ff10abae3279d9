"""Glasses whose tiles span more bins than a thread's private window holds (sites in row order,
narrow bins): values go to private or shared bins pair by pair.  Exact and inexact widths, with
and without dropped pairs, every tile width and warp count that meets it, against the FP64
oracle, and counts of the pairs against the plan's."""
import numpy as np
import pytest
import torch

import oracle
from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = {"split_bf16": 1e-5, "bf16": 4 * 2.0 ** -8}
T0, NT = 10, 2


@pytest.fixture(scope="module", params=[11, 17])
def glass(request):
    L = request.param     # 1331 sites: 128-wide tiles; 4913: 256- or 192-wide
    lat = synth.hypercubic(L, 3, False, pm_j=True, p=0.5, seed=7, jitter=0.1)
    tr = synth.traj_precess(lat.n_sites, T0 + NT, seed=41)
    return lat, tr, {}


def _ref(glass, w, nb):
    lat, tr, refs = glass
    if (w, nb) not in refs:
        refs[w, nb] = oracle.pair_corr(tr, T0, list(range(NT)), oracle.Geometry.of_lattice(lat), w, nb)
    return refs[w, nb]


@pytest.mark.parametrize("form", ["split_bf16", "bf16"])
@pytest.mark.parametrize("w,nb", [(0.0625, 512), (0.07, 400), (0.07, 120), (0.125, 100)])
@pytest.mark.parametrize("n_q,det", [(0, False), (9, False), (0, True)])
def test_bins_outside_the_window(glass, form, w, nb, n_q, det):
    from paper_2308_07487_gb300 import asd
    lat, tr, _ = glass
    ref = _ref(glass, w, nb)
    d = torch.from_numpy(np.ascontiguousarray(tr)).cuda()
    q = synth.rng(3).normal(size=(n_q, 3)) if n_q else None
    plan = asd.CorrPlan.for_lattice(lat, T0 + NT, T0, NT, w, nb, precision=form, q=q,
                                    deterministic=det)
    assert np.array_equal(plan.counts(), ref["counts"])
    C = torch.zeros((NT, nb), dtype=torch.float64, device="cuda")
    S = torch.zeros((NT, n_q), dtype=torch.float64, device="cuda") if n_q else None
    plan.run(d, C, S)
    assert asd.sync_status() == 0
    assert oracle.bin_error(C.cpu().numpy(), ref).max() <= TOL[form]
    # a static trajectory of unit spins along z: every product sum is T0, so the bins count pairs
    one = torch.zeros((lat.n_sites, T0 + NT, 3), device="cuda")
    one[..., 2] = 1.0
    C.zero_()
    plan.run(one, C, S)
    assert asd.sync_status() == 0
    assert np.array_equal(C.cpu().numpy(), np.tile(T0 * ref["counts"].astype(np.float64), (NT, 1)))
    plan.close()
