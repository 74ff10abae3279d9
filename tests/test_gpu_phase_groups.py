"""Phase sums are read out eight q-vectors at a time: counts at the edges of those groups, of half
passes (32) and of passes (64), with and without the sine part and bins, against the FP64
oracle.  Without bins no tile geometry is made, so plans with and without bins also run in turn
in one batch."""
import numpy as np
import pytest
import torch

import oracle
from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = {"split_bf16": 1e-5, "bf16": 4 * 2.0 ** -8}
T0, NT, L = 20, 3, 20


@pytest.fixture(scope="module")
def problem():
    lat = synth.hypercubic(L, 2, False)
    tr = synth.traj_precess(lat.n_sites, T0 + NT, seed=61)
    q = synth.rng(62).normal(size=(130, 3))
    ref = oracle.pair_corr(tr, T0, list(range(NT)), oracle.Geometry.of_lattice(lat), 1.0, 12, q=q)
    return lat, tr, q, ref


def _cut(ref, n):
    return {k: v[:, :n] if k in ("Sq_sum", "Sq_im", "Sq_abs", "Sq_im_abs") else v
            for k, v in ref.items()}


@pytest.mark.parametrize("form", ["split_bf16", "bf16"])
@pytest.mark.parametrize("n_q", [1, 7, 8, 9, 24, 25, 31, 32, 33, 56, 57, 63, 64, 65, 72, 97, 128, 130])
@pytest.mark.parametrize("nb,sine", [(0, False), (0, True), (12, True)])
def test_groups(problem, form, n_q, nb, sine):
    from paper_2308_07487_gb300 import asd
    lat, tr, q, ref = problem
    d = torch.from_numpy(np.ascontiguousarray(tr)).cuda()
    plan = asd.CorrPlan.for_lattice(lat, T0 + NT, T0, NT, 1.0, nb, precision=form, q=q[:n_q],
                                    phase_sine=sine)
    C = torch.zeros((NT, nb), dtype=torch.float64, device="cuda") if nb else None
    S = torch.zeros((NT, n_q, 1 + sine), dtype=torch.float64, device="cuda")
    plan.run(d, C, S)
    assert asd.sync_status() == 0
    cut, got = _cut(ref, n_q), S.cpu().numpy()
    assert oracle.phase_error(got[..., 0], cut).max() <= TOL[form]
    if sine:
        assert oracle.phase_error(got[..., 1], cut, "sin").max() <= TOL[form]
    if nb:
        assert oracle.bin_error(C.cpu().numpy(), ref).max() <= TOL[form]
    plan.close()


def test_batch_with_and_without_bins(problem):
    from paper_2308_07487_gb300 import asd
    lat, tr, q, ref = problem
    d = torch.from_numpy(np.ascontiguousarray(tr)).cuda()
    shapes = [(12, 0), (0, 9), (12, 9), (0, 64), (12, 0), (0, 1), (12, 33)] * 3
    plans = [asd.CorrPlan.for_lattice(lat, T0 + NT, T0, NT, 1.0, nb, q=q[:nq] if nq else None)
             for nb, nq in shapes]
    C = [torch.zeros((NT, nb), dtype=torch.float64, device="cuda") if nb else None
         for nb, _ in shapes]
    S = [torch.zeros((NT, nq), dtype=torch.float64, device="cuda") if nq else None
         for _, nq in shapes]
    asd.pair_corr_batched(plans, [d] * len(plans), C, S)
    assert asd.sync_status() == 0
    for (nb, nq), c, s in zip(shapes, C, S):
        if nb:
            assert oracle.bin_error(c.cpu().numpy(), ref).max() <= 1e-5
        if nq:
            assert oracle.phase_error(s.cpu().numpy(), _cut(ref, nq)).max() <= 1e-5
    for p in plans:
        p.close()
