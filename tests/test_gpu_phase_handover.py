"""Phase sums without bins: the epilogue then only converts a tile to BF16, far quicker than
the operands and phase weights arrive, so it runs as far ahead of the phase product as the
barriers between them let it.  One and two passes of q-vectors, one and two K chunks, both
tile widths with a phase product, CTA pairs, and batches that change problem at every hand-over,
against the FP64 oracle, several times over."""
import numpy as np
import pytest
import torch

import oracle
from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu

# BF16 operand rounding (2^-8 each); FP32-accurate split form
TOL = {"split_bf16": 1e-5, "tf32": 4 * 2.0 ** -11, "bf16": 4 * 2.0 ** -8}
T0, NT = 8, 4


@pytest.fixture(scope="module")
def asd():
    from paper_2308_07487_gb300 import asd as m
    return m


def _q(n):
    return synth.q_vectors_glass()[::5] if n == 13 else synth.rng(5).normal(size=(n, 3))


@pytest.fixture(scope="module")
def problem():
    """4225 sites in two dimensions (192-wide tiles by default), 1000 rows from mid-tile:
    more than five work items of one K block each per SM."""
    lat = synth.hypercubic(65, 2, False)
    tr = synth.traj_precess(lat.n_sites, T0 + NT, seed=81)
    rows = (70, 1070)
    ref = {n: oracle.pair_corr(tr, T0, list(range(NT)), oracle.Geometry.of_lattice(lat), 1.0, 1,
                               q=_q(n), rows=rows) for n in (13, 70)}
    return lat, tr, rows, ref


@pytest.mark.parametrize("form", ["split_bf16", "bf16", "tf32"])
@pytest.mark.parametrize("n_q", [13, 70])
@pytest.mark.parametrize("knobs", [dict(tile_n=192), dict(tile_n=128), dict(k_chunks=2),
                                   dict(cta_pair=True), dict(epi_warps=8, tile_n=192)],
                         ids=["192", "128", "chunks2", "pair", "warps8"])
def test_phase_only(asd, problem, form, n_q, knobs):
    lat, tr, rows, refs = problem
    ref = refs[n_q]
    # (a K block is 32 or 64 elements: two chunks need two samples of 24)
    d = torch.from_numpy(np.ascontiguousarray(tr)).cuda()
    if "k_chunks" in knobs:
        d = torch.stack([d, d], dim=1).contiguous()
    plan = asd.CorrPlan.for_lattice(lat, T0 + NT, T0, NT, 1.0, 0, precision=form, q=_q(n_q),
                                    S=2 if "k_chunks" in knobs else 1, **knobs)
    scale = 2.0 if "k_chunks" in knobs else 1.0
    for _ in range(5):
        S = torch.zeros((NT, n_q), dtype=torch.float64, device="cuda")
        plan.run(d, None, S, rows=rows)
        assert asd.sync_status() == 0
        assert oracle.phase_error(S.cpu().numpy() / scale, ref).max() <= TOL[form]
    plan.close()


@pytest.mark.parametrize("form", ["split_bf16", "bf16"])
def test_mixed_batch(asd, form):
    """Problems with q-vectors only, bins only, and both, so that successive work items of a CTA
    release their accumulators in different ways."""
    plans, trajs, Cs, Ss, refs = [], [], [], [], []
    for k in range(9):
        lat = synth.hypercubic(14 + 2 * k, 2, True)
        nb, n_q = [(0, 13), (9, 0), (9, 13)][k % 3]
        tr = synth.traj_precess(lat.n_sites, T0 + NT, seed=90 + k)
        q = _q(13) if n_q else None
        plans.append(asd.CorrPlan.for_lattice(lat, T0 + NT, T0, NT, 1.0, nb, precision=form, q=q,
                                              tile_n=128))
        trajs.append(torch.from_numpy(np.ascontiguousarray(tr[:, None])).cuda())
        Cs.append(torch.zeros((NT, nb), dtype=torch.float64, device="cuda") if nb else None)
        Ss.append(torch.zeros((NT, n_q), dtype=torch.float64, device="cuda") if n_q else None)
        refs.append(oracle.pair_corr(tr, T0, list(range(NT)), oracle.Geometry.of_lattice(lat), 1.0,
                                     max(nb, 1), q=q))
    for _ in range(5):
        for x in Cs + Ss:
            if x is not None:
                x.zero_()
        asd.pair_corr_batched(plans, trajs, Cs, Ss)
        assert asd.sync_status() == 0
        for C, S, ref in zip(Cs, Ss, refs):
            if C is not None:
                assert oracle.bin_error(C.cpu().numpy(), ref).max() <= TOL[form]
            if S is not None:
                assert oracle.phase_error(S.cpu().numpy(), ref).max() <= TOL[form]
    for p in plans:
        p.close()
