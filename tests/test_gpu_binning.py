"""Binning of the tensor-core epilogue against the plan's exact pair counts (counted by a
separate kernel with the two-sided threshold rule).  With every spin the same unit vector
each pair contributes exactly T0, so C_sum must equal counts * T0 to the last bit, on every
route: branch-free positions with computed or loaded thresholds, with and without dropped
pairs, one or two private windows, the general rule for coordinates outside the
branch-free range, and the byte-packed lattice distances."""
import numpy as np
import pytest
import torch

from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def asd():
    from paper_2308_07487_gb300 import asd as m
    return m


def _check(asd, N, T0, n_t, n_bins, **kw):
    F = T0 + n_t - 1
    tr = torch.from_numpy(synth.traj_static(N, F)).cuda()
    plan = asd.CorrPlan(N, F, T0, n_t, n_bins=n_bins, **kw)
    C = torch.zeros((n_t, n_bins), dtype=torch.float64, device="cuda")
    plan.run(tr, C)
    assert asd.sync_status() == 0
    want = plan.counts().astype(np.float64) * T0
    plan.close()
    for t in range(n_t):
        np.testing.assert_array_equal(C[t].cpu().numpy(), want)


@pytest.mark.parametrize("form", ["split_bf16", "bf16"])
@pytest.mark.parametrize("L,block,w,n_bins", [
    (9, None, 0.5, 32),                  # every bin kept and private, one ragged tile row
    (9, None, 0.7, 12),                  # loaded thresholds, dropped pairs
    (16, (4, 4, 8), 0.125, 226),         # private window, computed thresholds
    (16, (4, 4, 8), 0.1, 282),           # private window, loaded thresholds
    (16, (4, 4, 8), 0.125, 100),         # window and dropped pairs
    (24, (2, 2, 2), 0.0625, 700),        # two windows, and tiles that fit none
])
@pytest.mark.parametrize("jitter", [0.0, 0.1])   # 0: distances exactly on thresholds
def test_positions(asd, form, L, block, w, n_bins, jitter):
    lat = synth.hypercubic(L, 3, False, seed=5, block=block, jitter=jitter)
    _check(asd, lat.n_sites, 8, 2, n_bins, precision=form, pos=lat.pos, bin_width=w)


@pytest.mark.parametrize("bad", [3e19, np.inf, np.nan])
def test_positions_outside_the_fast_rule(asd, bad):
    lat = synth.hypercubic(9, 3, False, seed=5, jitter=0.1)
    pos = lat.pos.copy()
    pos[100, 1] = bad
    _check(asd, lat.n_sites, 8, 2, 12, precision="split_bf16", pos=pos, bin_width=0.5)


@pytest.mark.parametrize("L,dim,periodic,w,n_bins", [
    (255, 2, True, 1.0, 60), (254, 2, True, 0.7, 60), (128, 2, False, 1.0, 182),
    (10, 3, True, 0.5, 18), (11, 3, False, 0.5, 36), (11, 3, True, 0.7, 6)])
def test_lattices(asd, L, dim, periodic, w, n_bins):
    lat = synth.hypercubic(L, dim, periodic)
    _check(asd, lat.n_sites, 8, 1, n_bins, precision="bf16", coords=lat.coords, L=lat.L,
           periodic=periodic, bin_width=w)
