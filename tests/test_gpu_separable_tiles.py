"""Separable phase transform over its tile shapes and copy widths: q counts on both sides of
the tile heights, site counts on both sides of a slice of 4096 and a stage of 16, rows that
start on and off 16 bytes, several samples, against an FP64 transform."""
import numpy as np
import pytest
import torch

from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def asd():
    from paper_2308_07487_gb300 import asd as m
    return m


@pytest.mark.parametrize("N,n_q", [(1, 1), (15, 3), (17, 16), (4095, 17), (4097, 33), (9000, 48),
                                   (9000, 64), (4100, 65), (700, 250), (70000, 64)])
@pytest.mark.parametrize("F,T0,S,sine,center", [(8, 5, 1, False, False), (9, 7, 2, True, True),
                                                (640, 512, 1, False, False),
                                                (333, 200, 1, True, False)])
def test_tiles(asd, N, n_q, F, T0, S, sine, center):
    if N * F * S > 5_000_000 and F != 333:
        pytest.skip("one long case per size")
    g = synth.rng(N + n_q)
    pos = (g.random((N, 3)) * 20).astype(np.float32)
    q = g.normal(size=(n_q, 3))
    n_t = min(F - T0 + 1, 11)
    tr = torch.randn((N, S, F, 3), device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    plan = asd.CorrPlan(N, F, T0, n_t, S=S, pos=pos, q=q, phase_sine=sine, center=center)
    out = torch.full((n_t, n_q, 1 + sine), 0.5, dtype=torch.float64, device="cuda")
    plan.sq_separable(tr, out)
    assert asd.sync_status() == 0
    plan.close()
    ph = torch.from_numpy(pos).cuda().double() @ torch.from_numpy(q).cuda().T
    X = tr.double().reshape(N, -1)
    Fc, Fs = ((f(ph).T @ X).reshape(n_q, S, F, 3) for f in (torch.cos, torch.sin))
    mag = ((torch.cos(ph).abs() + torch.sin(ph).abs()).T @ X.abs()).reshape(n_q, S, F, 3)
    Bc, Bs = Fc[:, :, :T0], Fs[:, :, :T0]
    if center:
        Bc, Bs = (b - b.mean(dim=(1, 2), keepdim=True) for b in (Bc, Bs))
    for t in range(n_t):
        Ac, As = Fc[:, :, t:t + T0], Fs[:, :, t:t + T0]
        want = [(Ac * Bc + As * Bs).sum((1, 2, 3))] + [(As * Bc - Ac * Bs).sum((1, 2, 3))] * sine
        # FP32 sums of up to 4096 terms per transform: 4e-6 of the sums of magnitudes, with
        # the other factor's size
        size = (mag[:, :, t:t + T0] * (Bc.abs() + Bs.abs())
                + mag[:, :, :T0] * (Ac.abs() + As.abs())).sum((1, 2, 3)) + 1e-12
        for part, w in enumerate(want):
            assert ((out[t, :, part] - 0.5 - w).abs() / size).max() < 4e-6
