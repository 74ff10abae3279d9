"""asd_sq_omega makes its cosines in runs of 32 displacements: lengths at the edges of one and
several runs, against FP64 numpy."""
import numpy as np
import pytest
import torch

from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_t", [1, 2, 31, 32, 33, 64, 65, 4097])
@pytest.mark.parametrize("n_q", [1, 130])
def test_lengths(n_t, n_q):
    from paper_2308_07487_gb300 import asd
    g = synth.rng(n_t)
    S, om, dt = g.normal(size=(n_t, n_q)), g.uniform(0, 30, size=7), 0.1
    out = torch.zeros((7, n_q), dtype=torch.float64, device="cuda")
    asd.sq_omega(torch.from_numpy(S).cuda(), dt, torch.from_numpy(om).cuda(), out)
    assert asd.sync_status() == 0
    t = np.arange(n_t)
    v = 0.5 * (1 + np.cos(np.pi * t / n_t))
    w = np.where(t == 0, 1.0, 2.0) * v
    ref = dt * np.einsum("t,tq,kt->kq", w, S, np.cos(np.outer(om, t) * dt))
    # 32 rotations of a step add at most 32 rounding errors to a cosine, the phase itself
    # (up to 3 t) its own, the sum one per term
    tol = (64 + 3 * n_t + n_t) * 2.0 ** -53 * dt * np.abs(w[:, None] * S).sum(0).max() + 1e-300
    assert np.abs(out.cpu().numpy() - ref).max() <= 4 * tol
