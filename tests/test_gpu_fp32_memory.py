"""FP32 plans keep a copy of the trajectory by K where the device has room for it; without room
they read the trajectory itself.  Both must give the same sums bit for bit (deterministic mode)
over ragged rows, samples, centring and phase weights; and a plan of few sites must not pay for
whole tiles of them."""
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


@pytest.mark.parametrize("center", [False, True])
def test_plan_without_room_for_its_copy(asd, center):
    lat = synth.open_chain(602)
    S, F, T0, n_t, nb = 2, 20000, 45, 3, 40   # K = 135 per sample: a ragged last stage
    q = synth.rng(2).normal(size=(5, 3))
    copy = 4 * 604 * S * 3 * F                # 290 MB
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    tr = torch.randn((602, S, F, 3), generator=gen, device="cuda")

    def plan():
        return asd.CorrPlan.for_lattice(lat, F, T0, n_t, 1.0, nb, precision="fp32", S=S, q=q,
                                        center=center, phase_sine=True, deterministic=True)

    def run(p, rows):
        C = torch.zeros((n_t, nb), dtype=torch.float64, device="cuda")
        Q = torch.zeros((n_t, 5, 2), dtype=torch.float64, device="cuda")
        p.run(tr, C, Q, rows=rows)
        assert asd.sync_status() == 0
        return C, Q
    full = plan()
    ranges = [(0, 602), (1, 602), (3, 130), (128, 257), (601, 602)]
    want = [run(full, r) for r in ranges]
    big = full.workspace_bytes()
    assert big >= copy
    full.close()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    ballast = torch.empty(free - 160 * 2 ** 20, dtype=torch.uint8, device="cuda")
    try:
        direct = plan()
    finally:
        del ballast
        torch.cuda.empty_cache()
    assert direct.workspace_bytes() <= big - copy
    for r, (C, Q) in zip(ranges, want):
        c, s = run(direct, r)
        assert torch.equal(c, C) and torch.equal(s, Q)
    if not center:
        few = np.ascontiguousarray(tr[:, :, :T0 + n_t].cpu().numpy())
        ref = oracle.pair_corr(few, T0, list(range(n_t)), oracle.Geometry.of_lattice(lat), 1.0,
                               nb, q=q, rows=(3, 130))
        c, s = run(direct, (3, 130))
        assert oracle.rounding_ratio(c.cpu().numpy(), ref).max() <= 1e-6
        assert oracle.phase_error(s[..., 0].cpu().numpy(), ref).max() <= 1e-5
    direct.close()


@pytest.mark.parametrize("N", [1, 2, 5, 127, 1030])
def test_few_sites(asd, N):
    """Workspace in proportion to the sites, and the sums of a system smaller than a tile (and of
    one whose rows are whole lines but not whole tiles)."""
    lat = synth.open_chain(N)
    S, F, T0, n_t, nb = 3, 50, 20, 4, 6
    tr = synth.traj_precess(N, F, seed=3, S=S)
    p = asd.CorrPlan.for_lattice(lat, F, T0, n_t, 1.0, nb, precision="fp32", S=S)
    up = (N + 3) // 4 * 4 if N < 1024 else (N + 31) // 32 * 32
    assert p.workspace_bytes() <= 4 * up * (S * 3 * F + S * 64) + 12 * N + 3 * 256
    C = torch.zeros((n_t, nb), dtype=torch.float64, device="cuda")
    p.run(torch.from_numpy(np.ascontiguousarray(tr)).cuda(), C)
    assert asd.sync_status() == 0
    ref = oracle.pair_corr(tr, T0, list(range(n_t)), oracle.Geometry.of_lattice(lat), 1.0, nb)
    assert oracle.rounding_ratio(C.cpu().numpy(), ref).max() <= 1e-6
    p.close()
