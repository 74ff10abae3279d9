"""asd_ll_integrate with more samples of a small system than thread blocks fit the device: the
samples share blocks, and each follows the trajectory that it follows among few."""
import pytest
import torch

from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu

LATS = {
    "chain1": lambda: synth.open_chain(1),
    "chain2": lambda: synth.open_chain(2),
    "chain33": lambda: synth.open_chain(33),
    "square_dm": lambda: synth.with_dm_anisotropy(synth.hypercubic(4, 2, True), 0.3, 0.2),
    "cubic27": lambda: synth.hypercubic(3, 3, False),
    "chain128": lambda: synth.open_chain(128),
}


@pytest.mark.parametrize("name", list(LATS))
@pytest.mark.parametrize("F,stride", [(1, 1), (7, 2), (2, 4100)])
def test_many_samples(name, F, stride):
    from paper_2308_07487_gb300 import asd
    lat = LATS[name]()
    N, few = lat.n_sites, 300
    S = 32 * torch.cuda.get_device_properties(0).multi_processor_count + 37
    sysm = asd.System(lat)
    spins = torch.from_numpy(synth.random_unit(few * N, 7).reshape(few, N, 3)).cuda()
    ref = torch.empty((N, few, F, 3), device="cuda")
    ref_out = torch.empty_like(spins)
    sysm.ll_integrate(spins, 0.02, F, stride, ref, spins_out=ref_out)
    pick = torch.arange(S, device="cuda") * 7 % few
    many = spins[pick].contiguous()
    traj = torch.full((N, S, F, 3), float("nan"), device="cuda")
    out = torch.empty_like(many)
    sysm.ll_integrate(many, 0.02, F, stride, traj, spins_out=out)
    assert asd.sync_status() == 0
    assert torch.equal(traj, ref[:, pick]) and torch.equal(out, ref_out[pick])
    if N * S <= 262144:
        traj.fill_(float("nan"))
        sysm.ll_integrate_noalloc(many, 0.02, F, stride, traj, spins_out=many)   # in place
        assert asd.sync_status() == 0
        assert torch.equal(traj, ref[:, pick]) and torch.equal(many, out)
