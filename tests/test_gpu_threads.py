"""Calls of different sizes from two threads, each on its own stream, that launch the same kernel
with different amounts of shared memory: none may be refused, and results are those of one
thread alone."""
import threading

import pytest
import torch

from paper_2308_07487_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def asd():
    from paper_2308_07487_gb300 import asd as m
    return m


def _ll(asd, L, s):
    lat = synth.hypercubic(L, 2, True)
    sysm = asd.System(lat)
    y = torch.from_numpy(synth.random_unit(lat.n_sites, 3)[None]).cuda()
    tr = torch.empty((lat.n_sites, 1, 2, 3), device="cuda")
    return lambda: sysm.ll_integrate(y, 0.01, 2, 1, tr, stream=s), lambda: tr


def _mc(asd, L, s):
    lat = synth.hypercubic(L, 2, True)
    sysm = asd.System(lat)
    y0 = torch.from_numpy(synth.random_unit(lat.n_sites, 4)[None]).cuda()
    y = y0.clone()

    def call():
        with torch.cuda.stream(s):
            y.copy_(y0)
        sysm.thermalize(y, 0.7, 1, asd.ASD_HEATBATH, seed=1, stream=s)
    return call, lambda: y


def _learned(asd, depth, s):
    lat = synth.hypercubic(8, 2, True)
    sysm = asd.System(lat)
    net = asd.Mlp(12, seed=3, depth=depth)
    y0 = torch.from_numpy(synth.random_unit(lat.n_sites, 4)[None]).cuda()
    y = y0.clone()

    def call():
        with torch.cuda.stream(s):
            y.copy_(y0)
        sysm.thermalize(y, 0.7, 1, asd.ASD_LEARNED, net=net, seed=1, stream=s)
    return call, lambda: y


def _corr(asd, form, n_bins, s):
    lat = synth.hypercubic(8, 2, True)
    tr = torch.from_numpy(synth.traj_iid(lat.n_sites, 6, seed=1)).cuda()
    plan = asd.CorrPlan.for_lattice(lat, 6, 4, 1, 4.0 / n_bins, n_bins, precision=form,
                                    deterministic=True)
    C = torch.zeros((1, n_bins), dtype=torch.float64, device="cuda")

    def call():
        with torch.cuda.stream(s):
            C.zero_()
        plan.run(tr, C, stream=s)
    return call, lambda: C


def _omega(asd, n_t, s):
    S = torch.ones((n_t, 2), dtype=torch.float64, device="cuda")
    w = torch.zeros(1, dtype=torch.float64, device="cuda")
    out = torch.zeros((1, 2), dtype=torch.float64, device="cuda")
    return lambda: asd.sq_omega(S, 0.1, w, out, stream=s), lambda: out


KINDS = {
    "ll_block": lambda asd, k, s: _ll(asd, (6, 32)[k], s),        # one block per sample
    "ll_grid": lambda asd, k, s: _ll(asd, (50, 300)[k], s),       # one site per thread
    "mc_block": lambda asd, k, s: _mc(asd, (6, 62)[k], s),
    "learned": lambda asd, k, s: _learned(asd, (2, 3)[k], s),
    "corr_fp32": lambda asd, k, s: _corr(asd, "fp32", (4, 1000)[k], s),
    "corr_split": lambda asd, k, s: _corr(asd, "split_bf16", (4, 1000)[k], s),
    "omega": lambda asd, k, s: _omega(asd, (3200, 6000)[k], s),
}


@pytest.mark.parametrize("kind", list(KINDS))
def test_two_sizes_at_once(asd, kind):
    calls = 1500
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    jobs = [KINDS[kind](asd, k, streams[k]) for k in range(2)]
    torch.cuda.synchronize()
    alone = []
    for call, out in jobs:
        call()
        torch.cuda.synchronize()
        alone.append(out().clone())
    errors = []
    start = threading.Barrier(2)

    def work(k):
        try:
            start.wait()
            for i in range(calls):
                jobs[k][0]()
                if i % 100 == 99:
                    streams[k].synchronize()
        except Exception as e:   # (the thread's own; reported below)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[0]
    assert asd.sync_status() == 0
    for (_, out), ref in zip(jobs, alone):
        assert torch.equal(out(), ref)
