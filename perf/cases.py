"""The calls that a user's program makes, as cases that can be timed and compared.

A spin-dynamics study with this library samples spins by Monte Carlo (asd_thermalize),
integrates the Landau-Lifshitz equation into a trajectory (asd_ll_integrate), reduces the
trajectory to the pair correlation C(r, t) and the phase-weighted sum S(q, t)
(asd_pair_corr, asd_pair_corr_batched, asd_pair_corr_sq_separable, then
asd_pair_corr_normalize and asd_sq_omega), and may train and use a small network as the
Monte Carlo proposal (asd_mlp_loss_grad, asd_mlp_adam_step).  Every case is one of these
calls (or one with the normalisation that always follows it) through the package's
binding, with the plan, system or network that such a program makes once and keeps.

listed() gives the cases, draw() more of the same ranges, prepare() what the program has
in hand before the call, run() one pass, work() the bytes and operations that the call
cannot do without, exact() its result in FP64 from plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2308_07487_gb300 import asd, synth

DEV = "cuda"


# ---------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------

def listed():
    return [
        # the smallest study: 16 x 16 periodic square lattice, all 32 displacements; one call
        # is a few launches, so it stands for the cost of a call
        dict(name="corr_sq16", kind="corr", dim=2, L=16, glass=False, S=1, T0=64, n_t=32,
             w=1.0, n_bins=12, n_q=0, precision="split_bf16", center=False),
        # FP32-accurate tensor form on a simple-cubic lattice with the long time average
        # (1000 origins) of the throughput runs: bins by the lattice table
        dict(name="corr_cubic26", kind="corr", dim=3, L=26, glass=False, S=1, T0=1000, n_t=8,
             w=0.5, n_bins=46, n_q=0, precision="split_bf16", center=False),
        # the headline workload's form on a 32^3 jittered glass: FP32 positions, 256 bins and
        # 64 q-vectors, FP32-accurate tensor form
        dict(name="corr_glass32", kind="corr", dim=3, L=32, glass=True, S=1, T0=512, n_t=2,
             w=0.5, n_bins=256, n_q=64, precision="split_bf16", center=False),
        # a larger glass in the cheap BF16 form of the precision sweep (a survey run)
        dict(name="corr_glass48_bf16", kind="corr", dim=3, L=48, glass=True, S=1, T0=512, n_t=2,
             w=0.5, n_bins=256, n_q=64, precision="bf16", center=False),
        # plain FP32 form, connected correlation (Eq. 5), bins and q-vectors: the accuracy
        # reference that a user checks the tensor forms with
        dict(name="corr_glass24_fp32", kind="corr", dim=3, L=24, glass=True, S=1, T0=512, n_t=2,
             w=0.5, n_bins=96, n_q=32, precision="fp32", center=True),
        # an uneven ensemble of independent 2D / 3D samples in one batched launch
        dict(name="ensemble24", kind="ensemble", n=24, lo=1024, hi=16384, T0=256, n_t=8,
             precision="split_bf16"),
        # spectra without bins: separable S(q, t) of 128 displacements, normalised, then
        # S(q, omega)
        dict(name="spectrum_glass40", kind="separable", dim=3, L=40, glass=True, S=1, T0=512,
             n_t=128, n_q=64, n_w=256, center=False),
        # Landau-Lifshitz trajectories of 50 realisations of the small lattice (the paper's
        # M = 50)
        dict(name="ll_sq16_s50", kind="ll", dim=2, L=16, glass=False, S=50, F=96, stride=1,
             dm=0.0, aniso=0.0),
        # ... and of the 64^3 glass, the trajectory of the headline workload (a quarter of
        # its frames)
        dict(name="ll_glass64", kind="ll", dim=3, L=64, glass=True, S=1, F=160, stride=1,
             dm=0.0, aniso=0.0),
        # thermalisation of the 40^3 lattice: Metropolis sweeps with the adaptive cone
        dict(name="mc_cubic40", kind="mc", dim=3, L=40, glass=False, S=1, T=1.2, sweeps=100,
             proposal="metropolis", adapt=True, depth=2),
        # sweeps with the learned proposal on eight 128 x 128 chains
        dict(name="mc_learned_sq128", kind="mc", dim=2, L=128, glass=False, S=8, T=0.7, sweeps=10,
             proposal="learned", adapt=False, depth=2),
        # one training step of the proposal network at the usual batch of 16384 pairs
        dict(name="train_16384", kind="train", n=16384, z=4, depth=2),
    ]


def draw(rng):
    """One more case of the listed ranges."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["corr", "corr", "corr", "ensemble", "separable", "ll", "ll", "mc", "mc",
                       "train"])
    if kind == "corr":
        glass = rng.random() < 0.6
        dim = 3 if glass or rng.random() < 0.6 else 2
        precision = rng.choice(["split_bf16", "split_bf16", "split_bf16", "tf32", "bf16", "fp32"])
        if dim == 3:
            L = rng.randint(10, 22 if precision == "fp32" else 34)
        else:
            L = log_int(12, 100 if precision == "fp32" else 180)
        N = L ** dim
        S = 1 if rng.random() < 0.75 else rng.randint(2, 4)
        T0 = log_int(48, 1000) // S + 1
        # FP32-accurate tensor cost of at most 10^13 (10^12 for FP32) operations
        per_t = 2.0 * N * N * 3 * T0 * S
        n_t = max(1, min(rng.randint(1, 32), int((1e12 if precision == "fp32" else 1e13) / per_t)))
        w = rng.choice([0.5, 1.0, 0.7])
        rmax = math.sqrt(dim) * (L if glass else L / 2)
        n_bins = min(256, int(rmax / w) + 1)
        n_q = rng.choice([16, 37, 64, 100]) if glass and rng.random() < 0.7 else 0
        return dict(kind="corr", dim=dim, L=L, glass=glass, S=S, T0=T0, n_t=n_t, w=w,
                    n_bins=n_bins, n_q=n_q, precision=precision, center=rng.random() < 0.3)
    if kind == "ensemble":
        return dict(kind="ensemble", n=rng.randint(3, 24), lo=1024, hi=log_int(3000, 16384),
                    T0=log_int(64, 256), n_t=rng.randint(2, 8),
                    precision=rng.choice(["split_bf16", "split_bf16", "bf16"]))
    if kind == "separable":
        T0, S = log_int(100, 512), 1 if rng.random() < 0.7 else 2
        return dict(kind="separable", dim=3, L=rng.randint(14, 40), glass=True,
                    S=S, T0=T0 // S, n_t=rng.randint(16, 128),
                    n_q=rng.choice([16, 37, 64, 100]), n_w=rng.randint(64, 256),
                    center=rng.random() < 0.3)
    if kind == "ll":
        glass = rng.random() < 0.5
        dim = 3 if glass else rng.choice([2, 3])
        L = rng.randint(6, 60) if dim == 3 else log_int(10, 400)
        S = max(1, min(log_int(1, 64), 200000 // L ** dim))
        stride = rng.choice([1, 1, 1, 2])
        return dict(kind="ll", dim=dim, L=L, glass=glass, S=S, F=rng.randint(24, 120) // stride,
                    stride=stride, dm=rng.choice([0.0, 0.0, 0.3]),
                    aniso=rng.choice([0.0, 0.0, 0.2]))
    if kind == "mc":
        proposal = rng.choice(["metropolis", "heatbath", "learned"])
        glass = rng.random() < 0.4
        dim = 3 if glass else rng.choice([2, 3])
        # checkerboard colours need an even extent on periodic lattices
        L = 2 * (rng.randint(4, 20) if dim == 3 else log_int(6, 80))
        S = max(1, min(log_int(1, 64), 120000 // L ** dim))
        return dict(kind="mc", dim=dim, L=L, glass=glass, S=S, T=round(rng.uniform(0.4, 1.5), 3),
                    sweeps=rng.randint(2, 10) if proposal == "learned" else rng.randint(10, 100),
                    proposal=proposal, adapt=proposal == "metropolis" and rng.random() < 0.6,
                    depth=rng.choice([2, 3]))
    return dict(kind="train", n=log_int(700, 16384), z=rng.choice([4, 6]),
                depth=rng.choice([2, 2, 3]))


# ---------------------------------------------------------------------------------------
# inputs (from the seed alone)
# ---------------------------------------------------------------------------------------

def _lattice(case, seed):
    """The case's lattice: periodic with J = 1, or the open jittered +-J glass numbered in
    spatial blocks (at most 4 x 4 x 8 sites)."""
    L, dim = case["L"], case["dim"]
    if not case["glass"]:
        lat = synth.hypercubic(L, dim, True, J=1.0, seed=seed)
    else:
        def part(most):
            return max(b for b in range(1, most + 1) if L % b == 0)
        lat = synth.hypercubic(L, dim, False, pm_j=True, p=0.5, seed=seed,
                               block=(part(4), part(4), part(8)), jitter=0.1)
    if case.get("dm") or case.get("aniso"):
        lat = synth.with_dm_anisotropy(lat, case["dm"], case["aniso"])
    return lat


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _unit(shape, gen):
    v = torch.randn(shape, device=DEV, generator=gen)
    return v / v.norm(dim=-1, keepdim=True)


def _trajectory(N, S, F, seed):
    """[N][S][F][3]: unit spins tilted towards a common axis that precess about z at
    site-dependent rates (structure in r and t)."""
    g = _gen(seed)
    axis = torch.tensor([0.3, 0.2, 0.93], device=DEV)
    s0 = 0.6 * axis / axis.norm() + 0.4 * _unit((N, S, 3), g)
    s0 = s0 / s0.norm(dim=-1, keepdim=True)
    rate = 0.05 * (1.0 + 0.5 * torch.randn((N, S, 1), device=DEV, generator=g))
    ang = rate * torch.arange(F, device=DEV)
    c, s = torch.cos(ang), torch.sin(ang)
    tr = torch.empty((N, S, F, 3), device=DEV)
    tr[..., 0] = c * s0[..., 0:1] - s * s0[..., 1:2]
    tr[..., 1] = s * s0[..., 0:1] + c * s0[..., 1:2]
    tr[..., 2] = s0[..., 2:3]
    return tr


def _qs(n_q, seed):
    """n_q vectors along (100), (110), (111) and one more direction, |q| up to pi."""
    d = np.array([[1, 0, 0], [1, 1, 0], [1, 1, 1], [0.36, -0.48, 0.8]], np.float64)
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    m = math.pi * (np.arange(n_q) // 4 + 1e-3 * (seed % 97)) / max(1, n_q // 4)
    return d[np.arange(n_q) % 4] * m[:, None]


def _members(case, seed):
    """(lattice case, w, n_bins) of every sample of an ensemble: the sizes belong to the
    case, the spins to the seed."""
    out = []
    for d, L in synth.ensemble_sizes(case["n"], lo=case["lo"], hi=case["hi"]):
        w = 1.0 if d == 2 else 0.5
        out.append((dict(dim=d, L=L, glass=False), w,
                    int(math.floor(math.sqrt(d * (L // 2) ** 2) / w)) + 1))
    return out


def _net_params(z, depth, seed):
    """Glorot-uniform weights and small biases, packed as asd_mlp_init packs them."""
    g = synth.rng(seed)
    H, n_in = 64, 3 * z
    shapes = [(H, n_in)] + [(H, H)] * (depth - 1) + [(4, H)]
    out = []
    for o, i in shapes:
        a = math.sqrt(6.0 / (o + i))
        out += [g.uniform(-a, a, size=o * i), g.normal(0.0, 0.05, size=o)]
    return np.concatenate(out).astype(np.float32), shapes


def _pairs(case, seed):
    """Training pairs: neighbour spins and a site spin that leans against their sum."""
    g = _gen(seed)
    x = _unit((case["n"], case["z"], 3), g)
    y = -x.sum(1) + 0.8 * torch.randn((case["n"], 3), device=DEV, generator=g)
    return x.reshape(case["n"], -1).contiguous(), (y / y.norm(dim=1, keepdim=True)).contiguous()


def _frames(case):
    return case["T0"] + case["n_t"] - 1


# ---------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------

def prepare(case, seed):
    k = case["kind"]
    st = {"case": case}
    f64 = dict(dtype=torch.float64, device=DEV)
    if k == "corr":
        lat = _lattice(case, seed)
        q = _qs(case["n_q"], seed) if case["n_q"] else None
        st["traj"] = _trajectory(lat.n_sites, case["S"], _frames(case), seed)
        st["plan"] = asd.CorrPlan.for_lattice(
            lat, _frames(case), case["T0"], case["n_t"], case["w"], case["n_bins"],
            precision=case["precision"], S=case["S"], center=case["center"], q=q)
        st["C_sum"] = torch.empty((case["n_t"], case["n_bins"]), **f64)
        st["C"] = torch.empty_like(st["C_sum"])
        st["Sq_sum"] = torch.empty((case["n_t"], case["n_q"]), **f64) if q is not None else None
        st["Sq"] = torch.empty_like(st["Sq_sum"]) if q is not None else None
    elif k == "ensemble":
        st["trajs"], st["plans"], st["C_sums"], st["Cs"] = [], [], [], []
        for m, (c, w, nb) in enumerate(_members(case, seed)):
            lat = _lattice(c, seed)
            st["trajs"].append(_trajectory(lat.n_sites, 1, _frames(case), 1000 * seed + m))
            # one tile width for the whole batch, as its launch needs
            st["plans"].append(asd.CorrPlan.for_lattice(
                lat, _frames(case), case["T0"], case["n_t"], w, nb,
                precision=case["precision"], tile_n=256))
            st["C_sums"].append(torch.empty((case["n_t"], nb), **f64))
            st["Cs"].append(torch.empty((case["n_t"], nb), **f64))
    elif k == "separable":
        lat = _lattice(case, seed)
        st["traj"] = _trajectory(lat.n_sites, case["S"], _frames(case), seed)
        st["plan"] = asd.CorrPlan.for_lattice(
            lat, _frames(case), case["T0"], case["n_t"], 1.0, 0, S=case["S"],
            center=case["center"], q=_qs(case["n_q"], seed))
        st["Sq_sum"] = torch.empty((case["n_t"], case["n_q"]), **f64)
        st["Sq"] = torch.empty_like(st["Sq_sum"])
        st["omega"] = _omega(case)
        st["Sqw"] = torch.empty((case["n_w"], case["n_q"]), **f64)
    elif k == "ll":
        lat = _lattice(case, seed)
        st["sys"] = asd.System(lat)
        st["spins0"] = _unit((case["S"], lat.n_sites, 3), _gen(seed))
        st["traj"] = torch.empty((lat.n_sites, case["S"], case["F"], 3), device=DEV)
        st["last"] = torch.empty_like(st["spins0"])
    elif k == "mc":
        lat = _lattice(case, seed)
        st["sys"] = asd.System(lat)
        st["spins"] = _unit((case["S"], lat.n_sites, 3), _gen(seed))
        st["seed"], st["done"] = seed, 0
        st["net"] = None
        if case["proposal"] == "learned":
            z = lat.nbr.shape[1]
            st["net"] = asd.Mlp(3 * z, params=_net_params(z, case["depth"], seed)[0],
                                depth=case["depth"])
    else:
        st["x"], st["y"] = _pairs(case, seed)
        st["net"] = asd.Mlp(3 * case["z"], params=_net_params(case["z"], case["depth"], seed)[0],
                            depth=case["depth"])
    return st


_PROPOSALS = {"metropolis": asd.ASD_METROPOLIS, "heatbath": asd.ASD_HEATBATH,
              "learned": asd.ASD_LEARNED}


def run(st):
    case = st["case"]
    k = case["kind"]
    stream = torch.cuda.current_stream()
    if k == "corr":
        st["C_sum"].zero_()
        if st["Sq_sum"] is not None:
            st["Sq_sum"].zero_()
        st["plan"].run(st["traj"], st["C_sum"], st["Sq_sum"], stream=stream)
        st["plan"].normalize(st["C_sum"], st["Sq_sum"], st["C"], st["Sq"], stream=stream)
        return {"C": st["C"], "Sq": st["Sq"]}
    if k == "ensemble":
        for c in st["C_sums"]:
            c.zero_()
        asd.pair_corr_batched(st["plans"], st["trajs"], st["C_sums"], stream=stream)
        for p, s, c in zip(st["plans"], st["C_sums"], st["Cs"]):
            p.normalize(s, None, c, None, stream=stream)
        return st["Cs"]
    if k == "separable":
        st["Sq_sum"].zero_()
        st["plan"].sq_separable(st["traj"], st["Sq_sum"], stream=stream)
        st["plan"].normalize(None, st["Sq_sum"], None, st["Sq"], stream=stream)
        asd.sq_omega(st["Sq"], 0.01, st["omega"], st["Sqw"], window="hann", stream=stream)
        return {"Sq": st["Sq"], "Sqw": st["Sqw"]}
    if k == "ll":
        st["sys"].ll_integrate(st["spins0"], 0.01, case["F"], case["stride"], st["traj"],
                               spins_out=st["last"], stream=stream)
        return {"traj": st["traj"], "last": st["last"]}
    if k == "mc":
        # a chain goes on: the next call continues the counter-based random numbers
        st["sys"].thermalize(st["spins"], case["T"], case["sweeps"],
                             _PROPOSALS[case["proposal"]], net=st["net"], cone=0.0,
                             adapt=case["adapt"], seed=st["seed"], counter=st["done"],
                             stream=stream)
        st["done"] += case["sweeps"]
        return st["spins"]
    net = st["net"]
    net.grad.zero_()
    net.loss.zero_()
    net.loss_grad(st["x"], st["y"], stream=stream)
    net.adam(lr=1e-3, scale=1.0 / case["n"], stream=stream)
    return {"loss": net.loss, "grad": net.grad, "params": net.params, "weights": net.wb}


# ---------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------

def work(case):
    k = case["kind"]
    if k == "corr":
        N, F = case["L"] ** case["dim"], _frames(case)
        return {"bytes": 12.0 * N * case["S"] * F + 8.0 * case["n_t"] * (case["n_bins"] + case["n_q"]),
                "flops": 2.0 * N * N * 3 * case["T0"] * case["S"] * case["n_t"]}
    if k == "ensemble":
        b = f = 0.0
        for c, _, nb in _members(case, 0):
            N = c["L"] ** c["dim"]
            b += 12.0 * N * _frames(case) + 8.0 * case["n_t"] * nb
            f += 2.0 * N * N * 3 * case["T0"] * case["n_t"]
        return {"bytes": b, "flops": f}
    if k == "separable":
        N, F, S = case["L"] ** case["dim"], _frames(case), case["S"]
        return {"bytes": 12.0 * N * S * F + 8.0 * (case["n_t"] + case["n_w"]) * case["n_q"],
                "flops": 4.0 * case["n_q"] * (N * S * 3.0 * F + case["n_t"] * 3.0 * case["T0"] * S
                                              + case["n_w"] * case["n_t"])}
    if k == "ll":
        N, S = case["L"] ** case["dim"], case["S"]
        z = 2 * case["dim"]
        steps = (case["F"] - 1) * case["stride"]
        return {"bytes": 12.0 * N * S * (case["F"] + 2) + N * z * (20.0 if case["dm"] else 8.0),
                "flops": steps * 4.0 * N * S * (z * (21.0 if case["dm"] else 6.0) + 27.0)}
    if k == "mc":
        N, S = case["L"] ** case["dim"], case["S"]
        z = 2 * case["dim"]
        per = 6.0 * z + 100.0
        if case["proposal"] == "learned":
            per += 2.0 * (64 * 3 * z + (case["depth"] - 1) * 64 * 64 + 4 * 64)
        return {"bytes": 24.0 * N * S + 8.0 * N * z, "flops": case["sweeps"] * N * S * per}
    n_w = 64 * 3 * case["z"] + (case["depth"] - 1) * 64 * 64 + 4 * 64
    return {"bytes": 4.0 * case["n"] * (3 * case["z"] + 3) + 30.0 * n_w,
            "flops": 6.0 * case["n"] * n_w}


# ---------------------------------------------------------------------------------------
# the same results in FP64
# ---------------------------------------------------------------------------------------

def _omega(case):
    return torch.linspace(0.0, math.pi / 0.01 / 8, case["n_w"], dtype=torch.float64, device=DEV)


def _bins(d2, w, n_bins):
    """Largest k with (k w)^2 <= d2 (n_bins: dropped)."""
    thr = (torch.arange(n_bins + 1, dtype=torch.float64, device=d2.device) * w) ** 2
    return torch.bucketize(d2, thr, right=True) - 1


def _operands(tr, case):
    """A (every frame) and B (the origins, centred when asked), FP64 [N][S][.][3]."""
    A = tr.double()
    B = A[:, :, :case["T0"]]
    if case.get("center"):
        B = B - B.mean(dim=(1, 2), keepdim=True)
    return A, B


def _exact_periodic(case, lat, tr, w, n_bins):
    """C(r, t) of a periodic lattice from the spatial cross-correlation by FFT."""
    A, B = _operands(tr, case)
    N, S = tr.shape[:2]
    shape, T0 = tuple(lat.L[::-1]), case["T0"]
    dims = (0, 1, 2)
    Bf = torch.fft.fftn(B.reshape(shape + (-1,)), dim=dims)
    Af = torch.fft.fftn(A.reshape(shape + (-1,)), dim=dims).reshape(shape + (S, -1, 3))
    d = [torch.minimum(torch.arange(n, device=DEV), n - torch.arange(n, device=DEV)).double() ** 2
         for n in shape]
    d2 = d[0][:, None, None] + d[1][None, :, None] + d[2][None, None, :]
    b = _bins(d2, w, n_bins).reshape(-1)
    n_b = torch.bincount(b, minlength=n_bins + 1)[:n_bins].double() * N
    out = []
    for t in range(case["n_t"]):
        a = Af[..., t:t + T0, :].reshape(shape + (-1,))
        r = torch.fft.ifftn((a.conj() * Bf).sum(-1), dim=dims).real.reshape(-1)
        out.append(torch.zeros(n_bins + 1, dtype=torch.float64, device=DEV)
                   .index_add_(0, b, r)[:n_bins] / (S * T0 * n_b.clamp(min=1)))
    return torch.stack(out)


def _exact_pairs(case, lat, tr):
    """C(r, t) over all pairs of a glass, rows in blocks."""
    A, B = _operands(tr, case)
    N, S, T0, nb = lat.n_sites, case["S"], case["T0"], case["n_bins"]
    B = B.reshape(N, -1)
    pos = torch.from_numpy(lat.pos).to(DEV)
    out = torch.zeros((case["n_t"], nb + 1), dtype=torch.float64, device=DEV)
    n_b = torch.zeros(nb + 1, dtype=torch.float64, device=DEV)
    step = max(1, (1 << 26) // N)
    for i in range(0, N, step):
        d = (pos[None] - pos[i:i + step, None]).double() ** 2      # FP32 differences
        # fma(dz, dz, fma(dy, dy, dx dx)) with FP32 rounding of each result
        d2 = ((d[..., 0].float().double() + d[..., 1]).float().double() + d[..., 2]).float()
        b = _bins(d2.double(), case["w"], nb).reshape(-1)
        n_b += torch.bincount(b, minlength=nb + 1).double()
        for t in range(case["n_t"]):
            g = A[i:i + step, :, t:t + T0].reshape(-1, B.shape[1]) @ B.T
            out[t] += torch.bincount(b, weights=g.reshape(-1), minlength=nb + 1)
    n_b = n_b[:nb]
    return torch.where(n_b > 0, out[:, :nb] / (S * T0 * n_b.clamp(min=1)), 0.0)


def _exact_phase(case, lat, tr, q):
    """S(q, t) through the per-site transforms of every frame."""
    N, S, T0 = lat.n_sites, case["S"], case["T0"]
    r = torch.from_numpy(lat.pos).to(DEV).double()
    ph = r @ torch.from_numpy(q).to(DEV).T
    wt = torch.cat([torch.cos(ph), torch.sin(ph)], 1).T            # [2 n_q][N]
    Fa = sum(wt[:, i:i + 8192] @ tr[i:i + 8192].double().reshape(-1, S * _frames(case) * 3)
             for i in range(0, N, 8192)).reshape(-1, S, _frames(case), 3)
    Fb = Fa[:, :, :T0]
    if case["center"]:
        Fb = Fb - Fb.mean(dim=(1, 2), keepdim=True)
    out = [(Fa[:, :, t:t + T0] * Fb).sum(dim=(1, 2, 3)) for t in range(case["n_t"])]
    out = torch.stack(out)
    n_q = q.shape[0]
    return (out[:, :n_q] + out[:, n_q:]) / (N * S * T0)


def _exact_ll(case, lat, spins0):
    nbr = torch.from_numpy(lat.nbr).long().to(DEV)
    J = torch.where(nbr >= 0, torch.from_numpy(lat.J).to(DEV).double(), 0.0)
    D = None if lat.D is None else torch.from_numpy(lat.D).to(DEV).double()
    nbr = nbr.clamp(min=0)
    # (the constants as the FP32 values that the call receives)
    A, dt = float(np.float32(lat.A)), float(np.float32(0.01))

    def rhs(Y):
        h = torch.zeros_like(Y)
        h[..., 2] = -2.0 * A * Y[..., 2] - float(lat.Hz)
        for k in range(nbr.shape[1]):
            s = Y[:, nbr[:, k]]
            h = h + J[:, k, None] * s
            if D is not None:
                h = h + torch.cross(D[None, :, k].expand_as(s), s, dim=-1)
        return torch.cross(h, Y, dim=-1)

    Y = spins0.double()
    traj = torch.empty((lat.n_sites, case["S"], case["F"], 3), dtype=torch.float64, device=DEV)
    traj[:, :, 0] = Y.transpose(0, 1)
    for f in range(1, case["F"]):
        for _ in range(case["stride"]):
            k1 = rhs(Y)
            k2 = rhs(Y + 0.5 * dt * k1)
            k3 = rhs(Y + 0.5 * dt * k2)
            k4 = rhs(Y + dt * k3)
            Y = Y + dt / 6.0 * (k1 + 2 * k2 + 2 * k3 + k4)
        traj[:, :, f] = Y.transpose(0, 1)
    return {"traj": traj, "last": Y}


def _exact_train(case, seed):
    x, y = (v.double() for v in _pairs(case, seed))
    flat, shapes = _net_params(case["z"], case["depth"], seed)
    p = torch.from_numpy(flat).to(DEV)
    layers, o = [], 0
    for out, inp in shapes:
        W = p[o:o + out * inp].reshape(out, inp).bfloat16().double().requires_grad_()
        b = p[o + out * inp:o + out * inp + out].double().requires_grad_()
        layers.append((W, b))
        o += out * inp + out
    h = x
    for W, b in layers[:-1]:
        h = torch.tanh(h @ W.T + b)
    v = h @ layers[-1][0].T + layers[-1][1]
    kap = torch.nn.functional.softplus(v[:, 3]) + 1e-4
    mu = v[:, :3] / v[:, :3].norm(dim=1, keepdim=True)
    nll = (-torch.log(kap) + math.log(2 * math.pi) + kap + torch.log1p(-torch.exp(-2 * kap))
           - kap * (mu * y).sum(1))
    loss = nll.sum()
    loss.backward()
    grad = torch.cat([torch.cat([W.grad.reshape(-1), b.grad]) for W, b in layers])
    g = grad / case["n"]
    # the first Adam step: bias-corrected moments are g and g^2
    new = p.double() - 1e-3 * g / (g.abs() + 1e-8)
    return {"loss": loss.detach().reshape(1), "grad": grad, "params": new, "weights": None}


def exact(case, seed):
    """run()'s result for these inputs in FP64; None where that takes too long (pair sums of
    more than 8e12 operations) or is no computed number (a Monte Carlo chain's state)."""
    k = case["kind"]
    if k == "corr":
        lat = _lattice(case, seed)
        if case["glass"] and work(case)["flops"] > 8e12:
            return None
        tr = _trajectory(lat.n_sites, case["S"], _frames(case), seed)
        C = (_exact_pairs(case, lat, tr) if case["glass"]
             else _exact_periodic(case, lat, tr, case["w"], case["n_bins"]))
        Sq = _exact_phase(case, lat, tr, _qs(case["n_q"], seed)) if case["n_q"] else None
        return {"C": C, "Sq": Sq}
    if k == "ensemble":
        out = []
        for m, (c, w, nb) in enumerate(_members(case, seed)):
            lat = _lattice(c, seed)
            tr = _trajectory(lat.n_sites, 1, _frames(case), 1000 * seed + m)
            out.append(_exact_periodic(case, lat, tr, w, nb))
        return out
    if k == "separable":
        lat = _lattice(case, seed)
        tr = _trajectory(lat.n_sites, case["S"], _frames(case), seed)
        Sq = _exact_phase(case, lat, tr, _qs(case["n_q"], seed))
        t = torch.arange(case["n_t"], dtype=torch.float64, device=DEV)
        v = 0.5 * (1.0 + torch.cos(math.pi * t / case["n_t"]))
        v = torch.where(t > 0, 2.0 * v, v)
        Sqw = 0.01 * (torch.cos(_omega(case)[:, None] * t * 0.01) * v) @ Sq
        return {"Sq": Sq, "Sqw": Sqw}
    if k == "ll":
        lat = _lattice(case, seed)
        return _exact_ll(case, lat, _unit((case["S"], lat.n_sites, 3), _gen(seed)))
    if k == "mc":
        return None
    return _exact_train(case, seed)
