"""The work that users of this framework have it do, as measurable cases.

A case is a dict of plain values.  ``kind`` says which public calls one pass
makes:

* ``sample``    ``Plan.sample`` on a plan that the program keeps
* ``coeffs``    ``Plan.coeffs`` on a plan that the program keeps
* ``step``      a plan created, sampled and destroyed (what the benchmark times)
* ``plan``      a plan created, its tables read, destroyed
* ``fields``    ``Plan.field_from_coeffs`` on given coefficients
* ``batch``     ``Batch.run`` of a captured batch over uneven lattices
* ``stats``     ``Stats.add`` and ``Stats.read`` on given fields

The seed of a case's inputs sets the samples' Philox seeds and moves the
spectrum's parameters (wind speed, height, target) a little, so that plans of
different seeds differ.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2310_03979_gb300 import srm3
from paper_2310_03979_gb300 import workloads as W

FOUR_PI = 4 * math.pi


def listed():
    return [
        # a request of the serving loop's small class, its plan resident:
        # one 64 x 64 field, where launches and latency are everything
        dict(name="serve_small", kind="sample", nk=32, nw=32, nx=64, nt=64, n=1, ku=0.5,
             wu=FOUR_PI, U=30.0, z=20.0, target=0.5, precision="fp32", storage="recompute",
             envelope="gauss", interactions="sum"),
        # the plain method on the tiny lattice, FP64: a plan and one sample
        dict(name="tiny_step_fp64", kind="step", nk=32, nw=32, nx=64, nt=64, n=1, ku=0.5,
             wu=FOUR_PI, U=30.0, z=20.0, target=0.5, precision="fp64", storage="recompute",
             envelope="gauss", interactions="sum"),
        # the bridge-span wave with the stored W table, plan resident: the
        # sampling part of the default benchmark
        dict(name="bridge_table", kind="sample", nk=256, nw=512, nx=512, nt=1024, n=64, ku=0.25,
             wu=FOUR_PI, U=40.0, z=20.0, target=0.5, precision="fp32", storage="table",
             envelope="gauss", interactions="sum"),
        # the bridge lattice with W recomputed, plan built in the step: the
        # benchmark's form for spectra that are used once
        dict(name="bridge_step_recompute", kind="step", nk=256, nw=512, nx=512, nt=1024, n=64,
             ku=0.25, wu=FOUR_PI, U=40.0, z=20.0, target=0.5, precision="fp32",
             storage="recompute", envelope="gauss", interactions="sum"),
        # the large lattice, whose W table would not fit: 16 samples
        dict(name="large_sample", kind="sample", nk=512, nw=1024, nx=1024, nt=2048, n=16, ku=0.25,
             wu=FOUR_PI, U=40.0, z=20.0, target=0.5, precision="fp32", storage="recompute",
             envelope="gauss", interactions="sum"),
        # the large lattice's plan alone (the server's background builds)
        dict(name="large_plan", kind="plan", nk=512, nw=1024, nx=1024, nt=2048, n=0, ku=0.25,
             wu=FOUR_PI, U=40.0, z=20.0, target=0.5, precision="fp32", storage="recompute",
             envelope="gauss", interactions="sum"),
        # many spectra on uneven lattices in one captured graph
        dict(name="uneven_batch", kind="batch", spectra=32, mix=4),
        # the wind field along a long-span bridge (Sec. 5): fixed scale, the
        # separable envelope of i + j, one block of the 1000 fields
        dict(name="wind_field", kind="step", nk=256, nw=128, nx=1024, nt=2048, n=50,
             ku=2.0 * 255 * math.pi / 628.0, wu=math.pi, U=40.0, z=50.0, target=0.0, lam=20.0,
             precision="fp32", storage="recompute", envelope="sum", interactions="sum"),
        # ensemble statistics of a block of such fields
        dict(name="stats_fields", kind="stats", count=50 * 1024 * 2048, nbins=200,
             precision="fp32"),
        # fields of given FP64 coefficients (coefficients gathered from shards)
        dict(name="fields_fp64", kind="fields", nk=256, nw=512, nx=512, nt=1024, n=16, ku=0.25,
             wu=FOUR_PI, U=40.0, z=20.0, target=0.5, precision="fp64", storage="recompute",
             envelope="gauss", interactions="sum"),
        # FP64 coefficients on a ragged lattice (the audit of served fields)
        dict(name="audit_fp64", kind="coeffs", nk=90, nw=117, nx=128, nt=256, n=4, ku=0.5,
             wu=FOUR_PI, U=30.0, z=20.0, target=0.5, precision="fp64", storage="recompute",
             envelope="gauss", interactions="sum"),
        # mixed-sign interactions, plan and samples, on a ragged lattice
        dict(name="mixed_step", kind="step", nk=40, nw=70, nx=64, nt=256, n=16, ku=0.5,
             wu=FOUR_PI, U=30.0, z=20.0, target=0.5, precision="fp32", storage="recompute",
             envelope="gauss", interactions="mixed"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pow2(n):
    p = 2
    while p < n:
        p *= 2
    return p


def _pairs(nk, nw):
    return (nk * (nk + 1) // 2) * (nw * (nw + 1) // 2) // 2


def draw(rng):
    kind = rng.choice(["sample", "sample", "step", "step", "plan", "coeffs", "fields", "batch",
                       "stats"])
    if kind == "stats":
        return dict(kind=kind, count=_log_int(rng, 1000, 100_000_000), nbins=_log_int(rng, 10, 4000),
                    precision=rng.choice(["fp32", "fp32", "fp64"]))
    if kind == "batch":
        return dict(kind=kind, spectra=rng.randint(2, 32), mix=rng.randint(0, 1 << 20))
    precision = rng.choice(["fp32", "fp32", "fp32", "fp64"])
    envelope = rng.choice(["gauss", "gauss", "gauss", "separable", "sum"])
    mixed = envelope == "gauss" and kind in ("sample", "step", "coeffs") and rng.random() < 0.2
    if mixed:
        nk, nw = _log_int(rng, 12, 64), _log_int(rng, 12, 80)
    else:
        nk, nw = _log_int(rng, 16, 512), _log_int(rng, 16, 1024)
        if precision == "fp64" and envelope == "gauss" and kind not in ("fields", "plan"):
            nk, nw = min(nk, 160), min(nw, 200)
    nx, nt = _pow2(nk), _pow2(2 * nw - 1)
    if rng.random() < 0.5 and nx <= 512:
        nx *= 2
    if kind == "plan":
        n = 0
    else:  # within the listed cases' pair-terms, and 1 GB of fields
        terms = (2e9 if precision == "fp64" else 2.5e11) / (2.0 * _pairs(nk, nw))
        room = 2.5e8 / (nx * nt)
        n = _log_int(rng, 1, max(1, min(64, int(terms), int(room))))
    storage = "recompute"
    if precision == "fp32" and envelope == "gauss" and not mixed and nk * nw <= 1 << 17 \
            and rng.random() < 0.3:
        storage = "table"
    return dict(kind=kind, nk=nk, nw=nw, nx=nx, nt=nt, n=n, ku=rng.choice([0.25, 0.5]), wu=FOUR_PI,
                U=round(rng.uniform(22.0, 48.0), 3), z=round(rng.uniform(12.0, 58.0), 3),
                target=round(rng.uniform(0.15, 0.65), 3), precision=precision, storage=storage,
                envelope=envelope, interactions="mixed" if mixed else "sum")


def _workload(case, seed):
    """The case's workload with its spectrum moved by the seed."""
    r = random.Random(1_000_003 * seed + 17)
    target = case["target"]
    eps = 0.0
    if target > 0.0:
        target = min(0.7, target * r.uniform(0.97, 1.03))
    else:  # the fixed scale of the wind-field bispectrum
        eps = (4.0 / (3.0 * math.sqrt(3.0))) / math.sqrt(
            (case["ku"] / case["nk"]) * (case["wu"] / case["nw"]))
        target = 0.5
    return W.Workload(
        "case", case["nk"], case["nw"], case["ku"], case["wu"], case["U"] * r.uniform(0.97, 1.03),
        case["z"] * r.uniform(0.97, 1.03), case["nx"], case["nt"], _sample_seeds(seed, case["n"]),
        precision=case["precision"], storage=case["storage"], target=target,
        lam=case.get("lam", 7.0), envelope=case["envelope"], eps=eps,
        interactions=case["interactions"])


def _sample_seeds(seed, n):
    base = (seed * 2_654_435_761) % (1 << 48)
    return tuple(base + j for j in range(n))


def _batch_workloads(case, seed):
    """Spectra on power-of-two lattices, wind speeds, heights, targets and
    sample counts as the uneven benchmark draws them; the mix is the case's,
    the samples' seeds are the input seed's."""
    out = []
    for i, wl in enumerate(W.uneven_batch(case["spectra"], seed=case["mix"])):
        out.append(wl.with_seeds(_sample_seeds(seed + 7919 * (i + 1), wl.n_samples)))
    return out


class _Held:
    """A plan, batch or accumulator freed with the state that holds it."""

    def __init__(self, *things):
        self.things = things

    def __del__(self):
        for t in self.things:
            try:
                t.destroy()
            except Exception:
                pass


def _dtype(precision):
    return torch.float32 if precision == "fp32" else torch.float64


def _wave_values(case, seed):
    """A slightly skewed wave of standard deviation about 6."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.randn(case["count"], generator=g, device="cuda", dtype=_dtype(case["precision"]))
    u.mul_(6.0)
    return u.add_(0.05 * (u * u - 36.0) / 6.0)


def _given_coeffs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((case["n"], 2, case["nk"], case["nw"], 2), generator=g, device="cuda",
                       dtype=_dtype(case["precision"]))


def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind}
    if kind == "stats":
        u = _wave_values(case, seed)
        st = srm3.Stats(case["nbins"], -30.0, 30.0)
        return dict(state, u=u, stats=st, held=_Held(st))
    if kind == "batch":
        wls = _batch_workloads(case, seed)
        plans = [srm3.Plan.create(wl, storage="recompute") for wl in wls]
        outs = [torch.empty((wl.n_samples, wl.n_x, wl.n_t), device="cuda") for wl in wls]
        batch = srm3.Batch(plans, [wl.n_samples for wl in wls], outs)
        batch.capture()
        seeds = np.array([s for wl in wls for s in wl.seeds], dtype=np.uint64)
        return dict(state, batch=batch, seeds=seeds, outs=outs, held=_Held(batch, *plans))
    wl = _workload(case, seed)
    state["seeds"] = np.array(wl.seeds, dtype=np.uint64)
    if kind in ("step", "plan"):
        return dict(state, wl=wl)
    if kind == "fields":  # the transform takes any plan of the lattice: a fixed small scale
        plan = srm3.Plan.create(wl, eps=1e-3)
        return dict(state, plan=plan, C=_given_coeffs(case, seed), held=_Held(plan))
    plan = srm3.Plan.create(wl)
    return dict(state, plan=plan, held=_Held(plan))


def run(state):
    kind = state["kind"]
    if kind == "sample":
        return state["plan"].sample(state["seeds"])
    if kind == "coeffs":
        return state["plan"].coeffs(state["seeds"])
    if kind == "fields":
        return state["plan"].field_from_coeffs(state["C"])
    if kind == "step":
        with srm3.Plan.create(state["wl"]) as plan:
            u = plan.sample(state["seeds"])
            return {"u": u, "eps": plan.info().eps}
    if kind == "plan":
        with srm3.Plan.create(state["wl"]) as plan:
            S, q, sb2 = plan.tables()
            return {"S": S, "q": q, "sum_b2": sb2, "eps": plan.info().eps}
    if kind == "batch":
        state["batch"].run(state["seeds"])
        state["batch"].sync()
        return list(state["outs"])
    if kind == "stats":
        st = state["stats"]
        st.reset()
        st.add(state["u"])
        r = st.read()
        return {"hist": r["hist"].astype(np.int64), "below": r["below"], "above": r["above"],
                "power_sum": np.array(r["power_sum"]),
                "moments": np.array([r["mean"], r["variance"], r["skewness"], r["kurtosis"]])}
    raise ValueError(kind)


def _conv_flops(nk, nw, mixed):
    """Two complex 2-D transforms of the zero-padded lattice."""
    n = _pow2(2 * nk - 1) * _pow2((3 if mixed else 2) * nw - 1)
    return 2 * 5.0 * n * math.log2(n)


def _sampling_work(wl, n):
    """Coefficients and fields of n samples: the stored W table and its
    products where the user asks for it, else a self-convolution per sheet."""
    es = 4 if wl.precision == "fp32" else 8
    nl = wl.n_kappa * wl.n_omega
    if wl.storage == "table":
        flops, nbytes = 10.0 * wl.pair_terms_per_sample() * n, 4.0 * wl.pairs()
    else:
        flops, nbytes = 2.0 * n * _conv_flops(wl.n_kappa, wl.n_omega,
                                              wl.interactions == "mixed"), 0.0
    return nbytes + 3 * nl * es, flops


def _field_work(nk, nw, nx, nt, n, es):
    return n * nx * nt * es, n * 2.5 * nx * nt * math.log2(nx * nt)


def _plan_work(wl):
    """One evaluation of Eq. pure at the root: a real self-convolution."""
    return 3.0 * 8 * wl.n_kappa * wl.n_omega, 0.5 * _conv_flops(
        wl.n_kappa, wl.n_omega, wl.interactions == "mixed")


def work(case):
    kind = case["kind"]
    if kind == "stats":
        es = 4 if case["precision"] == "fp32" else 8
        return {"bytes": float(case["count"] * es + 8 * case["nbins"]), "flops": 9.0 * case["count"]}
    if kind == "batch":
        b = f = 0.0
        for wl in _batch_workloads(case, 0):
            sb, sf = _sampling_work(wl, wl.n_samples)
            fb, ff = _field_work(wl.n_kappa, wl.n_omega, wl.n_x, wl.n_t, wl.n_samples, 4)
            b, f = b + sb + fb, f + sf + ff
        return {"bytes": b, "flops": f}
    wl, n = _workload(case, 0), case["n"]
    es = 4 if case["precision"] == "fp32" else 8
    cbytes = 2.0 * n * 2 * case["nk"] * case["nw"] * es
    fb, ff = _field_work(case["nk"], case["nw"], case["nx"], case["nt"], n, es)
    pb, pf = _plan_work(wl)
    sb, sf = _sampling_work(wl, n)
    if kind == "fields":
        return {"bytes": cbytes + fb, "flops": ff}
    if kind == "plan":
        return {"bytes": pb, "flops": pf}
    if kind == "coeffs":
        return {"bytes": sb + cbytes, "flops": sf}
    if kind == "sample":
        return {"bytes": sb + fb, "flops": sf + ff}
    return {"bytes": pb + sb + fb, "flops": pf + sf + ff}


# ---------------------------------------------------------------------------
# The same quantities in 64 bits by plain torch: Eq. pure by fixed-point
# iteration with FFT self-convolutions, the coefficients by FFT
# self-convolutions, the fields by an inverse FFT.

def _spectrum(wl):
    dk, dw = wl.kappa_u / wl.n_kappa, wl.omega_u / wl.n_omega
    kap = torch.arange(wl.n_kappa, dtype=torch.float64, device="cuda")[:, None] * dk
    om = torch.arange(wl.n_omega, dtype=torch.float64, device="cuda")[None, :] * dw
    us = wl.k_vk * wl.U / math.log(wl.z / wl.z0)
    kaimal = 0.5 * (200 / (2 * math.pi)) * us * us * (wl.z / wl.U) / (
        1 + 50 * om * wl.z / (2 * math.pi * wl.U)) ** (5.0 / 3.0)
    a = wl.lam * om / (2 * math.pi * wl.U)
    S = kaimal * a / (math.pi * (a * a + kap * kap))
    S[:, 0] = 0.0
    return S


def _factors(wl):
    """a over (kappa index, omega index from -(n_omega - 1) on) and b over
    the lattice with g(i, j) = a(i) a(j) b(i + j).  The Gaussian envelope on
    i + j = k: (i - j)^2 = 2 (i - c)^2 + 2 (j - c)^2 - (k - 2c)^2, c a
    quarter of the lattice, where b stays near one."""
    nk, nw = wl.n_kappa, wl.n_omega
    if wl.envelope != "gauss":
        ta, tb = wl.envelope_tables()
        a = torch.zeros((nk, 2 * nw - 1), dtype=torch.float64, device="cuda")
        a[:, nw - 1:] = torch.from_numpy(ta).cuda()
        return a, torch.from_numpy(ta if tb is None else tb).cuda()
    sk, sw = wl.sigma_g * nk, wl.sigma_g * nw
    ck, cw = nk / 4.0, nw / 4.0
    ik = torch.arange(nk, dtype=torch.float64, device="cuda")[:, None]
    iw = torch.arange(-(nw - 1), nw, dtype=torch.float64, device="cuda")[None, :]
    a = torch.exp(-((ik - ck) / sk) ** 2 - ((iw - cw) / sw) ** 2)
    kw = iw[:, nw - 1:]
    b = torch.exp(0.5 * ((ik - 2 * ck) / sk) ** 2 + 0.5 * ((kw - 2 * cw) / sw) ** 2)
    return a, b


def _conv(h, nk, nw, mixed):
    """Sum over unordered pairs i + j = k of h_i h_j on the lattice; h over
    (..., kappa, signed omega)."""
    Nk, Nw = _pow2(2 * nk - 1), _pow2(4 * nw - 3 if mixed else 2 * nw - 1)
    x = h if mixed else h[..., nw - 1:]
    off = 2 * (nw - 1) if mixed else 0
    X = torch.fft.fftn(x, s=(Nk, Nw), dim=(-2, -1))
    c = torch.fft.ifftn(X * X, dim=(-2, -1))[..., :nk, off:off + nw]
    c = c if h.is_complex() else c.real
    c = c.clone()
    hp = h[..., nw - 1:]
    c[..., ::2, ::2] += (hp * hp)[..., :(nk + 1) // 2, :(nw + 1) // 2]
    if mixed:
        c[..., 0] = 0.0  # Kaimal spectra vanish at omega = 0: no sum pairs there
    return 0.5 * c


def _signed(pos, neg, mixed):
    """pos over omega >= 0 and neg over omega < 0 as one signed axis."""
    left = torch.flip(neg[..., 1:], dims=(-1,))
    return torch.cat([left if mixed else torch.zeros_like(left), pos], dim=-1)


def _exact_plan(wl):
    nk, nw, mixed = wl.n_kappa, wl.n_omega, wl.interactions == "mixed"
    dkdw = (wl.kappa_u / nk) * (wl.omega_u / nw)
    S = _spectrum(wl)
    a, b = _factors(wl)
    mask = (S > 0).double()
    origin = torch.ones_like(S)
    origin[0, 0] = 0.0
    q = mask.clone()
    x, near = wl.eps ** 2, 0
    for _ in range(400):
        h = a * a * _signed(q * origin, q * origin, mixed)
        g = torch.clamp(dkdw * b * b * _conv(h, nk, nw, mixed), min=0.0) * mask
        if wl.eps == 0.0:
            x = wl.target / float(g.max())
        new = mask / (1.0 - x * g)
        change = float((new - q).abs().max())
        q = new
        near = near + 1 if change < 2e-14 else 0
        if near >= 3:
            break
    return S, q, x * g, math.sqrt(x), a, b, dkdw


def _philox(seed, n):
    """n words of Philox4x32-10 with the given key, counters 0, 1, ..."""
    m32 = 0xFFFFFFFF
    c = [torch.arange((n + 3) // 4, dtype=torch.int64, device="cuda")]
    c += [torch.zeros_like(c[0]) for _ in range(3)]
    k0, k1 = seed & m32, (seed >> 32) & m32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        h0, h1 = (p0 >> 32) & m32, (p1 >> 32) & m32
        c = [h1 ^ c[1] ^ k0, p1 & m32, h0 ^ c[3] ^ k1, p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return torch.stack(c, dim=-1).reshape(-1)[:n]


def _exact_coeffs(wl, plan, seed):
    """Coefficients [2][nk][nw] (complex) of one sample."""
    S, q, sb2, eps, a, b, dkdw = plan
    nk, nw, mixed = wl.n_kappa, wl.n_omega, wl.interactions == "mixed"
    w = _philox(int(seed), 2 * nk * nw).reshape(2, nk, nw)
    y = torch.sqrt(q) * torch.polar(torch.ones((), dtype=torch.float64, device="cuda"),
                                    2 * math.pi * (w.double() + 0.5) * 2.0 ** -32)
    z = y.clone()
    z[:, 0, 0] = 0.0
    C = []
    for s in range(2):
        T = b * _conv(a * _signed(z[s], z[1 - s], mixed), nk, nw, mixed)
        C.append(2 * torch.sqrt(dkdw * S) * (1 - sb2) * y[s] + 2 * eps * dkdw * torch.sqrt(S) * T)
    return torch.stack(C)


def _exact_field(C, nk, nw, nx, nt):
    F = torch.zeros((nx, nt), dtype=torch.complex128, device="cuda")
    F[:nk, :nw] += C[0]
    F[:nk, (-torch.arange(nw, device="cuda")) % nt] += C[1]
    return torch.fft.ifft2(F).real * (nx * nt)


def _exact_samples(wl, plan):
    u = torch.empty((wl.n_samples, wl.n_x, wl.n_t), dtype=torch.float64, device="cuda")
    for i, s in enumerate(wl.seeds):
        u[i] = _exact_field(_exact_coeffs(wl, plan, s), wl.n_kappa, wl.n_omega, wl.n_x, wl.n_t)
    return u


def exact(case, seed):
    kind = case["kind"]
    if kind == "stats":
        u = _wave_values(case, seed).double()
        s = [float((u ** p).sum()) for p in (1, 2, 3, 4)]
        n = u.numel()
        m, e2, e3, e4 = (v / n for v in s)
        c2 = e2 - m * m
        c3 = e3 - 3 * m * e2 + 2 * m ** 3
        c4 = e4 - 4 * m * e3 + 6 * m * m * e2 - 3 * m ** 4
        return {"hist": None, "below": None, "above": None, "power_sum": np.array(s),
                "moments": np.array([m, c2, c3 / c2 ** 1.5, c4 / c2 ** 2])}
    if kind == "batch":
        return [_exact_samples(wl, _exact_plan(wl)) for wl in _batch_workloads(case, seed)]
    if kind == "fields":
        C = torch.view_as_complex(_given_coeffs(case, seed).double())
        return torch.stack([_exact_field(c, case["nk"], case["nw"], case["nx"], case["nt"])
                            for c in C])
    wl = _workload(case, seed)
    plan = _exact_plan(wl)
    if kind == "plan":
        S, q, sb2, eps = plan[:4]
        one = torch.where(S > 0, q, torch.ones_like(q))
        return {"S": S, "q": one, "sum_b2": sb2, "eps": eps}
    if kind == "coeffs":
        return torch.stack([torch.view_as_real(_exact_coeffs(wl, plan, s)) for s in wl.seeds])
    u = _exact_samples(wl, plan)
    return u if kind == "sample" else {"u": u, "eps": plan[3]}
