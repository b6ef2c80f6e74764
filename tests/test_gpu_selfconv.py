"""The pair sum as an FFT self-convolution (Gaussian envelope with W recomputed,
FP32 plans in double-float and FP64 plans in FP64) where it can go wrong: grids
just below, at and past a power of two, one-row and one-column lattices, more
samples than the scratch holds at a time, the widest range of the envelope's
factors that takes this form, a biphase, and mixed-sign interactions with
power at omega = 0.  Coefficients against the FP64 oracle at the tolerances
of the O(N^2) forms (tests/test_gpu_parity.py): 2e-6 of max|C| in FP32, whose
phasors are FP32, 1e-11 in FP64."""
from dataclasses import replace

import numpy as np
import pytest

import oracle
from paper_2310_03979_gb300 import srm3
from paper_2310_03979_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp32": 2e-6, "fp64": 1e-11}
pow2 = lambda n: 1 << max(1, (n - 1).bit_length())  # noqa: E731


def _case(nk, nw, precision, sigma_g=0.25, beta=0.0, interactions="sum"):
    return replace(W.small_case(nk=nk, nw=nw, nx=pow2(max(2, nk)), nt=pow2(max(2, 2 * nw)),
                                precision=precision, sigma_g=sigma_g, beta=beta),
                   interactions=interactions)


def _cplx(C):
    C = C.cpu().numpy()
    return C[..., 0] + 1j * C[..., 1]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nk,nw,sigma_g,beta,interactions", [
    (1, 9, 0.25, 0.0, "sum"), (9, 1, 0.25, 0.0, "sum"), (2, 2, 0.25, 0.3, "sum"),
    (16, 16, 0.25, 0.0, "sum"), (17, 33, 0.25, 1.1, "sum"), (33, 17, 0.6, 0.0, "sum"),
    (8, 129, 0.25, 0.0, "sum"), (64, 32, 0.225, 0.0, "sum"), (40, 64, 0.225, 2.0, "sum"),
    (1, 9, 0.25, 0.0, "mixed"), (9, 2, 0.25, 0.5, "mixed"), (11, 22, 0.25, 0.0, "mixed"),
    (12, 43, 0.225, 0.7, "mixed"),
])
def test_coefficients_against_oracle(oracle_lib, precision, nk, nw, sigma_g, beta, interactions):
    wl = _case(nk, nw, precision, sigma_g, beta, interactions)
    S = oracle.kaimal_lorentzian(nk, nw, wl.kappa_u, wl.omega_u, wl.U, wl.z)
    S[:, 0] = 0.4 * S.max() / (1.0 + np.arange(nk))  # power at omega = 0 as well
    S[nk // 2, nw // 2] = 0.0
    mixed = interactions == "mixed"
    eps = 0.1
    op = oracle.make_plan(S, wl.kappa_u, wl.omega_u, eps=eps, beta=beta, mixed=mixed,
                          env=oracle.Envelope("gauss", sigma_g))
    with srm3.Plan.create(wl, table=S, eps=eps) as p:
        C = _cplx(p.coeffs([3, 11]))
        info = p.info()
        assert bool(info.recursion_flags & srm3.SRM3_PAIRSUM_SEPARABLE) == (precision == "fp32")
    for i, s in enumerate((3, 11)):
        ref = op.coeffs(s)
        assert np.abs(C[i] - ref).max() <= TOL[precision] * np.abs(ref).max()


@pytest.mark.parametrize("precision,interactions,n", [("fp32", "sum", 100), ("fp32", "mixed", 100),
                                                      ("fp64", "sum", 100)])
def test_samples_do_not_depend_on_the_scratch(precision, interactions, n):
    """A lattice one past a power of two, whose padded rows are four times as
    long: the scratch takes fewer samples at a time than the call has."""
    wl = _case(24, 65, precision, interactions=interactions)
    with srm3.Plan.create(wl, eps=0.4) as p:
        C = p.coeffs(list(range(1, n + 1)))
        for j in (0, 41, 42, n - 1):
            assert torch.equal(C[j], p.coeffs([j + 1])[0])


@pytest.mark.parametrize("captured,timed", [(False, False), (True, False), (False, True)])
def test_batch_lanes_match_plans_alone(captured, timed):
    """More lattices than a batch has lanes, of every kind side by side (shape
    groups, FP64, mixed, a plan of the O(N^2) pair sum): each plan's fields
    are those of the plan alone, also when run again with other seeds."""
    wls = [_case(nk, nw, "fp32") for nk, nw in
           [(8, 8), (16, 8), (8, 16), (33, 20), (64, 40), (20, 64), (12, 12), (40, 9), (9, 40), (64, 40)]]
    wls += [_case(16, 16, "fp64"), _case(12, 9, "fp32", interactions="mixed"),
            _case(20, 24, "fp32", sigma_g=0.1)]
    wls[-4] = replace(wls[-4], U=25.0)
    plans = [srm3.Plan.create(w, storage="recompute") for w in wls]
    counts = [1 + i % 5 for i in range(len(wls))]
    outs = [torch.empty((c, w.n_x, w.n_t), device="cuda",
                        dtype=torch.float64 if w.precision == "fp64" else torch.float32)
            for c, w in zip(counts, wls)]
    batch = srm3.Batch(plans, counts, outs)
    batch.enable_timing(timed)
    if captured:
        batch.capture()
    for base in (3, 5000):
        seeds = [np.arange(base + 100 * i, base + 100 * i + c, dtype=np.uint64)
                 for i, c in enumerate(counts)]
        batch.run(np.concatenate(seeds))
        batch.sync()
        got = [o.clone() for o in outs]
        for p, s, g in zip(plans, seeds, got):
            assert torch.equal(p.sample(s), g)
    batch.destroy()
    for p in plans:
        p.destroy()


@pytest.mark.parametrize("nk,nw,sigma_g,interactions", [
    (90, 117, 0.25, "sum"), (90, 117, 0.2237, "sum"), (64, 65, 0.3, "sum"), (1, 50, 0.25, "sum"),
    (40, 33, 0.5, "mixed"), (20, 70, 0.2237, "mixed"),
])
def test_fp64_coefficients_keep_the_rounding_of_direct_sums(oracle_lib, nk, nw, sigma_g,
                                                            interactions):
    """FP64 coefficients as close to the oracle's as directly summed pairs are: 3e-16
    in the norm, the rounding of the phasors, tables and outputs of both sides.
    A transform in FP64, whose rounding is relative to its largest values and
    multiplied by the envelope's factor, leaves 8e-16 to 2e-15."""
    wl = _case(nk, nw, "fp64", sigma_g, 0.0, interactions)
    S = oracle.kaimal_lorentzian(nk, nw, wl.kappa_u, wl.omega_u, wl.U, wl.z)
    S[:, 0] = S.max() / (1.0 + np.arange(nk))
    op = oracle.make_plan(S, wl.kappa_u, wl.omega_u, target=0.5, mixed=interactions == "mixed",
                          env=oracle.Envelope("gauss", sigma_g))
    with srm3.Plan.create(wl, table=S, eps=op.eps) as p:
        C = _cplx(p.coeffs([1, 2, 3]))
    for i in range(3):
        ref = op.coeffs(i + 1)
        assert np.linalg.norm(C[i] - ref) <= 5e-16 * np.linalg.norm(ref)


@pytest.mark.parametrize("captured", [False, True])
def test_capped_batch_runs_in_small_launches_with_the_same_fields(captured):
    """A cap of one CTA leaves launches of one sample each, on the batch stream alone;
    the fields are the uncapped batch's, bit for bit."""
    wls = [_case(64, 40, "fp32"), replace(_case(64, 40, "fp32"), U=25.0), _case(20, 64, "fp32"),
           _case(12, 9, "fp32", interactions="mixed"), _case(16, 16, "fp64")]
    plans = [srm3.Plan.create(w, storage="recompute") for w in wls]
    counts = [5, 2, 3, 4, 2]
    outs = [torch.empty((c, w.n_x, w.n_t), device="cuda",
                        dtype=torch.float64 if w.precision == "fp64" else torch.float32)
            for c, w in zip(counts, wls)]
    seeds = np.arange(7, 7 + sum(counts), dtype=np.uint64)
    got = []
    for cap in (0, 1):
        with srm3.Batch(plans, counts, outs) as batch:
            batch.set_max_ctas(cap)
            if captured:
                batch.capture()
            for o in outs:
                o.fill_(float("nan"))
            batch.run(seeds)
            batch.sync()
            got.append([o.clone() for o in outs])
    for a, b in zip(*got):
        assert torch.equal(a, b)
    for p in plans:
        p.destroy()


@pytest.mark.parametrize("nk,nw,interactions", [(1, 2048, "sum"), (1, 2049, "sum"), (2048, 1, "sum"),
                                                (2049, 1, "sum"), (1, 1366, "mixed"),
                                                (1, 1367, "mixed")])
def test_fp64_coefficients_at_the_longest_transforms(oracle_lib, nk, nw, interactions):
    """Triple-float rows and columns reach 4096 points; the next lattice takes the
    direct sums."""
    wl = _case(nk, nw, "fp64", 0.25, 0.3, interactions)
    S = oracle.kaimal_lorentzian(nk, nw, wl.kappa_u, wl.omega_u, wl.U, wl.z)
    S[:, 0] = 1.0 / (1.0 + np.arange(nk))
    mixed = interactions == "mixed"
    op = oracle.make_plan(S, wl.kappa_u, wl.omega_u, eps=0.02, beta=0.3, mixed=mixed)
    with srm3.Plan.create(wl, table=S, eps=0.02) as p:
        C = _cplx(p.coeffs([5, 6]))
    for i in range(2):
        ref = op.coeffs(5 + i)
        assert np.abs(C[i] - ref).max() <= TOL["fp64"] * np.abs(ref).max()
