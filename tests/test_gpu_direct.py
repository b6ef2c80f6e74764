"""The forms that narrow envelopes (sigma_g below about 0.22) and targets out of the
whole-lattice solve's reach take: the O(N^2) pair sums with W recomputed, sum and
difference pairs, and the eps search by level passes, against the FP64 oracle.

Tolerances: coefficients 2e-6 of max|C| in FP32, whose phasors are FP32, 1e-11 in
FP64 (tests/test_gpu_parity.py); plans meet the target to 1e-9 in FP32 and 1e-13 in
FP64; tables against the oracle's at the plan's own eps."""
from dataclasses import replace

import numpy as np
import pytest

import oracle
from paper_2310_03979_gb300 import srm3
from paper_2310_03979_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pow2 = lambda n: 1 << max(1, (n - 1).bit_length())  # noqa: E731


@pytest.mark.parametrize("precision,storage", [("fp32", "recompute"), ("fp32", "table"),
                                               ("fp64", "recompute")])
@pytest.mark.parametrize("interactions", ["sum", "mixed"])
@pytest.mark.parametrize("n", [1, 16, 17, 70])
@pytest.mark.parametrize("nk,nw,tile", [(24, 37, 32), (33, 64, 32), (9, 100, 16), (1, 20, 32),
                                        (20, 1, 16)])
def test_direct_pair_sums_against_oracle(oracle_lib, precision, storage, interactions, n, nk, nw,
                                         tile):
    """Half groups (up to 16 samples), one full group and a ragged second one; rows
    short and long of the 32- and 16-wide tiles; power at omega = 0."""
    if interactions == "mixed" and (storage == "table" or nw < 3):
        pytest.skip("mixed plans recompute W, difference pairs need three columns")
    wl = replace(W.small_case(nk=nk, nw=nw, nx=pow2(max(2, nk)), nt=pow2(max(2, 2 * nw)),
                              precision=precision, storage=storage, sigma_g=0.15, beta=0.4),
                 interactions=interactions)
    S = oracle.kaimal_lorentzian(nk, nw, wl.kappa_u, wl.omega_u, wl.U, wl.z)
    S[:, 0] = 0.4 * (S.max() or 1.0) / (1.0 + np.arange(nk))
    S[nk // 2, nw // 2] = 0.0
    mixed = interactions == "mixed"
    op = oracle.make_plan(S, wl.kappa_u, wl.omega_u, eps=0.1, beta=0.4, mixed=mixed,
                          env=oracle.Envelope("gauss", 0.15))
    seeds = list(range(3, 3 + n))
    with srm3.Plan.create(wl, table=S, eps=0.1) as p:
        if precision == "fp32":
            p.set_tile_width(tile)
        C = p.coeffs(seeds).cpu().numpy()
        assert not p.info().recursion_flags & srm3.SRM3_PAIRSUM_SEPARABLE
    C = C[..., 0] + 1j * C[..., 1]
    tol = 2e-6 if precision == "fp32" else 1e-11
    for i in sorted({0, n // 2, n - 1}):
        ref = op.coeffs(seeds[i])
        assert np.abs(C[i] - ref).max() <= tol * np.abs(ref).max()


def _check_tables(p, wl, S, env, atol):
    _, q, sb2 = p.tables()
    info = p.info()
    assert not info.recursion_flags & srm3.SRM3_REC_LATTICE_SOLVE
    assert abs(info.max_sum_b2 - wl.target) <= (1e-9 if wl.precision == "fp32" else 1e-13)
    ref = oracle.make_plan(S, wl.kappa_u, wl.omega_u, eps=info.eps, env=env)
    np.testing.assert_allclose(sb2, ref.sum_b2, atol=atol)
    return info


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("mask", ["full", "no_coarse_pairs", "window_missed"])
def test_level_search_of_a_narrow_envelope(oracle_lib, precision, mask):
    """The search from the coarse lattice's root and its two misses (the supports of
    test_eps_search_coarse_start), with the FP32 tables moved to the root."""
    wl = W.small_case(nk=256, nw=256, nx=256, nt=512, precision=precision, sigma_g=0.15)
    S = oracle.kaimal_lorentzian(256, 256, wl.kappa_u, wl.omega_u, wl.U, wl.z)
    if mask == "no_coarse_pairs":
        S[:, 0::4] = 0.0
    elif mask == "window_missed":
        S[:, 2::4] = 0.0
    with srm3.Plan.create(wl, table=S) as p:
        info = _check_tables(p, wl, S, oracle.Envelope("gauss", 0.15),
                             1e-9 if precision == "fp32" else 1e-13)
    assert (info.coarse_fk, info.coarse_fw) == (4, 4)
    assert bool(info.recursion_flags & srm3.SRM3_REC_COARSE_START) == (mask == "full")
    assert (info.coarse_passes == 0) == (mask == "no_coarse_pairs")


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nk,nw,envelope,target", [(128, 96, "separable", 0.98),
                                                   (256, 256, "separable", 0.99),
                                                   (130, 70, "gauss", 0.99)])
def test_level_search_where_the_solve_does_not_reach(oracle_lib, precision, nk, nw, envelope,
                                                     target):
    """A target that the solve's iterations circle without reaching, one past its
    cut-off on a lattice with a coarse start (the self-convolution form of the
    bulk), and the Gaussian envelope's factors.  A sum's rounding of 1e-14 grows
    by 1/(1 - s)^2 on its way to the next point: 1e-9."""
    wl = replace(W.small_case(nk=nk, nw=nw, nx=256, nt=512, precision=precision, target=target),
                 envelope=envelope)
    S = oracle.kaimal_lorentzian(nk, nw, wl.kappa_u, wl.omega_u, wl.U, wl.z)
    env = oracle.Envelope("gauss", wl.sigma_g)
    if envelope == "separable":
        env = oracle.Envelope("separable", table=wl.envelope_tables()[0])
    with srm3.Plan.create(wl, table=S) as p:
        _check_tables(p, wl, S, env, 1e-8 if precision == "fp32" else 1e-9)
