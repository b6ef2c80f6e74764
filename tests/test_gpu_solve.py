"""Eq. pure on the whole lattice at once (FFT self-convolutions, the search for
eps folded into the iteration) and the direct iterations of small FP64 plans:
one-row and one-column lattices, lattices at and just past a power of two,
targets from 0.05 to 0.95, sparse supports, the three kinds of envelope and
mixed-sign interactions.  Tables and eps against the FP64 oracle (plain
bisection) at the tolerances of tests/test_gpu_parity.py."""
from dataclasses import replace

import numpy as np
import pytest

import oracle
from paper_2310_03979_gb300 import srm3
from paper_2310_03979_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

pow2 = lambda n: 1 << max(1, (n - 1).bit_length())  # noqa: E731


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nk,nw,target,envelope,interactions,holes", [
    (1, 9, 0.5, "gauss", "sum", 0), (9, 1, 0.5, "gauss", "sum", 0), (3, 2, 0.3, "gauss", "sum", 0),
    (16, 16, 0.95, "gauss", "sum", 0), (17, 33, 0.05, "gauss", "sum", 0),
    (40, 33, 0.6, "gauss", "sum", 3), (33, 65, 0.9, "gauss", "sum", 7),
    (16, 17, 0.9, "separable", "sum", 0), (33, 16, 0.5, "sum", "sum", 0),
    (9, 1, 0.4, "sum", "sum", 0), (20, 20, 0.7, "separable", "sum", 5),
    (1, 9, 0.3, "gauss", "mixed", 0), (12, 11, 0.5, "gauss", "mixed", 0),
    (9, 22, 0.6, "gauss", "mixed", 4),
])
def test_tables_and_eps_against_oracle(oracle_lib, precision, nk, nw, target, envelope,
                                       interactions, holes):
    wl = replace(W.small_case(nk=nk, nw=nw, nx=pow2(max(2, nk)), nt=pow2(max(2, 2 * nw)),
                              precision=precision, target=target),
                 envelope=envelope, interactions=interactions)
    S = oracle.kaimal_lorentzian(nk, nw, wl.kappa_u, wl.omega_u, wl.U, wl.z)
    S[:, 0] = (S.max() or 1.0) / (1.0 + np.arange(nk))
    if holes:
        S.ravel()[::holes] = 0.0
    env = oracle.Envelope("gauss", wl.sigma_g)
    if envelope != "gauss":
        ta, tb = wl.envelope_tables()
        env = oracle.Envelope("separable", table=ta, table_b=tb)
    mixed = interactions == "mixed"
    op = oracle.make_plan(S, wl.kappa_u, wl.omega_u, target=target, env=env, mixed=mixed)
    with srm3.Plan.create(wl, table=S) as p:
        _, q, sb2 = p.tables()
        info = p.info()
    tol, rel = (1e-13, 1e-11) if precision == "fp64" else (1e-9, 2e-8)
    assert info.eps == pytest.approx(op.eps, rel=rel)
    assert abs(info.max_sum_b2 - target) <= tol
    np.testing.assert_allclose(q, op.q, rtol=rel)
    np.testing.assert_allclose(sb2, op.sum_b2, rtol=rel, atol=1e-15)


def test_no_pairs_is_refused():
    """A support without pairs has no eps: the error of the level search."""
    wl = W.small_case(nk=8, nw=8, nx=8, nt=16)
    S = np.zeros((8, 8))
    S[7, 7] = 1.0
    for precision in ("fp32", "fp64"):
        with pytest.raises(srm3.SRM3Error) as ei:
            srm3.Plan.create(wl, table=S, precision=precision)
        assert ei.value.code == -4


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("interactions", ["sum", "mixed"])
@pytest.mark.parametrize("n,support", [
    (8, [(4, 6), (6, 3)]), (8, [(4, 2), (5, 1), (7, 2)]), (8, [(4, 3), (6, 2), (6, 5), (7, 6)]),
    (256, "upper half"),
])
def test_no_pairs_is_refused_whatever_the_rounding(precision, interactions, n, support):
    """Supports of several points, no two of which sum to a third: the
    transforms' rounding is not a pair sum."""
    S = np.zeros((n, n))
    if isinstance(support, str):
        if interactions == "mixed":
            pytest.skip("points of one half have difference pairs")
        r = np.random.default_rng(2)
        S[r.integers(n // 2 + 1, n, 500), r.integers(n // 2 + 1, n, 500)] = 1.0
    else:
        for k in support:
            S[k] = 1.0
    wl = replace(W.small_case(nk=n, nw=n, nx=n, nt=2 * n, precision=precision),
                 interactions=interactions)
    with pytest.raises(srm3.SRM3Error) as ei:
        srm3.Plan.create(wl, table=S)
    assert ei.value.code == -4


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_weak_pairs_among_many_points(oracle_lib, precision):
    """200 points with no pairs among them and one that has pairs with them, of
    weight 2e-7 and less: far below the largest sums the transforms could hold."""
    S = np.zeros((64, 64))
    r = np.random.default_rng(4)
    S[r.integers(43, 64, 200), r.integers(53, 64, 200)] = 1.0
    S[1, 1] = S[40, 50] = S[41, 51] = 1.0
    wl = W.small_case(nk=64, nw=64, nx=64, nt=128, precision=precision)
    op = oracle.make_plan(S, wl.kappa_u, wl.omega_u, target=wl.target)
    with srm3.Plan.create(wl, table=S) as p:
        _, q, sb2 = p.tables()
        info = p.info()
    rel = 1e-11 if precision == "fp64" else 2e-8
    assert info.eps == pytest.approx(op.eps, rel=rel)
    np.testing.assert_allclose(sb2, op.sum_b2, rtol=rel, atol=1e-15)
    np.testing.assert_allclose(q, op.q, rtol=rel)


@pytest.mark.parametrize("nk,nw", [(486, 202), (60, 44), (12, 9)])
def test_fp64_separable_tables_keep_fp64_accuracy(oracle_lib, nk, nw):
    """FP64 plans of the wind-field envelope, whose sums span the widest range:
    where the transform's rounding keeps the solve's sums moving the tables come
    from the level pass.  Against the oracle's tables at the plan's eps: 5e-13 of
    max sum_b2 (an accepted last change of 3e-14, converging at 0.3 or better,
    leaves 4e-14; as much again for eps, and room for the level pass's sums)."""
    wl = replace(W.small_case(nk=nk, nw=nw, nx=512, nt=512, precision="fp64"), envelope="sum")
    with srm3.Plan.create(wl) as p:
        S, q, sb2 = p.tables()
        info = p.info()
    assert abs(info.max_sum_b2 - wl.target) <= 1e-12
    ta, tb = wl.envelope_tables()
    ref = oracle.make_plan(S, wl.kappa_u, wl.omega_u, eps=info.eps,
                           env=oracle.Envelope("separable", table=ta, table_b=tb))
    assert np.abs(sb2 - ref.sum_b2).max() <= 5e-13 * ref.sum_b2.max()


class _Tables:
    """A workload with separable tables of its own."""
    envelope = "separable"

    def __init__(self, wl, a):
        self._wl, self._a = wl, a

    def __getattr__(self, name):
        return getattr(self._wl, name)

    def envelope_tables(self):
        return self._a, None


# Sums close to 1, where 1/(1 - s) must not be cut off.  Tolerances: a rounding of
# a sum (1e-14) reaches a dependent sum times q^2 = 1/(1 - s)^2, and FP32 plans
# move their tables to the root to first order (1e-9 of it); a cut-off q = 100
# is off by tens of per cent and its dependents by 1e-6 and more.
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nk,nw,peak", [(128, 96, 0.992), (32, 32, 0.992)])
def test_fixed_eps_with_sums_close_to_one(oracle_lib, precision, nk, nw, peak):
    """A separable bispectrum at a given eps: points above 0.99 feed others."""
    wl = replace(W.small_case(nk=nk, nw=nw, nx=pow2(nk), nt=pow2(2 * nw), precision=precision),
                 envelope="separable")
    S = oracle.kaimal_lorentzian(nk, nw, wl.kappa_u, wl.omega_u, wl.U, wl.z)
    env = oracle.Envelope("separable", table=wl.envelope_tables()[0])
    op = oracle.make_plan(S, wl.kappa_u, wl.omega_u, target=peak, env=env)
    with srm3.Plan.create(wl, table=S, eps=op.eps) as p:
        _, q, sb2 = p.tables()
    np.testing.assert_allclose(q, op.q, rtol=1e-8)
    np.testing.assert_allclose(sb2, op.sum_b2, atol=1e-9)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("kind", ["separable", "gauss", "mixed"])
@pytest.mark.parametrize("target", [0.992, 0.995])
def test_targets_close_to_one_on_sparse_supports(oracle_lib, precision, kind, target):
    """The largest sum feeds other points: tables at the plan's eps."""
    mixed = kind == "mixed"
    if kind == "separable":
        wl = W.small_case(nk=1, nw=6, nx=2, nt=16, precision=precision, target=target)
        S = np.ones((1, 6))
        a = np.sqrt(np.array([[0.0, 1.0, 1.0, 0.004, 0.0, 0.15]]))
        wl, env = _Tables(wl, a), oracle.Envelope("separable", table=a)
    else:
        wl = replace(W.small_case(nk=20, nw=20, nx=32, nt=64, precision=precision, target=target),
                     interactions="mixed" if mixed else "sum")
        S = oracle.kaimal_lorentzian(20, 20, wl.kappa_u, wl.omega_u, wl.U, wl.z)
        S[:, 0] = S.max() / (1.0 + np.arange(20))
        S[np.random.default_rng(5).random(S.shape) < 0.5] = 0.0
        env = oracle.Envelope("gauss", wl.sigma_g)
    with srm3.Plan.create(wl, table=S) as p:
        _, q, sb2 = p.tables()
        info = p.info()
    assert abs(info.max_sum_b2 - target) <= 1e-9
    ref = oracle.make_plan(S, wl.kappa_u, wl.omega_u, eps=info.eps, env=env, mixed=mixed)
    np.testing.assert_allclose(sb2, ref.sum_b2, atol=1e-6 if kind != "mixed" else 1e-9)
    np.testing.assert_allclose(q, ref.q, rtol=1e-5 if kind != "mixed" else 1e-6)


def test_mixed_fixed_point_reached_slowly(oracle_lib):
    """An eps 1e-7 below the largest that has a fixed point: 225 direct iterations
    (numpy), more than the small lattice's pass takes by itself.  Tolerance: there
    q moves by 1/sqrt(1e-7) of a relative change of the sums, 1e-15 each."""
    wl = replace(W.small_case(nk=4, nw=6, nx=4, nt=16, precision="fp64"), interactions="mixed")
    S = oracle.kaimal_lorentzian(4, 6, wl.kappa_u, wl.omega_u, wl.U, wl.z)
    eps = 1.1686150240765587
    op = oracle.make_plan(S, wl.kappa_u, wl.omega_u, eps=eps, mixed=True)
    with srm3.Plan.create(wl, table=S, eps=eps) as p:
        _, q, sb2 = p.tables()
        assert p.info().fixed_point_iterations > 96
    np.testing.assert_allclose(sb2, op.sum_b2, atol=1e-8)


def _timings(p):
    return srm3.get_timings(p.handle)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_info_says_where_the_tables_come_from(precision):
    """The whole-lattice solve has a flag of its own, counts as one search pass and,
    where the plan keeps its tables, as one evaluation of them; its time is in
    the passes' times.  Level passes (a target close to 1, a narrow envelope)
    report no solve."""
    wl = W.small_case(nk=40, nw=30, nx=64, nt=64, precision=precision)
    with srm3.Plan.create(wl) as p:
        i, t = p.info(), _timings(p)
        assert i.recursion_flags & srm3.SRM3_REC_LATTICE_SOLVE
        assert (i.root_passes_fp32, i.root_passes) == (1, 1)
        assert t.recursion_fp32_ms > 0 and (t.recursion_fp64_ms > 0) == (precision == "fp64")
    sep = replace(wl, envelope="separable")
    for eps in (None, 0.5):
        with srm3.Plan.create(sep, eps=eps) as p:
            i, t = p.info(), _timings(p)
            assert i.recursion_flags & srm3.SRM3_REC_LATTICE_SOLVE
            assert not i.recursion_flags & srm3.SRM3_REC_TABLES_MOVED
            assert i.root_passes_fp32 == (eps is None)
            assert t.recursion_fp32_ms > 0 and t.recursion_fp64_ms > 0
            assert t.recursion_ms == pytest.approx(t.recursion_fp32_ms + t.recursion_fp64_ms, rel=1e-3)
    for narrow in (replace(wl, target=0.995), replace(wl, sigma_g=0.15)):
        with srm3.Plan.create(narrow) as p:
            assert not p.info().recursion_flags & srm3.SRM3_REC_LATTICE_SOLVE


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nk,nw,envelope,eps", [(256, 128, "sum", 50.0), (94, 603, "sum", 63.0),
                                                (128, 256, "separable", 1.5)])
def test_separable_tables_at_a_given_eps_keep_fp64_rounding(oracle_lib, precision, nk, nw, envelope,
                                                           eps):
    """Tables of either precision's plans are FP64's.  Level passes are 1e-15 to 3e-15
    from the oracle here (a sum of some 1e4 pairs, rounded in another order)."""
    wl = replace(W.small_case(nk=nk, nw=nw, nx=512, nt=2048, precision=precision), envelope=envelope)
    ta, tb = wl.envelope_tables()
    with srm3.Plan.create(wl, eps=eps) as p:
        S, q, sb2 = p.tables()
    ref = oracle.make_plan(S, wl.kappa_u, wl.omega_u, eps=eps,
                           env=oracle.Envelope("separable", table=ta, table_b=tb))
    assert 0.01 < ref.sum_b2.max() < 0.5
    assert np.abs(sb2 - ref.sum_b2).max() <= 5e-15


@pytest.mark.parametrize("scale", [1e-25, 1e-9, 1e9, 1e25])
def test_separable_tables_of_any_magnitude(oracle_lib, scale):
    """Tables far outside FP32's range: eps alone answers for their magnitude."""
    wl = replace(W.small_case(nk=24, nw=20), envelope="separable")
    S = oracle.kaimal_lorentzian(24, 20, wl.kappa_u, wl.omega_u, wl.U, wl.z)
    with srm3.Plan.create(wl, table=S) as p:
        one = p.tables()[2]
        eps = p.info().eps
    with srm3.Plan.create(_Tables(wl, scale * wl.envelope_table()), table=S) as p:
        np.testing.assert_allclose(p.tables()[2], one, rtol=1e-12, atol=1e-18)
        assert p.info().eps == pytest.approx(eps / scale ** 3, rel=1e-12)


@pytest.mark.parametrize("nk,nw", [(12, 11), (40, 70), (100, 90)])
def test_fp32_mixed_tables_are_the_fp64_fixed_point(oracle_lib, nk, nw):
    """Tables of FP32 plans with mixed interactions at their own eps: FP64's fixed
    point, as those of FP64 plans (some 1e4 pairs a sum, iterated: 1e-14)."""
    wl = replace(W.small_case(nk=nk, nw=nw, nx=pow2(nk), nt=pow2(2 * nw)), interactions="mixed")
    with srm3.Plan.create(wl) as p:
        S, q, sb2 = p.tables()
        info = p.info()
    assert abs(info.max_sum_b2 - wl.target) <= 1e-9
    ref = oracle.make_plan(S, wl.kappa_u, wl.omega_u, eps=info.eps, mixed=True)
    assert np.abs(sb2 - ref.sum_b2).max() <= 3e-14


@pytest.mark.parametrize("nk,nw", [(2, 4096), (2048, 2), (2049, 2), (1025, 3), (3, 2049)])
def test_separable_tables_at_the_longest_transforms(oracle_lib, nk, nw):
    """The solve's transforms at 4096 points and just past 2048, and the level pass
    beyond: the tables of an FP32 plan against the oracle (some 1e3 pairs a sum)."""
    wl = replace(W.small_case(nk=nk, nw=nw, nx=pow2(nk), nt=pow2(2 * nw)), envelope="separable")
    ta, _ = wl.envelope_tables()
    S = np.ones((nk, nw))
    with srm3.Plan.create(wl, table=S) as p:
        _, q, sb2 = p.tables()
        info = p.info()
    assert bool(info.recursion_flags & srm3.SRM3_REC_LATTICE_SOLVE) == (nk <= 2048)
    ref = oracle.make_plan(S, wl.kappa_u, wl.omega_u, eps=info.eps,
                           env=oracle.Envelope("separable", table=ta))
    assert np.abs(sb2 - ref.sum_b2).max() <= 1e-13 * max(1.0, ref.q.max() ** 2)
