"""Sizes between the workloads: block and tile edges of the kernels that cut an
evaluation into padded tiles, odd electron counts per spin, the direct real-space
Ewald path, and slices of the reductions, against the FP64 oracle.

Tolerances are those of the parity tests: 1e-10 (FP64 form) and 1e-4 (mixed form)
relative to the largest magnitude, 1e-10 absolute for a Langevin step, 1e-12 for sums
taken in another order.
"""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1605_08423_gb300 import qmcmd as q
from paper_1605_08423_gb300 import synth

pytestmark = pytest.mark.gpu

ZETA = {1: (0.7,), 2: synth.ZETA_2, 3: (0.4446, 0.727, 1.962), 4: synth.ZETA_4}


def _workload(N, G, walkers, sweeps=1, seed=7):
    return synth.Workload(name="sizes", N=N, rs=1.3, zeta=ZETA[G], walkers=walkers, sweeps=sweeps, T_kelvin=1500.0,
                          seed=seed)


def _osys(wl, **kw):
    return orc.System(N=wl.N, L=wl.L, zeta=np.array(wl.zeta), coeff=wl.C, **kw)


def _sampled(wl, n, kappa=None):
    """|psi|^2-distributed configurations from the oracle's own chains."""
    X, _, _ = orc.vmc(_osys(wl, kappa=kappa), wl.R, W=n, n_sweeps=1, n_warmup=12, sigma=wl.sigma, seed=5, forces=False)
    return X


def _close(g, ref, tol):
    lp, el, dl, de = ref
    assert np.max(np.abs(g["el"] - el)) <= tol * np.max(np.abs(el))
    assert np.all(np.abs(g["lnpsi"] - lp) <= tol * np.maximum(np.abs(lp), 1.0))
    for key, v in (("dlnpsi", dl), ("del_", de)):
        rel = np.max(np.abs(g[key] - v), axis=(-1, -2)) / np.max(np.abs(v), axis=(-1, -2))
        assert np.all(rel <= tol), (key, rel)


# kappa L = 5 takes the tabulated real-space terms of the FP64 form, 6.5 the direct ones
@pytest.mark.parametrize("N,G,kl", [(2, 2, 5.0), (6, 1, 5.0), (10, 4, 6.5), (34, 3, 5.0), (46, 4, 6.5), (66, 1, 5.0),
                                    (66, 4, 5.0)])
def test_fp64_eval_config_between_tiles(N, G, kl):
    wl = _workload(N, G, 3)
    kappa = kl / wl.L
    X = _sampled(wl, 3, kappa)
    s = q.QMCSystem(q.Config.from_workload(wl, kappa=kappa), wl.R)
    _close(s.eval_config(X, wl.R), orc.eval_configs(_osys(wl, kappa=kappa), wl.R, X, derivs=True), 1e-10)


# n = 16 takes the FP64 elimination, above it the elimination on pairs of FP32 numbers;
# 4-column and 32-column edges, the largest block, kappa L with and without the short image polynomials
@pytest.mark.parametrize("N,G,kl", [(32, 2, 5.0), (34, 2, 5.0), (38, 3, 7.0), (64, 3, 5.0), (66, 2, 6.0), (126, 2, 5.0)])
def test_mixed_eval_config_between_tiles(N, G, kl):
    wl = _workload(N, G, 4)
    kappa = kl / wl.L
    X = _sampled(wl, 4, kappa)
    s = q.QMCSystem(q.Config.from_workload(wl, kappa=kappa, precision=q.QMC_MIXED), wl.R)
    _close(s.eval_config(X, wl.R), orc.eval_configs(_osys(wl, kappa=kappa), wl.R, X, derivs=True), 1e-4)


@pytest.mark.parametrize("N,G", [(2, 2), (10, 3), (34, 1), (66, 2)])
def test_twisted_eval_config_between_tiles(N, G):
    wl = _workload(N, G, 2)
    tw = synth.monkhorst_pack(4)[[11]]
    X = _sampled(wl, 2)
    g = q.QMCSystem(q.Config.from_workload(wl, twists=tw), wl.R).eval_config(X, wl.R)
    _close(g, orc.eval_configs_twist(_osys(wl, twist=np.asarray(tw[0])), wl.R, X, tw), 1e-10)


# 3N around the 32-wide tiles and each cluster size (1, 4, 8, 16 blocks)
@pytest.mark.parametrize("N", [2, 10, 22, 32, 34, 44, 64, 66, 76, 128])
def test_langevin_step_between_tiles(N):
    wl = _workload(N, 2, 2)
    s = q.QMCSystem(q.Config.from_workload(wl), wl.R)
    n = 3 * N
    rng = np.random.default_rng(N)
    R, Rprev, Sprev = wl.R.ravel().copy(), wl.R.ravel().copy(), None
    T = 1500.0 * synth.K_B_HARTREE_PER_KELVIN
    for step in range(2):
        A = rng.standard_normal((n, n))
        S = (A @ A.T / n + 0.3 * np.eye(n)) * 1e-2
        Sprev = S if Sprev is None else Sprev
        f = 0.1 * rng.standard_normal(n)
        ref = orc.langevin(R, Rprev, f, S, Sprev, T, 0.1, 30.0, orc.langevin_noise(wl.seed, step, n), box=wl.L)
        got = s.langevin_step(R, f, S, 1500.0, 0.1, s_mode=q.QMC_S_COV, alpha=30.0)
        assert np.max(np.abs(got - ref)) < 1e-10, step
        Rprev, Sprev, R = R, S, ref


def test_langevin_step_reports_a_late_negative_pivot():
    """S positive definite but for its last row: the factorisation fails in its last tile."""
    wl = _workload(128, 2, 2)
    s = q.QMCSystem(q.Config.from_workload(wl), wl.R)
    S = np.eye(384)
    S[383, 383] = -1.0
    with pytest.raises(q.QMCError):
        s.langevin_step(wl.R.ravel(), np.zeros(384), S, 1500.0, 0.1, s_mode=q.QMC_S_COV, alpha=30.0)


# fewer walkers than a slice, ragged slices, 16-wide tile edges of 3N, twists reduced together
@pytest.mark.parametrize("N,W,K", [(2, 2, 0), (6, 65, 0), (16, 333, 0), (34, 1000, 0), (10, 7 * 3, 3), (6, 130 * 2, 2)])
def test_reductions_match_the_accumulators(N, W, K):
    wl = _workload(N, 2, W, sweeps=3)
    tw = synth.monkhorst_pack(3)[1:1 + K] if K else None
    s = q.QMCSystem(q.Config.from_workload(wl, warmup=2, twists=tw), wl.R)
    g = s.energy_forces(wl.R)
    acc = s.accumulators()
    ref = orc.reduce_twists(acc, N, K) if K else orc.reduce(acc, N)
    for key in ("E", "E_err", "f", "S"):
        a, b = np.asarray(g[key]).ravel(), np.asarray(ref[key]).ravel()
        assert np.max(np.abs(a - b)) <= 1e-12 * W * np.max(np.abs(b)), key


# FP64 sweep with two warps a walker (few walkers, handle of its own) against one (many
# walkers): the same walkers' chains, to the bit
@pytest.mark.parametrize("N", [2, 10, 16, 34, 66, 128])
def test_sweep_does_not_depend_on_the_number_of_walkers(N):
    runs = []
    for W in (24, 640):
        wl = _workload(N, 2, W, sweeps=2)
        s = q.QMCSystem(q.Config.from_workload(wl, warmup=1, recompute_every=2), wl.R)
        g = s.energy_forces(wl.R)
        runs.append((s.walkers()[:24], s.accumulators()[:24], g["accept"]))
    assert np.array_equal(runs[0][0], runs[1][0])
    assert np.array_equal(runs[0][1], runs[1][1])
    assert runs[0][2] > 0.0
