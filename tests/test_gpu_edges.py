"""Calls at the edges of what the entry points take: no electron near a proton, the
largest reciprocal-space cutoff, very large meshes, far electrons, short runs.

Tolerances against the FP64 oracle are those of the parity tests: 1e-10 (FP64 form)
and 1e-4 (mixed form) relative to the largest magnitude.
"""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1605_08423_gb300 import qmcmd as q
from paper_1605_08423_gb300 import synth

pytestmark = pytest.mark.gpu

ZETA = {1: (0.7,), 2: synth.ZETA_2, 4: synth.ZETA_4, 8: (0.2, 0.3, 0.45, 0.7, 1.0, 1.5, 2.0, 3.0)}


def _workload(N, G, walkers, rs=1.3, **kw):
    return synth.Workload(name="edges", N=N, rs=rs, zeta=ZETA[G], walkers=walkers, T_kelvin=1500.0,
                          **{"seed": 7, "sweeps": 1, **kw})


def _osys(wl, **kw):
    return orc.System(N=wl.N, L=wl.L, zeta=np.array(wl.zeta), coeff=wl.C, **kw)


def _sampled(wl, n):
    """|psi|^2-distributed configurations from the oracle's own chains."""
    X, _, _ = orc.vmc(_osys(wl), wl.R, W=n, n_sweeps=1, n_warmup=12, sigma=wl.sigma, seed=5, forces=False)
    return X


def _close(g, ref, tol):
    lp, el, dl, de = ref
    assert np.max(np.abs(g["el"] - el)) <= tol * np.max(np.abs(el))
    assert np.all(np.abs(g["lnpsi"] - lp) <= tol * np.maximum(np.abs(lp), 1.0))
    for key, v in (("dlnpsi", dl), ("del_", de)):
        rel = np.max(np.abs(g[key] - v), axis=(-1, -2)) / np.max(np.abs(v), axis=(-1, -2))
        assert np.all(rel <= tol), (key, rel)


def _pushed_out(X, R, L, r_min):
    """X with every electron closer than r_min to its nearest proton moved out to r_min."""
    d = X[:, :, None, :] - R[None, None]
    d -= L * np.rint(d / L)
    r = np.linalg.norm(d, axis=-1)
    a = np.argmin(r, axis=-1)
    rmin = np.take_along_axis(r, a[..., None], -1)
    dmin = np.take_along_axis(d, a[..., None, None], 2)[:, :, 0]
    return np.where(rmin < r_min, R[a] + dmin * (r_min / rmin), X)


# the mixed sample without a single close pair (no electron within 0.3 bohr of a proton):
# its list of close pairs is empty and shares its place with the phase table built next
@pytest.mark.parametrize("N,G,W", [(16, 2, 300), (34, 2, 48), (128, 4, 4)])
def test_mixed_sample_without_close_pairs(N, G, W):
    wl = _workload(N, G, W)
    X = _pushed_out(_sampled(wl, 2 * W), wl.R, wl.L, 0.45)
    X = X[np.argsort([orc.slater_condition(_osys(wl), wl.R, x) for x in X])[:W]]   # FP32: away from the nodes
    s = q.QMCSystem(q.Config.from_workload(wl, precision=q.QMC_MIXED), wl.R)
    ref = orc.eval_configs(_osys(wl), wl.R, X, derivs=True)
    for _ in range(3):
        _close(s.eval_config(X, wl.R), ref, 1e-4)


# The order of the orbitals does not change |det|, only the order of the elimination: ln|psi|
# of two handles whose coefficients are column permutations of each other differs by the
# elimination's rounding.  First order, delta ln|det| = tr(A^-1 E) with rounding errors
# E_ij of random sign, some u sqrt(n) max|A| each after n steps: |delta| <~ u sqrt(n)
# |A^-1|_F max|A|; three times that per block (u = 2^-53), and the result's own last place.
@pytest.mark.parametrize("N", [34, 64, 126])
def test_mixed_determinant_is_eliminated_in_fp64(N):
    wl = _workload(N, 2, 24)
    X, n = _sampled(wl, 24), N // 2
    perm = np.random.default_rng(1).permutation(n)
    lp = [q.QMCSystem(q.Config.from_workload(wl, precision=q.QMC_MIXED, coeff=C), wl.R).eval_config(X, wl.R)["lnpsi"]
          for C in (wl.C, np.ascontiguousarray(wl.C[:, perm]))]
    u = 2.0 ** -53
    for k, x in enumerate(X):
        A = np.asarray(orc.slater_matrices(_osys(wl), wl.R, x)).reshape(2, n, n)
        tol = sum(3 * u * np.sqrt(n) * np.linalg.norm(np.linalg.inv(a)) * np.max(np.abs(a)) for a in A)
        assert abs(lp[0][k] - lp[1][k]) <= tol + 4 * u * abs(lp[0][k]), (k, lp[0][k] - lp[1][k], tol)


# the largest cutoff: 3576 reciprocal vectors beside the sample's work space in shared memory
@pytest.mark.parametrize("N,G,twisted", [(84, 1, True), (128, 1, True), (128, 1, False)])
def test_sample_at_the_largest_reciprocal_cutoff(N, G, twisted):
    wl = _workload(N, G, 2)
    tw = synth.monkhorst_pack(4)[[11]] if twisted else None
    X = _sampled(wl, 2)[:1]
    g = q.QMCSystem(q.Config.from_workload(wl, twists=tw, mmax=12), wl.R).eval_config(X, wl.R)
    if twisted:
        ref = orc.eval_configs_twist(_osys(wl, twist=np.asarray(tw[0]), mmax=12), wl.R, X, tw)
    else:
        ref = orc.eval_configs(_osys(wl, mmax=12), wl.R, X, derivs=True)
    _close(g, ref, 1e-10)


# more twists than a grid's second and third dimensions hold (65535): 65537 points of the
# 41 x 41 x 41 mesh, two walkers each, reduced on their own and averaged; the tolerance is
# that of sums taken in another order
def test_more_twists_than_a_grid_dimension_holds():
    K = 65537
    wl = _workload(2, 1, 2 * K)
    s = q.QMCSystem(q.Config.from_workload(wl, warmup=1, twists=synth.monkhorst_pack(41)[:K]), wl.R)
    g, ref = s.energy_forces(wl.R), orc.reduce_twists(s.accumulators(), 2, K)
    for key in ("E", "E_err", "f", "S"):
        a, b = np.asarray(g[key]).ravel(), np.asarray(ref[key]).ravel()
        assert np.max(np.abs(a - b)) <= 1e-12 * K * np.max(np.abs(b)), key


# every sum in a fixed order, also with the e-e-n-n Jastrow term: the same call on two
# handles gives the same accumulators to the bit
@pytest.mark.parametrize("N,G,mixed,twisted", [(54, 4, True, False), (128, 4, True, False), (126, 2, True, False),
                                               (30, 2, False, False), (66, 2, False, False), (22, 2, False, True)])
def test_eenn_samples_are_reproducible(N, G, mixed, twisted):
    wl = _workload(N, G, 200, sweeps=2)
    f = 0.02 * np.random.default_rng(3).standard_normal((N, N))
    runs = []
    for _ in range(3):
        s = q.QMCSystem(q.Config.from_workload(wl, warmup=2, fj=f + f.T, precision=q.QMC_MIXED if mixed else q.QMC_FP64,
                                               twists=synth.monkhorst_pack(2)[:2] if twisted else None), wl.R)
        s.energy_forces(wl.R)
        runs.append(s.accumulators())
    assert np.array_equal(runs[0], runs[1]) and np.array_equal(runs[0], runs[2])


# an electron so far from every proton that its orbitals are some 1e-302 (still normal numbers):
# the determinant is not singular and all terms are finite
def test_fp64_sample_of_a_far_electron():
    wl = synth.Workload(name="far", N=2, rs=39.0, zeta=(0.8,), walkers=2, sweeps=1, seed=3)
    X = np.random.default_rng(5).uniform(0.0, wl.L, (200000, 3))
    d = X[:, None] - wl.R
    t = np.min((wl.L / np.pi) ** 2 * np.sum(np.sin(np.pi * d / wl.L) ** 2, -1), -1)
    far = X[(0.8 * t > 691.0) & (0.8 * t < 699.0)][:2]
    X = np.stack([far, wl.R[1] + [[0.3, 0.2, 0.4], [0.5, -0.2, 0.1]]], 1)
    g = q.QMCSystem(q.Config.from_workload(wl), wl.R).eval_config(X, wl.R)
    # the oracle's dual numbers hold 1/phi^2: orbitals scaled by 2^500, which only shifts ln|psi|
    osys = orc.System(N=2, L=wl.L, zeta=np.array(wl.zeta), coeff=wl.C * 2.0 ** 500)
    lp, el, dl, de = orc.eval_configs(osys, wl.R, X, derivs=True)
    assert all(np.all(np.isfinite(v)) for v in (lp, el, dl, de))
    _close(g, (lp - 1000.0 * np.log(2.0), el, dl, de), 1e-10)


# the largest number of Gaussians, whose basis tiles take the most shared memory, at each
# size of the orbital kernels
@pytest.mark.parametrize("N,twisted", [(32, True), (34, True), (34, False), (66, False)])
def test_fp64_sample_with_eight_gaussians(N, twisted):
    wl = _workload(N, 8, 2)
    tw = synth.monkhorst_pack(4)[[11]] if twisted else None
    X = _sampled(wl, 2)[:1]
    g = q.QMCSystem(q.Config.from_workload(wl, twists=tw), wl.R).eval_config(X, wl.R)
    if twisted:
        ref = orc.eval_configs_twist(_osys(wl, twist=np.asarray(tw[0])), wl.R, X, tw)
    else:
        ref = orc.eval_configs(_osys(wl), wl.R, X, derivs=True)
    _close(g, ref, 1e-10)
