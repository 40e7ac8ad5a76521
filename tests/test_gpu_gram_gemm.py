"""The Gram matrices as one tensor-core product over the observation points (1,024 grid points and
more, LETKF_GRAM_AUTO and LETKF_MIXED): A and the counts against the FP64 oracle at the edges
of its tiles (16 x 16 points, 128 pairs, 32 observation slots, 8-row groups), the analysis (and
with it c) at the library's 1e-5 bar, and the values of points that a non-finite observation does
not reach.

Tolerance: the observations h(x) are FP32 moments of magnitude 0.02 (rounding 1e-9) under
perturbations of 5e-3, so dy carries about 2e-7 relative, A twice that; the products are
exact to 24 bits and the sums of at most 190 steps of 32 slots round to nearest: 2e-6 of the
largest entry bounds them.
"""
import numpy as np
import pytest

import synth
from oracle import lbm, letkf as oletkf, obs as oobs
from paper_2308_03310_gb300 import _build, letkf as L
from tests import _cases as C

pytestmark = pytest.mark.gpu

UV = L.LETKF_OBS_U | L.LETKF_OBS_V
RUV = UV | L.LETKF_OBS_RHO


@pytest.fixture(scope="module", autouse=True)
def _built():
    _build.build()


CASES = [
    # nx, ny, k, stride, radius (None: no localization), kind, obs_vars, precision
    (32, 32, 2, 4, 3.0, "gauss", UV, L.LETKF_FP32),       # smallest ensemble and grid
    (33, 47, 5, 3, 2.5, "gauss", UV, L.LETKF_FP32),       # ragged tiles, k off every width
    (47, 33, 15, 5, 4.0, "gc", RUV, L.LETKF_FP32),        # 135 pairs: a second, nearly empty tile
    (64, 17, 17, 1, 1.0, "gauss", L.LETKF_OBS_V, L.LETKF_FP32),   # dense, tiny cutoff
    (1100, 1, 8, 7, 6.0, "gauss", UV, L.LETKF_FP32),      # one row: y wraps onto itself
    (40, 30, 24, 4, None, "gauss", UV, L.LETKF_FP32),     # no localization
    (36, 30, 33, 2, 12.0, "gauss", UV, L.LETKF_FP32),     # cutoff wider than the grid
    (65, 49, 64, 4, 12.0, "gauss", UV, L.LETKF_FP32),
    (70, 40, 128, 3, 4.0, "gc", UV, L.LETKF_FP32),
    (50, 34, 40, 3, 4.0, "gauss", UV, L.LETKF_MIXED),
]


def _setup(nx, ny, k, stride, radius, kind, obs_vars, precision, **kw):
    f0 = C.perturb_nonequilibrium(C.ensemble_state(k, nx, ny, seed=900 + k), 1e-4, 901 + k)
    net = synth.regular_obs_network(nx, ny, stride)
    V = bin(obs_vars).count("1")
    var = np.full(len(net) * V, 1e-4, dtype=np.float32)
    yo = C.observations(C.ensemble_state(1, nx, ny, seed=902 + k), net, obs_vars, 0.01, 903 + k)[0]
    exp = L.Experiment(nx, ny, k, 0.6, net, var, obs_vars=obs_vars, loc_radius=radius,
                       loc_kind=L.LETKF_LOC_GC if kind == "gc" else L.LETKF_LOC_GAUSS,
                       precision=precision, **kw)
    exp.set_state(f0)
    return exp, f0, net, var, yo


@pytest.mark.parametrize("nx,ny,k,stride,radius,kind,obs_vars,precision", CASES)
def test_gram_and_counts_match_oracle(nx, ny, k, stride, radius, kind, obs_vars, precision):
    exp, f0, net, var, yo = _setup(nx, ny, k, stride, radius, kind, obs_vars, precision)
    assert exp.stats().gram_tile == L.LETKF_GRAM_TENSOR
    pts = sorted({(x, y) for x in (0, 1, 15, 16, nx // 2, nx - 1) for y in (0, 15, 16, ny - 1)
                  if 0 <= x < nx and 0 <= y < ny})
    lin = np.array([y * nx + x for x, y in pts])
    pr = exp.analyze_probe(yo, lin, want=("nloc", "gram"))
    assert exp.sync() == 0
    exp.close()
    Yf = C.observe_at_points(f0, net, obs_vars)
    ybar, dY = oobs.ensemble_obs(Yf)
    r = np.inf if radius is None else radius
    c2 = np.inf if radius is None else synth.loc_cutoff2(radius)
    for n, (x, y) in enumerate(pts):
        dYl, dl, rl, nloc = oletkf.point_inputs(x, y, Yf, yo.astype(np.float64), net,
                                                var.astype(np.float64), nx, ny, r, c2, obs_vars,
                                                ybar=ybar, dY=dY, loc=kind)
        dYl = dYl.reshape(-1, k)
        A = dYl.T @ (rl[:, None] * dYl)
        assert pr["nloc"][n] == nloc
        assert np.abs(pr["gram"][n] - A).max() <= 2e-6 * max(np.abs(A).max(), 1e-30), (x, y)


@pytest.mark.parametrize("case", [1, 4, 6, 7, 9])
def test_analysis_matches_oracle(case):
    nx, ny, k, stride, radius, kind, obs_vars, precision = CASES[case]
    exp, f0, net, var, yo = _setup(nx, ny, k, stride, radius, kind, obs_vars, precision)
    exp.analyze(yo)
    dev = C.dev64(exp.get_deviation())
    assert exp.sync() == 0
    exp.close()
    pts = [(x, y) for x in {0, 15, 16, nx // 2, nx - 1} for y in {0, 16, ny - 1} if x < nx and y < ny]
    ref = C.oracle_points(f0, C.observe_at_points(f0, net, obs_vars), yo, net, var, radius,
                          obs_vars, pts)
    W = lbm.W[:, None]
    got = np.concatenate([dev[:, :, y, x] for x, y in pts], axis=1)
    want = np.concatenate([(ref[p]["Xa"] - W).T for p in pts], axis=1)
    fore = np.concatenate([(f0[:, :, y, x].astype(np.float64).T - W).T for x, y in pts], axis=1)
    errs = C.point_parity(got, want, fore)
    assert max(errs) < 1e-5, errs


@pytest.mark.parametrize("kind,stride", [("gauss", 4), ("gc", 3)])
def test_non_finite_observation_stays_within_its_cutoff(kind, stride):
    nx, ny, k, radius = 60, 52, 20, 3.0
    args = (nx, ny, k, stride, radius, kind, UV, L.LETKF_FP32)
    pts = np.arange(nx * ny)
    exp, f0, net, var, yo = _setup(*args, eig_schedule=L.LETKF_EIG_FUSED)
    good = exp.analyze_probe(yo, pts, want=("gram", "cvec"))
    assert exp.sync() == 0
    o = len(net) // 2 + 3
    bad_yo = yo.copy()
    bad_yo[2 * o] = np.nan
    exp.set_state(f0)
    bad = exp.analyze_probe(bad_yo, pts, want=("gram", "cvec"))
    assert exp.sync() == L.LETKF_ENONFINITE
    exp.set_state(f0)                       # the flag does not outlive its analysis
    again = exp.analyze_probe(yo, pts, want=("gram", "cvec"))
    assert exp.sync() == 0
    exp.close()
    assert np.array_equal(good["gram"], again["gram"]) and np.array_equal(good["cvec"], again["cvec"])
    dx = (net[o, 0] - pts % nx + nx // 2) % nx - nx // 2
    dy = (net[o, 1] - pts // nx + ny // 2) % ny - ny // 2
    hit = dx * dx + dy * dy < synth.loc_cutoff2(radius)
    assert np.isnan(bad["cvec"][hit]).all() and np.isfinite(bad["cvec"][~hit]).all()
    # dy is finite everywhere, so the Gram matrices are too; both forms sum the same products
    scale = np.abs(good["gram"]).max()
    assert np.abs(bad["gram"] - good["gram"]).max() <= 2e-6 * scale
    assert np.abs((bad["cvec"] - good["cvec"])[~hit]).max() <= 4e-6 * np.abs(good["cvec"]).max()
