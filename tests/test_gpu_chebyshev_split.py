"""AUTO at k > 64 (the polynomial transform, from 4,096 points on) against SPLIT on the same inputs: the
errors of the mean increment and of the perturbations against the FP64 transform of the device's own A,
c and forecast, per class of the points' condition bound.  Only transformed points are in a class (its
limits are the last expansions in use: kappa 80 at k = 65, 180 at k = 100 and 400 at k = 128), and in
every class AUTO is to be no further off than SPLIT."""
import numpy as np
import pytest

import synth
from paper_2308_03310_gb300 import _build, letkf as L
from tests import _cases as C

pytestmark = pytest.mark.gpu

NX, NY = 72, 60
LIMITS = (1.04, 1.2, 2.0, 6.0, 16.0, 36.0, 80.0, 180.0, 400.0)


@pytest.fixture(scope="module", autouse=True)
def _built():
    _build.build()


def _smooth(rng, rms, scale):
    """A smooth divergence-free velocity field."""
    kx, ky = 2 * np.pi * np.fft.rfftfreq(NX)[None, :], 2 * np.pi * np.fft.fftfreq(NY)[:, None]
    psi = np.fft.rfft2(rng.normal(size=(NY, NX))) * np.exp(-0.25 * scale ** 2 * (kx ** 2 + ky ** 2))
    u = np.fft.irfft2(1j * ky * psi, s=(NY, NX))
    v = np.fft.irfft2(-1j * kx * psi, s=(NY, NX))
    f = rms * np.sqrt(2.0 / np.mean(u * u + v * v))
    return u * f, v * f


def _ensemble(k, smooth, seed):
    """FP32 deviations [k, 9, ny, nx]: a flow with smooth or pointwise perturbations of 5e-3."""
    from oracle import lbm
    rng = np.random.default_rng(seed)
    tu, tv = _smooth(rng, 0.02, 8.0)
    g = np.empty((k, 9, NY, NX), np.float32)
    for m in range(k):
        u, v = _smooth(rng, 5e-3, 6.0) if smooth else rng.normal(scale=5e-3, size=(2, NY, NX))
        rho = 1.0 + rng.normal(scale=5e-4, size=(NY, NX))
        g[m] = lbm.equilibrium(rho, tu + u, tv + v) - lbm.W[:, None, None]
    return g


def _transform(A, c, X, k):
    """(mean increment [n, 9], perturbations [n, 9, k]) of the FP64 analysis."""
    lam, U = np.linalg.eigh(A)
    q = np.maximum(lam, 0.0) + (k - 1)
    dX = X - X.mean(-1, keepdims=True)
    w = U @ ((U.transpose(0, 2, 1) @ c[:, :, None]) / q[:, :, None])
    T = U @ (np.sqrt((k - 1) / q)[:, :, None] * U.transpose(0, 2, 1))
    return (dX @ w)[:, :, 0], dX @ T


@pytest.mark.parametrize("smooth", [False, True])
@pytest.mark.parametrize("k", [65, 100, 128])
def test_auto_is_no_further_from_the_exact_transform_than_split(k, smooth):
    g0 = _ensemble(k, smooth, 17 + k)
    net = synth.regular_obs_network(NX, NY, 3)
    ramp = np.clip((net[:, 0] - 6) / 60.0, 0.0, 1.0)
    var = np.repeat(1e-2 * (1.5e-6 / 1e-2) ** ramp, 2).astype(np.float32)
    yo = (0.005 + 0.01 * np.random.default_rng(18 + k).normal(size=len(var))).astype(np.float32)
    got = {}
    for name, schedule in (("auto", L.LETKF_EIG_AUTO), ("split", L.LETKF_EIG_SPLIT)):
        e = L.Experiment(NX, NY, k, 0.6, net, var, loc_radius=2.5, eig_schedule=schedule)
        for _ in range(2):                    # the first analysis also times the schedules
            before = e.work_counts()
            e.set_deviation(g0)
            pr = e.analyze_probe(yo, np.arange(NX * NY), want=("gram", "cvec", "xf"))
        assert e.sync() == 0
        got[name] = C.dev64(e.get_deviation()).transpose(2, 3, 1, 0).reshape(-1, 9, k)
        transformed = e.work_counts()["cheb_points"] - before["cheb_points"]
        assert (transformed > NX * NY // 2) == (name == "auto")
        e.close()
    A = np.asarray(pr["gram"], np.float64)
    X = np.asarray(pr["xf"], np.float64)
    bound = np.minimum(np.abs(A).sum(-1).max(-1), np.minimum(np.sqrt((A * A).sum((1, 2))),
                                                             np.trace(A, axis1=1, axis2=2)))
    kappa = 1.0 + 1.001 * bound / (k - 1)
    inc, per = _transform(A, np.asarray(pr["cvec"], np.float64), X, k)
    full = X.mean(-1, keepdims=True) + inc[:, :, None] + per
    mean = full.mean(-1)
    lower, classes = 0.0, 0
    for limit in LIMITS:
        if limit > {65: 80.0, 100: 180.0, 128: 400.0}[k]:
            break
        s = (kappa > lower) & (kappa <= limit)
        lower = limit
        if s.sum() < 100:
            continue
        classes += 1
        err = {}
        for name, v in got.items():
            m = v[s].mean(-1)
            err[name] = (np.linalg.norm(m - mean[s]) / np.linalg.norm(mean[s] - X[s].mean(-1)),
                         C.rel_l2(v[s] - m[:, :, None], full[s] - mean[s][:, :, None]))
        assert err["auto"][0] <= err["split"][0] and err["auto"][1] <= err["split"][1], (limit, err)
    assert classes >= 6
