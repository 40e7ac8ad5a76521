"""Which Gram form AUTO takes by the sizes alone, and the forms without products on problems of several
tiles per block: LETKF_MIXED's split-FP16 form on 1,023 grid points (a tile is one to eight of
them), the CUDA-core schedules by name, and both where the one-product form's buffer would be
beyond 2 GiB.  The counts, A (1e-5 relative L2 per point) and the analysis (1e-5) against the FP64
oracle."""
import numpy as np
import pytest

import synth
from oracle import lbm, letkf as oletkf, obs as oobs
from paper_2308_03310_gb300 import _build, letkf as L
from tests import _cases as C

pytestmark = pytest.mark.gpu

UV = L.LETKF_OBS_U | L.LETKF_OBS_V


@pytest.fixture(scope="module", autouse=True)
def _built():
    _build.build()


def _check(nx, ny, k, stride, radius, tiles, **kw):
    f0 = C.big_ensemble_state(k, nx, ny, seed=7000 + k)
    net = synth.regular_obs_network(nx, ny, stride)
    var = np.full(len(net) * 2, 1e-4, dtype=np.float32)
    yo = C.observations(C.ensemble_state(1, nx, ny, seed=7001 + k), net, UV, 0.01, 7002 + k)[0]
    exp = L.Experiment(nx, ny, k, 0.6, net, var, loc_radius=radius, **kw)
    pts = sorted({(x, y) for x in (0, 1, nx // 2, nx - 2, nx - 1) for y in (0, ny // 2 + 1, ny - 1)
                  if 0 <= x < nx and y < ny})
    lin = np.array([y * nx + x for x, y in pts])
    for _ in range(2):                       # the first analysis may time the schedules
        exp.set_state(f0)
        pr = exp.analyze_probe(yo, lin, want=("nloc", "gram"))
    assert exp.sync() == 0
    assert exp.stats().gram_tile in tiles
    got = exp.get_deviation()
    exp.close()
    Yf = C.observe_at_points(f0, net, UV)
    ybar, dY = oobs.ensemble_obs(Yf)
    for n, (x, y) in enumerate(pts):
        dYl, _, rl, nloc = oletkf.point_inputs(x, y, Yf, yo.astype(np.float64), net,
                                               var.astype(np.float64), nx, ny, radius,
                                               synth.loc_cutoff2(radius), UV, ybar=ybar, dY=dY)
        dYl = dYl.reshape(-1, k)
        assert pr["nloc"][n] == nloc
        assert C.rel_l2(pr["gram"][n], dYl.T @ (rl[:, None] * dYl)) < 1e-5, (x, y)
    ref = C.oracle_points(f0, Yf, yo, net, var, radius, UV, pts)
    W = lbm.W[:, None]
    a = np.concatenate([C.dev64(got[:, :, y, x]) for x, y in pts], 1)
    b = np.concatenate([(ref[p]["Xa"] - W).T for p in pts], 1)
    f = np.concatenate([(f0[:, :, y, x].astype(np.float64).T - W).T for x, y in pts], 1)
    errs = C.point_parity(a, b, f)
    assert max(errs) < 1e-5, errs


CORES = (L.LETKF_GRAM_PIPE, L.LETKF_GRAM_TEAM)
TENSOR = (L.LETKF_GRAM_TENSOR,)


@pytest.mark.parametrize("precision", [L.LETKF_FP32, L.LETKF_MIXED])
@pytest.mark.parametrize("nx,ny,k,stride,radius,tiles", [
    (1200, 1, 40, 4, 3.0, CORES),           # grids one and two points wide: a tile is mostly empty
    (1, 1100, 64, 4, 3.0, CORES),
    (2, 600, 128, 4, 3.0, CORES),
    (400, 3, 64, 4, 4.0, TENSOR),
    (64, 48, 64, 1, 1.0, CORES),            # a short cutoff on a dense network
    (64, 48, 64, 2, 2.0, TENSOR),
])
def test_auto_picks_the_form_by_its_sizes(nx, ny, k, stride, radius, tiles, precision):
    _check(nx, ny, k, stride, radius, TENSOR if precision == L.LETKF_MIXED else tiles,
           precision=precision)


@pytest.mark.parametrize("k", [20, 40, 64, 65, 128])
def test_mixed_below_the_one_product_forms_grid_size(k):
    _check(31, 33, k, 3, 3.0, (L.LETKF_GRAM_TENSOR,), precision=L.LETKF_MIXED)


@pytest.mark.parametrize("tile", [L.LETKF_GRAM_PIPE, L.LETKF_GRAM_TEAM])
@pytest.mark.parametrize("nx,ny,k", [(161, 130, 20), (112, 96, 64), (72, 64, 128)])
def test_cuda_core_schedules_by_name(nx, ny, k, tile):
    _check(nx, ny, k, 4, 4.0, (tile,), gram_tile=tile)


@pytest.mark.parametrize("precision", [L.LETKF_FP32, L.LETKF_MIXED])
def test_networks_whose_products_exceed_the_buffer(precision):
    k, nx, ny = 128, 256, 164               # every point observed: 2.16e9 bytes
    _check(nx, ny, k, 1, 2.0, TENSOR if precision == L.LETKF_MIXED else CORES,
           precision=precision, eig_schedule=L.LETKF_EIG_FUSED)
