"""Non-finite observations and members through the one-product Gram form: the same entries are NaN and
infinite as in the CUDA-core form (which adds only the observations within a point's cutoff), every
other entry keeps its bits, and the launch takes no longer for it than a few times its own."""
import numpy as np
import pytest

import synth
from paper_2308_03310_gb300 import _build, letkf as L
from tests import _cases as C

pytestmark = pytest.mark.gpu

UV = L.LETKF_OBS_U | L.LETKF_OBS_V


@pytest.fixture(scope="module", autouse=True)
def _built():
    _build.build()


def _inputs(nx, ny, k, stride):
    f0 = C.perturb_nonequilibrium(C.ensemble_state(k, nx, ny, seed=300 + k), 1e-4, 301 + k)
    net = synth.regular_obs_network(nx, ny, stride)
    var = np.full(len(net) * 2, 1e-4, dtype=np.float32)
    yo = C.observations(C.ensemble_state(1, nx, ny, seed=302 + k), net, UV, 0.01, 303 + k)[0]
    return f0, net, var, yo


def _spoil(what, f0, net, yo):
    o = len(net) // 2 + 3
    x, y = net[o]
    if what == "nan_obs":
        yo[2 * o] = np.nan
    elif what == "inf_obs":
        yo[2 * o + 1] = -np.inf
    elif what == "nan_obs_edge":           # the last observation point, local across the edges
        yo[-1] = np.nan
    elif what == "nan_member":
        f0[1, 3, y, x] = np.nan
    elif what == "inf_member":
        f0[1, 3, y, x] = np.inf
    elif what == "all":
        f0[0] = np.nan


@pytest.mark.parametrize("what", ["nan_obs", "inf_obs", "nan_obs_edge", "nan_member", "inf_member",
                                  "all"])
@pytest.mark.parametrize("nx,ny,k,stride,radius,kind,chunk_rows", [
    (60, 52, 20, 4, 3.0, "gauss", 0), (47, 41, 40, 3, 2.5, "gc", 16), (40, 30, 24, 4, None, "gauss", 0),
])
def test_non_finite_entries_are_those_of_the_cuda_core_form(nx, ny, k, stride, radius, kind,
                                                            chunk_rows, what):
    pts = np.arange(nx * ny)
    out = {}
    for tile in (L.LETKF_GRAM_AUTO, L.LETKF_GRAM_PIPE):
        f0, net, var, yo = _inputs(nx, ny, k, stride)
        e = L.Experiment(nx, ny, k, 0.6, net, var, loc_radius=radius, gram_tile=tile,
                         loc_kind=L.LETKF_LOC_GC if kind == "gc" else L.LETKF_LOC_GAUSS,
                         eig_schedule=L.LETKF_EIG_FUSED, chunk_bytes=chunk_rows * nx * k * k * 4)
        for name in ("good", "bad"):
            if name == "bad":
                _spoil(what, f0, net, yo)
            e.set_state(f0)
            out[tile, name] = e.analyze_probe(yo, pts, want=("gram", "cvec"))
            assert e.sync() == (0 if name == "good" else L.LETKF_ENONFINITE)
        assert e.stats().gram_tile == (tile or L.LETKF_GRAM_TENSOR)
        e.close()
    hit = 0
    for part in ("gram", "cvec"):
        good, got, ref = (out[key][part] for key in ((L.LETKF_GRAM_AUTO, "good"),
                                                     (L.LETKF_GRAM_AUTO, "bad"),
                                                     (L.LETKF_GRAM_PIPE, "bad")))
        assert np.array_equal(np.isnan(got), np.isnan(ref))
        assert np.array_equal(np.isposinf(got), np.isposinf(ref))
        assert np.array_equal(np.isneginf(got), np.isneginf(ref))
        fin = np.isfinite(got)
        assert np.array_equal(got[fin], good[fin]) or what == "all"
        hit += np.count_nonzero(~fin)
    assert hit > 0


def test_non_finite_inputs_cost_no_more_than_a_few_launches():
    nx = ny = 256
    k, radius = 32, 8.0
    f0, net, var, yo = _inputs(nx, ny, k, 4)
    e = L.Experiment(nx, ny, k, 0.6, net, var, loc_radius=radius, eig_schedule=L.LETKF_EIG_RATIONAL)
    e.enable_timing()

    def gram_ms(f, y):
        best = np.inf
        for _ in range(5):
            e.set_state(f)
            e.analyze(y)
            best = min(best, e.timings()["gram_ms"])
            e.sync()
        return best

    good = gram_ms(f0, yo)
    bad_yo, bad_f, worst_f = yo.copy(), f0.copy(), f0.copy()
    bad_yo[len(yo) // 2] = np.nan
    bad_f[3, 2, 100, 100] = np.nan
    worst_f[0] = np.nan
    times = [gram_ms(f0, bad_yo), gram_ms(bad_f, yo), gram_ms(worst_f, yo)]
    e.close()
    # (the per-point CUDA-core form takes five times the finite launch's time here)
    assert max(times) < 5.0 * good, (good, times)
