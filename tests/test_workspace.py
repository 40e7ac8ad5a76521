"""letkf_config.chunk_bytes bounds the device memory of the Gram chunk on every grid (host only), and
the rows of a chunk of half a tile of the one-product Gram form are the bits of the whole grid's."""
import ctypes as C

import numpy as np
import pytest

import synth
from paper_2308_03310_gb300 import _build, letkf as L
from tests import _cases as T

GIB, MIB = 1 << 30, 1 << 20
# least rows of a chunk: the tile heights of the CUDA-core Gram schedules
LEAST = {8: 16, 16: 8, 32: 12, 64: 2, 128: 1}


@pytest.fixture(scope="module", autouse=True)
def _built():
    _build.build()


def _config(nx, ny, k, chunk_bytes, precision):
    obs = synth.regular_obs_network(nx, ny, 4)
    var = np.full(len(obs) * 2, 1e-4, dtype=np.float32)
    cfg = L.letkf_config()
    cfg.nx, cfg.ny, cfg.k, cfg.tau = nx, ny, k, 0.6
    cfg.n_obs = len(obs)
    cfg.obs_xy = obs.ctypes.data_as(C.POINTER(C.c_int32))
    cfg.obs_vars = L.LETKF_OBS_U | L.LETKF_OBS_V
    cfg.obs_err_var = var.ctypes.data_as(C.POINTER(C.c_float))
    cfg.loc_kind, cfg.loc_radius, cfg.infl = L.LETKF_LOC_GAUSS, 12.0, 1.0
    cfg.precision, cfg.eig_schedule = precision, L.LETKF_EIG_FUSED
    cfg.chunk_bytes = chunk_bytes
    cfg._keep = (obs, var)
    return cfg


@pytest.mark.parametrize("precision", [L.LETKF_FP32, L.LETKF_MIXED])
@pytest.mark.parametrize("nx,ny,k,chunk", [
    (8192, 64, 128, 0), (8192, 64, 128, 64 * MIB), (4096, 256, 128, 0), (4096, 512, 64, 64 * MIB),
    (1024, 1024, 64, 64 * MIB), (1024, 1024, 64, 256 * MIB), (1024, 1024, 64, 0),
    (4096, 64, 24, 16 * MIB), (512, 512, 32, 8 * MIB), (256, 256, 32, 4 * MIB),
])
def test_chunk_bytes_bounds_the_workspace(nx, ny, k, chunk, precision):
    kp = next(v for v in (8, 16, 32, 64, 128) if k <= v)
    budget = chunk or GIB
    rows = min(ny, max(LEAST[kp], budget // (nx * k * k * 4)))
    npts, n_obs = nx * ny, len(synth.regular_obs_network(nx, ny, 4))
    fixed = 3 * 9 * k * npts * 4 + npts * 4            # two states, the transposed one, counts
    # the chunk: A, c, eigenvalues, counts; observation buffers; rounding
    per_chunk = rows * nx * (4 * k * k + 8 * k + 4)
    obs = n_obs * (2 * (k + kp + 8) * 4 + 64)
    products = min(chunk, 2 * GIB) if chunk else 2 * GIB
    assert (L.letkf_workspace_size(_config(nx, ny, k, chunk, precision))
            <= fixed + per_chunk + obs + products + MIB)


def _run(nx, ny, k, chunk, precision):
    f0 = T.perturb_nonequilibrium(T.ensemble_state(k, nx, ny, seed=40 + k), 1e-4, 41 + k)
    net = synth.regular_obs_network(nx, ny, 4)
    var = np.full(len(net) * 2, 1e-4, dtype=np.float32)
    yo = T.observations(T.ensemble_state(1, nx, ny, seed=42 + k), net, T.VARS_UV, 0.01, 43 + k)[0]
    exp = L.Experiment(nx, ny, k, 0.6, net, var, loc_radius=3.0, precision=precision,
                       eig_schedule=L.LETKF_EIG_FUSED, chunk_bytes=chunk)
    exp.set_state(f0)
    exp.analyze(yo)
    out, st = exp.get_deviation(), exp.stats()
    assert exp.sync() == 0
    exp.close()
    return out, st


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [L.LETKF_FP32, L.LETKF_MIXED])
@pytest.mark.parametrize("nx,ny,k", [(36, 52, 20), (64, 45, 40), (33, 41, 70)])
def test_chunks_of_half_tiles_are_bitwise_identical(nx, ny, k, precision):
    whole, st = _run(nx, ny, k, 0, precision)
    assert (st.gram_tile, st.n_chunks) == (L.LETKF_GRAM_TENSOR, 1)
    row = nx * k * k * 4
    for rows, height in ((8, 8), (15, 8), (17, 16), (35, 32)):
        part, st = _run(nx, ny, k, rows * row, precision)
        assert (st.gram_tile, st.n_chunks) == (L.LETKF_GRAM_TENSOR, -(-ny // height)), rows
        assert np.array_equal(whole, part), rows


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [L.LETKF_FP32, L.LETKF_MIXED])
def test_smaller_chunks_take_the_schedules_without_products(precision):
    nx, ny, k = 36, 52, 40
    whole, _ = _run(nx, ny, k, 0, precision)
    part, st = _run(nx, ny, k, 7 * nx * k * k * 4, precision)
    assert st.n_chunks >= -(-ny // 7)
    assert precision == L.LETKF_MIXED or st.gram_tile in (L.LETKF_GRAM_PIPE, L.LETKF_GRAM_TEAM)
    # the same analysis up to the 1e-5 bar that both forms keep against the oracle
    assert T.rel_l2(part - part.mean(0), whole - whole.mean(0)) < 2e-5
