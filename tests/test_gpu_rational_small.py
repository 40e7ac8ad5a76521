"""The rational transform's instance for k <= 16 at its edges (one reflector, a ragged row, and 17, the
first size of the next instance) against the FP64 oracle at every grid point, at the library's FP32
bar (1e-5 relative L2)."""
import numpy as np
import pytest

import synth
from oracle import lbm
from paper_2308_03310_gb300 import _build, letkf as L
from tests import _cases as C

pytestmark = pytest.mark.gpu

UV = L.LETKF_OBS_U | L.LETKF_OBS_V


@pytest.fixture(scope="module", autouse=True)
def _built():
    _build.build()


@pytest.mark.parametrize("k", [3, 15, 17])
def test_small_ensembles_match_oracle(k):
    nx, ny, radius = 18, 13, 3.0
    f0 = C.perturb_nonequilibrium(C.ensemble_state(k, nx, ny, seed=300 + k), 1e-4, 301 + k)
    net = synth.regular_obs_network(nx, ny, 4)
    var = np.full(len(net) * 2, 1e-4, dtype=np.float32)
    yo = C.observations(C.ensemble_state(1, nx, ny, seed=307 + k), net, UV, 0.01, 309 + k)[0]
    exp = L.Experiment(nx, ny, k, 0.6, net, var, loc_radius=radius,
                       eig_schedule=L.LETKF_EIG_RATIONAL)
    exp.set_state(f0)
    exp.analyze(yo)
    dev = C.dev64(exp.get_deviation())
    assert exp.sync() == 0
    exp.close()
    Xa, _ = C.oracle_analysis(f0, yo, net, var, radius, UV)
    Wb = lbm.W[None, :, None, None]
    flat = [np.asarray(a).transpose(0, 2, 3, 1).reshape(k, -1)
            for a in (dev, Xa - Wb, f0.astype(np.float64) - Wb)]
    assert max(C.point_parity(*flat)) < 1e-5
