"""AUTO at k > 64 on a chunk of 4,104 points: the polynomial transform (k = 65 and 100: rows that are
not, and are, 16-byte multiples; 128: the largest) with the points beyond its expansions passed to
the split schedule, against the FP64 oracle.  The observation error variance falls across the domain,
so that the points' condition bounds run from 1 to beyond the last expansion in use (kappa 80, 180
and 400).  Tolerances: three times the error of the FP64 analysis at the same points when every
entry of A is off by 3e-7 of sqrt(A_ii A_jj) (FP32 inputs and accumulation) and c by 2e-7: 5.2e-6,
1.2e-5 and 1.6e-5 relative L2."""
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


@pytest.mark.parametrize("k,least_var,tol", [(65, 4e-7, 1.6e-5), (100, 1.5e-7, 3.6e-5),
                                             (128, 8e-8, 4.8e-5)])
def test_transformed_and_passed_on_points_match_oracle(k, least_var, tol):
    nx, ny = 72, 57
    f0 = C.perturb_nonequilibrium(C.ensemble_state(k, nx, ny, seed=201), 1e-4, 202)
    net = synth.regular_obs_network(nx, ny, 3)
    ramp = np.clip((net[:, 0] - 12) / 44.0, 0.0, 1.0)
    var = np.repeat(1e-3 * (least_var / 1e-3) ** ramp, 2).astype(np.float32)
    yo = C.observations(C.ensemble_state(1, nx, ny, seed=203), net, UV, 0.01, 204)[0]
    exp = L.Experiment(nx, ny, k, 0.6, net, var, loc_radius=2.0)
    got = None
    for _ in range(2):                       # the first analysis also times the schedules
        before = exp.work_counts()
        exp.set_state(f0)
        exp.analyze(yo)
        got = exp.get_deviation()
    counts = {n: v - before[n] for n, v in exp.work_counts().items()}
    assert exp.sync() == 0
    assert exp.stats().eig_schedule == L.LETKF_EIG_SPLIT
    exp.close()
    assert counts["cheb_points"] + counts["cheb_handed_on"] == nx * ny, counts
    assert min(counts["cheb_points"], counts["cheb_handed_on"]) > nx * ny // 20, counts
    pts = [(x, y) for x in range(1, nx, 5) for y in (0, 23, 56)]
    ref = C.oracle_points(f0, C.observe_at_points(f0, net, UV), yo, net, var, 2.0, UV, pts)
    bg = np.concatenate([C.dev64(got[:, :, y, x]) for x, y in pts], 1)
    bo = np.concatenate([ref[p]["Xa"].T - lbm.W[None, :] for p in pts], 1)
    bf = np.concatenate([f0[:, :, y, x].astype(np.float64) - lbm.W[None, :] for x, y in pts], 1)
    errs = C.point_parity(bg, bo, bf)
    assert max(errs) < tol, (errs, counts)
