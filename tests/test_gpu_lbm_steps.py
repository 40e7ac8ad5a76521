"""The four-step D2Q9 launch against four single steps, bit for bit: grids whose strips (64 columns)
and segments of rows are ragged, narrower than the halo, or wrap onto themselves, even widths
(8-byte copies) and odd ones (4-byte), with and without a force, and the rests of step counts
that are not multiples of four."""
import numpy as np
import pytest

import synth
from paper_2308_03310_gb300 import _build, letkf as L
from tests import _cases as C

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    _build.build()


def _forecasts(nx, ny, k, forced, steps):
    force = None
    if forced:
        force = np.stack(synth.kolmogorov_force(nx, ny, 1e-4, 2)).astype(np.float32)
        force[1] += synth.gaussian((ny, nx), 1e-5, 77).astype(np.float32)
    f0 = C.perturb_nonequilibrium(C.ensemble_state(k, nx, ny, seed=500 + nx), 1e-4, 501 + ny)
    out = []
    for chunks in ([steps], [1] * steps):
        exp = L.Experiment(nx, ny, k, 0.56, np.zeros((0, 2), np.int32), np.zeros(0, np.float32),
                           force=force)
        exp.set_state(f0)
        for n in chunks:
            exp.forecast(n)
        out.append(exp.get_deviation())
        assert exp.sync() == 0
        exp.close()
    return out


@pytest.mark.parametrize("forced", [True, False])
@pytest.mark.parametrize("nx,ny,k", [
    (64, 8, 2),       # one strip, one segment: both edges wrap
    (256, 64, 3),     # interior strips
    (192, 203, 2),    # a ragged last segment
    (132, 50, 2),     # a ragged last strip
    (130, 37, 2),     # an even width off the multiples of four
    (67, 29, 2),      # an odd width: 4-byte copies, a ragged last strip
    (20, 12, 2),      # narrower than a strip
    (3, 2, 2),        # narrower than the halo
    (1, 1, 2),
])
def test_four_step_launch_equals_single_steps(nx, ny, k, forced):
    many, single = _forecasts(nx, ny, k, forced, 8)
    assert np.array_equal(many, single)


@pytest.mark.parametrize("steps", [4, 5, 6, 7, 9, 10, 11])
def test_step_counts_with_rests_equal_single_steps(steps):
    many, single = _forecasts(140, 45, 2, True, steps)
    assert np.array_equal(many, single)
