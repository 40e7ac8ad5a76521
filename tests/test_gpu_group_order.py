"""A group cycle is ordered before the handles' later work, also the first one, which runs without
a captured graph while handles still pick a schedule: the states taken back right after the call
(on each handle's own stream) are those a synchronized copy returns."""
import numpy as np
import pytest

import synth
from paper_2308_03310_gb300 import _build, letkf as L
from tests import _cases as C

pytestmark = pytest.mark.gpu


def test_states_taken_back_after_the_first_group_cycle_are_its_results():
    import torch
    _build.build()
    n, ks = 64, (18, 26, 34, 42, 50, 58, 62, 22) * 2
    net = synth.regular_obs_network(n, n, 3)
    var = np.full(len(net) * 2, 1e-4, dtype=np.float32)
    exps, outs, yos = [], [], []
    for i, k in enumerate(ks):
        f0 = C.ensemble_state(k, n, n, seed=60 + i)
        e = L.Experiment(n, n, k, 0.55, net, var, loc_radius=3.0)
        e.set_state(f0)
        exps.append(e)
        outs.append(torch.empty((k, 9, n, n), device="cuda"))
        yos.append(torch.from_numpy(synth.gaussian(len(net) * 2, 0.01, 90 + i).astype(np.float32))
                   .cuda())
    torch.cuda.synchronize()
    L.letkf_group_cycle(exps, 25, yos)
    for e, out in zip(exps, outs):
        L.letkf_get_deviation(e.h, out.data_ptr(), 0, e.k, L.LETKF_DEVICE)
    torch.cuda.synchronize()
    for e, out in zip(exps, outs):
        assert np.array_equal(out.cpu().numpy(), e.get_deviation())
        assert e.sync() == 0
        e.close()
