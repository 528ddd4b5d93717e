"""Tuning a network whose scenarios fit clusters leaves it in clusters."""
import numpy as np
import pytest

from gpu_util import eta_tensor, gpu_net
from paper_2410_13055_gb300 import autotune, synth

pytestmark = pytest.mark.gpu


def test_tuned_network_keeps_the_librarys_choice():
    nets, sc = synth.medium(S=4, T=48)
    net = gpu_net(nets, sc, kappa=50.0, tol=1e-3, adj_tol=1e-3, max_iter=4000, adj_max_iter=4000)
    e = eta_tensor(nets[0]["eta_min"])
    before = net.persistent_info()
    assert min(before) > 0 and net.path_is_auto()
    autotune.tune_schedule(net, e, iters=40)
    assert net.persistent_info() == before and net.path_is_auto()
    net.solve(e)
    net.grad(e)
    out = autotune.tune_schedule_step(net, e, steps=1, reps=1)
    assert net.path_is_auto() == out["auto"]["kept"]
    net.set_schedule(bus_staged=1)
    assert net.persistent_info() == [0] * 4 and not net.path_is_auto()
    net.auto_path()
    assert net.persistent_info() == before and net.schedule()["bus_staged"] == 1
    net.use_persistent(False)
    assert net.persistent_info() == [0] * 4
    net.auto_path()
    assert net.persistent_info() == before
