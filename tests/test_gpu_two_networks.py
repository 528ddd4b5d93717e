"""A network bound while another lives leaves the other's launches as they were: the staged bus kernels'
shared-memory limit, which belongs to the kernel and not to a network, is not lowered.  The first
network's blocks have the largest stage (128 quads of 5 generators, 4 line ends and 2 batteries: 40 KB)
and records of about 10 KB, together above the 48 KB that any launch may take."""
import numpy as np
import pytest

from cases import network, scenario
from gpu_util import eta_tensor, gpu_net
from paper_2410_13055_gb300 import synth

pytestmark = pytest.mark.gpu

OPTS = dict(kappa=50.0, tol=1e-4, adj_tol=1e-4, max_iter=100, adj_max_iter=100, check_every=20)


def _large(N=52, T=24):
    rng = np.random.default_rng(1)
    net, eta = network(
        N, gens=[(n, float(rng.uniform(10, 80)), float(rng.uniform(20, 60))) for n in range(N) for _ in range(5)],
        lines=[(n, (n + d) % N, 300.0, 60.0) for n in range(N) for d in (1, 2)],
        bats=[(n, 10.0) for n in range(N) for _ in range(2)])
    return net, eta, scenario(rng.uniform(40.0, 160.0, (N, T)), cf=rng.uniform(0.3, 1.0, (5 * N, T)))


@pytest.mark.parametrize("bus_staged", [1, 2])
def test_second_network_with_shorter_records_leaves_the_first_running(bus_staged):
    import torch
    big, eta, sb = _large()
    small, ss = synth.custom(3, 2, 2, 1, 4, S=1, seed=4)
    e = eta_tensor(eta)
    out = []
    for mode in (0, bus_staged):
        a = gpu_net([big], [sb], **OPTS)
        a.set_schedule(bus_staged=mode)
        b = gpu_net([small], ss, **OPTS)
        b.set_schedule(bus_staged=mode)
        b.solve(eta_tensor(small["eta_min"]))
        a.solve(e)
        g = a.grad(e).clone()
        torch.cuda.synchronize()
        out.append([a.state(False).clone(), a.state(True).clone(), g])
    for x, y in zip(*out):
        assert torch.equal(x, y)
