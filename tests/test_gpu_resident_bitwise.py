"""The cluster-resident loops take bitwise the iterates of the per-iteration kernels, whichever
path the library picks and whenever it changes path or cluster size: state, iteration counts,
statuses and gradients are equal.  Sizes at the edges of the layout: one hour, horizons that
are no multiple of a quad, the first two-warp battery horizon (97) and the last one (192), more
batteries than warp groups, no batteries or lines, HVDC links, a batch subset, scenarios that
stop at different checks, and a batch with a network that fits no cluster.

Equality needs no tolerance: both paths evaluate the same expressions in the same order.  The
residual itself is summed in another order, so it is compared to 1e-4 (FP32 partial sums of up
to 1e5 terms)."""
import numpy as np
import pytest

from cases import network, scenario
from gpu_util import gpu_net
from paper_2410_13055_gb300 import synth

pytestmark = pytest.mark.gpu


def _one(N, L, G, B, T, S, hvdc=0):
    n, sc = synth.custom(N, L, G, B, T, S=S, seed=N + T)
    return [synth.add_hvdc(n, hvdc, seed=2) if hvdc else n], sc


def _single_bus():
    net, eta = network(1, gens=[(0, 20.0, 100.0), (0, 40.0, 100.0)])
    net["eta_min"] = eta
    return [net], [scenario([[150.0, 90.0, 120.0]], G=2)]


CASES = {
    "tiny": (lambda: synth.tiny(), None),
    "one-hour": (lambda: _one(60, 90, 180, 20, 1, 3), None),
    "ragged-13h-hvdc": (lambda: _one(30, 45, 90, 9, 13, 2, hvdc=2), None),
    "many-batteries-24h": (lambda: _one(40, 60, 100, 90, 24, 2), None),
    "ragged-45h": (lambda: _one(25, 40, 70, 7, 45, 1), None),
    "three-hours-per-lane-90h": (lambda: _one(20, 30, 60, 6, 90, 2), None),
    "two-warps-97h": (lambda: _one(12, 18, 36, 5, 97, 2), None),
    "two-warps-192h": (lambda: _one(12, 18, 36, 5, 192, 2), None),
    "no-batteries-7h": (lambda: _one(5, 6, 9, 0, 7, 1), None),
    "one-bus-no-lines": (lambda: _single_bus(), None),
    "staggered-stops": (lambda: synth.medium(S=16, T=24), None),
    "subset": (lambda: synth.medium(S=6, T=24), [1, 4]),
    "one-too-large": (lambda: synth.batching(seed=5, S=6), None),
}


def _run(nets, scens, batch, persistent):
    import torch
    net = gpu_net(nets, scens, kappa=50.0, tol=1e-3, adj_tol=1e-3, max_iter=1500, adj_max_iter=1500, check_every=20,
                  rho=0.2)
    if persistent is not None:
        net.use_persistent(persistent)
    e = torch.tensor(np.concatenate([n["eta_min"] for n in nets]) * 1.05, dtype=torch.float32, device="cuda")
    out, resid = [], []
    for _ in range(2):
        net.solve(e, batch=batch, warm="prev")
        out += [net.state(False).clone(), net.array("iters").clone(), net.array("status").clone()]
        resid.append(net.array("resid").clone())
        g = net.grad(e, warm="prev").clone()
        out += [net.state(True).clone(), net.array("adj_iters").clone(), net.array("status").clone(), g]
        e = e * 1.01
    torch.cuda.synchronize()
    return net, out, resid


@pytest.mark.parametrize("case", list(CASES))
def test_resident_iterates_are_bitwise_those_of_the_iteration_kernels(case):
    import torch
    make, batch = CASES[case]
    nets, scens = make()
    _, a, ra = _run(nets, scens, batch, False)
    for persistent in (None, True):
        net, b, rb = _run(nets, scens, batch, persistent)
        info = net.persistent_info()
        assert max(info) > 0 and (case != "one-too-large" or min(info) == 0), info
        for k, (x, y) in enumerate(zip(a, b)):
            assert torch.equal(x, y), (case, persistent, k)
        for x, y in zip(ra, rb):
            assert torch.all((x - y).abs() <= 1e-4 * x.abs()), (case, persistent)


def test_long_battery_horizons_and_explicit_choices_keep_the_iteration_kernels():
    nets, scens = _one(12, 18, 36, 5, 200, 1)
    assert gpu_net(nets, scens).persistent_info() == [0]
    nets, scens = synth.tiny()
    net = gpu_net(nets, scens)
    assert net.persistent_info() == [1]
    net.set_schedule(bus_staged=1)
    assert net.persistent_info() == [0]
