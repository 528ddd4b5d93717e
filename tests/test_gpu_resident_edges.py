"""The cluster-resident loops on networks whose device lists are empty at the end of the bus order:
a bus that no line reaches beside connected ones, several buses without lines, no generators.
State, iteration counts, statuses and gradients are bitwise those of the per-iteration kernels (both
paths evaluate the same expressions in the same order, so no tolerance is needed)."""
import numpy as np
import pytest

from cases import network, scenario
from gpu_util import eta_tensor, gpu_net

pytestmark = pytest.mark.gpu

LINES = [(0, 1, 400.0, 80.0), (1, 2, 300.0, 60.0), (0, 2, 350.0, 50.0)]
GENS = [(0, 20.0, 150.0), (1, 45.0, 90.0, 0.4), (2, 70.0, 120.0)]


def _lone(n_bus=4, gens=GENS, lines=LINES, bats=(), T=6):
    """The last bus stands alone; it has load, and what `gens` and `bats` give it."""
    net, eta = network(n_bus, gens=gens, lines=lines, bats=bats)
    rng = np.random.default_rng(n_bus + T)
    return net, eta, scenario(rng.uniform(20.0, 70.0, (n_bus, T)), cf=rng.uniform(0.6, 1.0, (len(gens), T)))


CASES = {
    "lone-load": lambda: _lone(T=5),
    "lone-load-battery": lambda: _lone(bats=[(3, 20.0), (1, 15.0)], T=24),
    "lone-generator-quads": lambda: _lone(gens=GENS + [(3, 30.0, 80.0)], bats=[(0, 10.0)], T=48),
    "two-lone-buses-100h": lambda: _lone(n_bus=5, bats=[(4, 20.0), (2, 15.0)], T=100),
    "no-lines": lambda: _lone(n_bus=3, lines=(), bats=[(0, 10.0)], T=13),
    "no-lines-no-batteries": lambda: _lone(n_bus=3, lines=(), T=8),
    "no-lines-one-hour": lambda: _lone(n_bus=3, lines=(), T=1),
    "no-generators": lambda: _lone(n_bus=4, gens=(), bats=[(1, 15.0)], T=6),
}


def _run(net, eta, sc, persistent):
    import torch
    h = gpu_net([net], [sc], kappa=50.0, tol=1e-4, adj_tol=1e-4, max_iter=800, adj_max_iter=800, check_every=20)
    if persistent is not None:
        h.use_persistent(persistent)
    e = eta_tensor(eta)
    out = []
    for warm in ("cold", "prev"):
        h.solve(e, warm=warm)
        out += [h.state(False).clone(), h.array("iters").clone(), h.array("status").clone()]
        out += [h.grad(e, warm=warm).clone(), h.state(True).clone(), h.array("adj_iters").clone()]
        e = e * 1.02
    torch.cuda.synchronize()
    return h, out


@pytest.mark.parametrize("case", list(CASES))
def test_empty_lists_take_the_iterates_of_the_iteration_kernels(case):
    import torch
    net, eta, sc = CASES[case]()
    _, a = _run(net, eta, sc, False)
    for persistent in (None, True):
        h, b = _run(net, eta, sc, persistent)
        assert h.persistent_info()[0] > 0
        for k, (x, y) in enumerate(zip(a, b)):
            assert torch.equal(x, y), (case, persistent, k)
        assert bool(torch.isfinite(b[0]).all())


def test_more_equal_scenarios_than_fit_change_path_bitwise():
    """More scenarios than the device holds side by side: the loop starts on the per-iteration kernels
    and the stragglers finish in clusters, with the iterates of the kernels alone."""
    import torch
    from paper_2410_13055_gb300 import synth
    nets, scens = synth.medium(S=320, T=24)
    e = eta_tensor(nets[0]["eta_min"] * 1.05)
    out, launches = [], []
    for persistent in (False, None, True):
        h = gpu_net(nets, scens, kappa=50.0, tol=1e-3, adj_tol=1e-3, max_iter=2000, adj_max_iter=2000, rho=0.2)
        if persistent is not None:
            h.use_persistent(persistent)
        h.solve(e)
        launches.append(h.last_stats["launches"])
        r = [h.state(False).clone(), h.array("iters").clone()]
        g = h.grad(e)
        out.append(r + [h.state(True).clone(), h.array("adj_iters").clone(), g.clone()])
        torch.cuda.synchronize()
    assert launches[2] < launches[1] < launches[0], launches
    for o in out[1:]:
        for k, (x, y) in enumerate(zip(out[0], o)):
            assert torch.equal(x, y), k
