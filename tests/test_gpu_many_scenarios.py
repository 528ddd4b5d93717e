"""Loops over very many scenarios that fit no cluster (here: a ramp-limited generator): each
scenario takes the iterations that it takes alone, whatever the count (32,768 is where a sum of 16-bit
weights would turn negative and 65,536 where it would be zero, and the loop would end unconverged)."""
import numpy as np
import pytest

from cases import network, scenario
from gpu_util import eta_tensor, gpu_net

pytestmark = pytest.mark.gpu

OPTS = dict(kappa=50.0, tol=1e-4, adj_tol=1e-4, max_iter=2000, adj_max_iter=2000, check_every=20)


@pytest.mark.parametrize("S", [32768, 65536])
def test_each_of_many_ramp_limited_scenarios_converges_as_alone(S):
    import torch
    net, eta = network(1, gens=[(0, 20.0, 100.0), (0, 60.0, 100.0, 0.3)], ramp={0: 0.3})
    sc = scenario([[60.0, 150.0]], G=2)
    e = eta_tensor(eta)
    one = gpu_net([net], [sc], **OPTS)
    assert one.solve(e) == 0
    g1 = one.grad(e).clone()
    want = one.last_stats["iters_max"]
    assert want > OPTS["check_every"], "the case must take several residual checks"
    many = gpu_net([net], [dict(sc, weight=1.0 / S)] * S, **OPTS)
    assert many.solve(e) == 0
    assert bool((many.array("iters") == want).all()) and many.last_stats["n_converged"] == S
    g = many.grad(e)
    assert bool((many.array("adj_iters") == one.last_grad_stats["iters_max"]).all())
    torch.cuda.synchronize()
    # the mean of S equal gradients: FP64 sums, one FP32 rounding each
    assert bool(((g - g1).abs() <= 1e-6 * g1.abs().max()).all()), np.abs((g - g1).cpu().numpy()).max()
