"""The ring bus kernel (a thread's next four devices in flight) against the per-thread-load one:
bitwise equal iterates for device lists shorter than the ring, longer than it, and empty ones."""
import numpy as np
import pytest

from gpu_util import eta_tensor, gpu_net
from paper_2410_13055_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,L,G,B,T", [
    (3, 2, 1, 1, 1),       # one or two line ends a bus, most buses without a generator
    (4, 6, 4, 1, 4),       # lists of about the ring's length, one full quad of hours
    (5, 10, 90, 7, 6),     # lists several rings long, a partly filled quad
    (43, 42, 50, 1, 31),   # a tree; more than one block
])
def test_ring_equals_per_thread_loads(N, L, G, B, T):
    import torch
    net, sc = synth.custom(N, L, G, B, T, S=2, seed=N)
    out = []
    for mode in (0, 2):
        h = gpu_net([net], sc, kappa=50.0, tol=1e-4, adj_tol=1e-4, max_iter=61, adj_max_iter=61, check_every=20)
        h.set_schedule(bus_staged=mode)
        eta = eta_tensor(net["eta_min"] * 1.05)
        h.solve(eta)
        g = h.grad(eta).clone()
        torch.cuda.synchronize()
        out.append((h.state(False).cpu().numpy().copy(), h.state(True).cpu().numpy().copy(), g.cpu().numpy()))
    for a, b in zip(*out):
        assert np.array_equal(a, b)
