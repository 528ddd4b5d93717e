"""Equal calls take equal steps: the loops that move scenarios between the per-iteration kernels and
clusters of changing size give the same iterations, residuals and states, bit for bit, every time, also
beside other work on the device that delays some of the clusters.  (Stops are staggered, so clusters
change size on the way; a change that depended on how far each cluster had got would show in the last
bits of the residuals.)"""
import numpy as np
import pytest

from gpu_util import eta_tensor, gpu_net
from paper_2410_13055_gb300 import synth

pytestmark = pytest.mark.gpu

CASES = {
    "weeks": lambda: synth.medium(S=16),
    "days": lambda: synth.medium(S=32, T=24),
    "uneven": lambda: synth.batching(S=24, seed=9),
}


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("persistent", [None, True])
def test_equal_calls_take_equal_steps(case, persistent):
    import torch
    nets, scens = CASES[case]()
    h = gpu_net(nets, scens, kappa=50.0, tol=1e-3, adj_tol=1e-3, max_iter=2000, adj_max_iter=2000, rho=0.2)
    if persistent is not None:
        h.use_persistent(persistent)
    e = eta_tensor(np.concatenate([n["eta_min"] for n in nets]) * 1.05)
    side = torch.cuda.Stream()
    a = torch.ones(4096, 4096, dtype=torch.bfloat16, device="cuda")
    b = torch.empty_like(a)
    first = None
    for k in range(6):
        if k % 2:
            with torch.cuda.stream(side):
                for _ in range(40):
                    torch.mm(a, a, out=b)
        h.solve(e, warm="cold")
        out = [h.state(False).clone(), h.array("iters").clone(), h.array("resid").clone()]
        g = h.grad(e, warm="cold")
        out += [h.state(True).clone(), h.array("adj_iters").clone(), h.array("resid").clone(), g.clone()]
        torch.cuda.synchronize()
        if first is None:
            first = out
            assert len(set(out[1].tolist())) > 2, "the stops must be staggered"
        for q, (x, y) in enumerate(zip(first, out)):
            assert torch.equal(x, y), (k, q)
