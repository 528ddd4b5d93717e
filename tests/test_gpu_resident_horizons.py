"""Which horizons the cluster-resident loops take: any without batteries, up to 192 hours with them
by the library's choice and all on request."""
import numpy as np
import pytest

from gpu_util import eta_tensor, gpu_net
from paper_2410_13055_gb300 import synth

pytestmark = pytest.mark.gpu


def _run(net, sc, persistent):
    import torch
    h = gpu_net([net], sc, kappa=50.0, tol=1e-4, adj_tol=1e-4, max_iter=400, adj_max_iter=400, check_every=20)
    if persistent is not None:
        h.use_persistent(persistent)
    e = eta_tensor(net["eta_min"] * 1.05)
    h.solve(e)
    g = h.grad(e).clone()
    torch.cuda.synchronize()
    return h, [h.state(False), h.state(True), g, h.array("iters"), h.array("adj_iters")]


@pytest.mark.parametrize("T", [97, 200, 256])
@pytest.mark.parametrize("S", [1, 3])
def test_long_horizons_without_batteries_take_clusters_bitwise(T, S):
    import torch
    net, sc = synth.custom(12, 18, 30, 0, T, S=S, seed=T)
    _, a = _run(net, sc, False)
    for persistent in (None, True):
        h, b = _run(net, sc, persistent)
        assert min(h.persistent_info()) > 0
        for k, (x, y) in enumerate(zip(a, b)):
            assert torch.equal(x, y), (persistent, k)


@pytest.mark.parametrize("T,B", [(193, 5), (224, 40), (256, 5)])
def test_battery_horizons_over_192_hours_take_clusters_on_request(T, B):
    """Up to the rounding of four hours a lane, where the two paths fuse differently: 100 iterations of
    a few hundred roundings of 2^-24 each, on state of the loads' size."""
    net, sc = synth.custom(12, 18, 36, B, T, S=1, seed=T)
    out = []
    for persistent in (False, True):
        h = gpu_net([net], sc, kappa=50.0, tol=1e-12, adj_tol=1e-12, max_iter=100, adj_max_iter=100, check_every=20)
        assert h.persistent_info() == [0]  # not by the library's choice
        h.use_persistent(persistent)
        assert (h.persistent_info()[0] > 0) == persistent
        e = eta_tensor(net["eta_min"] * 1.05)
        h.solve(e)
        g = h.grad(e).double().cpu().numpy()
        out.append([h.state(False).double().cpu().numpy(), g])
    for x, y in zip(*out):
        assert np.abs(x - y).max() <= 100 * 300 * 2.0 ** -24 * np.abs(x).max()


def test_cluster_query_only_reads():
    """From several threads beside a solve: the answer is worked out when the network is bound."""
    import threading

    import torch
    net, sc = synth.custom(5, 7, 6, 2, 24, S=512, seed=2)
    h = gpu_net([net], sc, kappa=50.0, tol=1e-3, adj_tol=1e-3, max_iter=200, adj_max_iter=200)
    got = []
    threads = [threading.Thread(target=lambda: got.append(h.persistent_info())) for _ in range(4)]
    for th in threads:
        th.start()
    h.solve(eta_tensor(net["eta_min"]))
    for th in threads:
        th.join()
    torch.cuda.synchronize()
    want = h.persistent_info()
    assert min(want) > 0 and got == [want] * 4
