"""The sums of the residual that stops a cluster-resident loop, against FP64 sums of the same FP32 terms.

Without lines and batteries the primal residual is sqrt(sum cnt_n p_bar^2) / |load|, and p_bar of the
last iteration is a row of the state.  An item's term is FP32: up to four hours of a bus, each
fma(cnt p_bar, p_bar, sum), or one hour where the network takes one-hour items.  Given the terms, the
kernel's sum is pairs of floats (the error of every addition kept, the errors summed in FP32) and FP64:
k additions are off by at most k^2 2^-48 relative, and a thread adds fewer than 50.  The residual is
half that: 5e-12.  Plain FP32 sums over a CTA are off by some 1e-8."""
import numpy as np
import pytest

from cases import network, scenario
from gpu_util import eta_tensor, gpu_net

pytestmark = pytest.mark.gpu


def _terms(pbar, quad):
    """FP32 items of cnt p_bar^2, hours padded to quads: the fused multiply-add's product is exact in
    FP64 and its sum rounds once more there, 2^-53."""
    cnt = np.float32(1.0) / (np.float32(1.0) / np.float32(3.0))  # 3 terminals a bus
    c = (cnt * pbar).astype(np.float32)
    if not quad:
        return (c.astype(np.float64) * pbar).astype(np.float32)
    N, T = pbar.shape
    pad = np.zeros((N, -T % 4), np.float32)
    p, c = (np.concatenate([a, pad], axis=1).reshape(N, -1, 4) for a in (pbar, c))
    s = np.zeros(p.shape[:2], np.float32)
    for h in range(4):
        s = (c[..., h].astype(np.float64) * p[..., h] + s).astype(np.float32)
    return s


@pytest.mark.parametrize("N,T", [(1, 1), (120, 12), (200, 24), (300, 40), (40, 160), (500, 4), (700, 1)])
def test_primal_residual_sums_the_terms_in_more_than_fp32(N, T):
    import torch
    rng = np.random.default_rng(N + T)
    gens = [(n, float(rng.uniform(10.0, 90.0)), float(rng.uniform(40.0, 120.0))) for n in range(N) for _ in range(2)]
    net, eta = network(N, gens=gens)
    sc = scenario(np.float32(rng.uniform(20.0, 200.0, (N, T))), cf=rng.uniform(0.3, 1.0, (2 * N, T)))
    h = gpu_net([net], [sc], tol=1e-12, adj_tol=1e-12, max_iter=60, adj_max_iter=60, check_every=20)
    assert h.persistent_info()[0] > 0
    e = eta_tensor(eta)
    h.solve(e, warm="cold")
    worst = 0.0
    for _ in range(6):
        h.solve(e, warm="prev")
        torch.cuda.synchronize()
        th = h.array("theta")  # the state's last bus row block; p_bar's is the one before it
        Tp = h.info[0]["Tp"]
        off = th.data_ptr() - h.ws.data_ptr() - (4 * N * Tp + 255) // 256 * 256
        pbar = h.ws[off:off + 4 * N * Tp].view(torch.float32).view(N, Tp)[:, :T].cpu().numpy()
        norm = np.sqrt((sc["load"].astype(np.float64) ** 2).sum())
        got = float(h.array("resid").cpu()[0])
        err = [abs(np.sqrt(_terms(pbar, q).astype(np.float64).sum()) / norm - got) for q in (True, False)]
        assert got > 1e-9
        worst = max(worst, min(err) / got)
    print(f"N {N} T {T}: {worst:.1e}")
    assert worst <= 5e-12
