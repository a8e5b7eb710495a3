"""The adaptive router's window score (Eq. redundancy) is a function of the
window alone: one prompt's scores, read off bit by bit through the routes they
give, are the same alone and in batches whose windows the GPU splits in other
ways."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sls():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_19368_gb300 as m
    m.lib()
    return m


def scores(route, nwin):
    """The float32 score of each window: the largest tau that still routes it to
    the spectral path, by bisection over the float32 values of [2^-20, 2)."""
    out = []
    for w in range(nwin):
        lo = int(np.float32(2.0 ** -20).view(np.int32))
        hi = int(np.float32(2.0).view(np.int32))
        while hi - lo > 1:
            mid = (lo + hi) // 2
            if route(float(np.int32(mid).view(np.float32)))[w]:
                lo = mid
            else:
                hi = mid
        out.append(lo)
    return out


@pytest.mark.parametrize("N,d,window,dtype", [(2 * 2048 + 331, 256, 2048, torch.bfloat16),
                                              (1500, 1032, 700, torch.float32),
                                              (300, 2056, 2048, torch.bfloat16)])
def test_score_does_not_depend_on_the_batch(sls, N, d, window, dtype):
    g = torch.Generator(device="cuda").manual_seed(N)
    nwin = -(-N // window)
    cfg = sls.Config.make(backend=sls.BACKEND_ADAPTIVE, rho=8.0, D=64, r=4, window=window,
                          preserve_last=0)
    cfg.tau_schedule = 0
    W = torch.randn(64, d, generator=g, device="cuda").to(dtype)
    b = torch.rand(64, generator=g, device="cuda")
    R = torch.randn(32, 4, generator=g, device="cuda")
    X = (torch.randn(N, d, generator=g, device="cuda") +
         0.3 * torch.randn(1, d, generator=g, device="cuda")).to(dtype)

    def routes(B):
        batch = torch.randn(B, N, d, generator=g, device="cuda").to(dtype)
        batch[B - 1] = X
        q1 = torch.ones(B, N, dtype=torch.float64, device="cuda")
        ws = sls.Workspace(cfg, B, N, d, X.device)

        def route(tau):
            cfg.tau = tau
            return sls.compress(batch, cfg, W, b, R, q1, workspace=ws)[4][(B - 1) * nwin:].cpu()

        return route

    alone = scores(routes(1), nwin)
    assert all(0.0 < np.int32(s).view(np.float32) < 1.0 for s in alone)
    x = X.double()
    for w, s in enumerate(alone):  # and it is the score: a chain of float32 sums
        xw = x[w * window:(w + 1) * window]
        c = xw.sum(0)
        want = float((xw / xw.norm(dim=1, keepdim=True)).sum(0) @ c / (xw.shape[0] * c.norm()))
        assert abs(float(np.int32(s).view(np.float32)) - want) <= 4e-6
    for B in (5, 130):
        assert scores(routes(B), nwin) == alone, B
