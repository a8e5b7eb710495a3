"""Failure detection on the GPU without a GPU fault: a wait that is never
satisfied (an mbarrier nothing arrives at, a group barrier one CTA never
reaches) must give up after its limit of about a second, report
SLS_ERR_TIMEOUT through the status word, and leave the context usable."""
import time

import numpy as np
import pytest
import torch

import oracle as O
import workloads as WL
from tests.gpu_util import feature_tolerance, to_torch_x

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sls():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_19368_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("which", [0, 1])
def test_stuck_wait_ends_with_timeout_status(sls, which):
    t0 = time.time()
    st = sls.selftest_wait_limit(which)
    elapsed = time.time() - t0
    assert st == 5, st                      # SLS_ERR_TIMEOUT
    assert elapsed < 30.0, elapsed          # about one second of clock cycles
    # the context still works: a small feature map against the oracle
    w = WL.scaled(WL.WORKLOADS["tiny"], N=200, D=256)
    p, prm = WL.make_prompt(w), WL.params_for(w)
    phi = sls.feature_map(to_torch_x(p.X, w.dtype), to_torch_x(prm.W, w.dtype),
                          torch.from_numpy(prm.b).cuda())
    got = phi.cpu().numpy().astype(np.float64)
    want = O.rff_features(p.x_f64(), prm.w_f64(), prm.b)
    assert np.all(np.abs(got - want) <= feature_tolerance(p.x_f64(), prm.w_f64(),
                                                          prm.b.astype(np.float64)))


def test_lanczos_giveup_leaves_empty_result_and_usable_context(sls):
    """The persistent Lanczos kernel's own give-up path: one CTA reports a
    failed wait at its first exchange (as a wait that ran out would), so the
    other CTAs' polls stop, every copy in flight lands, the status reads
    SLS_ERR_TIMEOUT, r_eff stays -1 and the later kernels treat the problem as
    empty (theta and U zero) instead of reading stale values.
    The same problem then runs normally and matches the oracle."""
    g = np.random.default_rng(5)
    N, D, r = 3000, 512, 24
    X = g.standard_normal((N, 24)) / np.sqrt(24)
    W = g.standard_normal((D, 24)) * 24 ** -0.25
    b = g.random(D) * 2 * np.pi
    phi32 = O.rff_features(X, W, b).astype(np.float32)
    q1 = g.standard_normal(N)
    Phi, Q1 = torch.from_numpy(phi32).cuda(), torch.from_numpy(q1).cuda()
    t0 = time.time()
    status, theta, U, r_eff = sls.selftest_lanczos_giveup(Phi, Q1, r)
    torch.cuda.synchronize()
    assert time.time() - t0 < 30.0
    assert status == 5, status
    assert int(r_eff.item()) == -1
    assert float(theta.abs().max().item()) == 0.0
    assert float(U.abs().max().item()) == 0.0
    # the context still works, and a normal call gives the oracle's result
    th, U2, k, _, _ = sls.lanczos_topr(Phi, Q1, r)
    a, be, Q, ko = O.lanczos(phi32.astype(np.float64), q1, r)
    th_o, _, U_o = O.ritz_pairs(a, be, Q)
    assert int(k.item()) == ko
    t = th.cpu().numpy()[:ko]
    assert np.all(np.abs(t - th_o) <= 1e-4 * np.abs(th_o) + 1e-12 * abs(th_o[0]))


def test_feature_map_giveup_reaches_the_pass_status(sls):
    """A wait of the float32 tensor-core feature map that gives up inside
    compress() is reported by the workspace's status word, as it is for bf16;
    the same workspace then serves a normal pass."""
    g = torch.Generator(device="cuda").manual_seed(9)
    N, d, D, r = 1500, 512, 256, 16
    X = torch.randn(N, d, generator=g, device="cuda") / d ** 0.5
    W = torch.randn(D, d, generator=g, device="cuda") * d ** -0.25
    b = torch.rand(D, generator=g, device="cuda") * 6.28
    R = torch.randn(32, r, generator=g, device="cuda")
    q1 = torch.randn(N, generator=g, device="cuda", dtype=torch.float64)
    cfg = sls.Config.make(rho=4.0, D=D, r=r, bits=8)
    ws = sls.Workspace(cfg, 1, N, d, X.device)
    t0 = time.time()
    assert sls.selftest_compress_giveup(X, cfg, W, b, R, q1, ws) == 5
    assert time.time() - t0 < 30.0
    Xt, pos, t2m, _, _ = sls.compress(X, cfg, W, b, R, q1, workspace=ws)
    assert sls.workspace_status(ws) == 0
    again = sls.compress(X, cfg, W, b, R, q1)
    assert torch.equal(t2m, again[2]) and torch.equal(Xt, again[0])
    # shapes without that kernel are refused instead of passing untested
    with pytest.raises(sls.SLSError):
        sls.selftest_compress_giveup(X[:, :256].contiguous(), cfg, W[:, :256].contiguous(), b, R, q1,
                                     sls.Workspace(cfg, 1, N, 256, X.device))
