"""The Lanczos kernel at the edges of its launch shapes, against the oracle.

A row of Phi is split over NV float4 groups of 32 lanes and WPR warps, rows are
taken R (2 or 4) at a time by 8 / WPR teams, and the basis in tiles of 32: the
widths here are the first and last of each (NV, WPR) and ragged ones, the row
counts leave teams without rows, batches of fewer than R rows and odd strips
over the CTAs, and the ranks sit at and beside the tile edges.  Bars as in the
other parity tests: Ritz values 1e-4 relative (float32 Phi on both sides),
subspace angle 1e-3 rad, and the same r_eff."""
import numpy as np
import pytest
import torch

import oracle as O
from tests.gpu_util import max_subspace_angle

pytestmark = pytest.mark.gpu

RITZ_RTOL, ANGLE_TOL, ZERO_FLOOR = 1e-4, 1e-3, 1e-12


@pytest.fixture(scope="module")
def sls():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_19368_gb300 as m
    m.lib()
    return m


def _phi(N, D, seed):
    g = np.random.default_rng(seed)
    X = g.standard_normal((N, 24)) / np.sqrt(24)
    W = g.standard_normal((D, 24)) * 24 ** -0.25
    phi = O.rff_features(X, W, g.random(D) * 2 * np.pi).astype(np.float32)
    return phi, g.standard_normal(N)


def _check(theta, U, k_gpu, phi64, q1, r):
    a, be, Q, k = O.lanczos(phi64, q1, r)
    th_o, _, U_o = O.ritz_pairs(a, be, Q)
    assert k_gpu == k
    th = theta[:k]
    assert np.all(np.abs(th - th_o) <= RITZ_RTOL * np.abs(th_o) + ZERO_FLOOR * abs(th_o[0]))
    assert max_subspace_angle(U[:, :k].astype(np.float64), U_o) <= ANGLE_TOL


@pytest.mark.parametrize("N,D,r", [
    (33, 4, 2), (65, 36, 16), (100, 256, 1), (333, 256, 33), (401, 260, 24), (515, 384, 32),
    (258, 388, 31), (700, 512, 64), (129, 516, 16), (611, 768, 65), (260, 772, 24),
    (1031, 1024, 32), (77, 1024, 64), (1030, 1028, 32), (903, 1536, 33), (517, 1540, 17),
    (1283, 2048, 64), (97, 2048, 48), (451, 2052, 24), (301, 4096, 65), (203, 4100, 12),
    (333, 8192, 128), (161, 1024, 128)])
def test_lanczos_shapes_match_oracle(sls, N, D, r):
    phi, q1 = _phi(N, D, N + D)
    theta, U, k, _, _ = sls.lanczos_topr(torch.from_numpy(phi).cuda(), torch.from_numpy(q1).cuda(), r)
    _check(theta.cpu().numpy(), U.cpu().numpy(), int(k.item()), phi.astype(np.float64), q1, r)


@pytest.mark.parametrize("N,D,r", [(333, 256, 33), (401, 264, 24), (611, 768, 32), (1031, 1024, 33),
                                   (517, 1544, 17), (1283, 2048, 64), (301, 4096, 65),
                                   (203, 8192, 40)])
def test_lanczos_bf16_shapes_match_oracle(sls, N, D, r):
    phi, q1 = _phi(N, D, N + D)
    phib = torch.from_numpy(phi).cuda().to(torch.bfloat16)
    theta, U, k, _, _ = sls.lanczos_topr(phib, torch.from_numpy(q1).cuda(), r)
    _check(theta.cpu().numpy(), U.cpu().numpy(), int(k.item()),
           phib.double().cpu().numpy(), q1, r)


@pytest.mark.parametrize("sizes,D,r", [([33, 47, 1, 64, 50, 2, 35], 128, 16),
                                       ([1024, 1025, 300, 2047], 1024, 24),
                                       ([700, 1, 1100, 33], 768, 32)])
def test_lanczos_batched_uneven_problems_match_oracle(sls, sizes, D, r):
    phi, q1 = _phi(sum(sizes), D, D + len(sizes))
    row0 = np.concatenate([[0], np.cumsum(sizes)[:-1]])
    theta, U, k, _, _ = sls.lanczos_topr_batched(torch.from_numpy(phi).cuda(),
                                                 torch.from_numpy(q1).cuda(), r, row0, sizes)
    theta, U, k = theta.cpu().numpy(), U.cpu().numpy(), k.cpu().numpy()
    for p, (s, n) in enumerate(zip(row0, sizes)):
        _check(theta[p], U[s:s + n], int(k[p]), phi[s:s + n].astype(np.float64), q1[s:s + n], r)


@pytest.mark.parametrize("N,D,r", [(7677, 768, 16), (5823, 1024, 16), (14000, 512, 24)])
def test_lanczos_bf16_full_grid_matches_oracle(sls, N, D, r):
    """Every SM's CTA at work and rings deeper than a team's batches: the whole next
    pass is issued ahead while the exchanges run."""
    phi, q1 = _phi(N, D, N + D)
    phib = torch.from_numpy(phi).cuda().to(torch.bfloat16)
    theta, U, k, alpha, _ = sls.lanczos_topr(phib, torch.from_numpy(q1).cuda(), r)
    phi64 = phib.double().cpu().numpy()
    _check(theta.cpu().numpy(), U.cpu().numpy(), int(k.item()), phi64, q1, r)
    # (a row left out of a pass would show in the first step already)
    a = O.lanczos(phi64, q1, 2)[0]
    assert np.all(np.abs(alpha.cpu().numpy()[:2] - a) <= 1e-12 * np.abs(a).max())
