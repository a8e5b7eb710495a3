"""alpha and beta of the Lanczos kernel against the float64 oracle, for the
widths whose rows one warp holds (D <= 512).  The kernel's vectors and sums are
double-float (roundings of 2^-49 and 2^-48) and beta, its reciprocal and alpha
float64, so T agrees to a few of those roundings, as far as the recurrence itself
does not amplify them: the bound is 2^-46 of |T| (four sums' roundings) and sixteen
times (one per step) what the oracle's own T moves by when its start vector is
rounded to 2^-49."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


def check(phi, q1, r, alpha, beta, k, steps=None):
    """alpha and beta (of the first `steps` steps) against the oracle's."""
    phi = phi.astype(np.float64)
    a, b, _, ko = O.lanczos(phi, q1, r)
    wobble = np.random.default_rng(1).choice([-1.0, 1.0], q1.size) * 2.0 ** -49
    a2, b2, _, _ = O.lanczos(phi, q1 * (1.0 + wobble), r)
    n = steps or ko
    if steps is None:
        assert int(k) == ko
    scale = np.abs(a).max()
    bound = 2.0 ** -46 * scale + 16 * max(np.abs(a2[:n] - a[:n]).max(),
                                          np.abs(b2[:n - 1] - b[:n - 1]).max())
    assert np.abs(alpha.cpu().numpy()[:n] - a[:n]).max() <= bound
    assert np.abs(beta.cpu().numpy()[:n - 1] - b[:n - 1]).max() <= bound


@pytest.fixture(scope="module")
def sls():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_19368_gb300 as m
    m.lib()
    return m


def features(g, N, D, dims, scale):
    X, W = g.standard_normal((N, dims)), g.standard_normal((dims, D)) * scale
    return (np.sqrt(2.0 / D) * np.cos(X @ W + g.random(D) * 2 * np.pi)).astype(np.float32)


@pytest.mark.parametrize("N,D,r,dims", [(400, 128, 16, 24), (1000, 256, 24, 24), (700, 260, 16, 24),
                                        (2000, 384, 24, 24), (1500, 512, 16, 24),
                                        (1000, 256, 24, 3), (33, 64, 8, 8)])
def test_alpha_beta_to_float64(sls, N, D, r, dims):
    g = np.random.default_rng(N + D)
    phi, q1 = features(g, N, D, dims, 0.4), g.standard_normal(N)
    _, _, k, alpha, beta = sls.lanczos_topr(torch.from_numpy(phi).cuda(),
                                            torch.from_numpy(q1).cuda(), r)
    check(phi, q1, r, alpha, beta, k)


def test_alpha_of_a_rank_deficient_matrix(sls):
    """Rank 7: alpha and beta up to the last step before the breakdown."""
    g = np.random.default_rng(7)
    phi = (g.standard_normal((1000, 7)) @ g.standard_normal((7, 256))).astype(np.float32)
    q1 = g.standard_normal(1000)
    _, _, k, alpha, beta = sls.lanczos_topr(torch.from_numpy(phi).cuda(),
                                            torch.from_numpy(q1).cuda(), 24)
    check(phi, q1, 24, alpha, beta, k, steps=7)


def test_batched_windows(sls):
    g = np.random.default_rng(11)
    phi, q1 = features(g, 1800, 256, 24, 0.4), g.standard_normal(1800)
    _, _, k, alpha, beta = sls.lanczos_topr_batched(torch.from_numpy(phi).cuda(),
                                                    torch.from_numpy(q1).cuda(), 16,
                                                    [0, 900, 1500], [900, 600, 300])
    for i, (s, n) in enumerate(((0, 900), (900, 600), (1500, 300))):
        check(phi[s:s + n], q1[s:s + n], 16, alpha[i], beta[i], k[i])
