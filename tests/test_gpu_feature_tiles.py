"""The feature map (Sec. 3.2, Eq. rff_map) at the edges of its tiles: the float32
kernel's three tile sizes with ragged rows, features and depth, unaligned and
strided inputs, and the three-product kernel that takes deep float32
contractions.  Every feature within the float32 bound of the oracle."""
import math

import numpy as np
import pytest
import torch

import oracle as O
from tests.gpu_util import feature_tolerance

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sls():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_19368_gb300 as m
    m.lib()
    return m


def _inputs(N, d, D, seed):
    g = np.random.default_rng(seed)
    X = (g.standard_normal((N, d)) / math.sqrt(d)).astype(np.float32)
    W = (g.standard_normal((D, d)) * d ** -0.25).astype(np.float32)
    return X, W, (g.random(D) * 2 * math.pi).astype(np.float32)


def _check(phi, X64, W64, b):
    want = O.rff_features(X64, W64, b)
    tol = feature_tolerance(X64, W64, b.astype(np.float64))
    err = np.abs(phi.cpu().numpy().astype(np.float64) - want)
    assert np.all(err <= tol), float(np.max(err / tol))


# 32 x 32, 64 x 64 and 128 x 64 tiles (by the number of tiles), the depth a
# multiple of the 16-wide slice, of four, and odd
@pytest.mark.parametrize("N,d,D", [(31, 16, 32), (33, 17, 36), (65, 5, 100), (1500, 31, 1300),
                                   (1793, 40, 1028), (2500, 36, 3076), (3000, 7, 2560)])
def test_feature_map_f32_tiles(sls, N, d, D):
    X, W, b = _inputs(N, d, D, N + D)
    _check(sls.feature_map(torch.from_numpy(X).cuda(), torch.from_numpy(W).cuda(),
                           torch.from_numpy(b).cuda()), X.astype(np.float64),
           W.astype(np.float64), b)


def test_feature_map_f32_strided_rows(sls):
    """Rows of a wider matrix: a row stride that forbids 16-byte loads, and one
    that allows them."""
    for pad in (1, 4):
        X, W, b = _inputs(333, 64, 256, pad)
        wide = torch.zeros((333, 64 + pad), device="cuda")
        wide[:, :64] = torch.from_numpy(X)
        _check(sls.feature_map(wide[:, :64], torch.from_numpy(W).cuda(), torch.from_numpy(b).cuda()),
               X.astype(np.float64), W.astype(np.float64), b)


# the smallest and ragged shapes of the float32 inputs that go to the tensor cores
@pytest.mark.parametrize("phi", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("N,d,D", [(897, 512, 128), (129, 516, 484), (1000, 1028, 132),
                                   (2000, 2044, 260), (513, 600, 4096)])
def test_feature_map_f32_split(sls, N, d, D, phi):
    X, W, b = _inputs(N, d, D, N + d)
    X *= np.exp2(np.random.default_rng(D).integers(-12, 4, X.shape)).astype(np.float32)
    guard = torch.full((N + 1, D), 7.0, device="cuda", dtype=phi)
    wide = torch.zeros((N, d + 4), device="cuda")
    wide[:, :d] = torch.from_numpy(X)
    got = sls.feature_map(wide[:, :d], torch.from_numpy(W).cuda(), torch.from_numpy(b).cuda(),
                          out=guard[:N])
    assert torch.all(guard[N] == 7.0)
    X64, W64 = X.astype(np.float64), W.astype(np.float64)
    if phi == torch.float32:
        _check(got, X64, W64, b)
    else:
        want = O.rff_features(X64, W64, b)
        tol = feature_tolerance(X64, W64, b.astype(np.float64)) + 2.0 ** -8 * np.abs(want)
        assert np.all(np.abs(got.float().cpu().numpy() - want) <= tol)


def test_feature_map_f32_split_special_rows(sls):
    """A NaN, an infinity, the largest float32 and a subnormal stay in their rows."""
    N, d, D = 1100, 520, 128
    X, W, b = _inputs(N, d, D, 3)
    clean = sls.feature_map(torch.from_numpy(X).cuda(), torch.from_numpy(W).cuda(),
                            torch.from_numpy(b).cuda()).cpu().numpy()
    Y = X.copy()
    Y[5, 7], Y[300, 519], Y[777] = np.nan, -np.inf, 0.0
    Y[777, 3] = 1e-41
    Y[778] = 0.0
    Y[778, 0] = np.finfo(np.float32).max
    W[:, 0] = np.exp2(-120.0)
    X[:, 0] = Y[:, 0]
    ref = sls.feature_map(torch.from_numpy(X).cuda(), torch.from_numpy(W).cuda(),
                          torch.from_numpy(b).cuda()).cpu().numpy()
    got = sls.feature_map(torch.from_numpy(Y).cuda(), torch.from_numpy(W).cuda(),
                          torch.from_numpy(b).cuda()).cpu().numpy()
    assert np.isnan(got[[5, 300]]).all() and np.isfinite(clean).all()
    scale = math.sqrt(2.0 / D)
    assert np.allclose(got[777], scale * np.cos(b), rtol=0, atol=1e-7)
    big = float(np.finfo(np.float32).max) * 2.0 ** -120   # 256 (1 - 2^-24)
    want = scale * np.cos(big + b.astype(np.float64))
    assert np.allclose(got[778], want, rtol=0, atol=scale * (big + 8) * 2.0 ** -22)
    keep = [i for i in range(N) if i not in (5, 300, 777, 778)]
    assert np.array_equal(got[keep], ref[keep])
