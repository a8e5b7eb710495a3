"""The feature map (Sec. 3.2, Eq. rff_map) at the edges of its tiles: the float32
kernel's three tile sizes with ragged rows, features and depth, unaligned and
strided inputs, and the tensor-core kernel's ragged last feature block.  Every
feature within the float32 bound of the oracle."""
import math

import numpy as np
import pytest
import torch

import oracle as O
import workloads as WL
from tests.gpu_util import feature_tolerance, to_torch_x, widen

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


# 32 x 32, 64 x 64 and 128 x 128 tiles (by the number of tiles), the depth a
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


@pytest.mark.parametrize("phi", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("N,d,D", [(129, 72, 4), (300, 64, 100), (257, 200, 260), (128, 64, 316),
                                   (400, 128, 776)])
def test_feature_map_tc_ragged_features(sls, N, d, D, phi):
    X, W, b = _inputs(N, d, D, D)
    Xb, Wb = WL.f32_to_bf16_bits(X), WL.f32_to_bf16_bits(W)
    guard = torch.full((N + 1, D), 7.0, device="cuda", dtype=phi)
    got = sls.feature_map(to_torch_x(Xb, "bf16"), to_torch_x(Wb, "bf16"),
                          torch.from_numpy(b).cuda(), out=guard[:N])
    assert torch.all(guard[N] == 7.0)
    X64, W64 = widen(Xb, "bf16"), widen(Wb, "bf16")
    if phi == torch.float32:
        _check(got, X64, W64, b)
    else:
        want = O.rff_features(X64, W64, b)
        tol = feature_tolerance(X64, W64, b.astype(np.float64)) + 2.0 ** -8 * np.abs(want)
        assert np.all(np.abs(got.float().cpu().numpy() - want) <= tol)
