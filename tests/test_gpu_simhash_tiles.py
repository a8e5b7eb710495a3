"""SimHash codes (Sec. 3.3, Eq. simhash) at the edges of the kernel's tiles, bit
for bit against the oracle: one and two rows per thread, one, two and four
threads per row, row lengths that are no multiple of four, and rows whose stride
forbids 16-byte copies."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sls():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2607_19368_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("N,k,bits,pad", [
    (1, 1, 1, 0), (127, 16, 8, 0), (129, 17, 9, 0), (65, 30, 16, 2), (33, 64, 17, 0),
    (1000, 128, 32, 0), (1000, 128, 8, 1), (78000, 64, 16, 0), (155700, 5, 8, 3),
    (40001, 33, 20, 3)])
def test_simhash_tiles_bit_exact(sls, N, k, bits, pad):
    g = np.random.default_rng(N + k)
    U = g.standard_normal((N, k)).astype(np.float32)
    U[::7, 0] = 0.0
    U[::11] = 0.0            # dots of exactly +-0
    U[5::13, k // 2] = np.float32(1e-42)
    R = g.standard_normal((bits, k)).astype(np.float32)
    wide = torch.full((N, k + pad), float("nan"), device="cuda")
    wide[:, :k] = torch.from_numpy(U)
    got = sls.simhash(wide, torch.from_numpy(R).cuda(), bits, k=k)
    assert np.array_equal(got.cpu().numpy().view(np.uint32), O.simhash(U, R))
