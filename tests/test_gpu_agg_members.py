"""Macro-token embeddings (Eq. macro_embed) where the launch expects few members per
macro-token: the averages at which the member kernel changes (3 and 6), rows of
one to eight 16-byte words per thread, a last row word that some threads lack, one
work item and more than the GPU holds, and a macro-token of many items among
singletons."""
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


def check(sls, X, lens):
    """Groups of consecutive tokens of the given lengths."""
    lens = np.asarray(lens)
    M, N = lens.size, int(lens.sum())
    assert X.shape[0] == N
    codes = torch.from_numpy(np.repeat(np.arange(M, dtype=np.int32), lens)).cuda()
    Xt, pos, t2m = sls.aggregate(X, codes, M)
    assert np.array_equal(t2m.cpu().numpy(), np.repeat(np.arange(M), lens))
    assert np.array_equal(pos.cpu().numpy(), np.cumsum(lens) - 1)
    x, lab = X.double(), codes.long()
    n = torch.from_numpy(lens).cuda().double()
    mean = torch.zeros(M, X.shape[1], dtype=torch.float64, device="cuda").index_add_(0, lab, x)
    mean /= n[:, None]
    eta = torch.zeros(M, dtype=torch.float64, device="cuda").index_add_(0, lab, x.norm(dim=1)) / n
    nrm = mean.norm(dim=1)
    scale = torch.where(n > 1, eta / nrm, torch.ones_like(nrm))
    # a chain of len additions and a scale of a few roundings
    tol = 2.0 ** -24 * (lens.max() + 16) * float((x.abs().max() * scale.max()).item())
    assert float((Xt.double() - mean * scale[:, None]).abs().max()) <= tol
    assert torch.equal(Xt[torch.from_numpy(lens == 1).cuda()],
                       X[torch.from_numpy(np.repeat(lens == 1, lens)).cuda()].float())


@pytest.mark.parametrize("d,dtype", [(8, torch.bfloat16), (2048, torch.bfloat16),
                                     (2056, torch.bfloat16), (4096, torch.bfloat16),
                                     (5120, torch.bfloat16), (8192, torch.bfloat16),
                                     (4, torch.float32), (1028, torch.float32),
                                     (2048, torch.float32), (8192, torch.float32)])
@pytest.mark.parametrize("members", [1, 2, 3, 5, 6])
def test_few_members(sls, d, dtype, members):
    g = torch.Generator(device="cuda").manual_seed(d + members)
    M = 1500
    X = torch.randn(M * members, d, generator=g, device="cuda").to(dtype)
    check(sls, X, [members] * M)


@pytest.mark.parametrize("d,dtype", [(264, torch.bfloat16), (3584, torch.bfloat16),
                                     (5120, torch.bfloat16), (1536, torch.float32)])
@pytest.mark.parametrize("lens", [[1], [2, 1], [3] * 7 + [1], [1] * 900 + [700] + [1] * 5,
                                  [129, 64, 65] + [2] * 400, [2, 1] * 9000])
def test_mixed_lengths(sls, d, dtype, lens):
    g = torch.Generator(device="cuda").manual_seed(d + len(lens))
    check(sls, torch.randn(sum(lens), d, generator=g, device="cuda").to(dtype), lens)
