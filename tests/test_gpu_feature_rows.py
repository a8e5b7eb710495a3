"""A row's float32 features keep their bits whatever the number of rows in the
call: the kernel that computes them is chosen by d and D."""
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


@pytest.mark.parametrize("phi_dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("d,D", [(64, 256), (508, 256), (512, 64), (512, 1024), (516, 260),
                                 (2048, 512)])
def test_bits_do_not_depend_on_the_row_count(sls, d, D, phi_dtype):
    g = torch.Generator(device="cuda").manual_seed(d + D)
    X = torch.randn(4000, d, generator=g, device="cuda") / d ** 0.5
    W = torch.randn(D, d, generator=g, device="cuda")
    b = torch.rand(D, generator=g, device="cuda") * 6.28
    full = sls.feature_map(X, W, b, phi_dtype=phi_dtype)
    for n in (1, 31, 127, 300, 1500):
        part = sls.feature_map(X[:n].contiguous(), W, b, phi_dtype=phi_dtype)
        assert torch.equal(part, full[:n]), n


def test_row_limit(sls):
    """More than 64 * 65535 float32 rows are refused at every depth."""
    X = torch.empty(64 * 65535 + 1, 512, device="cuda")
    W, b = torch.zeros(4, 512, device="cuda"), torch.zeros(4, device="cuda")
    with pytest.raises(sls.SLSError):
        sls.feature_map(X, W, b)


@pytest.mark.parametrize("dtype,d,D", [(torch.float32, 512, 128), (torch.bfloat16, 256, 256)])
def test_a_row_of_huge_arguments_leaves_its_neighbours(sls, dtype, d, D):
    """Arguments beyond the fast cosine's range take another cosine by themselves."""
    g = torch.Generator(device="cuda").manual_seed(5)
    X = (torch.randn(200, d, generator=g, device="cuda") / d ** 0.5).to(dtype)
    W = torch.randn(D, d, generator=g, device="cuda").to(dtype)
    b = torch.rand(D, generator=g, device="cuda") * 6.28
    ref = sls.feature_map(X, W, b)
    X[70] *= 1e6
    got = sls.feature_map(X, W, b)
    keep = [i for i in range(200) if i != 70]
    assert torch.equal(got[keep], ref[keep])
    want = (2.0 / D) ** 0.5 * torch.cos(X[70].double() @ W.double().T + b.double())
    # float32 sums of about 1e6 leave 2^-24 of that in the argument, a few times over
    assert (got[70].double() - want).abs().max() <= (2.0 / D) ** 0.5 * 8 * 5e6 * 2.0 ** -24


@pytest.mark.parametrize("phi_dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("N,d,D", [(40, 64, 36), (900, 72, 700), (5000, 65, 1060)])
def test_unaligned_output(sls, N, d, D, phi_dtype):
    """Phi at an address that forbids wide stores, in each tile size of the float32
    kernel; the elements around it stay as they are."""
    g = torch.Generator(device="cuda").manual_seed(N)
    X = torch.randn(N, d, generator=g, device="cuda") / d ** 0.5
    W = torch.randn(D, d, generator=g, device="cuda")
    b = torch.rand(D, generator=g, device="cuda") * 6.28
    ref = sls.feature_map(X, W, b, phi_dtype=phi_dtype)
    for off in (1, 2, 3):
        buf = torch.full((N * D + 8,), 7.0, device="cuda", dtype=phi_dtype)
        got = sls.feature_map(X, W, b, out=buf[off:off + N * D].view(N, D))
        assert torch.equal(got, ref)
        assert torch.all(buf[:off] == 7.0) and torch.all(buf[off + N * D:] == 7.0)
