"""What sls_lanczos_topr_noalloc accepts, without a GPU: exactly the problems whose
basis, coefficients, one set of column partials per CTA and w_k fit
SLS_NOALLOC_MAX_BYTES, whatever the kernel's exchange slots take on top.  An
accepted call then stops at the missing device (SLS_ERR_CUDA), a refused one has
SLS_ERR_WORKSPACE before that."""
import ctypes

import pytest
import torch

SMS = 152  # planned for when no device is visible


def al(x):
    return (x + 255) & ~255


def problem_bytes(N, D, r):
    g = max(1, min(SMS, -(-N // 32)))
    return (256 + al(8 * N * ((r + 1) & ~1)) + 2 * al(8 * r) + al(8 * r * r) + 256 +
            al(16 * (r + 4)) + al(8 * g * D) + al(8 * D) + al(8 * D * r))


def test_accepted_problems():
    if torch.cuda.is_available():
        pytest.skip("the answers here are those of a machine without a GPU")
    import paper_2607_19368_gb300 as sls
    L = sls.lib()
    p = ctypes.c_void_p(256)
    seen = set()
    for D in (4, 64, 1024, 4096, 7000, 8192):
        for r in (1, 16, 64, 127, 128):
            lo, hi = 1, 5_000_000  # the largest N that fits, and a few around
            while hi - lo > 1:
                mid = (lo + hi) // 2
                lo, hi = (mid, hi) if problem_bytes(mid, D, r) <= 32 << 20 else (lo, mid)
            # (4065 .. 4160 rows: 128 to 130 CTAs, the widest padding of the slots)
            for N in sorted({1, 33, 4064, 4065, 4096, 4160, 4864, lo - 1, lo, lo + 1, 2 * lo}):
                if N < 1 or L.sls_lanczos_workspace_size(N, D, r) == 0:
                    continue
                st = L.sls_lanczos_topr_noalloc(p, N, D, r, p, 1e-10, p, p, p, None, None, None)
                want = 4 if problem_bytes(N, D, r) <= 32 << 20 else 3
                assert st == want, (N, D, r)
                seen.add(st)
    assert seen == {3, 4}
