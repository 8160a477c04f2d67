"""cis coordinates out of order are refused before the scan is launched: the caller's lists
stay as they were."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("where", ["snp first", "snp last", "trait", "outside the range", "no SNPs", "with a bad code"])
@pytest.mark.parametrize("missing", [False, True])
def test_lists_untouched(where, missing):
    import torch
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    T, S, N, cap = 300, 2000, 60, 300 * 2000
    rng = np.random.default_rng(7)
    g = rng.integers(0, 3, (S, N)).astype(np.int8)
    if missing:
        g[::50, 3] = -1
    snp, trait = np.arange(S, dtype=np.int64) * 10, np.arange(T, dtype=np.int64) * 60
    begin, end = 100, 1900
    if where == "snp first":
        snp[[100, 101]] = snp[[101, 100]]
    elif where == "snp last":
        snp[1899] = 0
    elif where == "trait":
        trait[-1] = 0
    elif where == "outside the range":
        snp[5] = 10 ** 9
    elif where == "no SNPs":
        snp[5], end = 10 ** 9, 100
    elif where == "with a bad code":
        snp[200], g[300, 2] = 0, 7
    geno, snp, trait = (torch.from_numpy(a).cuda() for a in (g, snp, trait))
    expr = torch.from_numpy(rng.standard_normal((T, N)).astype(np.float32)).cuda()
    kx = k.Krux(0)
    rs = kx.krux_rank(expr)
    hits = torch.full((cap, 4), -7, dtype=torch.int32, device="cuda")
    H, p = (torch.full((cap,), -7.0, dtype=torch.float64, device="cuda") for _ in range(2))
    o = k.Opts()
    o.pthresh, o.hit_capacity, o.snp_begin, o.snp_end = 0.5, cap, begin, end
    n = ctypes.c_int64(-1)

    def call():
        ptr = lambda t: ctypes.c_void_p(t.data_ptr())
        return kx.lib.krux_scan_cis(kx.handle, rs.handle, ptr(geno), S, N, ptr(snp), ptr(trait), 10 ** 6,
                                    ctypes.byref(o), ptr(hits), ptr(H), ptr(p), ctypes.byref(n),
                                    ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))

    assert call() == 1 and n.value == 0  # KRUX_EINVAL
    assert b"nondecreasing" in kx.lib.krux_last_error(kx.handle)
    assert bool((hits == -7).all()) and bool((H == -7).all()) and bool((p == -7).all())
    snp.copy_(torch.arange(S, device="cuda") * 10)
    trait.copy_(torch.arange(T, device="cuda") * 60)
    if where == "with a bad code":
        assert call() == 1 and b"genotype code" in kx.lib.krux_last_error(kx.handle)
    else:
        assert call() == 0 and (n.value > 0) == (where != "no SNPs")
    rs.free()
    kx.close()
