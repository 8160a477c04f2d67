"""As many missing-genotype patterns as SNPs that carry one, on both sides of the 256
whose sizes are read back in one trip."""
import numpy as np
import pytest

import synth
from kwcheck import check_hits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_patterns", [1, 255, 256, 257, 400])
def test_scan_with_many_missing_patterns(oracle_mod, n_patterns):
    import torch
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    rng = np.random.default_rng(n_patterns)
    T, S, N = 24, 450, 40
    geno = rng.integers(0, 3, (S, N), dtype=np.int8)
    pairs = [(i, j) for i in range(N) for j in range(i)]
    for s, q in zip(rng.permutation(S)[:n_patterns], rng.permutation(len(pairs))):
        geno[s, list(pairs[q])] = -1
    expr = synth.expression_lognormal(rng, T, N)
    kx = k.Krux(0)
    rs = kx.krux_rank(torch.from_numpy(expr).cuda())
    for pth in (0.05, 1e-3):  # (a second call on the same context)
        r = kx.krux_scan(rs, torch.from_numpy(geno).cuda(), pth, capacity=T * S)
        orc = oracle_mod.scan(expr, geno, pth)
        check_hits(r, orc, np.arange(T), np.arange(S), pth, must_have_hits=False)
        assert r["n_hits"] == int(orc["hit"].sum())
    rs.free()
    kx.close()


@pytest.mark.parametrize("N", [7, 31, 102, 128, 129, 256, 257, 384, 512])
def test_reranked_rows_with_ties_and_nan(oracle_mod, N):
    """Every way a dropped sample meets a row: tied with others, alone, absent itself;
    rows without ties; up to a quarter of the samples dropped."""
    import torch
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    rng = np.random.default_rng(N)
    T, S = 140, 130
    expr = rng.standard_normal((T, N)).astype(np.float32)
    expr[:40] = np.round(expr[:40], 1)
    expr[40:60] = np.round(expr[40:60])
    expr[60] = 1.0
    expr[20:80:3][rng.random((20, N)) < 0.05] = np.nan
    geno = rng.integers(0, 3, (S, N), dtype=np.int8)
    for s in range(0, S, 2):
        geno[s, rng.permutation(N)[:1 + s % max(1, N // 4)]] = -1
    kx = k.Krux(0)
    rs = kx.krux_rank(torch.from_numpy(expr).cuda())
    orc = oracle_mod.scan(expr, geno, 0.3)
    r = kx.krux_scan(rs, torch.from_numpy(geno).cuda(), 0.3, capacity=T * S)
    check_hits(r, orc, np.arange(T), np.arange(S), 0.3)
    assert r["n_hits"] == int(orc["hit"].sum())
    rs.free()
    kx.close()
