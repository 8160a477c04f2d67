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
