"""cis scans with SNP lists out of order (missing-genotype patterns, NaN expression),
sample counts of every plain shape, and windows that reach no trait or every trait."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("window", [0, 40_000_000, 1 << 62])
@pytest.mark.parametrize("N,kind", [(60, "missing"), (102, "missing"), (102, "nan"), (150, "plain"),
                                    (210, "plain"), (300, "plain")])
def test_cis_hits_equal_the_full_scan_inside_the_window(oracle_mod, N, kind, window):
    import torch
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    T, S, pth = 333, 1500, 0.01
    rng = np.random.default_rng(N + len(kind))
    geno = rng.binomial(2, rng.uniform(0.05, 0.5, S)[:, None], (S, N)).astype(np.int8)
    expr = rng.standard_normal((T, N)).astype(np.float32)
    if kind == "missing":
        synth.add_missing_genotypes(rng, geno, n_patterns=9)
    if kind in ("missing", "nan"):
        synth.add_missing_expression(rng, expr, 0.01)
    snp, trait = synth.genome_positions(rng, S, T, n_chrom=3)
    kx = k.Krux(0)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    rs = kx.krux_rank(dev(expr))
    r = kx.krux_scan_cis(rs, dev(geno), dev(snp), dev(trait), window, pth, capacity=T * S)
    orc = oracle_mod.scan(expr, geno, pth)
    want = orc["hit"] & (np.abs(snp[None, :] - trait[:, None]) <= window)
    near = np.abs(orc["p"] / pth - 1.0) < 1e-12
    h = r["hits"].cpu().numpy().astype(np.int64)
    got = np.zeros_like(want)
    got[h[:, 0], h[:, 1]] = True
    assert not ((got != want) & ~near).any()
    assert r["n_hits"] == len(h) == int(got.sum())
    rs.free()
    kx.close()
