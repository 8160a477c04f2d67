"""Permutation batches over markers with two genotype groups alone (inbred lines) and
monomorphic ones among them, whose class of three-group SNPs is empty."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,S,N,P", [(700, 6000, 102, 8), (300, 2005, 200, 16)])
def test_monomorphic_markers_cost_nothing(oracle_mod, T, S, N, P):
    import torch
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    rng = np.random.default_rng(S)
    geno = (2 * (rng.random((S, N)) < rng.uniform(0.1, 0.5, S)[:, None])).astype(np.int8)
    mono = geno.copy()
    mono[rng.random(S) < 0.3] = 2
    expr = rng.standard_normal((T, N)).astype(np.float32)
    perms = k.krux_make_perms(N, P, N)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    kx = k.Krux(0)
    kx.set_profiling(True)
    rs, pm = kx.krux_rank(dev(expr)), dev(perms)
    ms, got = [], []
    for g in (geno, mono, mono[(mono != 2).any(1)]):
        d = dev(g)
        t = []
        for _ in range(5):
            r = kx.krux_permute(rs, d, pm, 1e-3, T * S, fdr_bins=12)
            t.append(kx.profile()["ms_scan"])
        ms.append(min(t))
        got.append((r["minp"].cpu(), r["fdr_hist"].cpu(), r["n_hits"]))
    # the same results without the monomorphic markers, and the oracle's minimum p
    assert torch.equal(got[1][0], got[2][0]) and torch.equal(got[1][1], got[2][1]) and got[1][2] == got[2][2]
    traits = np.arange(0, T, 37)
    want = oracle_mod.perm_minp(expr, mono, perms, traits=traits)
    assert np.all(np.abs(got[1][0].numpy()[:, traits] - want) <= 1e-6 * want)
    # (they took 10 to 50 times as long when every block that holds one went to the event warps)
    assert ms[1] < 3 * ms[0]
    rs.free()
    kx.close()
