"""A large permutation batch packs its SNPs by df class (from about 2^30 permuted
pairs): minimum p, hits and FDR counts equal those of the two halves of its SNPs,
which are below that and keep their order."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,S,P,N,two", [(300, 44003, 64, 51, 0.5),   # mixed classes, odd last chunk
                                         (100, 270001, 32, 20, 0.02),  # more than one lap of the prefix sums
                                         (260, 44000, 64, 33, 1.0)])   # one class only
def test_ordered_batch_equals_its_halves(T, S, P, N, two):
    import torch
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    rng = np.random.default_rng(T + N)
    geno = rng.integers(0, 3, (S, N), dtype=np.int8)
    geno[:, 0], geno[:, 1], geno[:, 2] = 0, 1, 2
    pick = rng.random(S) < two
    geno[pick] = np.minimum(geno[pick], 1)
    geno[5] = 1  # one group: never tested
    expr = rng.standard_normal((T, N)).astype(np.float32)
    perms = torch.from_numpy(synth.make_perms(5, P, N)).cuda()
    g = torch.from_numpy(geno).cuda()
    pth = 1e-5
    kx = k.Krux(0)
    rs = kx.krux_rank(torch.from_numpy(expr).cuda())
    assert P * ((T + 127) // 128 * 128) * S >= 2 ** 30 > P * ((T + 127) // 128 * 128) * (S // 2 + 1)
    out = []
    for lo, hi in ((0, S), (0, S // 2), (S // 2, S)):
        r = kx.krux_permute(rs, g[lo:hi], perms, pth, capacity=200000, fdr_bins=8)
        h = r["hits"].cpu().numpy().astype(np.int64)
        h[:, 1] += lo
        out.append((r["minp"].cpu().numpy(), {tuple(x) for x in h.tolist()},
                    r["fdr_hist"].cpu().numpy().astype(np.int64)))
    full, a, b = out
    assert np.array_equal(full[0], np.minimum(a[0], b[0]))
    assert full[1] == a[1] | b[1]
    assert np.array_equal(full[2], a[2] + b[2])
    rs.free()
    kx.close()
