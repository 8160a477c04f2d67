"""The FP64 pass of the dense output: every p from 1 down to the smallest the sample
count allows, both degrees of freedom, missing-genotype patterns, odd row lengths and
slices, and the hits it appends."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("N,S,missing", [(30, 701, False), (102, 513, True), (190, 640, False),
                                         (300, 333, False), (500, 257, False)])
def test_dense_values_and_hits(oracle_mod, N, S, missing):
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    rng = np.random.default_rng(N)
    T, pth = 150, 1e-3
    maf = rng.uniform(0.01, 0.5, S)
    geno = rng.binomial(2, maf[:, None], (S, N)).astype(np.int8)
    geno[::9] = np.minimum(geno[::9], 1)  # two groups
    geno[5] = 1                           # one group
    if missing:
        synth.add_missing_genotypes(rng, geno, n_patterns=7)
    shift = rng.uniform(0, 6, T)[:, None] * (rng.random(T) < 0.7)[:, None]
    expr = (rng.standard_normal((T, N)) + shift * np.abs(geno[rng.integers(0, S, T)])).astype(np.float32)
    expr[3] = 1.0  # constant: H = 0, p = 1
    kx = k.Krux(0)
    rs = kx.krux_rank(_dev(expr))
    orc = oracle_mod.scan(expr, geno, pth)
    for b, e in ((0, S), (7, S - 3)):
        r = kx.krux_scan(rs, _dev(geno), pth, capacity=T * S, snp_begin=b, snp_end=e, dense=True)
        H, p = r["dense_H"].cpu().numpy(), r["dense_p"].cpu().numpy()
        oH, op = orc["H"][:, b:e], orc["p"][:, b:e]
        assert np.all(np.abs(H - oH) <= 1e-12 + 1e-10 * oH)
        # the tails of the reported H itself, to a few units in the last place
        from scipy.special import erfc
        df = np.broadcast_to(orc["df"][:, b:e], H.shape)
        ref = np.where(df == 1, erfc(np.sqrt(H / 2)), np.where(df == 2, np.exp(-H / 2), 1.0))
        ref = np.where(H > 0, ref, 1.0)
        assert np.all(np.abs(p - ref) <= 4e-14 * ref)  # (x up to 250 through exp: 250 ulps)
        small = ref > 1e-6
        assert np.all(np.abs(p - ref)[small] <= 4e-15 * ref[small])
        assert p.min() < (1e-12 if N >= 102 else 1e-4)
        h = r["hits"].cpu().numpy().astype(np.int64)
        got = np.zeros_like(orc["hit"])
        got[h[:, 0], h[:, 1]] = True
        want = orc["hit"].copy()
        want[:, :b] = want[:, e:] = False
        near = np.abs(orc["p"] / pth - 1.0) < 1e-12
        assert not ((got != want) & ~near).any()
        assert r["n_hits"] == len(h) == int(got.sum())
        assert np.array_equal(h[:, 2], orc["d"][h[:, 0], h[:, 1], 0])
    rs.free()
    kx.close()


@pytest.mark.parametrize("N", [40, 102, 200])
def test_hits_at_a_threshold_of_the_data(N):
    """P_c that is a p of the data, or next to one: the dense form lists the hits that the
    plain scan lists, and its p values say the same."""
    import torch
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    T, S = 60, 600
    rng = np.random.default_rng(N)
    geno = rng.integers(0, 3, (S, N)).astype(np.int8)
    geno[::4] = np.minimum(geno[::4], 1)
    geno, expr = _dev(geno), _dev(rng.standard_normal((T, N)).astype(np.float32))
    kx = k.Krux(0)
    rs = kx.krux_rank(expr)
    p = kx.krux_scan(rs, geno, 0.3, T * S, dense=True)["dense_p"].cpu().numpy().ravel()
    for v in rng.choice(p[p < 0.2], 100, replace=False):
        for pth in (float(v), float(np.nextafter(v, 1)), float(np.nextafter(v, 0))):
            d = kx.krux_scan(rs, geno, pth, T * S, dense=True)
            s = kx.krux_scan(rs, geno, pth, T * S)
            key = lambda r: (r["hits"][:, 0].long() * S + r["hits"][:, 1].long()).sort().values
            assert torch.equal(key(d), key(s)) and int((d["dense_p"] < pth).sum()) == d["n_hits"]
    rs.free()
    kx.close()
