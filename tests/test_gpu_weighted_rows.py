"""The plain form's weighted indicator rows: every hit found and every rank sum
recovered, at the sample counts where the weights' precision changes, for group sizes
from 1 to N - 2, two-group markers, and traits whose order follows the genotype (the
largest sums)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pth", [0.3, 1e-4])
@pytest.mark.parametrize("N", [7, 16, 90, 91, 102, 128, 129, 160, 181, 182, 200, 256, 257, 300, 362, 363, 512])
def test_sums_and_hits_at_every_group_shape(oracle_mod, N, pth):
    import torch
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    rng = np.random.default_rng(N)
    sizes = []
    for a in sorted({1, 2, 3, N // 7, N // 4, N // 3, N // 2, N - 2} - {0}):
        for b in sorted({0, 1, 2, N // 5, (N - a) // 2, N - a - 1}):
            if 0 <= b <= N - a:
                sizes.append((a, b, N - a - b))
    geno = []
    for n in sizes:
        base = np.repeat(np.array([0, 1, 2], dtype=np.int8), n)
        for codes in ([0, 1, 2], [1, 0, 2], [2, 1, 0], [1, 2, 0]):
            g = np.array(codes, dtype=np.int8)[base]
            geno.append(g)  # in sample order: the traits below follow it
            geno.append(rng.permutation(g))
    geno = np.ascontiguousarray(np.stack(geno))
    up = np.arange(N, dtype=np.float32)
    expr = [up, -up, np.abs(up - N // 2), np.floor(up / 3)]
    expr += [up + rng.normal(0, s * N, N).astype(np.float32) for s in (0.05, 0.2, 0.5, 1, 2) for _ in range(12)]
    expr += [np.round(rng.standard_normal(N), 1) for _ in range(70)]
    expr = np.ascontiguousarray(np.stack(expr).astype(np.float32))
    kx = k.Krux(0)
    rs = kx.krux_rank(torch.from_numpy(expr).cuda())
    r = kx.krux_scan(rs, torch.from_numpy(geno).cuda(), pth, capacity=expr.shape[0] * geno.shape[0])
    orc = oracle_mod.scan(expr, geno, pth)
    h = r["hits"].cpu().numpy().astype(np.int64)
    got = np.zeros_like(orc["hit"])
    got[h[:, 0], h[:, 1]] = True
    near = np.abs(orc["p"] / pth - 1.0) < 1e-12
    assert not ((got != orc["hit"]) & ~near).any()
    assert r["n_hits"] == len(h) == int(got.sum())
    assert np.array_equal(h[:, 2], orc["d"][h[:, 0], h[:, 1], 0])
    assert np.array_equal(h[:, 3], orc["d"][h[:, 0], h[:, 1], 1])
    rs.free()
    kx.close()


@pytest.mark.parametrize("T", [100, 129, 300])  # one trait tile, an odd and an even last step
@pytest.mark.parametrize("S", [40, 64, 65, 700])  # one chunk, a whole one, an odd last chunk
@pytest.mark.parametrize("N", [193, 224, 240, 257, 336, 352, 512])
def test_wide_shapes_at_the_edges_of_their_tiles(oracle_mod, N, S, T):
    """K blocks (up to 224 samples) and pairs of CTAs (from 240): every number of K
    blocks, a last shorter one, odd numbers of trait tiles and of chunks."""
    import torch
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    rng = np.random.default_rng(N + S + T)
    geno = rng.binomial(2, rng.uniform(0.02, 0.5, S)[:, None], (S, N)).astype(np.int8)
    expr = rng.standard_normal((T, N)).astype(np.float32)
    kx = k.Krux(0)
    rs = kx.krux_rank(torch.from_numpy(expr).cuda())
    r = kx.krux_scan(rs, torch.from_numpy(geno).cuda(), 0.02, capacity=T * S)
    orc = oracle_mod.scan(expr, geno, 0.02)
    h = r["hits"].cpu().numpy().astype(np.int64)
    got = np.zeros_like(orc["hit"])
    got[h[:, 0], h[:, 1]] = True
    near = np.abs(orc["p"] / 0.02 - 1.0) < 1e-12
    assert not ((got != orc["hit"]) & ~near).any()
    assert r["n_hits"] == len(h) == int(got.sum())
    assert np.array_equal(h[:, 2], orc["d"][h[:, 0], h[:, 1], 0])
    rs.free()
    kx.close()


def test_pairs_of_ctas_report_a_wait_that_ran_out():
    """A one-cycle wait limit ends a launch over pairs of CTAs with KRUX_ETIMEOUT; the
    next call on the context is right again."""
    import torch
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    rng = np.random.default_rng(5)
    geno = torch.from_numpy(rng.integers(0, 3, (9000, 300)).astype(np.int8)).cuda()
    expr = torch.from_numpy(rng.standard_normal((2000, 300)).astype(np.float32)).cuda()
    kx = k.Krux(0)
    rs = kx.krux_rank(expr)
    want = kx.krux_scan(rs, geno, 1e-3, capacity=200_000)["n_hits"]
    kx.set_wait_limit(1)
    with pytest.raises(k.KruxError) as e:
        kx.krux_scan(rs, geno, 1e-3, capacity=200_000)
    assert e.value.status == k.KRUX_ETIMEOUT
    kx.set_wait_limit(0)
    assert kx.krux_scan(rs, geno, 1e-3, capacity=200_000)["n_hits"] == want
    rs.free()
    kx.close()


@pytest.mark.parametrize("pth", [0.3, 1e-4])
@pytest.mark.parametrize("N", [9, 31, 102, 128, 160, 181, 193, 256, 300, 340])
def test_multiallelic_sums_and_hits_at_every_group_shape(oracle_mod, N, pth):
    import itertools
    import torch
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    rng = np.random.default_rng(2 * N)
    geno = []
    for n0, n1, n2, n3 in itertools.product((0, 1, N // 5, N // 2), (0, 1, 2, N // 4), (0, 1, N // 6), (0, 1)):
        if n0 + n1 + n2 + n3 > N:
            continue
        n = [n0, n1, n2, n3, N - n0 - n1 - n2 - n3]
        codes = rng.permutation(5)
        g = np.repeat(codes, n).astype(np.int8)
        geno += [g, rng.permutation(g)]
    geno = np.ascontiguousarray(np.stack(geno))
    up = np.arange(N, dtype=np.float32)
    expr = [up, -up, np.floor(up / 3)] + [up + rng.normal(0, s * N, N) for s in (0.1, 0.4, 1) for _ in range(10)]
    expr += [np.round(rng.standard_normal(N), 1) for _ in range(100)]
    expr = np.ascontiguousarray(np.stack(expr).astype(np.float32))
    kx = k.Krux(0)
    rs = kx.krux_rank(torch.from_numpy(expr).cuda())
    r = kx.krux_scan(rs, torch.from_numpy(geno).cuda(), pth, capacity=expr.shape[0] * geno.shape[0],
                     multiallelic=True)
    orc = oracle_mod.scan(expr, geno, pth, max_code=4)
    h = r["hits"].cpu().numpy().astype(np.int64)
    got = np.zeros_like(orc["hit"])
    got[h[:, 0], h[:, 1]] = True
    near = np.abs(orc["p"] / pth - 1.0) < 1e-12
    assert not ((got != orc["hit"]) & ~near).any()
    assert r["n_hits"] == len(h) == int(got.sum())
    H, p = r["H"].cpu().numpy(), r["p"].cpu().numpy()
    assert np.all(np.abs(H - orc["H"][h[:, 0], h[:, 1]]) <= 1e-10 + 1e-9 * H)  # (all four sums)
    assert np.all(np.abs(p - orc["p"][h[:, 0], h[:, 1]]) <= 1e-6 * p)
    rs.free()
    kx.close()
