"""The wait limit bounds single waits, not the length of a launch: one that runs several
times the limit without a candidate pair is right, in every plain form."""
import pytest

pytestmark = pytest.mark.gpu

LIMIT = 2_000_000  # cycles, about a millisecond; every launch below takes at least two


@pytest.mark.parametrize("kind,T,S,N", [
    ("scan", 20_000, 1_000_000, 102), ("scan", 15_000, 300_000, 300), ("nan", 20_000, 400_000, 102),
    ("multi", 20_000, 300_000, 102), ("anova", 20_000, 800_000, 102), ("permute", 20_000, 60_000, 102)])
def test_a_launch_may_take_longer_than_a_wait(kind, T, S, N):
    import torch
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    g = torch.Generator(device="cuda").manual_seed(N + len(kind))
    geno = torch.randint(0, 5 if kind == "multi" else 3, (S, N), generator=g, device="cuda", dtype=torch.int8)
    expr = torch.randn((T, N), generator=g, device="cuda")
    if kind == "nan":
        expr[torch.rand((T, N), generator=g, device="cuda") < 0.005] = float("nan")
    kx = k.Krux(0)
    kx.set_profiling(True)

    def call():
        if kind == "anova":
            return kx.krux_scan_parametric(expr, geno, "anova", 1e-40, 1024)["n_hits"]
        rs = kx.krux_rank(expr)
        if kind == "permute":
            perms = torch.from_numpy(k.krux_make_perms(3, 16, N)).cuda()
            n = kx.krux_permute(rs, geno, perms, 1e-40, 1024)["minp"]
        else:
            n = kx.krux_scan(rs, geno, 1e-40, 1024, multiallelic=kind == "multi")["n_hits"]
        rs.free()
        return n

    want = call()
    assert kx.profile()["ms_scan"] > 1.5  # (of a permutation batch the second, shorter pass)
    kx.set_wait_limit(LIMIT)
    got = call()
    assert bool((torch.as_tensor(got) == torch.as_tensor(want)).all())
    kx.close()


@pytest.mark.parametrize("limit", [1, 1000, 3000, 10_000, 30_000])
@pytest.mark.parametrize("N", [257, 300, 400, 512])  # one to three K blocks, a shorter last one
def test_pairs_of_ctas_drain_what_they_asked_for(N, limit):
    """After a wait that gave up, the two CTAs of a pair may have stopped at different
    tiles: the launch ends with KRUX_ETIMEOUT without any drain giving up too (sites from
    32 on), and the next call is right."""
    import re
    import torch
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    g = torch.Generator(device="cuda").manual_seed(N)
    geno = torch.randint(0, 3, (20_000, N), generator=g, device="cuda", dtype=torch.int8)
    expr = torch.randn((2300, N), generator=g, device="cuda")
    kx = k.Krux(0)
    rs = kx.krux_rank(expr)
    want = kx.krux_scan(rs, geno, 1e-3, capacity=200_000)["n_hits"]
    for _ in range(3):
        kx.set_wait_limit(limit)
        try:
            assert kx.krux_scan(rs, geno, 1e-3, capacity=200_000)["n_hits"] == want
        except k.KruxError as e:
            assert e.status == k.KRUX_ETIMEOUT
            assert int(re.search(r"site (\d+)", str(e)).group(1)) < 32
        else:
            assert limit > 1
        kx.set_wait_limit(0)
        assert kx.krux_scan(rs, geno, 1e-3, capacity=200_000)["n_hits"] == want
    rs.free()
    kx.close()
