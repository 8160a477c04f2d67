"""The kernel form that a call takes where the plain and the general form meet, and the same
results on both sides of the line."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kx():
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    ctx = k.Krux(0)
    ctx.set_profiling(True)
    yield ctx
    ctx.close()


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _data(N, T=200, S=700, codes=3):
    rng = np.random.default_rng(N)
    return rng.standard_normal((T, N)).astype(np.float32), rng.integers(0, codes, (S, N)).astype(np.int8)


@pytest.mark.parametrize("N,form", [(102, 4), (304, 4), (320, 4), (321, 4), (336, 4), (337, 2), (368, 2), (400, 2)])
def test_wide_permutation_batches(kx, oracle_mod, N, form):
    """The plain form up to the width where its K blocks hold 32 samples."""
    import paper_1307_3519_gb300 as k
    expr, geno = _data(N)
    perms = k.krux_make_perms(N, 3, N)
    rs = kx.krux_rank(_dev(expr))
    r = kx.krux_permute(rs, _dev(geno), _dev(perms), 5e-3, capacity=200 * 700)
    assert kx.profile()["scan_form"] == form
    orc = oracle_mod.scan(expr, geno, 5e-3)
    h = r["hits"].cpu().numpy().astype(np.int64)
    got = np.zeros_like(orc["hit"])
    got[h[:, 0], h[:, 1]] = True
    near = np.abs(orc["p"] / 5e-3 - 1.0) < 1e-12
    assert not ((got != orc["hit"]) & ~near).any() and r["n_hits"] == len(h)
    want = oracle_mod.perm_minp(expr, geno, perms)
    assert np.all(np.abs(r["minp"].cpu().numpy() - want) <= 1e-6 * want)
    rs.free()


@pytest.mark.parametrize("N,scan,dense,multi,cis,anova,nan", [
    (60, 0, 9, 8, 0, 0, 5), (102, 0, 9, 8, 0, 0, 5), (224, 0, 9, 8, 0, 0, 5), (240, 7, 9, 8, 0, 7, 5),
    (336, 7, 9, 8, 0, 7, 5), (368, 7, 9, 8, 0, 7, 3), (369, 7, 3, 1, 3, 7, 3), (512, 7, 3, 1, 3, 7, 3)])
def test_the_profile_names_the_form_that_ran(kx, N, scan, dense, multi, cis, anova, nan):
    import torch
    expr, geno = _data(N)
    e, g, g5 = _dev(expr), _dev(geno), _dev(_data(N, codes=5)[1])
    rs = kx.krux_rank(e)
    T, S = 200, 700
    got = []
    for call in (lambda: kx.krux_scan(rs, g, 1e-4, T * S),
                 lambda: kx.krux_scan(rs, g, 1e-4, T * S, dense=True),
                 lambda: kx.krux_scan(rs, g5, 1e-4, T * S, multiallelic=True),
                 lambda: kx.krux_scan_cis(rs, g, torch.arange(S, device="cuda"), torch.arange(T, device="cuda"),
                                          300, 1e-4, T * S),
                 lambda: kx.krux_scan_parametric(e, g, "anova", 1e-4, T * S)):
        call()
        got.append(kx.profile()["scan_form"])
    e[3, 5] = float("nan")
    rn = kx.krux_rank(e)
    kx.krux_scan(rn, g, 1e-4, T * S)
    got.append(kx.profile()["scan_form"])
    assert got == [scan, dense, multi, cis, anova, nan]
    rs.free()
    rn.free()


@pytest.mark.parametrize("kind,pth,form", [("cis", 1.5e-3, 0), ("cis", 1.6e-3, 3), ("cis", 0.2, 3),
                                           ("anova", 1.5e-3, 0), ("anova", 1.6e-3, 3), ("anova", 0.2, 3),
                                           ("linear", 1.5e-3, 0), ("linear", 1.6e-3, 3), ("linear", 0.2, 3),
                                           ("multi", 4e-3, 8), ("multi", 4.1e-3, 1), ("multi", 0.2, 1),
                                           ("scan", 0.2, 0)])
def test_calls_with_many_hits(kx, oracle_mod, kind, pth, form):
    """cis, parametric and five-group scans leave the plain form where P_c lets through more
    hits than its event warps write in time."""
    import torch
    T, S, N = 200, 700, 102
    expr, geno = _data(N, codes=5 if kind == "multi" else 3)
    e, g = _dev(expr), _dev(geno)
    rs = kx.krux_rank(e)
    if kind in ("anova", "linear"):
        r = kx.krux_scan_parametric(e, g, kind, pth, T * S)
        orc = oracle_mod.parametric_scan(expr, geno, pth, kind)
        want = orc["hit"]
    else:
        orc = oracle_mod.scan(expr, geno, pth, max_code=4 if kind == "multi" else 2)
        want = orc["hit"]
        if kind == "cis":
            r = kx.krux_scan_cis(rs, g, torch.arange(S, device="cuda"), torch.arange(T, device="cuda"), 150, pth, T * S)
            want = want & (np.abs(np.arange(S)[None, :] - np.arange(T)[:, None]) <= 150)
        else:
            r = kx.krux_scan(rs, g, pth, T * S, multiallelic=kind == "multi")
    assert kx.profile()["scan_form"] == form
    h = r["hits"].cpu().numpy().astype(np.int64)
    got = np.zeros_like(want)
    got[h[:, 0], h[:, 1]] = True
    near = np.abs(orc["p"] / pth - 1.0) < 1e-9
    assert not ((got != want) & ~near).any() and r["n_hits"] == len(h) == int(got.sum())
    p = r["p"].cpu().numpy()
    assert np.all(np.abs(p - orc["p"][h[:, 0], h[:, 1]]) <= 1e-6 * p)
    rs.free()


@pytest.mark.parametrize("missing", [False, True])
@pytest.mark.parametrize("N", [176, 193, 240, 257, 305, 321, 337, 352])  # whole K, K blocks of 128 to 16 samples
def test_nan_expression_at_wide_shapes(kx, oracle_mod, N, missing):
    import synth
    T, S, pth = 200, 700, 4e-3
    rng = np.random.default_rng(N)
    expr, geno = _data(N)
    geno[::5] = np.minimum(geno[::5], 1)
    geno[::7, 1:] = np.where(rng.random((100, N - 1)) < 0.02, 2, 0)  # small groups that NaN samples may empty
    if missing:
        synth.add_missing_genotypes(rng, geno, n_patterns=9)
    for t in range(T):  # up to the last coefficient set's count, one trait beyond it
        expr[t, rng.choice(N, 11 if t == 40 else t % 7, replace=False)] = np.nan
    rs = kx.krux_rank(_dev(expr))
    r = kx.krux_scan(rs, _dev(geno), pth, capacity=T * S)
    assert kx.profile()["scan_form"] == 5
    orc = oracle_mod.scan(expr, geno, pth)
    h = r["hits"].cpu().numpy().astype(np.int64)
    got = np.zeros_like(orc["hit"])
    got[h[:, 0], h[:, 1]] = True
    near = np.abs(orc["p"] / pth - 1.0) < 1e-12
    assert not ((got != orc["hit"]) & ~near).any() and r["n_hits"] == len(h) == int(got.sum())
    assert np.array_equal(h[:, 2], orc["d"][h[:, 0], h[:, 1], 0])
    rs.free()


@pytest.mark.parametrize("kind,N,pth,form", [
    ("scan", 176, 0.2, 0), ("scan", 177, 2.5e-3, 0), ("scan", 177, 2.6e-3, 3), ("scan", 300, 2.5e-3, 7),
    ("scan", 300, 2.6e-3, 3), ("nan", 160, 0.2, 5), ("nan", 161, 4e-3, 5), ("nan", 161, 4.1e-3, 3),
    ("nan", 300, 0.2, 3), ("dense", 300, 0.2, 9), ("permute", 176, 0.2, 4), ("permute", 300, 7e-3, 4),
    ("permute", 300, 7.1e-3, 2), ("fdr", 177, 7.1e-3, 4), ("fdr", 300, 0.03, 4), ("fdr", 177, 0.031, 2)])
def test_wide_calls_with_many_hits(kx, oracle_mod, kind, N, pth, form):
    import paper_1307_3519_gb300 as k
    T, S = 200, 700
    expr, geno = _data(N)
    if kind == "nan":
        expr[::3, 4] = np.nan
    rs, g = kx.krux_rank(_dev(expr)), _dev(geno)
    if kind in ("permute", "fdr"):
        perms = k.krux_make_perms(N, 3, N)
        r = kx.krux_permute(rs, g, _dev(perms), pth, T * S, fdr_bins=9 if kind == "fdr" else 0)
        want = oracle_mod.perm_minp(expr, geno, perms, traits=np.arange(0, T, 20))
        assert np.all(np.abs(r["minp"].cpu().numpy()[:, ::20] - want) <= 1e-6 * want)
    else:
        r = kx.krux_scan(rs, g, pth, T * S, dense=kind == "dense")
    assert kx.profile()["scan_form"] == form
    orc = oracle_mod.scan(expr, geno, pth)
    h = r["hits"].cpu().numpy().astype(np.int64)
    got = np.zeros_like(orc["hit"])
    got[h[:, 0], h[:, 1]] = True
    near = np.abs(orc["p"] / pth - 1.0) < 1e-12
    assert not ((got != orc["hit"]) & ~near).any() and r["n_hits"] == len(h) == int(got.sum())
    rs.free()
