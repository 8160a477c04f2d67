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


@pytest.mark.parametrize("N,form", [(102, 4), (304, 4), (320, 4), (321, 2), (336, 2), (368, 2), (400, 2)])
def test_wide_permutation_batches(kx, oracle_mod, N, form):
    """The plain form up to the width where its K blocks hold 48 samples."""
    import paper_1307_3519_gb300 as k
    expr, geno = _data(N)
    perms = k.krux_make_perms(N, 3, N)
    rs = kx.krux_rank(_dev(expr))
    r = kx.krux_permute(rs, _dev(geno), _dev(perms), 1e-2, capacity=200 * 700)
    assert kx.profile()["scan_form"] == form
    orc = oracle_mod.scan(expr, geno, 1e-2)
    h = r["hits"].cpu().numpy().astype(np.int64)
    got = np.zeros_like(orc["hit"])
    got[h[:, 0], h[:, 1]] = True
    near = np.abs(orc["p"] / 1e-2 - 1.0) < 1e-12
    assert not ((got != orc["hit"]) & ~near).any() and r["n_hits"] == len(h)
    want = oracle_mod.perm_minp(expr, geno, perms)
    assert np.all(np.abs(r["minp"].cpu().numpy() - want) <= 1e-6 * want)
    rs.free()
