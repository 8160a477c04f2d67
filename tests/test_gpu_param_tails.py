"""The finalisation's tails of the parametric statistics over their whole range: strong
and weak effects, two and three groups, odd and even sample counts, thresholds from near
1 (the library's tails) to 1e-30."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", ["anova", "linear"])
@pytest.mark.parametrize("N,pth", [(4, 0.9), (5, 0.5), (20, 0.9), (21, 0.3), (102, 0.5), (129, 1e-6), (512, 1e-30)])
def test_tails_match_the_host_ones(model, N, pth):
    import torch
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    from scipy import stats
    rng = np.random.default_rng(N)
    T, S = 150, 90
    geno = rng.integers(0, 3, (S, N), dtype=np.int8)
    geno[::3] = np.minimum(geno[::3], 1)
    effect = np.exp(rng.uniform(-3, 4, T)) * (rng.random(T) < 0.8)
    base = geno[rng.integers(0, S, T)].astype(np.float64)
    expr = (rng.standard_normal((T, N)) + effect[:, None] * base).astype(np.float32)
    kx = k.Krux(0)
    r = kx.krux_scan_parametric(torch.from_numpy(expr).cuda(), torch.from_numpy(geno).cuda(), model, pth,
                                capacity=T * S)
    h = r["hits"].cpu().numpy().astype(np.int64)
    stat, p = r["stat"].cpu().numpy(), r["p"].cpu().numpy()
    assert len(h) and r["n_hits"] == len(h)
    groups = np.array([len(np.unique(g)) for g in geno])[h[:, 1]]
    if model == "anova":
        d1 = groups - 1
        ref = stats.f.sf(stat, d1, N - groups)
    else:
        ref = 2 * stats.t.sf(np.abs(stat), N - 2)
    # the statistic's rounding (1e-15) enters p times at most N / 2, either way, and the
    # reference's own tail is good to about 1e-12
    ok = (ref > 1e-300) & np.isfinite(stat)
    assert np.all(np.abs(p - ref)[ok] <= 1e-11 * ref[ok])
    assert (p < pth).all()
    kx.close()
