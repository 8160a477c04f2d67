"""A parametric call that is refused after its tail's table has been queued leaves nothing
under way: the next call on the context, whose values lie where that table was, is right."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("refused", ["nan", "missing"])
def test_call_after_a_refused_one(refused):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    rng = np.random.default_rng(11)
    T, S, N = 300, 400, 60
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    expr = dev(rng.standard_normal((T, N)).astype(np.float32))
    geno = dev(synth.hwe_genotypes(rng, S, N, 0.1, 0.5)[0])
    bad_e = rng.standard_normal((1, 12)).astype(np.float32)
    bad_g = rng.integers(0, 3, (5, 12)).astype(np.int8)
    if refused == "nan":
        bad_e[0, 3] = np.nan
    else:
        bad_g[2, 3] = -1
    bad_e, bad_g = dev(bad_e), dev(bad_g)
    kx = k.Krux(0)
    try:
        def run():
            r = kx.krux_scan_parametric(expr, geno, "anova", 0.001, capacity=10_000)
            h = r["hits"].cpu().numpy().astype(np.int64)
            o = np.lexsort((h[:, 1], h[:, 0]))
            return h[o, :2], r["stat"].cpu().numpy()[o], r["p"].cpu().numpy()[o]
        want = run()
        assert len(want[0]) > 20
        for _ in range(30):
            with pytest.raises(k.KruxError):
                kx.krux_scan_parametric(bad_e, bad_g, "anova", 0.001, capacity=100)
            got = run()
            for a, b in zip(want, got):
                assert np.array_equal(a, b)
    finally:
        kx.close()
