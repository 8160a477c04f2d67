"""An autotuned shape is the scan's: calls of other kinds keep their plain forms whatever
the tuner picked (inputs full of hits may make a general shape the fastest scan), with the
results of an untuned context."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_tuned_shape_leaves_other_calls_their_forms():
    import torch
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    rng = np.random.default_rng(11)
    T, S, N = 520, 3000, 102
    geno = torch.from_numpy(rng.integers(0, 3, (S, N), dtype=np.int8)).cuda()
    expr = torch.from_numpy(rng.standard_normal((T, N)).astype(np.float32)).cuda()
    perms = torch.from_numpy(synth.make_perms(3, 3, N)).cuda()
    pos = torch.arange(S, dtype=torch.int64, device="cuda")
    out = []
    for tuned in (False, True):
        kx = k.Krux(0)
        rs = kx.krux_rank(expr)
        if tuned:
            kx.autotune(rs, geno, 0.4)
        kx.set_profiling(True)
        p = kx.krux_permute(rs, geno, perms, 1e-3, capacity=T * S)
        forms = [kx.profile()["scan_form"]]
        c = kx.krux_scan_cis(rs, geno, pos, torch.arange(T, dtype=torch.int64, device="cuda") * 5, 200, 0.05, T * S)
        forms.append(kx.profile()["scan_form"])
        a = kx.krux_scan_parametric(expr, geno, "anova", 1e-2, T * S)
        forms.append(kx.profile()["scan_form"])
        out.append((p["minp"].cpu(), p["n_hits"], c["n_hits"], a["n_hits"], forms))
        rs.free()
        kx.close()
    assert torch.equal(out[0][0], out[1][0])
    assert out[0][1:] == out[1][1:]
