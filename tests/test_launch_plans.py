"""Launch plans on the CPU: what a form keeps in shared memory beside its operands must not
cost it resident chunks or rank stages."""
import pytest


@pytest.fixture(scope="module")
def k():
    from paper_1307_3519_gb300 import build
    build.build()
    import paper_1307_3519_gb300 as k
    return k


@pytest.mark.parametrize("nan,lo,hi,ka,nA,nc", [
    (0, 145, 160, 160, 2, 3), (0, 257, 272, 64, 4, 2), (0, 289, 304, 64, 3, 2), (0, 321, 336, 64, 2, 2),
    (1, 97, 112, 112, 3, 4), (1, 257, 272, 64, 3, 2), (1, 289, 304, 64, 2, 2), (1, 481, 496, 64, 3, 1)])
def test_general_forms_keep_their_chunks_and_stages(k, nan, lo, hi, ka, nA, nc):
    """(the widths where 768 bytes more per chunk, weights that only the plain forms read,
    would not fit)"""
    for N in range(lo, hi + 1):
        st, plan = k.krux_debug_plan(N, nan)
        assert st == 0 and (plan["ka"], plan["nA"], plan["nc"]) == (ka, nA, nc), (N, plan)


@pytest.mark.parametrize("mode,least,most", [(5, 1, 368), (6, 1, 352), (7, 193, 512)])
def test_plain_plans_with_k_blocks_and_pairs_of_ctas(k, mode, least, most):
    """Every sample count of the form's range (pairs of CTAs: from where the whole K beside a
    chunk pair does not fit one) has a sound plan (the check that each
    launch runs): whole or blocked K, a pair of chunks at least, three rank stages of it when it is
    blocked, four and boxes of at most eight atoms over pairs of CTAs."""
    for N in range(1, 513):
        st, plan = k.krux_debug_plan(N, mode)
        assert (st == 0) == (least <= N <= most), (N, st)
        if st:
            continue
        Np = (N + 15) // 16 * 16
        assert plan["smem"] <= 232448 and plan["b_region"] % 1024 == 0
        assert plan["ka"] % 16 == 0 and plan["nkb"] == -(-Np // plan["ka"]) and plan["nc"] in (2, 4)
        assert plan["b_stride"] == 256 * Np and 2 <= plan["nA"] <= 8
        if mode == 7:
            assert plan["nc"] == 2 and plan["nA"] >= 4 and plan["ka"] <= 128 and plan["b_region"] == plan["b_stride"]
        else:
            assert plan["nc"] * plan["b_stride"] <= plan["b_region"]
            assert plan["nkb"] == 1 or (plan["nc"] == 2 and plan["nA"] >= 3)
        assert plan["nA"] * 256 * plan["ka"] + plan["b_region"] < plan["smem"]
