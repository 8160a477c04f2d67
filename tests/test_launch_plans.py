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
