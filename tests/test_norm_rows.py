"""CPU-only: which kernel the append with the norm takes.  On both sides of each line of the rule, 148 SMs, tokens per
SM; the sizes beside them are where the other kernel was measured faster."""
import pytest

from paper_2509_22622_b200 import binding as B


@pytest.mark.parametrize("heads,dim,with_q,streamed,registers", [
    (4, 128, True, (), (1, 6, 12, 48)),
    (5, 128, True, (1, 6), (7, 13, 14, 16, 24, 32, 48)),
    (9, 64, True, (1, 6), (7, 14, 48)),
    (8, 128, True, (1, 10, 19, 20, 32, 48), (11, 12, 14, 18, 49)),
    (8, 128, False, (), (1, 6, 16, 20, 48)),
    (10, 128, True, (1, 12, 17, 48), (13, 16, 49)),
    (12, 128, True, (1, 11, 17, 32, 48), (12, 14, 16, 49, 98)),
    (24, 64, False, (1, 11, 17, 48), (12, 16, 49)),
    (14, 128, True, (1, 24), (25, 32)),
    (16, 128, True, (1, 24, 25, 98), ()),
    (16, 128, False, (1, 24), (25, 32)),
    (17, 128, True, (1, 16), (17, 32)),
    (17, 128, False, (1, 16), (17,)),
    (24, 128, False, (1, 15), (16, 32)),
    (32, 128, False, (1, 12), (13, 16)),
    (32, 128, True, (1, 16), (17,)),
    (33, 128, True, (), (1, 16, 48)),
])
def test_where_rows_are_streamed(heads, dim, with_q, streamed, registers):
    for per_sm in streamed + registers:
        for n in {148 * (per_sm - 1) + 1, 148 * per_sm}:
            assert B.ll_debug_norm_rows(heads, dim, n, with_q, 148) == (per_sm in streamed), (per_sm, n)


def test_the_default_is_148_sms():
    assert B.ll_debug_norm_rows(5, 128, 6 * 148) and not B.ll_debug_norm_rows(5, 128, 6 * 148 + 1)
    assert not B.ll_debug_norm_rows(5, 128, 6 * 148, sm_count=132)


@pytest.mark.parametrize("bad", [(0, 128, 1), (4, 96, 1), (4, 128, 0)])
def test_bad_arguments(bad):
    with pytest.raises(Exception):
        B.ll_debug_norm_rows(*bad)
