"""Which attention schedule a call takes (csrc/attn_schedule.h), on the host: the lines that
were measured, what never cuts units, and that the launcher and the share kernel agree on a
bank that is full."""
import random

import pytest

import attn_schedule as A


@pytest.mark.parametrize("n_sm", [148, 152])
@pytest.mark.parametrize("H,M,Nq,W,want", [
    (12, 9360, 4680, 4680, A.WHOLE),     # 249 us whole | 264 shares
    (12, 9360, 1560, 4680, A.SHARES),    # 170 | 112
    (12, 9360, 256, 4680, A.SHARES),     # 95 | 37
    (7, 5903, 1846, 0, A.WHOLE),         # 40 | 47
    (123, 7745, 182, 8087, A.WHOLE),     # 212 | 301: keys of all heads past L2
    (160, 9360, 128, 4680, A.SHARES),    # 232 | 189: the same, one query tile a head
    (24, 9360, 1560, 4680, A.SHARES),    # 242 | 206
    (40, 9360, 1560, 4680, A.WHOLE),     # 326 | 507
    (1, 15000, 16, 500, A.SHARES),
    (160, 18720, 4680, 4680, A.TWO),
])
def test_the_measured_lines(H, M, Nq, W, want, n_sm):
    assert A.launched([M] * H, Nq, W, n_sm) == want


def test_the_two_tile_line():
    assert A.launched([9360] * 16, 4680, 4680, 152) == A.TWO      # 341 us shares | 315 two tiles
    assert A.launched([9360] * 17, 4680, 4680, 152) == A.SHARES   # 406 | 460


def test_what_is_never_cut_and_what_both_sides_agree_on():
    rng = random.Random(5)
    seen = set()
    for _ in range(4000):
        H, n_sm = rng.choice([1, 2, 5, 12, 40, 150]), rng.choice([148, 152])
        budgets = [rng.choice([100, 1000, 5000, 20000]) for _ in range(H)]
        Nq, W = int(2 ** rng.uniform(0, 13)), rng.choice([0, 77, 4680])
        got = A.launched(budgets, Nq, W, n_sm)
        seen.add(got)
        assert A.launched(budgets, Nq, W, n_sm, scratch=False) != A.SHARES
        if got == A.SHARES:
            assert A.cuts(budgets, Nq, W, n_sm)
            assert H * ((Nq + 127) // 128) < 1024
            assert (max(budgets) + 127) // 128 + (W + 127) // 128 >= 16
        short = [min(b, 700) for b in budgets]
        if W < 1000:
            assert not A.cuts(short, Nq, W, n_sm)   # at most 7 key tiles
    assert seen == {A.WHOLE, A.SHARES, A.TWO}
