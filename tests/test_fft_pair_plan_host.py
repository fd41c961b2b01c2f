"""The planner of the passes that run two lines at once (mm_fft_pair_plan), no
GPU: orders multiply out with the fewest stages of radices up to 12, start with
four or more where they can (the twiddle tables count on it), and the lengths the
y pass is compiled for are the planner's own choice for them."""

import numpy as np
import pytest

from paper_1801_04181_gb300 import _native

RADICES = (2, 3, 4, 5, 6, 8, 9, 10, 12)


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_1801_04181_gb300.build import build

    build()
    return _native.load()


def _smooth(L):
    for p in (2, 3, 5):
        while L % p == 0:
            L //= p
    return L == 1


def _fewest_stages(L):
    best = {1: 0}
    for n in range(2, L + 1):
        if L % n == 0:
            best[n] = min((best[n // r] + 1 for r in RADICES if n % r == 0 and (n // r) in best), default=10 ** 9)
    return best[L]


def test_pair_plans_multiply_out_with_fewest_stages():
    from paper_1801_04181_gb300 import fft_pair_plan

    for L in filter(_smooth, range(2, 2400, 2)):
        plan, _ = fft_pair_plan(L)
        assert int(np.prod(plan)) == L and all(r in RADICES for r in plan)
        assert len(plan) == _fewest_stages(L)
        assert plan[0] >= 4 or max(plan) < 4


def test_the_compiled_lengths_are_the_planners_choice():
    """64, 128, 256, 512 and 1024 cells at a margin of four, and no others."""
    from paper_1801_04181_gb300 import fft_pair_plan

    assert [L for L in filter(_smooth, range(2, 4000, 2)) if fft_pair_plan(L)[1]] == [160, 288, 540, 1080, 2160]


def test_pair_plan_rejects_lengths_outside_2_3_5():
    from paper_1801_04181_gb300 import MMError, fft_pair_plan

    for L in (0, 7, 14, 22):
        with pytest.raises(MMError):
            fft_pair_plan(L)
