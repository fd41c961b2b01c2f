"""The fused y pass on two columns per CTA and on one, where the rule between
them (ypass_pairs) draws its lines.  A whole evaluation and the two single calls
may take different passes of one source, so its H_eff (no exchange, anisotropy or
applied field) is compared with their sum, and at sizes the oracle does in
seconds with the oracle.

Bars: relative L2 <= 1e-5 of each against the FP64 oracle; between two of them
the sum of their bars, 2e-5."""

import pytest

import workloads
from oracle import fields as OF
from oracle.interaction import stray_interaction
from tests.pair_setup import gpu_pair, rel_l2

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _pair(n, n1=None):
    fp, _, _ = workloads.film_pair_plain(n, 2, 7)
    fp.n_slider = n1 or n
    fp.mat_base.Aex = fp.mat_slider.Aex = 0.0
    fp.u0 = (0.3, -0.2, 0.0)
    m0, m1 = workloads.random_unit(n, 7), workloads.random_unit(fp.n_slider, 8)
    return fp, m0, m1, gpu_pair(fp, m0, m1, mech=False)


def _fields(mm, g):
    """Whole evaluation, own field, other's field of magnet g."""
    whole = mm.compute_torque(g)[1].double().cpu().numpy()
    return whole, mm.compute_demag(g).double().cpu().numpy(), mm.compute_stray_field(1 - g).double().cpu().numpy()


@pytest.mark.parametrize("n,n1", [
    ((296, 33, 1), None),              # many columns: pairs in every call
    ((296, 20, 2), (297, 31, 3)),      # two and three layers, odd column counts
    ((140, 33, 1), (133, 21, 3)),      # a whole evaluation on pairs, single calls on columns
    ((140, 33, 2), None),              # columns in every call
    ((296, 190, 1), (296, 190, 2)),    # longer lines: columns
    ((9, 60, 2), (9, 125, 1)),         # few columns of compiled lengths: pairs
])
def test_fields_match_oracle(n, n1):
    fp, m0, m1, mm = _pair(n, n1)
    M = (fp.mat_base.Ms * m0, fp.mat_slider.Ms * m1)
    for g in (0, 1):
        whole, own, other = _fields(mm, g)
        ref_own = OF.demag_conv(M[g], fp.cell)
        ref = stray_interaction(M[1 - g], M[g], fp.cell, fp.offsets[1 - g], fp.offsets[g], fp.u0, g == 1)["H"]
        assert rel_l2(own, ref_own) < TOL
        assert rel_l2(other, ref) < TOL
        assert rel_l2(whole, ref_own + ref) < TOL
    mm.close()


@pytest.mark.parametrize("n", [
    (300, 256, 1), (640, 250, 1),                   # lines of up to 640 points, few and many columns
    (450, 512, 1), (450, 512, 2), (450, 512, 3),    # 1080 points: pairs in whole evaluations
    (450, 1024, 1), (770, 256, 2), (770, 256, 3),   # 2160 points, 540 points of two layers (and three: columns)
])
def test_whole_evaluation_is_the_sum_of_the_single_calls(n):
    _, _, _, mm = _pair(n)
    for g in (0, 1):
        whole, own, other = _fields(mm, g)
        assert rel_l2(whole, own + other) < 2 * TOL
    mm.close()
