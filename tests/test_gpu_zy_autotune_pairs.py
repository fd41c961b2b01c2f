"""Autotuned orders in the passes on two lines at once: whichever of sixteen
candidates is kept, the fields still match.  Collected late: tuned plans are
process-wide."""

import pytest

import workloads
from oracle import fields as OF
from oracle.interaction import stray_interaction
from paper_1801_04181_gb300 import fft_pair_plan
from tests.pair_setup import gpu_pair, rel_l2

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _tuned(n):
    fp, m0, m1 = workloads.film_pair_plain(n, 2, 4)
    fp.mat_base.Aex = fp.mat_slider.Aex = 0.0
    fp.u0 = (0.3, 0.6, 0.0)
    mm = gpu_pair(fp, m0, m1, mech=False)
    assert fft_pair_plan(mm.plan_info(0)["fft"][1])[1]
    mm.autotune(candidates=16, reps=2)
    return fp, m0, m1, mm


def test_fields_after_tuning_match_oracle():
    fp, m0, m1, mm = _tuned((6, 64, 2))
    ref = stray_interaction(fp.mat_base.Ms * m0, fp.mat_slider.Ms * m1, fp.cell, fp.offsets[0], fp.offsets[1], fp.u0, True)
    assert rel_l2(mm.compute_stray_field(0).double().cpu().numpy(), ref["H"]) < TOL
    assert rel_l2(mm.compute_demag(0).double().cpu().numpy(), OF.demag_conv(fp.mat_base.Ms * m0, fp.cell)) < TOL
    mm.close()


def test_long_lines_after_tuning():
    """512 cells in y: 1080 points, where the candidates hold the radices of a
    compiled plan in another order.  A whole evaluation runs on pairs of lines, a
    single call on single lines; each is within 1e-5 of the exact field."""
    _, _, _, mm = _tuned((450, 512, 1))
    for g in (0, 1):
        whole = mm.compute_torque(g)[1].double().cpu().numpy()
        parts = mm.compute_demag(g).double().cpu().numpy() + mm.compute_stray_field(1 - g).double().cpu().numpy()
        assert rel_l2(whole, parts) < 2 * TOL
    mm.close()


def test_each_kind_of_pass_keeps_what_was_timed_in_it():
    """The same lengths in passes on pairs of lines (a film of one layer) and, in y, on
    single lines (one of six): what the first run kept for y says nothing about the second."""
    kept = []
    for n, fresh in (((21, 128, 1), 2), ((21, 128, 6), 1), ((21, 128, 1), 0), ((21, 128, 6), 0)):
        fp, m0, m1 = workloads.film_pair_plain(n, 2, 4)
        mm = gpu_pair(fp, m0, m1, mech=False)
        kept.append(mm.plan_info(0)["fft"])
        assert mm.autotune(candidates=2, reps=1) == fresh
        mm.close()
    assert len(set(kept)) == 1 and kept[0][0] != kept[0][1]
