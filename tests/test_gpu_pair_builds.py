"""The passes on two lines at once at the lengths they are compiled for, which
run no other plan: fields against the FP64 oracle, relative L2 <= 1e-5."""

import pytest

import workloads
from oracle import fields as OF
from oracle.interaction import stray_interaction
from tests.pair_setup import gpu_pair, rel_l2

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _check(fp, m0, m1, mm):
    M0, M1 = fp.mat_base.Ms * m0, fp.mat_slider.Ms * m1
    ref = stray_interaction(M0, M1, fp.cell, fp.offsets[0], fp.offsets[1], fp.u0, True)
    assert rel_l2(mm.compute_stray_field(0).double().cpu().numpy(), ref["H"]) < TOL
    assert rel_l2(mm.compute_demag(1).double().cpu().numpy(), OF.demag_conv(M1, fp.cell)) < TOL


@pytest.mark.parametrize("n,Qy", [((5, 64, 3), 160), ((5, 128, 1), 288), ((5, 128, 2), 288), ((5, 256, 2), 540),
                                  ((5, 512, 1), 1080), ((5, 512, 2), 1080), ((5, 1024, 1), 2160)])
def test_y_pass(n, Qy):
    fp, m0, m1 = workloads.film_pair_plain(n, 2, 7)
    fp.u0 = (0.3, -0.2, 0.0)
    mm = gpu_pair(fp, m0, m1, mech=False)
    assert mm.plan_info(0)["fft"][1] == Qy
    _check(fp, m0, m1, mm)
    mm.close()


@pytest.mark.parametrize("nz,Qz", [(64, 160), (128, 288)])
def test_z_pass(nz, Qz):
    fp, m0, m1 = workloads.cube_pair((4, 3, nz), 2, 7)
    fp.u0 = (0.0, 0.3, -0.2)
    mm = gpu_pair(fp, m0, m1, mech=False)
    assert mm.plan_info(0)["Qz"] == Qz
    _check(fp, m0, m1, mm)
    mm.close()
