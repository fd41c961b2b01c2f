"""The passes that run two lines at once, at the sizes where they can go wrong:
odd column counts, chunks of coefficient planes, lines too long for a pair, the
edge between the short and long x builds, tiles and remainders of the z pass,
the plane mixing and its transpose, and the SOR on degenerate grids.

Bar: the FP32 fields' relative L2 <= 1e-5 against the FP64 oracle.
"""

import numpy as np
import pytest
import torch

import workloads
from oracle import eddy as OE
from oracle import fields as OF
from oracle.adjoint import energy_gradients
from oracle.interaction import stray_interaction
from tests.pair_setup import gpu_pair, rel_l2

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _pair(n0, n1, seed, gap=2, u=(0.3, -0.2, 0.0)):
    fp, _, _ = workloads.film_pair_plain(n0, gap, seed)
    fp.n_slider = n1
    fp.u0 = u
    return fp, workloads.random_unit(n0, seed), workloads.random_unit(n1, seed + 1)


@pytest.mark.parametrize("n0,n1", [
    ((9, 33, 1), (9, 33, 1)),        # fused y pass, one layer: two outputs per batch of quads
    ((7, 20, 1), (7, 20, 2)),        # an odd number of outputs
    ((8, 310, 2), (8, 310, 2)),      # coefficient planes in chunks of three and two
    ((6, 1024, 1), (6, 1024, 1)),    # one CTA per SM, chunks of two
    ((6, 330, 3), (6, 330, 3)),      # one CTA per SM, all planes at once
    ((6, 140, 4), (6, 140, 4)),      # four layers: one column per CTA
    ((5, 700, 3), (5, 256, 1)),      # a column source beside a pair source
    ((5, 1760, 1), (5, 1760, 1)),    # lines too long for a pair
    ((1, 1, 1), (2, 3, 1)),          # the smallest lines
    ((113, 9, 2), (113, 9, 2)),      # x lines of at most 256 points
    ((117, 9, 2), (117, 9, 2)),      # and just beyond
    ((15, 14, 5), (11, 13, 7)),      # plane mixing of odd layer counts, odd columns
    ((12, 70, 8), (12, 70, 6)),      # its last chunk of frequencies
    ((6, 5, 9), (7, 5, 12)),         # z pass: the fewest layers
    ((5, 21, 70), (5, 21, 70)),      # whole and partial tiles of positions
    ((4, 3, 190), (4, 3, 190)),      # the longest z lines: four positions a tile
])
def test_fields_match_oracle(n0, n1):
    fp, m0, m1 = _pair(n0, n1, 11)
    mm = gpu_pair(fp, m0, m1, mech=False)
    Ms = fp.mat_base.Ms
    ms = (m0, m1)
    for src in (0, 1):
        t = 1 - src
        H = mm.compute_stray_field(src).double().cpu().numpy()
        ref = stray_interaction(Ms * ms[src], Ms * ms[t], fp.cell, fp.offsets[src], fp.offsets[t], fp.u0, t == 1)
        assert rel_l2(H, ref["H"]) < TOL
        assert rel_l2(mm.compute_demag(src).double().cpu().numpy(), OF.demag_conv(Ms * ms[src], fp.cell)) < TOL
    # a whole evaluation takes both kinds of plane through the passes at once
    mm.compute_fields()
    H2 = mm.compute_stray_field(1).double().cpu().numpy()
    assert rel_l2(H2, ref["H"]) < TOL
    mm.close()


@pytest.mark.parametrize("n0,n1", [((6, 7, 1), (5, 6, 1)), ((7, 6, 8), (6, 5, 3)), ((5, 9, 17), (6, 4, 11)),
                                   ((3, 40, 25), (3, 35, 4))])
def test_energy_gradients_match_oracle(n0, n1):
    """Layers in whole and partial groups of eight, box planes in whole and partial stages of 32."""
    fp, m0, m1 = _pair(n0, n1, 5)
    mm = gpu_pair(fp, m0, m1, mech=False)
    Ms = fp.mat_base.Ms
    _, gs, gt = mm.backward_energy(0)
    ref = energy_gradients(Ms * m0, Ms * m1, fp.cell, fp.offsets[0], fp.offsets[1], fp.u0, True)
    assert rel_l2(gs.double().cpu().numpy(), Ms * ref["dE_dMs"]) < TOL
    assert rel_l2(gt.double().cpu().numpy(), Ms * ref["dE_dMt"]) < TOL
    mm.close()


@pytest.mark.parametrize("n", [(1, 7, 5), (6, 1, 3), (2, 2, 1), (5, 3, 2), (33, 5, 4)])
def test_eddy_currents_on_degenerate_grids(n):
    """Axes of one or two cells and odd rows: every count of neighbours of the SOR update."""
    fp, m0, m1 = _pair(n, n, 3)
    mm = gpu_pair(fp, m0, m1, mech=False)
    dB = np.random.default_rng(2).standard_normal((3, n[2], n[1], n[0])) * 1e9
    H, J, sweeps = mm.eddy_field(0, torch.as_tensor(dB, dtype=torch.float32, device="cuda"), 1e6)
    ref = OE.eddy_field(dB.astype(np.float32).astype(np.float64), fp.cell, 1e6, return_all=True)
    assert sweeps > 0
    assert rel_l2(J.double().cpu().numpy(), ref["J"]) < TOL
    assert rel_l2(H.double().cpu().numpy(), ref["H"]) < TOL
    mm.close()
