"""A context whose materials are set again answers like a new one: every kernel
spectrum carries the source's saturation magnetisation.  Same kernels on the same
values: compared bit for bit."""

import numpy as np
import pytest
import torch

import workloads
from tests.pair_setup import gpu_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(14, 9, 2), (9, 7, 6)])
def test_every_field_after_a_second_set_material(n):
    fp, _, _ = workloads.film_pair_plain(n, 2, 3)
    fp.u0 = (0.3, -0.2, 0.0)
    m0, m1 = workloads.random_unit(n, 3), workloads.random_unit(n, 4)
    dB = torch.as_tensor(np.random.default_rng(2).standard_normal((3, n[2], n[1], n[0])) * 1e9, dtype=torch.float32,
                         device="cuda")

    def fields(mm):
        _, J, _ = mm.eddy_field(0, dB, 1e6)
        return [mm.compute_stray_field(0), mm.compute_demag(0), mm.compute_potential(0)[0],
                mm.compute_stray_field_componentwise(0), mm.compute_stray_field_fd4(0), mm.backward_energy(0)[1],
                mm.eddy_field(0, dB, 1e6)[0], J, mm.eddy_field_on_other(0, J)]

    used = gpu_pair(fp, m0, m1, mech=False)
    fields(used)
    fp.mat_base.Ms = 3e5
    for g in (0, 1):
        used.set_material(g, fp.mat_base.Ms, Aex=fp.mat_base.Aex, alpha=fp.mat_base.alpha)
    got = fields(used)
    fresh = gpu_pair(fp, m0, m1, mech=False)
    for i, (a, b) in enumerate(zip(got, fields(fresh))):
        assert torch.equal(a, b), i
    used.close()
    fresh.close()
