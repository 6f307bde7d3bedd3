"""A handle's first gauge force splits the links where they are used on lattices of 1821 to 16384 sites (limbs
above 1 MB); later calls and other lattices split them in a pass before.  The arithmetic is the same: equal bits.
"""
import numpy as np
import pytest

import odwf_synth as syn
import paper_1811_08095_gb300 as odwf
from gpu_common import M0, from_dev, to_dev, torch_cuda
from oracle import hmc, zolotarev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(6, 6, 6, 8), (6, 6, 8, 8), (16, 8, 8, 16), (16, 8, 10, 16)])  # both sides of the edges
def test_first_call_equals_later_ones(dims):
    torch = torch_cuda()
    U = syn.gauge_field(dims, 0.7, 3)
    U[:, :, 1] = syn.gauge_field(dims, 1e-4, 4)[:, :, 1]  # some links for the FP64 kernel
    with odwf.Handle(dims, 4, M0, 0.1, zolotarev.omega(4, 0.05, 6.2, True)[0]) as h:
        out = []
        for _ in range(3):
            F = torch.empty(U.shape, dtype=torch.complex128, device="cuda")
            out.append((h.gauge_force(to_dev(torch, U), 6.2, F), from_dev(F)))
    for act, F in out[1:]:
        assert act == out[0][0] and np.array_equal(F, out[0][1])
    ref = hmc.gauge_force(U, 6.2)
    assert np.abs(out[0][1] - ref).max() <= 3e-14 * np.abs(ref).max()
