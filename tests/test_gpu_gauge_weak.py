"""The gauge force where it is small: links near the unit field.

There the force comes from the off-diagonal entries and imaginary parts of the links, of size eps, and FP64
keeps it to its relative accuracy.  An entry of U Sigma sums six staples of three products; to first order in
eps each carries at most 28 roundings of terms that add up to 24 eps, a force entry is beta / 3 of that and
the largest entry is not below beta / 3 x 5 eps: 28 x 24 / 5 x 2^-53 = 1.5e-14 of the largest entry for either of
the two evaluations compared, bar 3e-14.
"""
import numpy as np
import pytest

import odwf_synth as syn
import paper_1811_08095_gb300 as odwf
from gpu_common import M0, from_dev, to_dev, torch_cuda
from oracle import hmc, zolotarev

pytestmark = pytest.mark.gpu

BETA = 6.2


def _force(U, dims):
    torch = torch_cuda()
    with odwf.Handle(dims, 4, M0, 0.1, zolotarev.omega(4, 0.05, 6.2, True)[0]) as h:
        F = torch.empty(U.shape, dtype=torch.complex128, device="cuda")
        act = h.gauge_force(to_dev(torch, U), BETA, F)
        assert act == h.gauge_force(to_dev(torch, U), BETA)  # the action alone
    return act, from_dev(F)


@pytest.mark.parametrize("eps", [0.3, 0.1, 1e-2, 1e-4, 1e-6, 1e-8])
@pytest.mark.parametrize("dims", [(4, 4, 2, 6), (2, 6, 4, 2)])
def test_weak_field(eps, dims):
    U = syn.gauge_field(dims, eps, 5)
    act, F = _force(U, dims)
    ref, ract = hmc.gauge_force(U, BETA), hmc.gauge_action(U, BETA)
    assert np.abs(F - ref).max() <= 3e-14 * np.abs(ref).max()
    assert abs(act - ract) <= 1e-12 * BETA * U[..., 0, 0].size


def test_weak_and_rough_regions():
    """Each region of a field keeps the accuracy of its own size: links are weak for t < 6 and rough beyond."""
    dims = (2, 4, 2, 12)
    U, weak = syn.gauge_field(dims, 0.7, 6), syn.gauge_field(dims, 1e-5, 7)
    U[:, :6] = weak[:, :6]
    act, F = _force(U, dims)
    ref, ract = hmc.gauge_force(U, BETA), hmc.gauge_action(U, BETA)
    inside = np.abs(F - ref)[:, 1:5].max(), np.abs(ref)[:, 1:5].max()  # links whose staples are all weak
    assert inside[1] < 1e-3 and inside[0] <= 3e-14 * inside[1]
    assert np.abs(F - ref).max() <= 3e-14 * np.abs(ref).max()
    assert abs(act - ract) <= 1e-12 * BETA * U[..., 0, 0].size
