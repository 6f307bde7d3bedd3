"""The force contraction shares a link's s between four lanes and eight sites between a warp's lanes: its
edges are fewer s than lanes (Ns = 2), many (Ns = 32) and the smallest lattices.

Tolerance as in test_gpu_pf_force.py: an inner FP64 solve to 1e-12 differs from the oracle's by at most
kappa * 1e-12, which every force component inherits: 2e-8 of the largest.
"""
import numpy as np
import pytest

import odwf_synth as syn
import paper_1811_08095_gb300 as odwf
from gpu_common import M0, from_dev, make_case, to_dev, torch_cuda
from oracle import hmc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,ns,tbc", [((2, 2, 2, 2), 2, True), ((4, 2, 2, 6), 2, False), ((2, 2, 2, 2), 32, True),
                                         ((2, 6, 2, 2), 16, True)])
def test_force_lanes(dims, ns, tbc):
    torch = torch_cuda()
    U, w = make_case(dims, ns, 0.1, eps=0.5, seed=11)
    h = odwf.Handle(dims, ns, M0, 0.1, w, t_antiperiodic=tbc)
    h.set_gauge(to_dev(torch, U))
    phi = syn.gaussian_spinor_even(ns, dims, 12)
    ref, s_ref = hmc.pf_force(U, phi, M0, 0.1, 0.5, w, tbc)
    F = torch.zeros(U.shape, dtype=torch.complex128, device="cuda")
    act, st = h.pf_force(to_dev(torch, phi), 0.1, 0.5, F, tol=1e-12, max_iter=100000, prec="f64")
    assert st["status"] == 0
    assert abs(act - s_ref) < 1e-9 * s_ref
    assert np.abs(from_dev(F) - ref).max() < 2e-8 * np.abs(ref).max()
    h.close()
