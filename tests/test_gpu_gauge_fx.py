"""The fixed-point gauge force against the oracle, and the fields it hands to the FP64 kernel.

Links are split into 60 fraction bits when every row and column is of unit length to 2^-16; any other
field (the entry point takes any matrices) runs in FP64.  Bar 1e-12 of the largest force component, as
in test_gpu_md.py.
"""
import numpy as np
import pytest

import odwf_synth as syn
import paper_1811_08095_gb300 as odwf
from gpu_common import M0, from_dev, to_dev, torch_cuda
from oracle import hmc, zolotarev

pytestmark = pytest.mark.gpu


def _field(kind, dims):
    U = syn.gauge_field(dims, 0.7, 3)
    if kind == "unit":
        U = np.zeros_like(U)
        U[..., range(3), range(3)] = 1.0
    elif kind == "signed permutation":  # entries exactly -1, 0, 1
        U = np.zeros_like(U)
        U[..., 0, 1], U[..., 1, 2], U[..., 2, 0] = -1.0, 1j, 1j
    elif kind == "nearly unitary":
        U = U * (1.0 + 2e-6)
    elif kind == "scaled":
        U = U * 3.0
    elif kind == "one bad link":
        U[1, 1, 0, 1, 0] *= 1e3
    return U


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 2, 6, 4)])
@pytest.mark.parametrize("kind", ["random", "unit", "signed permutation", "nearly unitary", "scaled", "one bad link"])
def test_gauge_force_fields(kind, dims):
    torch = torch_cuda()
    U, beta = _field(kind, dims), 6.2
    with odwf.Handle(dims, 4, M0, 0.1, zolotarev.omega(4, 0.05, 6.2, True)[0]) as h:
        F = torch.empty(U.shape, dtype=torch.complex128, device="cuda")
        act = h.gauge_force(to_dev(torch, U), beta, F)
        act2 = h.gauge_force(to_dev(torch, U), beta)  # the action alone
    ref, ract = hmc.gauge_force(U, beta), hmc.gauge_action(U, beta)
    scale = max(np.abs(ref).max(), beta * np.abs(U).max() ** 4)
    assert np.abs(from_dev(F) - ref).max() <= 1e-12 * scale
    assert act == act2 and abs(act - ract) <= 1e-12 * max(abs(ract), scale * U[..., 0, 0].size)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_link(bad):
    torch = torch_cuda()
    dims = (4, 4, 4, 4)
    U = syn.gauge_field(dims, 0.7, 3)
    U[2, 1, 0, 3, 2, 1, 0] = bad
    with odwf.Handle(dims, 4, M0, 0.1, zolotarev.omega(4, 0.05, 6.2, True)[0]) as h:
        F = torch.empty(U.shape, dtype=torch.complex128, device="cuda")
        act = h.gauge_force(to_dev(torch, U), 6.2, F)
    with np.errstate(invalid="ignore"):
        links = np.isfinite(hmc.gauge_force(U, 6.2)).all(axis=(-2, -1))
    assert not np.isfinite(act)
    assert np.array_equal(np.isfinite(from_dev(F)).all(axis=(-2, -1)), links)
