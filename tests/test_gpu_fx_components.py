"""The FP64-accuracy hops component by component, where components of very different size do not mix.

Unit or diagonal links never mix colours, so a colour far below the others has a result of its own size, and
an FP64 operator gives it to its own relative accuracy.  An output component sums 16 products, the operators
along s at most 2 Ns terms more with a norm of M^-1 of a few, and a Schur operator does both twice: some 200
roundings of parts of the size of the largest value of that colour, 2e-14 for either of the two evaluations
compared; bar 1e-13 of the colour's largest value.
"""
import numpy as np
import pytest

import odwf_synth as syn
import oracle
import paper_1811_08095_gb300 as odwf
from gpu_common import M0, from_dev, make_case, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

MQ = 0.05


def _check_colours(got, ref):
    for c in range(3):
        assert np.abs(got[..., c] - ref[..., c]).max() <= 1e-13 * np.abs(ref[..., c]).max(), c


def _ops(torch, dims, ns, U, w, psi, full):
    """(got, ref) of the operator, its adjoint and the normal operator."""
    x = to_dev(torch, psi)
    mode = odwf.ODWF_MODE_FULL if full else odwf.ODWF_MODE_SCHUR_EVEN
    system = odwf.ODWF_SYS_FULL_NORMAL if full else odwf.ODWF_SYS_SCHUR_NORMAL
    with odwf.Handle(dims, ns, M0, MQ, w) as h:
        h.set_gauge(to_dev(torch, U))
        for dagger in (False, True):
            out = torch.empty_like(x)
            (h.apply_dagger if dagger else h.apply)(out, x, mode)
            yield from_dev(out), (oracle.d5(U, psi, M0, MQ, w, True, dagger=dagger) if full
                                  else oracle.schur(U, psi, M0, MQ, w, True, dagger=dagger))
        out = torch.empty_like(x)
        h.apply_normal(out, x, system)
        yield from_dev(out), oracle.normal_op(U, psi, M0, MQ, w, True, oracle.FULL_NORMAL if full else oracle.SCHUR_NORMAL)


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


def test_noise_off_the_diagonal(torch):
    """A free field as an eigendecomposition makes it: 1e-15 off the diagonal, a colour at that level."""
    dims, ns = (4, 4, 2, 6), 16
    U, w = make_case(dims, ns, MQ, eps=0.0, seed=1)
    psi = syn.gaussian_spinor_even(ns, dims, 11)
    psi[..., 1] *= 1e-15
    for got, ref in _ops(torch, dims, ns, U, w, psi, False):
        _check_colours(got, ref)
