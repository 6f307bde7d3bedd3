"""Flow.get_gauge against the stored pairs, entry by entry.

A link entry is stored as two FP32 values, u = h + l with |u - h - l| <= 2^-48 |u|, and comes back as their
FP64 sum (one rounding, 2^-53), whatever its size.  The third row is conj(row0 x row1): two products of two
complex numbers per entry, of size D = |a1| |b2| + |a2| |b1|, at most eight roundings of parts of D in either
of the two FP64 evaluations compared here: bar 16 x 2^-53 D.
"""
import numpy as np
import pytest

import odwf_synth as syn
import paper_1811_08095_gb300 as odwf
from gpu_common import from_dev, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

DIMS = (4, 3, 2, 6)


def _round_trip(U):
    torch = torch_cuda()
    with odwf.Flow(DIMS) as f:
        out = torch.empty(U.shape, dtype=torch.complex128, device="cuda")
        f.set_gauge(to_dev(torch, U))
        f.get_gauge(out)
    return from_dev(out)


def _check_third_row(got):
    a, b = got[..., 0, :], got[..., 1, :]
    n, p = [1, 2, 0], [2, 0, 1]
    ref = np.conj(a[..., n] * b[..., p] - a[..., p] * b[..., n])
    D = np.abs(a[..., n]) * np.abs(b[..., p]) + np.abs(a[..., p]) * np.abs(b[..., n])
    err = np.abs(got[..., 2, :] - ref)
    assert (err <= 16 * 2.0 ** -53 * D).all(), np.max(err / np.where(D > 0, D, 1.0))


@pytest.mark.parametrize("size", [1.24, 1.26, 1.41, 1.42, 1.45, 1.49, 1.51])
def test_entries_above_one(size):
    """Entries of either sign up to the sizes at which the products of two entries add up to 8 and more."""
    rng = np.random.default_rng(4)
    shape = (4, DIMS[3], DIMS[2], DIMS[1], DIMS[0], 3, 3)
    U = size * (rng.choice([-1.0, 1.0], shape) + 1j * rng.choice([-1.0, 1.0], shape))
    _check_third_row(_round_trip(U))


@pytest.mark.parametrize("eps", [0.3, 2.0 ** -5, 1e-3, 1e-6, 1e-12])
def test_small_entries_keep_their_bits(eps):
    """Links near the unit field: entries off the diagonal and imaginary parts of size eps."""
    U = syn.gauge_field(DIMS, eps, 7)
    got = _round_trip(U)
    rows, ref = got[..., :2, :].view(np.float64), np.ascontiguousarray(U[..., :2, :]).view(np.float64)
    assert (np.abs(rows - ref) <= (2.0 ** -48 + 2.0 ** -53) * np.abs(ref)).all()
    _check_third_row(got)


@pytest.mark.parametrize("scale", [2.0 ** -60, 2.0 ** -30, 2.0 ** -14])
def test_one_small_row(scale):
    U = syn.gauge_field(DIMS, 0.8, 8)
    U[..., 0, :] *= scale
    got = _round_trip(U)
    rows, ref = got[..., :2, :].view(np.float64), np.ascontiguousarray(U[..., :2, :]).view(np.float64)
    assert (np.abs(rows - ref) <= (2.0 ** -48 + 2.0 ** -53) * np.abs(ref)).all()
    _check_third_row(got)
