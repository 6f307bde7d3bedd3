"""Flow.set_gauge / get_gauge: the split of FP64 links into pairs of FP32 and their sums, in integers.

A pair resolves 2^-48 of an entry (the sum 2^-60 of 1 in fixed point); the third row is rebuilt from the
first two.  Entries of 1.5 or more, zeros and entries below 2^-60 take the FP64 branches.
"""
import numpy as np
import pytest

import odwf_synth as syn
import paper_1811_08095_gb300 as odwf
from gpu_common import from_dev, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (5, 3, 7, 4)])  # 420 sites: a ragged last block
@pytest.mark.parametrize("kind", ["random", "unit", "tiny entries", "times 3", "not a number"])
def test_round_trip(dims, kind):
    torch = torch_cuda()
    U = syn.gauge_field(dims, 0.8, 3)
    if kind == "unit":
        U = np.zeros_like(U)
        U[..., range(3), range(3)] = 1.0
    elif kind == "tiny entries":
        U[..., 0, :] *= 2.0 ** -70
    elif kind == "times 3":
        U = U * 3.0
    elif kind == "not a number":
        U[2, 1, 0, 1, 0, 1, 2] = np.nan
    with odwf.Flow(dims) as f:
        out, host = torch.empty(U.shape, dtype=torch.complex128, device="cuda"), np.empty_like(U)
        f.set_gauge(to_dev(torch, U))
        f.get_gauge(out)
        f.set_gauge(U)  # host pointers
        f.get_gauge(host)
    got = from_dev(out)
    assert np.array_equal(got, host, equal_nan=True)
    rows, ref = got[..., :2, :].view(np.float64), np.ascontiguousarray(U[..., :2, :]).view(np.float64)
    ok = np.isfinite(ref)
    assert np.array_equal(np.isfinite(rows), ok)
    assert (np.abs(rows - ref)[ok] <= 2.0 ** -48 * np.abs(ref[ok]) + 2.0 ** -59).all()
    third = np.conj(np.cross(got[..., 0, :], got[..., 1, :]))
    fin = np.isfinite(third)
    assert np.array_equal(np.isfinite(got[..., 2, :]), fin)
    assert np.abs(got[..., 2, :] - third)[fin].max() <= 1e-15 * max(1.0, np.abs(third[fin]).max())
