"""What the timings of single kernels count: the sums over block partials that a mixed CG iteration makes are
part of them.  Lattices with more than 256 partials form beta in a launch of its own, between K4 and the p
update; smaller ones in the p update and the next K1.
"""
import ctypes

import pytest

import odwf_synth as syn
import paper_1811_08095_gb300 as odwf
from gpu_common import M0, make_case, to_dev, torch_cuda
from paper_1811_08095_gb300 import _lib

pytestmark = pytest.mark.gpu

LARGE, SMALL = ((8, 8, 8, 32), 16), ((4, 4, 4, 4), 8)


def _handle(torch, dims, ns):
    U, w = make_case(dims, ns, 0.5)
    h = odwf.Handle(dims, ns, M0, 0.5, w)
    h.set_gauge(to_dev(torch, U))
    return h, to_dev(torch, syn.gaussian_spinor_even(ns, dims, 3))


@pytest.mark.parametrize("nsys", [1, 3])
@pytest.mark.parametrize("lattice,kind,per_rep", [(LARGE, 3, 1), (LARGE, 4, 2), (LARGE, 5, 1), (SMALL, 4, 1), (SMALL, 1, 1)])
def test_time_kernel_counts_the_sums(lattice, kind, per_rep, nsys):
    torch, lib = torch_cuda(), odwf.load()
    h, fill = _handle(torch, *lattice)
    h.time_kernel(kind, fill, prec="f16", nsys=nsys, reps=1)  # makes the low-precision links
    n = []
    for reps in (5, 15):
        before = lib.odwf_launch_count()
        r = h.time_kernel(kind, fill, prec="f16", nsys=nsys, reps=reps)
        n.append(lib.odwf_launch_count() - before)
        assert r["launches"] == reps and r["system_launches"] == reps * nsys and r["total_ms"] > 0
    h.close()
    assert n[1] - n[0] == 10 * per_rep


@pytest.mark.parametrize("lattice", [LARGE, SMALL])
def test_profile_of_a_solve_has_every_launch_of_the_iteration(lattice):
    torch, lib = torch_cuda(), odwf.load()
    h, b = _handle(torch, *lattice)
    x = torch.zeros_like(b)
    _lib.check(lib.odwf_profile_enable(1))
    st = h.cg_solve(x, b, tol=1e-8, prec="f16")
    arr, n = (_lib.odwf_kernel_prof * 64)(), ctypes.c_int(0)
    _lib.check(lib.odwf_profile_read(ctypes.cast(arr, ctypes.c_void_p), 64, ctypes.byref(n)))
    _lib.check(lib.odwf_profile_enable(0))
    h.close()
    prof = {arr[i].name.decode().split(".v2.")[-1]: arr[i].launches for i in range(n.value)}
    assert st["status"] == 0
    k4 = prof["K4_normal_cg"]
    assert prof["K1_chi_minv"] == prof["K2_schur_norm_mdinv"] == prof["K3_dag_minvdag"] == k4
    if lattice is LARGE:
        assert prof["beta_sum"] == k4
    else:
        assert 0 < prof["beta_sum"] < k4  # the last iteration of every chunk
