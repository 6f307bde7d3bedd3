"""The FP64-accuracy hops in block fixed point against the oracle, at the edges of their number format.

A 5D site is stored as integers with one exponent and resolves 2^-57 of its largest component, sums
of eight neighbours 2^-55; bars below are 1e-12 of the component scale, as for the FP64 operators
(test_gpu_operator.py).  Sites whose components span more than 2^32, non-finite values and values
near the ends of the FP64 range keep their FP64 bits and go through FP64 arithmetic.
"""
import numpy as np
import pytest

import odwf_synth as syn
import oracle
import paper_1811_08095_gb300 as odwf
from gpu_common import M0, assert_close_componentwise, from_dev, make_case, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


def _apply(torch, dims, ns, mq, w, U, psi, dagger):
    with odwf.Handle(dims, ns, M0, mq, w) as h:
        h.set_gauge(to_dev(torch, U))
        out = torch.empty(psi.shape, dtype=torch.complex128, device="cuda")
        (h.apply_dagger if dagger else h.apply)(out, to_dev(torch, psi), odwf.ODWF_MODE_SCHUR_EVEN)
        return from_dev(out)


@pytest.mark.parametrize("dagger", [False, True])
@pytest.mark.parametrize("dims,ns", [((2, 2, 2, 2), 2), ((2, 2, 2, 2), 32), ((6, 2, 4, 2), 4), ((4, 6, 2, 10), 16)])
def test_lane_groups_and_ragged_blocks(torch, dims, ns, dagger):
    U, w = make_case(dims, ns, 0.05, eps=0.6, seed=3)
    psi = syn.gaussian_spinor_even(ns, dims, 5)
    ref = oracle.schur(U, psi, M0, 0.05, w, True, dagger=dagger)
    assert_close_componentwise(_apply(torch, dims, ns, 0.05, w, U, psi, dagger), ref, 1e-12)


@pytest.mark.parametrize("scale", [1e-300, 1e-200, 1e200])
@pytest.mark.parametrize("dagger", [False, True])
def test_field_scale(torch, scale, dagger):
    dims, ns = (4, 2, 2, 4), 8
    U, w = make_case(dims, ns, 0.05, eps=0.6, seed=4)
    psi = syn.gaussian_spinor_even(ns, dims, 6)
    ref = oracle.schur(U, psi, M0, 0.05, w, True, dagger=dagger)
    got = _apply(torch, dims, ns, 0.05, w, U, psi * scale, dagger) / scale
    assert_close_componentwise(got, ref, 1e-12)


@pytest.mark.parametrize("links", ["unit", "times 3", "times 1e-3", "dense", "mixed scales"])
def test_links_outside_su3(torch, links):
    """The FP64 operators take any 3 x 3 matrices."""
    dims, ns = (4, 2, 4, 4), 8
    U, w = make_case(dims, ns, 0.05, eps=0.6, seed=5)
    rng = np.random.default_rng(9)
    if links == "unit":
        U = np.zeros_like(U)
        U[..., range(3), range(3)] = 1.0
    elif links == "dense":
        U = rng.uniform(0.9, 1.0, U.shape) + 1j * rng.uniform(-1.0, -0.9, U.shape)
    elif links == "mixed scales":
        U = U * np.exp2(rng.integers(-8, 9, U.shape[:5]))[..., None, None]
    else:
        U = U * float(links.split()[1])
    psi = syn.gaussian_spinor_even(ns, dims, 7)
    for dagger in (False, True):
        ref = oracle.schur(U, psi, M0, 0.05, w, True, dagger=dagger)
        assert_close_componentwise(_apply(torch, dims, ns, 0.05, w, U, psi, dagger), ref, 1e-12)


@pytest.mark.parametrize("dagger", [False, True])
def test_wide_range_keeps_small_colours(torch, dagger):
    """Unit links never mix colours: a colour 1e-15 below another keeps its own relative accuracy."""
    dims, ns = (4, 4, 2, 2), 4
    U, w = make_case(dims, ns, 0.05, eps=0.0, seed=1)
    U = np.zeros_like(U)  # exactly 1 (the generator's eigendecomposition leaves 1e-15 off the diagonal)
    U[..., range(3), range(3)] = 1.0
    psi = syn.gaussian_spinor_even(ns, dims, 8)
    psi[..., 1] *= 1e-15
    psi[..., 2] = 0.0
    ref = oracle.schur(U, psi, M0, 0.05, w, True, dagger=dagger)
    got = _apply(torch, dims, ns, 0.05, w, U, psi, dagger)
    for c in (0, 1):
        assert_close_componentwise(got[..., c], ref[..., c], 1e-12)
    assert not got[..., 2].any()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_values_reach_the_same_sites(torch, bad):
    dims, ns = (4, 4, 4, 4), 8
    U, w = make_case(dims, ns, 0.05, eps=0.6, seed=6)
    psi = syn.gaussian_spinor_even(ns, dims, 9)
    psi[3, 5, 1, 2] = bad
    for dagger in (False, True):
        ref = oracle.schur(U, psi, M0, 0.05, w, True, dagger=dagger)
        got = _apply(torch, dims, ns, 0.05, w, U, psi, dagger)
        # the oracle's dense M^-1 multiplies exact zeros along s and spin, so the two agree on the sites
        # a non-finite value reaches, not on its components there
        sites = np.isfinite(ref).all(axis=(0, 2, 3))
        assert sites.any() and not sites.all()
        assert np.array_equal(np.isfinite(got).all(axis=(0, 2, 3)), sites)
        scale = np.abs(ref[:, sites]).max()
        assert np.abs(got[:, sites] - ref[:, sites]).max() <= 1e-12 * scale
    Ub = U.copy()
    Ub[1, 2, 1, 3, 0, 1, 1] = bad
    got = _apply(torch, dims, ns, 0.05, w, Ub, syn.gaussian_spinor_even(ns, dims, 9), False)
    assert not np.isfinite(got).all() and np.isfinite(got).any()


@pytest.mark.parametrize("ns", [4, 32])
def test_full_fields_and_in_place(torch, ns):
    """Operators read and write the caller's fields directly: full fields of both parities on a ragged
    lattice, and out = in."""
    dims = (4, 6, 2, 6)
    U, w = make_case(dims, ns, 0.05, eps=0.6, seed=7)
    rng = np.random.default_rng(11)
    shape = (ns, dims[3], dims[2], dims[1], dims[0], 4, 3)
    psi = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    even = syn.gaussian_spinor_even(ns, dims, 12)
    with odwf.Handle(dims, ns, M0, 0.05, w) as h:
        h.set_gauge(to_dev(torch, U))
        for op in ("apply", "apply_dagger", "apply_normal"):
            for f in (psi, even):
                arg = ((odwf.ODWF_SYS_FULL_NORMAL if f is psi else odwf.ODWF_SYS_SCHUR_NORMAL) if op == "apply_normal"
                       else (odwf.ODWF_MODE_FULL if f is psi else odwf.ODWF_MODE_SCHUR_EVEN))
                x = to_dev(torch, f)
                out = torch.empty_like(x)
                getattr(h, op)(out, x, arg)
                host = np.empty_like(f)
                getattr(h, op)(host, f, arg)  # host pointers
                getattr(h, op)(x, x, arg)
                assert np.array_equal(from_dev(out), host) and np.array_equal(from_dev(out), from_dev(x))
                if f is even:
                    ref = (oracle.normal_op(U, f, M0, 0.05, w) if op == "apply_normal"
                           else oracle.schur(U, f, M0, 0.05, w, True, dagger=op == "apply_dagger"))
                    assert_close_componentwise(host, ref, 1e-12)
