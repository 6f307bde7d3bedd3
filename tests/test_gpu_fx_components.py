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
from gpu_common import M0, from_dev, make_case, rel_norm, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

MQ = 0.05


def _links(kind, dims):
    U = np.zeros((4, dims[3], dims[2], dims[1], dims[0], 3, 3), dtype=np.complex128)
    if kind == "unit":
        U[..., range(3), range(3)] = 1.0
    else:
        ph = np.random.default_rng(2).uniform(-np.pi, np.pi, U.shape[:5] + (3,))
        U[..., range(3), range(3)] = np.exp(1j * ph)
    return U


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


@pytest.mark.parametrize("full", [False, True])
@pytest.mark.parametrize("links", ["unit", "diagonal"])
@pytest.mark.parametrize("ratio", [1e-2, 1e-3, 1e-6, 1e-9, 1e-13, 1e-30])
def test_colours_of_different_size(torch, ratio, links, full):
    dims, ns = (4, 2, 4, 6), 8
    U, (_, w) = _links(links, dims), make_case((2, 2, 2, 2), ns, MQ)
    psi = syn.gaussian_spinor(ns, dims, 8) if full else syn.gaussian_spinor_even(ns, dims, 8)
    psi[..., 1] *= ratio
    psi[..., 2] *= ratio ** 2 if ratio > 1e-10 else 1.0
    for got, ref in _ops(torch, dims, ns, U, w, psi, full):
        _check_colours(got, ref)


@pytest.mark.parametrize("ns", [4, 32])
@pytest.mark.parametrize("ratio", [1e-1, 1e-3, 1e-6, 1e-9])
def test_one_small_colour(torch, ratio, ns):
    dims = (4, 4, 2, 4)
    U, (_, w) = _links("diagonal", dims), make_case((2, 2, 2, 2), ns, MQ)
    psi = syn.gaussian_spinor_even(ns, dims, 13)
    psi[..., 0] *= ratio
    for got, ref in _ops(torch, dims, ns, U, w, psi, False):
        _check_colours(got, ref)


@pytest.mark.parametrize("ns", [2, 16, 32])
@pytest.mark.parametrize("ratio", [1e-3, 1e-9, 1e-13])
def test_neighbours_of_different_size(torch, ratio, ns):
    """Colour 0 lives on one site, colour 1 is `ratio` everywhere else: next to that site the sums over the
    eight neighbours hold terms of both sizes, in different colours."""
    dims = (4, 4, 2, 4)
    U, (_, w) = _links("unit", dims), make_case((2, 2, 2, 2), ns, MQ)
    psi = syn.gaussian_spinor(ns, dims, 9)
    psi[..., 2] = 0.0
    psi[..., 1] *= ratio
    one = psi[:, 1, 0, 2, 1].copy()
    psi[..., 0] = 0.0
    psi[:, 1, 0, 2, 1] = one
    psi[:, 1, 0, 2, 1, :, 1:] = 0.0
    for got, ref in _ops(torch, dims, ns, U, w, psi, True):
        _check_colours(got, ref)


@pytest.mark.parametrize("ratio", [1e-3, 1e-6, 1e-9])
def test_spins_of_different_size(torch, ratio):
    """One large spin on sites whose neighbours hold none: D sends it to the same spin of its own site and to
    spins of the neighbours, and what is left at its own site keeps its own size."""
    dims, ns = (4, 4, 4, 4), 8
    U, w = make_case(dims, ns, MQ, eps=0.6, seed=5)  # dense links
    psi = syn.gaussian_spinor(ns, dims, 10) * ratio
    lone = np.zeros(psi.shape[1:5], dtype=bool)
    lone[1, 1, 1, 1] = lone[3, 3, 3, 3] = True
    psi[:, lone, 0] /= ratio
    near = lone.copy()
    for ax in range(4):
        near |= np.roll(lone, 1, ax) | np.roll(lone, -1, ax)
    for k, (got, ref) in enumerate(_ops(torch, dims, ns, U, w, psi, True)):
        if k == 2:
            break
        far = np.abs(got - ref)[:, ~near].max(), np.abs(ref)[:, ~near].max()
        assert far[0] <= 1e-13 * far[1]
        for sp in (1, 2, 3):  # the other spins of the lone sites
            err, size = np.abs(got - ref)[:, lone, sp].max(), np.abs(ref)[:, lone, sp].max()
            assert size < 1e3 * ratio and err <= 1e-13 * size


@pytest.mark.parametrize("ns", [2, 16, 32])
@pytest.mark.parametrize("ratio", [2.0 ** -7, 1e-3, 1e-12, 1e-40])
def test_small_colours_on_dense_links(torch, ratio, ns):
    """Links that mix colours: sites keep FP64 bits, and the fixed-point stencil converts them where it reads them.
    Every other site, so that both kinds of neighbours meet."""
    dims = (4, 2, 6, 4)
    U, w = make_case(dims, ns, MQ, eps=0.7, seed=6)
    psi = syn.gaussian_spinor(ns, dims, 14)
    psi[:, :, ::2, :, :, :, 1:] *= ratio
    for got, ref in _ops(torch, dims, ns, U, w, psi, True):
        _check_colours(got, ref)


def test_noise_off_the_diagonal(torch):
    """A free field as an eigendecomposition makes it: 1e-15 off the diagonal, a colour at that level."""
    dims, ns = (4, 4, 2, 6), 16
    U, w = make_case(dims, ns, MQ, eps=0.0, seed=1)
    psi = syn.gaussian_spinor_even(ns, dims, 11)
    psi[..., 1] *= 1e-15
    for got, ref in _ops(torch, dims, ns, U, w, psi, False):
        _check_colours(got, ref)


def test_solve_of_colours_of_different_size(torch):
    """FP64 CG runs the same hops with its own epilogues; colours decouple, so the solution of the sum is the
    sum of the solutions."""
    dims, ns = (4, 4, 2, 4), 8
    U, (_, w) = _links("diagonal", dims), make_case((2, 2, 2, 2), ns, 0.5)
    b = syn.gaussian_spinor_even(ns, dims, 12)
    b[..., 1] *= 1e-9
    x_ref, _, _ = oracle.cg(U, b, M0, 0.5, w, tol=1e-13)
    with odwf.Handle(dims, ns, M0, 0.5, w) as h:
        h.set_gauge(to_dev(torch, U))
        x = torch.zeros(b.shape, dtype=torch.complex128, device="cuda")
        st = h.cg_solve(x, to_dev(torch, b), tol=1e-12, max_iter=10000, prec="f64")
    assert st["status"] == 0 and st["true_resid"] <= 1e-12
    assert rel_norm(from_dev(x), x_ref) <= 1e-9
