"""The settings of the reliable updates' arithmetic (auto, f64, ff) are names of one operator, odwf_apply_normal:
equal bits from each, and FP64 accuracy (1e-12 of the component scale, as test_gpu_operator.py) from all.
"""
import numpy as np
import pytest

import odwf_synth as syn
import oracle
import paper_1811_08095_gb300 as odwf
from gpu_common import M0, assert_close_componentwise, from_dev, make_case, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,ns", [((6, 4, 2, 10), 8), ((2, 4, 2, 4), 32)])
def test_operator_of_the_updates(dims, ns):
    torch = torch_cuda()
    U, w = make_case(dims, ns, 0.1, eps=0.6, seed=1)
    b = syn.gaussian_spinor_even(ns, dims, 2)
    with odwf.Handle(dims, ns, M0, 0.1, w) as h:
        h.set_gauge(to_dev(torch, U))
        x = to_dev(torch, b)
        a, n = torch.empty_like(x), torch.empty_like(x)
        h.apply_normal_prec(a, x, "ff")
        h.apply_normal(n, x)
    assert np.array_equal(from_dev(a), from_dev(n))
    assert_close_componentwise(from_dev(a), oracle.normal_op(U, b, M0, 0.1, w), 1e-12)


@pytest.mark.parametrize("prec,ns", [("f16", 8), ("bf16", 16), ("f32", 4)])
def test_settings_give_the_same_solution(prec, ns):
    torch = torch_cuda()
    dims = (4, 4, 2, 6)
    U, w = make_case(dims, ns, 0.1, eps=0.3, seed=2)
    b = to_dev(torch, syn.gaussian_spinor_even(ns, dims, 3))
    out = []
    with odwf.Handle(dims, ns, M0, 0.1, w) as h:
        h.set_gauge(to_dev(torch, U))
        for updates in ("auto", "f64", "ff"):
            x = torch.zeros_like(b)
            st = h.cg_solve(x, b, tol=1e-10, prec=prec, updates=updates)
            out.append((from_dev(x), st["iters"], st["n_reliable"], st["true_resid"]))
    for o in out[1:]:
        assert np.array_equal(o[0], out[0][0]) and o[1:] == out[0][1:]
