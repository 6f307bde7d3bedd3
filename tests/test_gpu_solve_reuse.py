"""Solves on one handle share streams, pinned memory and captured iteration graphs: a later solve with
other storage, batch size, mass, gauge field or workspace sizes must not see an earlier one's, and gives
the bits of the same solve on a fresh handle."""
import pytest

import odwf_synth as syn
import paper_1811_08095_gb300 as odwf
from gpu_common import M0, from_dev, make_case, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def test_solves_in_any_order_match_fresh_handles():
    torch = torch_cuda()
    dims, ns = (4, 4, 4, 6), 8
    fields = [make_case(dims, ns, 0.1, eps=0.3, seed=s)[0] for s in (1, 2)]
    w = make_case(dims, ns, 0.1)[1]
    bs = [syn.gaussian_spinor_even(ns, dims, 30 + k) for k in range(3)]
    runs = [  # gauge field, storage, links, masses
        (0, "f16", "f32", [0.1]), (0, "f16", "f32", [0.3]), (1, "f16", "f32", [0.1]), (1, "bf16", "f32", [0.1]),
        (0, "f16", "f16", [0.1]), (0, "f64", "f32", [0.1]), (0, "f16", "f32", [0.1, 0.2, 0.5]), (0, "f32", "f32", [0.2]),
        (0, "f16", "f32", [0.1]), (1, "f64", "f32", [0.4]), (0, "f16", "f32", [0.5, 0.1]),
    ]

    def solve(h, run):
        u, prec, links, ms = run
        h.set_gauge(to_dev(torch, fields[u]))
        b = [to_dev(torch, f) for f in bs[:len(ms)]]
        x = [torch.empty_like(t) for t in b]
        st = h.cg_solve_batched(x, b, ms, tol=1e-10, prec=prec, link_prec=links, check_every=4)
        assert all(s["status"] == 0 for s in st)
        return [from_dev(t) for t in x], [s["iters"] for s in st]

    with odwf.Handle(dims, ns, M0, 0.1, w) as shared:
        for run in runs:
            with odwf.Handle(dims, ns, M0, 0.1, w) as fresh:
                xa, ia = solve(fresh, run)
            xb, ib = solve(shared, run)
            assert ia == ib
            for a, b in zip(xa, xb):
                assert (a == b).all(), run
