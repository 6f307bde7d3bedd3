"""The mixed iteration on either side of the kernels' size rules, with the per-stage bounds of
test_gpu_mixed_step.py: lattices of at most 16384 five-dimensional sites take the one-s-per-lane hops
that fetch every neighbour up front (the small cases there), larger ones the two-s-per-lane hops;
reductions of more than 256 blocks sum in two levels, with a ragged last group here.
"""
import pytest

from gpu_common import torch_cuda
from test_gpu_mixed_step import _step_and_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,ns,mq,tbc,prec,recon,link_prec", [
    ((4, 4, 8, 32), 8, 0.5, True, "f16", 12, "f32"),     # 16384 sites: the last size of the small kernels
    ((2, 6, 10, 18), 16, 0.5, True, "f16", 12, "f32"),   # 17280: the next, ragged blocks
    ((6, 10, 12, 14), 16, 0.5, True, "bf16", 18, "f32"),  # 80640: 315 and 158 blocks in the reducing hops
    ((6, 10, 12, 14), 8, 0.04, False, "f16", 12, "f16"),
    ((6, 10, 12, 14), 16, 0.5, True, "f32", 12, "f32"),  # FP32 storage has no small variant
])
def test_mixed_step_across_size_rules(dims, ns, mq, tbc, prec, recon, link_prec):
    _step_and_check(torch_cuda(), dims, ns, mq, tbc, prec, recon, link_prec=link_prec)
