"""The FP32 nearfield entries of the mixed mode against the FP64 ones, through products on the CUDA cores."""
import pytest
import torch

from paper_2106_15911_gb300 import pfmm as P
from paper_2106_15911_gb300.inputs import cube_mesh, random_density

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n_a,Et,alpha", [(4, 16, 0.5), (8, 64, 0.5), (8, 256, 0.5), (8, 512, 1.0), (5, 32, 1.5)])
def test_fp32_entries_carry_no_common_rounding(n_a, Et, alpha):
    V, T = cube_mesh(n_a)
    kw = dict(m_t=2, m_x=2, quad_regular=2, quad_singular=3, nf_engine=P.PFMM_NF_CUDA_CORES)
    mixed = P.Operator(V, T, 1.0, Et, alpha, precision=P.PFMM_MIXED, **kw)
    fp64 = P.Operator(V, T, 1.0, Et, alpha, **kw)
    for call, n in (("V", len(T)), ("K", len(V))):
        x = torch.tensor(random_density(Et, n, 1, seed=3), device=DEV)
        a, b = getattr(mixed, call)(x, parts=P.PFMM_PART_NEAR), getattr(fp64, call)(x, parts=P.PFMM_PART_NEAR)
        # the terms of the second differences in time are up to some 20 times the entries, a few of their 6e-8
        # roundings each: 1e-6 an entry, independent from entry to entry and so a third of it over a row
        assert float((a - b).norm() / b.norm()) <= 4.5e-7
    mixed.close()
    fp64.close()
