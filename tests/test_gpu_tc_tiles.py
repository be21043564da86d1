"""The mixed-precision tensor-core nearfield at the edges of its tiling (128 target triangles, blocks of
32 columns, of 64 or 128 leaf intervals, FP32 sums over 4 and 16 column blocks, up to 16 K chunks)
against the CUDA-core engine on the same FP32 panels."""
import numpy as np
import pytest
import torch

from paper_2106_15911_gb300 import pfmm as P
from paper_2106_15911_gb300.inputs import cube_mesh, cube_sphere_mesh, random_density

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("mesh,n_a,Et,nrhs", [
    (cube_mesh, 1, 4, 1),           # 12 triangles: one row tile, one pair of column blocks, 2 leaf intervals
    (cube_mesh, 3, 64, 3),          # 108 rows, 32 intervals: half a block
    (cube_sphere_mesh, 5, 128, 2),  # 300 rows: two tiles and 44 rows; a full narrow block
    (cube_mesh, 7, 256, 1),         # 588 rows, 128 intervals: the wide block
    (cube_sphere_mesh, 9, 512, 2),  # 972 rows, 256 intervals: two blocks
    (cube_mesh, 16, 64, 9),         # 3072 rows: 96 column blocks, several FP32 sums a chunk
])
def test_mixed_nearfield_at_tile_edges(mesh, n_a, Et, nrhs):
    V, T = mesh(n_a)
    kw = dict(m_t=2, m_x=2, c_st=1.0, quad_regular=2, quad_singular=2, precision=P.PFMM_MIXED)
    op = P.Operator(V, T, 1.0, Et, **kw)
    ref = P.Operator(V, T, 1.0, Et, nf_engine=P.PFMM_NF_CUDA_CORES, **kw)
    assert op.info()["nf_tensor_cores"] == 3 and ref.info()["nf_tensor_cores"] == 0
    for call, n in (("V", T.shape[0]), ("K", V.shape[0])):
        x = torch.tensor(random_density(Et, n, nrhs, seed=17), device=DEV)
        near = lambda o, v: getattr(o, call)(v, parts=P.PFMM_PART_NEAR).cpu().numpy()
        a = near(op, x)
        P.pfmm_check(op.h)
        assert np.array_equal(a, near(op, x))
        one = near(op, x[-1:].contiguous())[0]  # its own number of K chunks in the same workspace
        # The blocks of both layers keep one sign on a convex body: sum |A| |x| is the product with |x|.
        # 96 truncated sums of 2^-23, a few roundings of 2^-24, and 2^-22 for each part of the split and
        # the product of the low parts; the other engine's FP32 sums are shorter.  Entries far below the
        # largest have subnormal low parts: 2^-39 of the largest, of A and of x, per product
        top = np.max(np.abs(near(ref, torch.full_like(x, float(x.abs().max())))))
        tol = 1.3e-5 * np.abs(near(ref, x.abs())) + 4 * n * 2.0**-38 * top
        b = near(ref, x)
        assert np.all(np.abs(a - b) <= tol)
        assert np.all(np.abs(one - b[-1]) <= tol[-1])
    op.close()
    ref.close()
