"""The FP64 tensor-core nearfield at the edges of its tiling (128 target triangles, 64 columns, blocks
of 32, 64 or 128 leaf intervals, reductions every 2 to 18 column blocks): row and column counts that
leave remainders, one to several column blocks, interval counts on both sides of a block, one to four
steps per leaf.  The two forms of the kernel are the same but for one and two steps per leaf and more than 64
intervals, and are told apart only there."""
import numpy as np
import pytest
import torch

from paper_2106_15911_gb300 import pfmm as P
from paper_2106_15911_gb300.inputs import cube_mesh, cube_sphere_mesh, random_density

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


SAME = [                               # forms that are the same kernel
    (cube_mesh, 1, 4, 1, 2),           # 12 triangles: one row tile, one column block, 2 leaf intervals
    (cube_mesh, 3, 64, 3, 2),          # 108 rows, 32 intervals: a full block of 32
    (cube_sphere_mesh, 5, 128, 2, 2),  # 300 rows: two tiles and 44 rows, 5 column blocks, 64 intervals
    (cube_mesh, 9, 128, 1, 2),         # 972 rows, 16 column blocks (8 for K): reductions on the last block
    (cube_mesh, 2, 4, 2, 1),           # one step per leaf: 4 and 64 intervals
    (cube_sphere_mesh, 5, 64, 1, 1),
    (cube_mesh, 1, 3, 1, 3),           # three steps per leaf: one interval, 64 intervals
    (cube_sphere_mesh, 9, 192, 2, 3),
    (cube_mesh, 2, 16, 1, 4),          # four steps per leaf: 4 and 64 intervals
    (cube_sphere_mesh, 9, 256, 2, 4),
]
APART = [
    (cube_mesh, 7, 256, 1, 2),         # 588 rows, 10 column blocks, 128 intervals
    (cube_sphere_mesh, 3, 512, 2, 2),  # 108 rows, 256 intervals: two blocks of 128 or four of 64
    (cube_mesh, 9, 256, 1, 1),         # one step per leaf: 256 and 128 intervals
    (cube_mesh, 2, 128, 3, 1),
]


@pytest.mark.parametrize("form,mesh,n_a,Et,nrhs,ls", [(0,) + c for c in SAME] + [(f,) + c for f in (0, 1, 2) for c in APART])
def test_residue_nearfield_at_tile_edges(form, mesh, n_a, Et, nrhs, ls):
    V, T = mesh(n_a)
    kw = dict(m_t=2, m_x=2, c_st=1.0, quad_regular=2, quad_singular=2, leaf_steps=ls)
    op = P.Operator(V, T, 1.0, Et, nf_form=form, **kw)
    ref = P.Operator(V, T, 1.0, Et, nf_engine=P.PFMM_NF_CUDA_CORES, **kw)
    info = op.info()
    assert info["nf_tensor_cores"] == 3 and ref.info()["nf_tensor_cores"] == 0
    if ls > 2 or Et // ls <= 64:  # one kernel: nothing to time
        assert info["nf_form"] == 1 and info["nf_form_ms"] == [0, 0]
    else:
        assert info["nf_form"] in ((form,) if form else (1, 2)) and (min(info["nf_form_ms"]) > 0) == (form == 0)
    for call, n in (("V", T.shape[0]), ("K", V.shape[0])):
        x = torch.tensor(random_density(Et, n, nrhs, seed=17), device=DEV)
        a = getattr(op, call)(x, parts=P.PFMM_PART_NEAR).cpu().numpy()
        P.pfmm_check(op.h)
        b = getattr(ref, call)(x, parts=P.PFMM_PART_NEAR).cpu().numpy()
        # operands rounded to 52 bits of each row's and right-hand side's largest, exact sums
        assert np.max(np.abs(a - b)) <= 1e-13 * np.max(np.abs(b))
    op.close()
    ref.close()
