"""The CUDA-core nearfield (8 rows of a panel per CTA, 32 to 256 leaf intervals, columns two stages at a
time) on panels of their own columns, against the oracle's nearfield: one to four steps per leaf, interval
counts of one, below and past a CTA's, panels of fewer than 8 rows and of several groups."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2106_15911_gb300 import pfmm as P
from paper_2106_15911_gb300.inputs import cube_mesh, cube_sphere_mesh, random_density, sample_triangles

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("precision", [P.PFMM_FP64, P.PFMM_MIXED])
@pytest.mark.parametrize("mesh,n_a,ls,nint,nrhs,c_st", [
    (cube_mesh, 4, 1, 64, 2, 0.15),         # half a CTA's intervals
    (cube_mesh, 4, 2, 32, 1, 0.15),         # one warp, half of it
    (cube_sphere_mesh, 5, 3, 16, 2, 0.15),  # one interval per thread
    (cube_mesh, 6, 4, 8, 1, 0.15),
    (cube_mesh, 3, 1, 1, 1, 1.0),           # one interval
    (cube_mesh, 2, 1, 512, 1, 1.0),         # two CTAs of 256 intervals
])
def test_nearfield_rows_match_oracle(precision, mesh, n_a, ls, nint, nrhs, c_st):
    V, T = mesh(n_a)
    Et = ls * nint
    kw = dict(m_t=2, m_x=2, c_st=c_st, n_tr=1 if c_st < 1 else -1, leaf_steps=ls)
    op = P.Operator(V, T, 1.0, Et, precision=precision, nf_engine=P.PFMM_NF_CUDA_CORES, **kw)
    Pr = O.make_problem(V, T, 1.0, Et, **kw)
    rows = sample_triangles(T.shape[0], 12, seed=3)
    tol = 1e-12 if precision == P.PFMM_FP64 else 1e-5
    for k, (call, n) in enumerate((("V", T.shape[0]), ("K", V.shape[0]))):
        w = random_density(Et, n, nrhs, seed=5)
        out = getattr(op, call)(torch.tensor(w, device=DEV), parts=P.PFMM_PART_NEAR).cpu().numpy()
        for r in range(nrhs):
            ref = O.pfmm_apply(Pr, k, w[r], targets=rows, parts=P.PFMM_PART_NEAR)[:, rows]
            assert np.max(np.abs(out[r][:, rows] - ref)) <= tol * np.max(np.abs(ref))
    op.close()
