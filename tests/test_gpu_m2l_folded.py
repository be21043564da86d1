"""The folded M2L of the levels with 4^3 cells (every direction split into its even and odd part)
against the oracle's literal pFMM: all degrees that take it, a truncated and a full interaction
area, the split launch (few right-hand sides) and the whole one (many)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2106_15911_gb300 import pfmm as P
from paper_2106_15911_gb300.inputs import cube_mesh, cube_sphere_mesh, random_density, sample_triangles

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("precision,m_x", [(P.PFMM_FP64, m) for m in (0, 1, 2, 3, 5, 6)] +
                         [(P.PFMM_MIXED, m) for m in (0, 1, 2, 4, 6, 7, 8)])
@pytest.mark.parametrize("mesh,n_tr", [(cube_mesh, -1), (cube_sphere_mesh, 1)])
def test_folded_m2l_matches_oracle(precision, m_x, mesh, n_tr):
    V, T = mesh(4)
    Et, nrhs = 32, 16  # 16 leaf intervals x 5 nodes x 16 rhs: past the eight CTAs per SM of the split launch
    kw = dict(m_t=4, m_x=m_x, c_st=0.15, n_tr=n_tr)
    op = P.Operator(V, T, 1.0, Et, precision=precision, **kw)
    info = op.info()
    lv4 = [l for l in range(2, info["p"] + 1) if info["lx"][l] == 2]
    engine = P.PFMM_M2L_FUSED_SLICED if m_x == 8 else P.PFMM_M2L_FUSED
    assert lv4 and all(info["m2l_engine"][l] == engine for l in lv4), info
    w = random_density(Et, T.shape[0], nrhs, seed=70 + m_x)
    wt = torch.tensor(w, device=DEV)
    many = op.V(wt, parts=P.PFMM_PART_FAR).cpu().numpy()
    Pr = O.make_problem(V, T, 1.0, Et, **kw)
    rows = sample_triangles(T.shape[0], 12, seed=3)
    # FP64: 48-bit sums of a few thousand terms; mixed: FP32 sums
    tol = 1e-12 if precision == P.PFMM_FP64 else 1e-5
    for r in (0, nrhs - 1):
        one = op.V(wt[r:r + 1].contiguous(), parts=P.PFMM_PART_FAR).cpu().numpy()[0]
        ref = O.pfmm_apply(Pr, 0, w[r], targets=rows, parts=P.PFMM_PART_FAR)[:, rows]
        den = np.max(np.abs(ref))
        assert den > 0
        assert np.max(np.abs(many[r][:, rows] - ref)) <= tol * den
        assert np.max(np.abs(one[:, rows] - ref)) <= tol * den
    op.close()
