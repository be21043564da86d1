"""Far-field launches whose form depends on how much there is to do, against the oracle's literal pFMM:
trees of coarse levels only (their M2L is one launch) and deeper ones, M2M and L2L with fewer and more
parents than SMs and with more moments than one CTA's shared memory holds, S2M in chunks of 32 and of 192
moments, the 8^3 M2L with its folded moments whole, in chunks of right-hand sides, and in what a bounded
scratch array leaves."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2106_15911_gb300 import pfmm as P
from paper_2106_15911_gb300.inputs import cube_mesh, random_density, sample_triangles

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
BOTH = [P.PFMM_FP64, P.PFMM_MIXED]


def _compare(V, T, Et, nrhs, precision, check=None, noalloc=0, **kw):
    op = P.Operator(V, T, 1.0, Et, precision=precision, **kw)
    if check:
        check(op.info())
    Pr = O.make_problem(V, T, 1.0, Et, **kw)
    rows = sample_triangles(T.shape[0], 8, seed=3)
    w = random_density(Et, T.shape[0], nrhs, seed=70)
    wt = torch.tensor(w, device=DEV)
    many = op.V(wt, parts=P.PFMM_PART_FAR).cpu().numpy()
    # FP64: 48-bit sums of a few thousand terms; mixed: FP32 sums
    tol = 1e-12 if precision == P.PFMM_FP64 else 1e-5
    for r in (0, nrhs - 1):
        one = op.V(wt[r:r + 1].contiguous(), parts=P.PFMM_PART_FAR).cpu().numpy()[0]
        ref = O.pfmm_apply(Pr, 0, w[r], targets=rows, parts=P.PFMM_PART_FAR)[:, rows]
        den = np.max(np.abs(ref))
        assert den > 0
        assert np.max(np.abs(many[r][:, rows] - ref)) <= tol * den
        assert np.max(np.abs(one[:, rows] - ref)) <= tol * den
    if noalloc:
        full = op.V(wt[:noalloc].contiguous())
        out = torch.full_like(full, float("nan"))
        P.pfmm_apply_V_noalloc(op.h, wt[:noalloc].contiguous(), out, noalloc)
        torch.cuda.synchronize()
        assert float((out - full).abs().max() / full.abs().max()) <= tol
    op.close()


@pytest.mark.parametrize("precision", BOTH)
@pytest.mark.parametrize("n_a,Et,c_st,m_x,nrhs", [(4, 16, 1.0, 6, 1), (2, 8, 1.0, 0, 3), (4, 128, 8.0, 3, 40)])
def test_trees_of_coarse_levels(precision, n_a, Et, c_st, m_x, nrhs):
    def check(info):
        assert info["p"] >= 2 and info["lx"][info["p"]] <= 1, info
    _compare(*cube_mesh(n_a), Et, nrhs, precision, check, m_t=4, m_x=m_x, c_st=c_st)


@pytest.mark.parametrize("precision", BOTH)
@pytest.mark.parametrize("m_x,nrhs", [(1, 24), (6, 24), (12, 3)])
def test_space_time_passes_few_and_many_parents(precision, m_x, nrhs):
    def check(info):
        assert max(info["lx"]) >= 2, info
    _compare(*cube_mesh(4), 32, nrhs, precision, check, m_t=4, m_x=m_x, c_st=0.15)


@pytest.mark.parametrize("m_x,nrhs", [(2, 1), (6, 3), (6, 34)])
def test_8_cubed_m2l(m_x, nrhs):
    def check(info):
        assert P.PFMM_M2L_SLAB in info["m2l_engine"], info
    _compare(*cube_mesh(12), 32, nrhs, P.PFMM_MIXED, check, noalloc=min(nrhs, 3), m_t=4, m_x=m_x, c_st=0.1)
