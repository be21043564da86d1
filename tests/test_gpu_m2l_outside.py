"""M2L on levels whose interaction radius leaves cells out (Eq. 03:Iarea): a density in one box reaches the boxes
within the radius and leaves the others at zero, and one that is not finite spoils those within the radius only."""
import numpy as np
import pytest
import torch

from paper_2106_15911_gb300 import pfmm as P
from paper_2106_15911_gb300.inputs import cube_mesh, random_density

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _cells(V, T, G):
    lo, hi = V.min(0), V.max(0)
    H = 0.5 * (hi - lo).max()
    cen = ((V[T[:, 0]] + V[T[:, 1]]) + V[T[:, 2]]) / 3.0
    return np.clip(np.ceil((cen - (0.5 * (lo + hi) - H)) / (2 * H / G)).astype(int) - 1, 0, G - 1)


@pytest.mark.parametrize("precision,n_a,c_st,m_x", [
    (P.PFMM_FP64, 4, 0.15, 4), (P.PFMM_MIXED, 4, 0.15, 4), (P.PFMM_MIXED, 4, 0.15, 8),  # 4^3, sliced too
    (P.PFMM_FP64, 12, 0.1, 2), (P.PFMM_MIXED, 12, 0.1, 2)])                             # 8^3
@pytest.mark.parametrize("n_tr,nrhs", [(1, 1), (2, 24)])
def test_the_interaction_radius_bounds_what_a_density_reaches(precision, n_a, c_st, m_x, n_tr, nrhs):
    V, T = cube_mesh(n_a)
    Et, ls = 32, 2
    op = P.Operator(V, T, 1.0, Et, precision=precision, m_t=3, m_x=m_x, c_st=c_st, n_tr=n_tr, quad_regular=2,
                    quad_singular=2, leaf_steps=ls)
    info = op.info()
    G = 2 ** info["lx"][info["p"]]
    assert G == (4 if n_a == 4 else 8)
    cell = _cells(V, T, G)
    src = int(np.argmin(cell.sum(1)))
    box = (cell == cell[src]).all(1)
    inside = np.abs(cell - cell[src]).max(1) <= n_tr
    J = 8  # only the leaf level reaches the intervals J + 2 and J + 3
    steps = slice((J + 2) * ls, (J + 4) * ls)
    x = np.zeros((nrhs, Et, len(T)))
    x[:, J * ls:(J + 1) * ls, box] = random_density(ls, int(box.sum()), nrhs, seed=41)
    f = op.V(torch.tensor(x, device=DEV), parts=P.PFMM_PART_FAR).cpu().numpy()[:, steps]
    assert (f[:, :, inside] != 0).all() and (f[:, :, ~inside] == 0).all()
    # all boxes; then one entry of the same that is not finite
    x[:, J * ls:(J + 1) * ls] = random_density(ls, len(T), nrhs, seed=43)
    x[:, :, box] = 0.0
    f = op.V(torch.tensor(x, device=DEV), parts=P.PFMM_PART_FAR).cpu().numpy()[:, steps]
    x[0, J * ls, src] = np.nan
    x[nrhs - 1, J * ls + 1, src] = np.inf
    g = op.V(torch.tensor(x, device=DEV), parts=P.PFMM_PART_FAR).cpu().numpy()[:, steps]
    tol = 1e-12 if precision == P.PFMM_FP64 else 1e-5  # 48-bit and FP32 sums
    for r in range(nrhs):
        if r in (0, nrhs - 1):
            assert np.isnan(g[r][:, inside]).all()
            assert np.max(np.abs(g[r] - f[r])[:, ~inside]) <= tol * np.max(np.abs(f[r]))
        else:
            assert np.max(np.abs(g[r] - f[r])) <= tol * np.max(np.abs(f[r]))
    op.close()
