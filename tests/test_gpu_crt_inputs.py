"""The FP64 tensor-core nearfield on inputs that its fixed point could lose, against the CUDA-core FP64
engine: entries that are not finite (they reach the outputs whose products read them, and no others),
densities that grow or decay over the steps by far more than FP64's 53 bits, and magnitudes near both ends
of FP64's range."""
import numpy as np
import pytest
import torch

from paper_2106_15911_gb300 import pfmm as P
from paper_2106_15911_gb300.inputs import cube_mesh, random_density

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
LS = [1, 2, 3, 4]


def _pair(ls, nint):
    V, T = cube_mesh(4)
    Et = ls * nint
    kw = dict(m_t=2, m_x=2, c_st=1.0, quad_regular=2, quad_singular=2, leaf_steps=ls)
    op = P.Operator(V, T, 1.0, Et, **kw)
    ref = P.Operator(V, T, 1.0, Et, nf_engine=P.PFMM_NF_CUDA_CORES, **kw)
    assert op.info()["nf_tensor_cores"] == 3 and ref.info()["nf_tensor_cores"] == 0
    return V, T, Et, op, ref


def _near(op, call, x):
    return getattr(op, call)(x, parts=P.PFMM_PART_NEAR).cpu().numpy()


@pytest.mark.parametrize("ls", LS)
def test_entries_that_are_not_finite(ls):
    V, T, Et, op, ref = _pair(ls, 8)
    for call, n in (("V", len(T)), ("K", len(V))):
        for bad in ({(0, ls, 3): np.nan}, {(0, Et - 1, n - 1): np.inf, (1, 0, 0): -np.inf},
                    {(1, 4 * ls, 5): np.inf, (1, 4 * ls, 6): -np.inf, (2, 0, 1): 1e300}):
            w = random_density(Et, n, 3, seed=23)
            for at, v in bad.items():
                w[at] = v
            x = torch.tensor(w, device=DEV)
            a, b = _near(op, call, x), _near(ref, call, x)
            assert not np.isfinite(b).all() and np.isfinite(b).any()
            np.testing.assert_array_equal(np.isnan(a), np.isnan(b))
            np.testing.assert_array_equal(a[np.isinf(b)], b[np.isinf(b)])
            # 52 bits of the largest finite input that a step's outputs read
            for r in range(3):
                for t in range(Et):
                    ok = np.isfinite(b[r, t])
                    if ok.any():
                        assert np.max(np.abs(a[r, t] - b[r, t])[ok]) <= 1e-13 * np.max(np.abs(b[r, t])[ok])
    op.close()
    ref.close()


@pytest.mark.parametrize("ls", LS)
@pytest.mark.parametrize("first,rate", [(0, 6), (0, -6), (-992, 6), (990, -6)])
def test_inputs_of_wide_range_over_the_steps(ls, first, rate):
    # leaf interval i is scaled by 2^(first + rate i), 186 binary orders over the 32 intervals
    V, T, Et, op, ref = _pair(ls, 32)
    for call, n in (("V", len(T)), ("K", len(V))):
        w = random_density(Et, n, 2, seed=29) * np.ldexp(1.0, first + rate * (np.arange(Et) // ls))[None, :, None]
        x = torch.tensor(w, device=DEV)
        a, b = _near(op, call, x), _near(ref, call, x)
        # 52 bits of the larger of two neighbouring intervals, 2^6 apart, on the scale of each step's outputs
        err, size = np.max(np.abs(a - b), axis=2), np.max(np.abs(b), axis=2)
        assert np.isfinite(b).all() and (size > 0).all()
        assert (err <= 2 ** 6 * 1e-13 * size).all(), (err / size).max()
    op.close()
    ref.close()


@pytest.mark.parametrize("ls,nint", [(1, 256), (2, 256), (3, 64), (4, 64)])
@pytest.mark.parametrize("steps", [(0.25, -30), (0.25, 30), (0.5, -30), (0.75, 30)])
def test_one_jump_among_several_tiles_of_intervals(ls, nint, steps):
    # intervals from the fraction on are 2^30 smaller or larger: the jump within a tile or between two
    V, T, Et, op, ref = _pair(ls, nint)
    first, e = int(steps[0] * nint), steps[1]
    for call, n in (("V", len(T)), ("K", len(V))):
        w = random_density(Et, n, 2, seed=31) * np.where(np.arange(Et) // ls < first, 1.0, 2.0 ** e)[None, :, None]
        x = torch.tensor(w, device=DEV)
        a, b = _near(op, call, x), _near(ref, call, x)
        err, size = np.max(np.abs(a - b), axis=2), np.max(np.abs(b), axis=2)
        # 50 bits of the larger interval; right after a fall the outputs still hold the larger one's products
        t = np.arange(Et) // ls
        tol = np.where((t == first) & (e < 0), 1e-10, 1e-12)
        assert (err <= tol[None] * size).all(), (err / size).max()
    op.close()
    ref.close()


def test_more_right_hand_sides_than_the_residues_hold():
    V, T = cube_mesh(2)
    Et, nrhs = 512, 2600  # 2 MiB of input residues each, 4 GiB at a time
    op = P.Operator(V, T, 1.0, Et, m_t=2, m_x=2, c_st=1.0, quad_regular=2, quad_singular=2)
    assert op.info()["nf_tensor_cores"] == 3
    x = torch.tensor(random_density(Et, len(T), 7, seed=37), device=DEV)[torch.arange(nrhs, device=DEV) % 7].contiguous()
    f = op.V(x, parts=P.PFMM_PART_NEAR)
    g = op.V(x[:7].contiguous(), parts=P.PFMM_PART_NEAR)
    assert all(torch.equal(f[r], g[r % 7]) for r in range(nrhs))
    op.close()
