"""The CUDA-core nearfield (8 rows of a panel per CTA, 32 to 256 leaf intervals, columns two stages at a
time), from the FP16 parts of a tensor-core handle against its tensor-core product and the FP32 panels, and on panels of their own columns, against the oracle's nearfield: one to four steps per leaf, interval
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


@pytest.mark.parametrize("mesh,n_a,Et,nrhs", [
    (cube_mesh, 1, 2, 1),          # 12 rows: 8 and 4; one interval
    (cube_mesh, 2, 64, 2),         # 48 rows: six times 8
    (cube_sphere_mesh, 4, 16, 3),  # 192 rows: a tile of 128 and a half
    (cube_sphere_mesh, 5, 512, 1), # 300 rows: two tiles and 44 = 5 times 8 and 4; 256 intervals
])
def test_rows_from_the_fp16_parts(mesh, n_a, Et, nrhs):
    # the blocks of a mixed handle on the tensor cores exist as FP16 parts only
    V, T = mesh(n_a)
    kw = dict(m_t=2, m_x=2, quad_regular=2, quad_singular=2, precision=P.PFMM_MIXED)
    op, panels = P.Operator(V, T, 1.0, Et, **kw), P.Operator(V, T, 1.0, Et, nf_engine=P.PFMM_NF_CUDA_CORES, **kw)
    assert op.info()["nf_tensor_cores"] == 3
    for k, (call, n) in enumerate((("V", len(T)), ("K", len(V)))):
        x = torch.tensor(random_density(Et, n, nrhs, seed=9), device=DEV)
        P.pfmm_set_nf_engine(op.h, P.PFMM_NF_AUTO)
        tc = getattr(op, call)(x, parts=P.PFMM_PART_NEAR)
        P.pfmm_set_nf_engine(op.h, P.PFMM_NF_CUDA_CORES)
        got = getattr(op, call)(x, parts=P.PFMM_PART_NEAR)
        ref = getattr(panels, call)(x, parts=P.PFMM_PART_NEAR)
        # the parts hold a block to 2^-22, a row's sums are the same FP32 ones; the tensor cores also round the input
        # to two parts and sum in another order
        assert float((got - ref).abs().max()) <= 1e-6 * float(ref.abs().max())
        assert float((got - tc).abs().max()) <= 1e-5 * float(ref.abs().max())
        # three kernels instead of six
        assert P.pfmm_count_apply_kernels(op.h, k, x, torch.empty_like(ref), nrhs, P.PFMM_PART_NEAR) == 3
    for h in (op, panels):
        h.close()


@pytest.mark.parametrize("ls,n_a", [(1, 8), (2, 8), (3, 6), (4, 6)])
def test_sums_beyond_the_fp32_range(ls, n_a):
    # products and the sums of 128 of them are FP32 numbers, the outputs are not: FP64 sums
    V, T = cube_mesh(n_a)
    V = 100.0 * V  # entries of order one
    Et = 8 * ls
    kw = dict(m_t=2, m_x=2, c_st=1.0, leaf_steps=ls, quad_regular=2, quad_singular=2)
    op = P.Operator(V, T, 1e4, Et, precision=P.PFMM_MIXED, nf_engine=P.PFMM_NF_CUDA_CORES, **kw)
    ref = P.Operator(V, T, 1e4, Et, nf_engine=P.PFMM_NF_CUDA_CORES, **kw)
    x = torch.ones(1, Et, len(T), device=DEV, dtype=torch.float64)
    one = ref.V(x, parts=P.PFMM_PART_NEAR)
    x *= 5e38 / float(one.max())
    assert float(x.max()) < 3e38
    a, b = op.V(x, parts=P.PFMM_PART_NEAR), ref.V(x, parts=P.PFMM_PART_NEAR)
    assert float(b.max()) > 4.9e38
    assert float((a - b).abs().max()) <= 1e-5 * float(b.max())  # FP32 blocks and sums
    op.close()
    ref.close()


@pytest.mark.parametrize("ns", [1, 32, 33])  # one slice of a CTA's 32, all, and a second CTA
@pytest.mark.parametrize("kw", [dict(precision=P.PFMM_MIXED, c_st=1.0),   # FP16 parts
                                dict(precision=P.PFMM_MIXED, c_st=0.15, n_tr=1),  # FP32 panels of their own columns
                                dict(precision=P.PFMM_FP64, c_st=0.15, n_tr=1)])
def test_same_step_block_of_slices(kw, ns):
    V, T = cube_mesh(4)
    Et = 32
    kw = dict(kw, m_t=2, m_x=2)
    op = P.Operator(V, T, 1.0, Et, **kw)
    otf = P.Operator(V, T, 1.0, Et, nearfield=P.PFMM_NEARFIELD_ONTHEFLY, **dict(kw, precision=P.PFMM_FP64))
    net = P.Mpnn(V, T, 1.0, Et, width=16, layers=1, seed=1)
    net.output_scale = 1.0
    R = torch.tensor(random_density(Et, len(T), 2, seed=32), device=DEV)
    sl = (np.arange(ns) * 7 % (2 * Et)).astype(np.int32)
    l1, g1 = net.loss_grad(R, None, sl, handle=op.h)
    l2, g2 = net.loss_grad(R, None, sl, handle=otf.h)
    # the panels' FP32 rounding and FP32 sums enter the residual and its gradient
    assert l1 == pytest.approx(l2, rel=1e-5)
    assert np.max(np.abs(g1 - g2)) <= 1e-5 * np.max(np.abs(g2))
    for h in (net, op, otf):
        h.close()
