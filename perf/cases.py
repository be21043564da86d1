"""The work that users of this framework have it do, as cases that can be timed and checked.

A case is a dict of plain values: its "kind" names the entry point, the rest the mesh, the steps and
the options.  Sizes follow the repository's own configurations (cube and cube-sphere meshes of 192 to
12288 triangles, 16 to 1024 steps, one to eight right-hand sides, FP64 and mixed precision, spatial
degrees up to 10).  The quadrature orders of large meshes are kept low: they decide how long the
assembly takes and not what a product costs.

`exact` is a second implementation in plain torch FP64: the nearfield by direct quadrature, the FMM on
dense coefficient cubes of every grid cell, one total source degree at a time.
"""
import itertools
import math

import numpy as np
import torch

from paper_2106_15911_gb300 import pfmm as P
from paper_2106_15911_gb300.inputs import cube_mesh, cube_sphere_mesh, heat_source_datum, shell_sources

DEV = "cuda:0"
F8 = torch.float64
BASE = dict(shape="cube", split="diag", alpha=1.0, T=1.0, m_t=4, m_x=6, c_st=1.0, leaf_steps=2, leaf_tris=16,
            n_tr=-1, precision="fp64", quad_regular=2, quad_singular=3, nrhs=1)


def listed():
    c = []
    # the smallest problem a user starts with: a handful of blocks per kernel, launches and latency
    c.append(dict(BASE, name="v_fp64_192x16", kind="V", n_a=4, steps=16))
    # the single large problem of the headline benchmark, the product of every GMRES iteration
    c.append(dict(BASE, name="v_fp64_12288x256", kind="V", n_a=32, steps=256, quad_regular=1, quad_singular=2))
    # the same mesh in mixed precision with four data sets at once
    c.append(dict(BASE, name="v_mixed_12288x256_r4", kind="V", n_a=32, steps=256, precision="mixed", nrhs=4,
                  quad_regular=1, quad_singular=2))
    # a coarse mesh at the degree the autotuner picks for tighter targets, eight data sets
    c.append(dict(BASE, name="v_mixed_768x256_deg8_r8", kind="V", n_a=8, steps=256, precision="mixed", m_x=8,
                  nrhs=8))
    # a long time interval: 8^3 leaf grids, truncated nearfield
    c.append(dict(BASE, name="v_mixed_1728x1024", kind="V", n_a=12, steps=1024, precision="mixed"))
    # the double layer, which every direct formulation applies to its Dirichlet datum
    c.append(dict(BASE, name="k_fp64_3072x128", kind="K", n_a=16, steps=128, quad_regular=1, quad_singular=2))
    # odd sizes throughout: 1176 triangles, 96 steps in leaves of 3, other degrees and heat capacity
    c.append(dict(BASE, name="v_fp64_sphere_1176x96_r2", kind="V", shape="sphere", split="cross", n_a=7, steps=96,
                  leaf_steps=3, m_t=3, m_x=5, alpha=0.7, nrhs=2))
    # the whole solve of the direct formulation: mixed FGMRES refined in FP64 to 1e-8
    c.append(dict(BASE, name="solve_768x64", kind="solve", n_a=8, steps=64))
    # one training step of the learned preconditioner: loss and gradient in the same-step form
    c.append(dict(BASE, name="net_grad_3072x128_s32", kind="net", n_a=16, steps=128, precision="mixed", width=64,
                  layers=4, slices=32, quad_regular=1, quad_singular=2))
    # independent problems through one call
    c.append(dict(BASE, name="batch_6", kind="batch", count=6, largest=16, precision="mixed", which=3))
    # graded steps, fine near t = 0 where the kernel is steepest
    c.append(dict(BASE, name="general_768x32", kind="general", n_a=8, steps=32, grading=1.5, n_max=200,
                  quad_regular=1, quad_singular=2))
    # a new mesh: set-up with the default quadrature and the first product
    c.append(dict(BASE, name="build_fp64_768x64", kind="build", n_a=8, steps=64, quad_regular=3, quad_singular=6))
    return c


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ones' ranges: sizes spread over their logarithm, odd ones among them."""
    most = {}
    for c in listed():
        w = work(c)
        for k in w:
            most[k] = max(most.get(k, 0.0), w[k])
    while True:
        kind = rng.choice(["V", "V", "V", "V", "K", "K", "solve", "net", "batch", "general", "build"])
        c = dict(BASE, kind=kind, shape=rng.choice(["cube", "sphere"]), split=rng.choice(["diag", "diag", "cross"]),
                 alpha=round(rng.uniform(0.5, 1.5), 3))
        if kind in ("V", "K"):
            ls = rng.choice([2, 2, 2, 1, 3, 4])
            c.update(n_a=_log_int(rng, 3, 28), leaf_steps=ls, steps=ls * 2 ** rng.randint(3, 8),
                     precision=rng.choice(["fp64", "mixed"]), m_x=rng.choice([4, 5, 6, 6, 6, 7, 8, 10]),
                     m_t=rng.choice([3, 4, 4, 4]), nrhs=rng.choice([1, 1, 1, 2, 3, 5, 8]),
                     n_tr=rng.choice([-1, -1, -1, 2]))
            if c["split"] == "cross":
                c["n_a"] = min(c["n_a"], 18)
            if c["n_a"] > 10:
                c.update(quad_regular=1, quad_singular=2)
            nt = _n_tri(c)
            # products of the listed largest size: elements of the nearfield, and moments of the far field
            if nt * c["steps"] * c["nrhs"] > 4 * 12288 * 256 or c["nrhs"] * c["steps"] * math.comb(c["m_x"] + 5, 5) > \
                    4 * 256 * math.comb(13, 5) // (4 if c["precision"] == "fp64" else 1):
                continue
            # FP64 blocks that only the FP64 pipe applies: no more time than the listed long interval takes
            if c["precision"] == "fp64" and (c["leaf_steps"] != 2 or c["n_tr"] >= 0) and work(c)["flops"] > 1e10:
                continue
        elif kind == "solve":
            c.update(n_a=_log_int(rng, 2, 8), split="diag", shape="cube", alpha=1.0, steps=2 ** rng.randint(4, 6))
        elif kind == "net":
            c.update(n_a=_log_int(rng, 3, 16), split="diag", steps=2 ** rng.randint(4, 7), precision="mixed",
                     width=rng.choice([16, 32, 64]), layers=rng.randint(1, 4), slices=rng.randint(3, 32),
                     quad_regular=1, quad_singular=2)
        elif kind == "batch":
            c.update(count=rng.randint(2, 6), largest=_log_int(rng, 6, 16), precision=rng.choice(["mixed", "fp64"]),
                     which=rng.randrange(1000))
            if c["precision"] == "fp64":
                c["largest"] = min(c["largest"], 10)
        elif kind == "general":
            c.update(n_a=_log_int(rng, 3, 8), split="diag", steps=rng.randint(9, 32), n_max=rng.choice([60, 100, 200]),
                     grading=round(rng.uniform(1.0, 2.0), 2), quad_regular=1, quad_singular=2, m_x=rng.choice([4, 5, 6]))
        else:
            c.update(n_a=_log_int(rng, 2, 8), split="diag", steps=2 ** rng.randint(4, 6), quad_regular=3,
                     quad_singular=rng.choice([4, 5, 6]), precision=rng.choice(["fp64", "mixed"]))
        w = work(c)
        if all(w[k] <= most[k] for k in w):
            return c


# ---- meshes, trees and counts ----------------------------------------------------------------
def _n_tri(c):
    return (12 if c["split"] == "diag" else 24) * c["n_a"] ** 2


def _mesh(c):
    return (cube_mesh if c["shape"] == "cube" else cube_sphere_mesh)(c["n_a"], c["split"])


def _params(c, **more):
    p = dict(m_t=c["m_t"], m_x=c["m_x"], c_st=c["c_st"], n_tr=c["n_tr"], leaf_steps=c["leaf_steps"],
             leaf_tris=c["leaf_tris"], precision=P.PFMM_FP64 if c["precision"] == "fp64" else P.PFMM_MIXED,
             quad_regular=c["quad_regular"], quad_singular=c["quad_singular"])
    return dict(p, **more)


def _problems(c):
    """The problems of a batch case, as cases of kind V."""
    r = np.random.default_rng(c["which"])
    out = []
    for _ in range(c["count"]):
        n_a = int(round(math.exp(r.uniform(math.log(4), math.log(c["largest"])))))
        out.append(dict(c, kind="V", shape=str(r.choice(["cube", "sphere"])), split="diag", n_a=n_a,
                        steps=int(2 ** r.integers(5, 9 if c["precision"] == "mixed" else 8)),
                        nrhs=int(r.integers(1, 5)), m_x=int(r.choice([6, 6, 8])) if c["precision"] == "mixed" else 6,
                        quad_regular=1, quad_singular=2))
    return out


class _Tree:
    """Box cluster tree of Alg. 1 on uniform steps: per level the spatial grid, sizes and padding."""

    def __init__(self, c, V, T):
        al, Tend, Et, ls = c["alpha"], c["T"], c["steps"], c["leaf_steps"]
        lo, hi = V.min(0), V.max(0)
        self.H = H = 0.5 * float((hi - lo).max())
        corner = 0.5 * (lo + hi) - H
        cen = ((V[T[:, 0]] + V[T[:, 1]]) + V[T[:, 2]]) / 3.0
        self.p = p = int(round(math.log2(Et // ls)))
        lx = 0
        while (H / 2 ** lx) ** 2 > c["c_st"] * 4 * al * (Tend / 2):
            lx += 1
        self.lv = []
        for l in range(p + 1):
            ht = Tend / 2 ** (l + 1)
            if l and not (hx * hx <= c["c_st"] * 4 * al * ht or count <= c["leaf_tris"]):
                lx += 1
            G, hx = 2 ** lx, H / 2 ** lx
            w = 2 * H / G
            cell = np.clip(np.ceil((cen - corner) / w).astype(int) - 1, 0, G - 1)
            lin = (cell[:, 0] * G + cell[:, 1]) * G + cell[:, 2]
            count = int(np.bincount(lin).max())
            low = (corner + cell * w)[:, None, :]
            pad = max(0.0, float(np.maximum(low - V[T], V[T] - (low + w)).max()))
            self.lv.append(dict(G=G, hx=hx, ht=ht, nint=2 ** l, lin=lin, pad=pad, corner=corner))
        for l in range(p - 1, -1, -1):
            self.lv[l]["pad"] = max(self.lv[l]["pad"], self.lv[l + 1]["pad"])
        for L in self.lv:
            L["hxp"] = L["hx"] + L["pad"]
            L["ntr"] = self._radius(c, L, 8 * L["ht"])
        self.ntr_near = self._radius(c, self.lv[p], 2 * ls * Tend / Et)

    @staticmethod
    def _radius(c, L, dmax):
        if c["n_tr"] >= 0:
            return c["n_tr"]
        for n in range(1, L["G"]):
            s = max(0.0, 2 * n * L["hx"] - 2 * L["pad"])
            if math.exp(-s * s / (4 * c["alpha"] * dmax)) <= 1e-12:
                return n
        return max(L["G"] - 1, 0)


def work(case):
    """Bytes: input, output and the stored blocks once, in the precision's own format.  Flops: the nearfield
    product and the separable sums of M2L, S2M and L2T."""
    c = case
    if c["kind"] == "batch":
        ws = [work(q) for q in _problems(c)]
        return {k: float(sum(w[k] for w in ws)) for k in ws[0]}
    nt, Et, nrhs = _n_tri(c), c["steps"], c["nrhs"]
    es = 8 if c["precision"] == "fp64" else 4
    if c["kind"] == "net":
        rows, W = nt * c["slices"], c["width"]
        return {"bytes": float(nt * nt * es + 3 * rows * 8), "flops": 6.0 * rows * c["layers"] * 2 * W * W + 4.0 * nt * rows}
    if c["kind"] == "general":
        n = nt * Et
        return {"bytes": 16.0 * n + 8.0 * nt * nt * Et * 3, "flops": 2.0 * nt * nt * Et * 3}
    V, T = _mesh(c)
    tree = _Tree(c, V, T)
    ls, m, na = c["leaf_steps"], c["m_x"], c["m_t"] + 1
    lp = tree.lv[tree.p]
    G = lp["G"]
    cnt = np.bincount(lp["lin"], minlength=G ** 3).reshape(G, G, G).astype(float)
    near = cnt.copy()
    for ax in range(3):
        k = min(tree.ntr_near, G - 1)
        near = sum(np.take(np.pad(near, [(k, k) if i == ax else (0, 0) for i in range(3)]),
                           np.arange(s, s + G), axis=ax) for s in range(2 * k + 1))
    pairs = float((cnt * near).sum())
    cols = V.shape[0] / nt if c["kind"] == "K" else 1.0
    nk, ne, n5 = math.comb(m + 3, 3), math.comb(m + 4, 4), math.comb(m + 5, 5)
    flops = 2.0 * pairs * cols * Et * (3 * ls + 1) / 2 + 8.0 * nt * Et * nk * (3 if c["kind"] == "K" else 1)
    for L in tree.lv[2:]:
        q = sum(0 if k < 2 else 1 + k % 2 for k in range(L["nint"]))
        flops += 2.0 * q * na * na * min(L["G"], 2 * L["ntr"] + 1) * L["G"] ** 3 * (2 * ne + n5)
    b = pairs * cols * 2 * ls * es + nrhs * 8.0 * Et * (nt + nt * cols)
    if c["kind"] == "solve":  # about 80 products at this size; g in, x out
        return {"bytes": 80.0 * b, "flops": 80.0 * flops}
    if c["kind"] == "build":  # the values of the regular pairs, about 60 operations per point pair and offset
        npt = c["quad_regular"] ** 4
        return {"bytes": pairs * 2 * ls * es * (1 + V.shape[0] / nt) + b, "flops": 60.0 * 2 * pairs * npt * 2 * ls + flops}
    return {"bytes": b, "flops": nrhs * flops}


def tolerance(case):
    """About four times the distance from `exact` measured over the listed and some drawn cases: FP64 up to
    1e-14, mixed up to 6e-6 (FP32 far field, degree 8), the network's gradient up to 6e-7, solutions 3e-8."""
    c = case
    if c["kind"] == "solve":  # the residual is below 1e-8; the condition number scales what that leaves
        return {"rel": 5e-7, "max": 1e-5}
    if c["kind"] == "net":  # BF16 weights in both, FP32 sums
        return {"rel": 5e-6, "max": 2e-4}
    if c["precision"] == "fp64":
        return {"rel": 5e-14, "max": 2e-12}
    return {"rel": 2.5e-5, "max": 1e-3}


# ---- the calls -------------------------------------------------------------------------------
def _gen(seed, *shape):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return torch.randn(*shape, generator=g, device=DEV, dtype=F8)


def _graded(c):
    return c["T"] * (np.arange(c["steps"] + 1) / c["steps"]) ** c["grading"]


def _datum(c, V, seed):
    src = shell_sources(1, center=tuple(0.5 * (V.min(0) + V.max(0))), seed=seed)
    return torch.tensor(heat_source_datum(V, c["T"], c["steps"], src, c["alpha"])[None], device=DEV, dtype=F8)


def _net_inputs(c, seed):
    n = c["width"]
    num = 6 * n + c["layers"] * 2 * n * n + n
    g = np.random.default_rng(seed)
    # weights as a trained network holds them: representable in BF16, layers close to the identity's size
    w = torch.tensor((g.standard_normal(num) * 0.5 / math.sqrt(n)).astype(np.float32)).bfloat16().float().numpy()
    nvec = 2
    R = _gen(seed, nvec, c["steps"], _n_tri(c))
    sl = np.sort(g.choice(nvec * c["steps"], size=c["slices"], replace=False)).astype(np.int32)
    return w, R, sl


def prepare(case, seed):
    c = case
    k = c["kind"]
    if k == "batch":
        qs = _problems(c)
        probs, ws = [], []
        for i, q in enumerate(qs):
            V, T = _mesh(q)
            prm = P.pfmm_default_params()
            for key, v in _params(q).items():
                setattr(prm, key, v)
            probs.append((V, T, q["T"], q["steps"], q["alpha"], prm))
            ws.append(_gen(seed * 100 + i, q["nrhs"], q["steps"], _n_tri(q)))
        return dict(kind=k, batch=P.Batch(probs), ws=ws, fs=[torch.empty_like(w) for w in ws])
    V, T = _mesh(c)
    nt = T.shape[0]
    s = dict(kind=k)
    if k == "general":
        s["op"] = P.GeneralOperator(V, T, _graded(c), c["n_max"], c["alpha"], m_t=c["m_t"], m_x=c["m_x"],
                                    c_st=c["c_st"], quad_regular=c["quad_regular"], quad_singular=c["quad_singular"])
        s["x"] = _gen(seed, c["nrhs"], c["steps"], nt)
        return s
    if k == "build":
        s.update(V=V, T=T, c=c, x=_gen(seed, c["nrhs"], c["steps"], nt))
        return s
    s["op"] = P.Operator(V, T, c["T"], c["steps"], c["alpha"], **_params(c, **(dict(precision=P.PFMM_MIXED) if k == "solve" else {})))
    if k == "solve":
        s["fine"] = P.Operator(V, T, c["T"], c["steps"], c["alpha"], **_params(c))
        s["g"] = _datum(c, V, seed)
        s["x"] = torch.empty(1, c["steps"], nt, device=DEV, dtype=F8)
        s["opts"] = P.pfmm_default_solve_opts()
        s["opts"].refine = s["fine"].h
    elif k == "net":
        w, s["R"], s["sl"] = _net_inputs(c, seed)
        s["net"] = P.Mpnn(V, T, c["T"], c["steps"], c["alpha"], width=c["width"], layers=c["layers"])
        s["net"].set_params(w)
        s["net"].output_scale = 40.0
    else:
        s["x"] = _gen(seed, c["nrhs"], c["steps"], nt if k == "V" else V.shape[0])
    return s


def run(s):
    k = s["kind"]
    if k == "V" or k == "general":
        return s["op"].V(s["x"])
    if k == "K":
        return s["op"].K(s["x"])
    if k == "solve":
        P.pfmm_solve(s["op"].h, P.PFMM_DIRECT, s["g"], s["x"], 1, s["opts"])
        return s["x"]
    if k == "net":
        loss, grad = s["net"].loss_grad(s["R"], None, s["sl"], handle=s["op"].h)
        return {"loss": loss, "grad": grad}
    if k == "batch":
        s["batch"].apply_V(s["ws"], s["fs"])
        return s["fs"]
    c = s["c"]
    op = P.Operator(s["V"], s["T"], c["T"], c["steps"], c["alpha"], **_params(c))
    f = op.V(s["x"])
    op.close()
    return f


# ---- the same results in plain torch FP64 ----------------------------------------------------
def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), device=DEV)


def _gauss01(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (x + 1.0), 0.5 * w


def _triangle_rule(n):
    """Collapsed Gauss points (s1, s2, weight) on 0 <= s2 <= s1 <= 1."""
    x, w = _gauss01(n)
    return [(u, u * v, wu * wv * u) for u, wu in zip(x, w) for v, wv in zip(x, w)]


def _erfs(u):
    ef, efc = torch.erf(u), torch.special.erfc(u)
    return ef, efc, torch.exp(-u * u)


def _G2(r, s, al):
    """Second time antiderivative of the heat kernel and its bounded form (less the part linear in s)."""
    if s <= 0:
        z = torch.zeros_like(r)
        return z, z
    ss, a32 = math.sqrt(s), al * math.sqrt(al)
    u = r / (2 * math.sqrt(al) * ss)
    ef, efc, ex = _erfs(u)
    u2 = u * u
    small = 2 / math.sqrt(math.pi) * (1 + u2 * (-1 / 3 + u2 * (1 / 10 + u2 * (-1 / 42 + u2 / 216))))
    eou = torch.where(u < 0.05, small, ef / u.clamp_min(1e-300))
    gt = r * efc / (8 * math.pi * al * al) - ss * eou / (8 * math.pi * a32) - ss * ex / (4 * math.pi ** 1.5 * a32)
    g = ((s + r * r / (2 * al)) * efc - r * ss / math.sqrt(math.pi * al) * ex) / (4 * math.pi * al * r.clamp_min(1e-300))
    return torch.where(r > 0, g, torch.zeros_like(g)), gt


def _D2(r, s, al):
    """The double layer's factor of (x - y).n and its bounded form."""
    if s <= 0:
        z = torch.zeros_like(r)
        return z, z
    u = r / (2 * math.sqrt(al * s))
    ef, efc, ex = _erfs(u)
    g = ((s / (r * r) - 1 / (2 * al)) * efc + math.sqrt(s / (math.pi * al)) * ex / r) / (4 * math.pi * r)
    u2 = u * u
    acc = torch.zeros_like(u)
    for n in range(12, 0, -1):
        acc = acc * u2 + (1 if n % 2 else -1) * 2 * n / (math.factorial(n) * (2 * n + 1))
    phi = torch.where(u < 0.5, 2 / math.sqrt(math.pi) * acc, (ef - 2 / math.sqrt(math.pi) * u * ex) / (u2 * u))
    return g, -(0.5 * u * phi + efc) / (8 * math.pi * al * r)


def _time_factors(r, h, al, nd, op):
    """Integrals over a target and a source step at offsets 0 .. nd-1 (second differences)."""
    f = _G2 if op == "V" else _D2
    rr = r if op == "V" else torch.where(r > 0, r, torch.ones_like(r))
    g = [f(rr, k * h, al) for k in range(nd + 1)]
    out = [g[1][0]]
    for d in range(1, nd):
        u = rr / (2 * math.sqrt(al * (d + 1) * h))
        a, b = ((g[d + 1][i] - g[d][i]) - (g[d][i] - g[d - 1][i]) for i in (0, 1))
        out.append(torch.where(u < 1, b, a))
    return out if op == "V" else [torch.where(r > 0, o, torch.zeros_like(o)) for o in out]


def _ss_points(cls, xi, a, b, c):
    """Sauter-Schwab points (s1, s2, t1, t2) and Jacobian factors for identical (3), edge (2) and vertex (1)."""
    if cls == 3:
        j = xi ** 3 * a * a * b
        q = [(1, 1 - a + a * b, 1 - a * b * c, 1 - a), (1 - a * b * c, 1 - a, 1, 1 - a + a * b),
             (1, a * (1 - b + b * c), 1 - a * b, a * (1 - b)), (1 - a * b, a * (1 - b), 1, a * (1 - b + b * c)),
             (1 - a * b * c, a * (1 - b * c), 1, a * (1 - b)), (1, a * (1 - b), 1 - a * b * c, a * (1 - b * c))]
        js = [j] * 6
    elif cls == 2:
        j = xi ** 3 * a * a
        q = [(1, a * c, 1 - a * b, a * (1 - b)), (1, a, 1 - a * b * c, a * b * (1 - c)),
             (1 - a * b, a * (1 - b), 1, a * b * c), (1 - a * b * c, a * b * (1 - c), 1, a),
             (1 - a * b * c, a * (1 - b * c), 1, a * b)]
        js = [j] + [j * b] * 4
    else:
        j = xi ** 3 * b
        q, js = [(1, a, b, b * c), (b, b * c, 1, a)], [j, j]
    return [tuple(xi * v for v in p) for p in q], js


def _touching(T):
    """Pairs sharing vertices, by their number, with the local vertex order of the singular rules."""
    star = {}
    for x, t in enumerate(T.tolist()):
        for v in t:
            star.setdefault(v, []).append(x)
    got = {1: [], 2: [], 3: []}
    for x, t in enumerate(T.tolist()):
        for y in sorted({y for v in t for y in star[v]}):
            s = T[y].tolist()
            com = [(i, s.index(v)) for i, v in enumerate(t) if v in s]
            ox, oy = [i for i, _ in com], [j for _, j in com]
            if len(com) == 2:
                ox, oy = ox + [3 - sum(ox)], oy + [3 - sum(oy)]
            elif len(com) == 1:
                ox, oy = [(ox[0] + k) % 3 for k in range(3)], [(oy[0] + k) % 3 for k in range(3)]
            got[len(com)].append((x, y, ox, oy))
    return got


class _Geometry:
    def __init__(self, c, V, T):
        self.c, self.V, self.T = c, V, T
        self.nt, self.nv = T.shape[0], V.shape[0]
        self.X = _dev(V[T])  # [nt][3 vertices][3]
        e1, e2 = self.X[:, 1] - self.X[:, 0], self.X[:, 2] - self.X[:, 1]
        cr = torch.linalg.cross(e1, e2)
        self.J = cr.norm(dim=1)
        self.n = cr / self.J[:, None]
        self.e1, self.e2 = e1, e2
        self.touch = _touching(T)
        t = torch.zeros(self.nt, self.nt, dtype=torch.bool, device=DEV)
        for prs in self.touch.values():
            if prs:
                t[_dev([q[0] for q in prs]), _dev([q[1] for q in prs])] = True
        self.touching = t

    def regular(self, factors, nout, op, rows):
        """Sum over the collapsed rule of factors(r) [list of nout] for target rows and every source triangle:
        V: [nout][rows][nt]; K: [nout][rows][nt][3 hat functions]."""
        rule = _triangle_rule(self.c["quad_regular"])
        out = torch.zeros((nout, len(rows), self.nt) + ((3,) if op == "K" else ()), device=DEV, dtype=F8)
        X, J = self.X[rows], self.J[rows]
        for s1, s2, wi in rule:
            xp = X[:, 0] + s1 * self.e1[rows] + s2 * self.e2[rows]
            for t1, t2, wj in rule:
                yp = self.X[:, 0] + t1 * self.e1 + t2 * self.e2
                dx = xp[:, None] - yp[None]
                r = dx.norm(dim=2)
                wt = wi * wj * J[:, None] * self.J[None]
                if op == "K":
                    wt = wt * (dx * self.n[None]).sum(2)
                for d, v in enumerate(factors(r)):
                    if op == "V":
                        out[d] += wt * v
                    else:
                        for i, b in enumerate((1 - t1, t1 - t2, t2)):
                            out[d][..., i] += wt * v * b
        return out

    def singular(self, factors, nout, op):
        """(rows, cols, values) of the touching pairs: V [nout][n], K [nout][n][3]."""
        x1, w1 = _gauss01(self.c["quad_singular"])
        rows, cols, vals = [], [], []
        g4 = list(itertools.product(range(len(x1)), repeat=4))
        q4 = _dev(np.array([[x1[i] for i in g] for g in g4]))
        w4 = _dev(np.array([math.prod(w1[i] for i in g) for g in g4]))
        for cls, prs in self.touch.items():
            for at in range(0, len(prs), 4096):
                part = prs[at:at + 4096]
                if not part:
                    continue
                ix, iy = _dev([q[0] for q in part]), _dev([q[1] for q in part])
                ox, oy = _dev([q[2] for q in part]), _dev([q[3] for q in part])
                PX = torch.gather(self.X[ix], 1, ox[:, :, None].expand(-1, -1, 3))
                PY = torch.gather(self.X[iy], 1, oy[:, :, None].expand(-1, -1, 3))
                acc = torch.zeros((nout, len(part)) + ((3,) if op == "K" else ()), device=DEV, dtype=F8)
                pts, js = _ss_points(cls, *(q4[:, i] for i in range(4)))
                for (s1, s2, t1, t2), j in zip(pts, js):
                    ex = lambda p, u, v: p[:, None, 0] + u[None, :, None] * (p[:, None, 1] - p[:, None, 0]) + \
                        v[None, :, None] * (p[:, None, 2] - p[:, None, 1])  # noqa: E731
                    dx = ex(PX, s1, s2) - ex(PY, t1, t2)
                    wt = (w4 * j)[None] * (self.J[ix] * self.J[iy])[:, None]
                    if op == "K":
                        wt = wt * (dx * self.n[iy][:, None]).sum(2)
                    for d, v in enumerate(factors(dx.norm(dim=2))):
                        if op == "V":
                            acc[d] += (wt * v).sum(1)
                        else:
                            b = torch.stack([(wt * v * q[None]).sum(1) for q in (1 - t1, t1 - t2, t2)], 1)
                            acc[d] += torch.zeros_like(b).scatter_(1, oy, b)
                rows.append(ix)
                cols.append(iy)
                vals.append(acc)
        return torch.cat(rows), torch.cat(cols), torch.cat(vals, 1)


class _Reference:
    """The pFMM product of Alg. 2 on uniform steps in torch FP64."""

    def __init__(self, c):
        self.c = c
        self.V, self.T = _mesh(c)
        self.geo = _Geometry(c, self.V, self.T)
        self.tree = _Tree(c, self.V, self.T)
        self.nt, self.nv = self.geo.nt, self.geo.nv
        self.h = c["T"] / c["steps"]
        self.m, self.na = c["m_x"], c["m_t"] + 1
        m1 = self.m + 1
        i = torch.arange(m1, device=DEV)
        self.deg = i[:, None, None] + i[None, :, None] + i[None, None, :]
        self.near, self.moments = {}, {}

    def blocks(self, op, rows, nd):
        """Nearfield entries [nd][rows][nt or nv] at step offsets 0 .. nd-1."""
        c, geo = self.c, self.geo
        f = lambda r, n=nd: _time_factors(r, self.h, c["alpha"], n, op)  # noqa: E731
        A = geo.regular(f, nd, op, rows)
        A[:min(nd, 2), geo.touching[rows]] = 0.0
        if op not in self.near:
            self.near[op] = geo.singular(lambda r: f(r, 2), 2, op)
        sr, sc, sv = self.near[op]
        inv = torch.full((self.nt,), -1, device=DEV, dtype=torch.long)
        inv[rows] = torch.arange(len(rows), device=DEV)
        keep = inv[sr] >= 0
        for d in range(min(nd, 2)):
            A[d][inv[sr[keep]], sc[keep]] += sv[d][keep]
        lp = self.tree.lv[self.tree.p]
        G = lp["G"]
        lin = _dev(lp["lin"])
        g = torch.stack([lin // (G * G), (lin // G) % G, lin % G], 1)
        far = (g[rows][:, None] - g[None]).abs().amax(2) > self.tree.ntr_near
        A[:, far] = 0.0
        if op == "K":
            B = torch.zeros(nd, len(rows), self.nv, device=DEV, dtype=F8)
            for v in range(3):
                B.index_add_(2, _dev(self.T[:, v].astype(np.int64)), A[..., v])
            A = B
        return A

    def nearfield(self, op, x):
        ls, Et = self.c["leaf_steps"], self.c["steps"]
        f = torch.zeros(x.shape[0], Et, self.nt, device=DEV, dtype=F8)
        t = torch.arange(Et, device=DEV)
        step = max(1, int(2e7) // self.nt)
        for r0 in range(0, self.nt, step):
            rows = torch.arange(r0, min(r0 + step, self.nt), device=DEV)
            A = self.blocks(op, rows, 2 * ls)
            for d in range(2 * ls):
                ok = (d <= ls + t % ls) & (t >= d)
                xs = torch.zeros_like(x)
                xs[:, ok] = x[:, t[ok] - d]
                f[:, :, rows] += xs @ A[d].T
        return f

    def cheb(self, z):
        T = [torch.ones_like(z), z]
        dT = [torch.zeros_like(z), torch.ones_like(z)]
        for k in range(2, self.m + 1):
            T.append(2 * z * T[-1] - T[-2])
            dT.append(2 * T[k - 1] + 2 * z * dT[-1] - dT[-2])
        return torch.stack(T[:self.m + 1], -1), torch.stack(dT[:self.m + 1], -1)

    def space_moments(self, op):
        """[nt][m1^3] integrals of the Chebyshev products, or [nt][3][m1^3] of their conormal derivatives."""
        if op in self.moments:
            return self.moments[op]
        L, geo, m1 = self.tree.lv[self.tree.p], self.geo, self.m + 1
        G, lin = L["G"], _dev(L["lin"])
        g = torch.stack([lin // (G * G), (lin // G) % G, lin % G], 1)
        cen = _dev(L["corner"]) + (2.0 * g + 1.0) * L["hx"]
        out = torch.zeros((self.nt,) + ((3,) if op == "K" else ()) + (m1, m1, m1), device=DEV, dtype=F8)
        for s1, s2, w in _triangle_rule(self.m // 2 + 2):
            T, dT = self.cheb((geo.X[:, 0] + s1 * geo.e1 + s2 * geo.e2 - cen) / L["hxp"])
            prod = lambda a, b, c: a[:, :, None, None] * b[:, None, :, None] * c[:, None, None, :]  # noqa: E731
            wj = (w * geo.J)[:, None, None, None]
            if op == "V":
                out += wj * prod(T[:, 0], T[:, 1], T[:, 2])
                continue
            n = self.c["alpha"] / L["hxp"] * geo.n
            q = n[:, 0, None, None, None] * prod(dT[:, 0], T[:, 1], T[:, 2]) + \
                n[:, 1, None, None, None] * prod(T[:, 0], dT[:, 1], T[:, 2]) + \
                n[:, 2, None, None, None] * prod(T[:, 0], T[:, 1], dT[:, 2])
            for v, b in enumerate((1 - s1, s1 - s2, s2)):
                out[:, v] += wj * b * q
        out *= (self.deg <= self.m)
        self.moments[op] = out
        return out

    def node(self, i, m):
        return math.cos((2 * i + 1) * math.pi / (2 * m + 2))

    def lagrange(self, b, x):
        mt = self.na - 1
        v, xb = 1.0, self.node(b, mt)
        for k in range(mt + 1):
            if k != b:
                v = v * (x - self.node(k, mt)) / (xb - self.node(k, mt))
        return v

    def step_weights(self):
        ls, na = self.c["leaf_steps"], self.na
        gx, gw = _gauss01(na)
        S = [[sum(w * self.h * self.lagrange(a, 2 * (s + x) / ls - 1) for x, w in zip(gx, gw)) for a in range(na)]
             for s in range(ls)]
        return _dev(np.array(S))

    def shifts(self, l):
        """q^(x)[bit][kappa][nu] from a child of level l into its parent, q^(t)[c][a_c][a_p]."""
        L, Lp, m = self.tree.lv[l], self.tree.lv[l - 1], self.m
        qx = np.zeros((2, m + 1, m + 1))
        tn = lambda k, x: math.cos(k * math.acos(x)) if abs(x) <= 1 else float(np.polynomial.chebyshev.chebval(x, [0] * k + [1]))  # noqa: E731
        for bit in range(2):
            for ka in range(m + 1):
                for nu in range(ka, m + 1):
                    qx[bit, ka, nu] = (1 if ka == 0 else 2) / (m + 1) * sum(
                        tn(nu, ((2 * bit - 1) * L["hx"] + L["hxp"] * self.node(n, m)) / Lp["hxp"]) * tn(ka, self.node(n, m))
                        for n in range(m + 1))
        qt = np.array([[[self.lagrange(ap, 0.5 * (2 * c - 1) + 0.5 * self.node(ac, self.na - 1)) for ap in range(self.na)]
                        for ac in range(self.na)] for c in range(2)])
        return _dev(qx), _dev(qt)

    def m2l(self, l, mu):
        """Locals of level l from its moments [R][nint][na][G][G][G][m1][m1][m1]."""
        L, m, na, al = self.tree.lv[l], self.m, self.na, self.c["alpha"]
        G, N = L["G"], L["nint"]
        lam = torch.zeros_like(mu)
        xs = np.array([self.node(i, m) for i in range(m + 1)])
        Tn = np.cos(np.outer(np.arange(m + 1), np.arccos(xs)))  # [k][node]
        sc = np.where(np.arange(m + 1) == 0, 1.0, 2.0)
        off = np.arange(-(G - 1), G)
        z = 2 * L["hx"] * off[:, None, None] / L["hxp"] + xs[None, :, None] - xs[None, None, :]
        i = np.arange(G)
        at = i[:, None] - i[None, :] + G - 1
        for D in (2, 3):
            k = [q for q in range(2, N) if D == 2 or (q % 2 and q >= 3)]
            if not k:
                continue
            tgt, src = _dev(k), _dev([q - D for q in k])
            for a in range(na):
                for b in range(na):
                    dt = D * 2 * L["ht"] + L["ht"] * (self.node(b, na - 1) - self.node(a, na - 1))
                    E = np.einsum("onm,ln,km->okl", np.exp(-z * z / (4 * al * dt / L["hxp"] ** 2)), Tn, Tn)
                    E *= (sc[:, None] * sc[None]) / (m + 1) ** 2
                    E[np.abs(off) > L["ntr"]] = 0.0
                    M = _dev(E[at])  # [X][Y][kappa][nu]
                    S = mu[:, src, a]
                    add = torch.zeros_like(S)
                    for q in range(m + 1):
                        n, w = m - q + 1, q + 1
                        s = S[..., :w, :w, :w] * (self.deg[:w, :w, :w] == q)
                        s = torch.einsum("RBYVWijk,XYiu->RBXVWujk", s, M[:, :, :w, :n])
                        s = torch.einsum("RBXVWujk,YVjv->RBXYWuvk", s, M[:, :, :w, :n])
                        s = torch.einsum("RBXYWuvk,ZWkw->RBXYZuvw", s, M[:, :, :w, :n])
                        add[..., :n, :n, :n] += s * (self.deg[:n, :n, :n] <= m - q)
                    lam[:, tgt, b] += (4 * math.pi * al * dt) ** -1.5 * add
        return lam

    def farfield(self, op, x):
        tree, m1, na, ls = self.tree, self.m + 1, self.na, self.c["leaf_steps"]
        p, R, Et = tree.p, x.shape[0], self.c["steps"]
        f = torch.zeros(R, Et, self.nt, device=DEV, dtype=F8)
        if p < 2:
            return f
        S = self.step_weights()
        L = tree.lv[p]
        G, cube = L["G"], (m1, m1, m1)
        Sx = self.space_moments("V").reshape(self.nt, -1)
        part = torch.zeros(R, Et, G ** 3, m1 ** 3, device=DEV, dtype=F8)
        T = self.T.astype(np.int64)
        for cell in np.unique(L["lin"]):
            idx = np.nonzero(L["lin"] == cell)[0]
            if op == "V":
                part[:, :, cell] = x[:, :, _dev(idx)] @ Sx[_dev(idx)]
            else:
                part[:, :, cell] = x[:, :, _dev(T[idx].reshape(-1))] @ self.space_moments("K")[_dev(idx)].reshape(-1, m1 ** 3)
        mu = {p: torch.einsum("sa,RNscq->RNacq", S, part.view(R, Et // ls, ls, G ** 3, m1 ** 3)).reshape(
            (R, Et // ls, na, G, G, G) + cube)}
        del part
        qs = {l: self.shifts(l) for l in range(3, p + 1)}
        for l in range(p - 1, 1, -1):
            qx, qt = qs[l + 1]
            c = mu[l + 1]
            N, Gc, Gp = c.shape[1], c.shape[3], tree.lv[l]["G"]
            c = torch.einsum("cap,RNcaq->RNpq", qt, c.reshape(R, N // 2, 2, na, -1)).reshape((R, N // 2, na, Gc, Gc, Gc) + cube)
            if Gc != Gp:
                c = c.reshape((R, N // 2, na, Gp, 2, Gp, 2, Gp, 2) + cube)
                c = torch.einsum("RNaXxYyZzijk,xiu->RNaXYyZzujk", c, qx)
                c = torch.einsum("RNaXYyZzujk,yjv->RNaXYZzuvk", c, qx)
                c = torch.einsum("RNaXYZzuvk,zkw->RNaXYZuvw", c, qx) * (self.deg <= self.m)
            mu[l] = c
        lam = None
        for l in range(2, p + 1):
            new = self.m2l(l, mu.pop(l))
            if lam is not None:
                qx, qt = qs[l]
                Gp, Gc, N = lam.shape[3], new.shape[3], lam.shape[1]
                c = lam
                if Gc != Gp:
                    c = torch.einsum("RNaXYZuvw,xiu->RNaXxYZivw", c, qx)
                    c = torch.einsum("RNaXxYZivw,yjv->RNaXxYyZijw", c, qx)
                    c = torch.einsum("RNaXxYyZijw,zkw->RNaXxYyZzijk", c, qx)
                    c = c.reshape((R, N, na, Gc, Gc, Gc) + cube) * (self.deg <= self.m)
                new += torch.einsum("cap,RNpq->RNcaq", qt, c.reshape(R, N, na, -1)).reshape(new.shape)
            lam = new
        q = torch.einsum("sa,RNacq->RNscq", S, lam.reshape(R, Et // ls, na, G ** 3, m1 ** 3)).reshape(R, Et, G ** 3, m1 ** 3)
        for cell in np.unique(L["lin"]):
            idx = _dev(np.nonzero(L["lin"] == cell)[0])
            f[:, :, idx] = q[:, :, cell] @ Sx[idx].T
        return f

    def apply(self, op, x):
        return self.nearfield(op, x) + self.farfield(op, x)

    def mass(self, g):
        area = 0.5 * self.geo.J
        T = _dev(self.T.astype(np.int64))
        return self.h * area / 3 * g[:, :, T].sum(3)


def _exact_general(c, x):
    """The dense Galerkin product on general steps; the FMM's truncation error is in the difference."""
    V, T = _mesh(c)
    geo = _Geometry(c, V, T)
    ts, Et, al = _graded(c), c["steps"], c["alpha"]
    f = torch.zeros_like(x)
    rows = torch.arange(geo.nt, device=DEV)

    def factors(k, j):
        def g(r):
            if j == k:
                return [_G2(r, ts[k + 1] - ts[k], al)[0]]
            s = (ts[k + 1] - ts[j], ts[k + 1] - ts[j + 1], ts[k] - ts[j], ts[k] - ts[j + 1])
            q = [_G2(r, v, al) for v in s]
            a, b = ((q[0][i] - q[1][i]) - (q[2][i] - q[3][i]) for i in (0, 1))
            return [torch.where(r / (2 * math.sqrt(al * s[0])) < 1, b, a)]
        return g
    for k in range(Et):
        for j in range(k + 1):
            A = geo.regular(factors(k, j), 1, "V", rows)[0]
            if k - j < 2:
                sr, sc, sv = geo.singular(factors(k, j), 1, "V")
                A[geo.touching] = 0.0
                A[sr, sc] = sv[0]
            f[:, k] += x[:, j] @ A.T
    return f


def _exact_net(c, seed):
    w, R, sl = _net_inputs(c, seed)
    ref = _Reference(c)
    geo, n, S = ref.geo, c["width"], c["slices"]
    A0 = torch.cat([ref.blocks("V", torch.arange(r, min(r + 1024, ref.nt), device=DEV), 1)[0] for r in range(0, ref.nt, 1024)])
    edge = {}
    for x, t in enumerate(ref.T.tolist()):
        for i in range(3):
            edge.setdefault(frozenset((t[i], t[(i + 1) % 3])), []).append(x)
    M = torch.zeros(ref.nt, ref.nt, device=DEV, dtype=F8)
    for q in edge.values():
        for x, y in itertools.permutations(q, 2):
            M[x, y] = 1.0
    M /= M.sum(1, keepdim=True).clamp_min(1.0)
    p = _dev(w.astype(np.float64)).requires_grad_()
    at = 0

    def take(*shape):
        nonlocal at
        v = p[at:at + math.prod(shape)].view(*shape)
        at += math.prod(shape)
        return v
    Wg, bg = take(5, n), take(n)
    layers = [(take(n, n), take(n, n)) for _ in range(c["layers"])]
    wo = take(n)
    area = 0.5 * geo.J
    s = _dev(sl.astype(np.int64))
    r = R.view(-1, ref.nt)[s]
    t = (s % c["steps"]).to(F8)
    feat = torch.cat([(area / area.mean())[:, None], geo.n], 1)
    rms = r.square().mean(1).sqrt() + 1e-30
    e = feat @ Wg[:4] + bg
    e = torch.nn.functional.silu(e[None] + ((t + 0.5) / c["steps"])[:, None, None] * Wg[4])
    h = (r / rms[:, None])[..., None] * e
    for Ws, Wn in layers:
        h = h + h @ Ws + torch.einsum("xy,byo->bxo", M, h) @ Wn
    z = 40.0 * rms[:, None] * (h @ wo)
    res = z.detach() @ A0.T - r
    den = r.square().sum(1) + 1e-30
    loss = (res.square().sum(1) / den).mean()
    z.backward(2.0 / S * (res / den[:, None]) @ A0.T)
    return {"loss": float(loss), "grad": p.grad}


def exact(case, seed):
    c = case
    k = c["kind"]
    if k == "batch":
        return [_Reference(q).apply("V", _gen(seed * 100 + i, q["nrhs"], q["steps"], _n_tri(q)))
                for i, q in enumerate(_problems(c))]
    nt = _n_tri(c)
    if k == "net":
        return _exact_net(c, seed)
    if k == "general":
        return _exact_general(c, _gen(seed, c["nrhs"], c["steps"], nt))
    ref = _Reference(c)
    if k == "solve":
        n = nt * c["steps"]
        if n > 6000:  # the dense matrix takes too long
            return None
        g = _datum(c, ref.V, seed)
        b = 0.5 * ref.mass(g) + ref.apply("K", g)
        eye = torch.eye(n, device=DEV, dtype=F8)
        A = torch.cat([ref.apply("V", q.view(-1, c["steps"], nt)).view(-1, n) for q in eye.split(256)])
        return torch.linalg.solve(A.T, b.view(n)).view(1, c["steps"], nt)
    x = _gen(seed, c["nrhs"], c["steps"], ref.nv if k == "K" else nt)
    return torch.cat([ref.apply("K" if k == "K" else "V", x[i:i + 1]) for i in range(c["nrhs"])])
