"""Performance cases: the calls a program that solves H x = lambda S x with this library makes.

Most cases are single steps of the LABPSD iteration through their own entry points, at the sizes
of the 8^3, 32^3 and 64^3 workloads and between them; two are whole solves from host arrays.
listed() names them, draw() gives further ones of the same ranges, prepare() / run() set one up
and make one pass, work() counts what the pass cannot do without and exact() gives the 64-bit
result where there is one.
"""
import functools
import math

import numpy as np
import torch

from paper_1308_2445_gb300 import hbsd
from paper_1308_2445_gb300 import pufe_inputs as pufe

TOL = 1e-8
# (elements per edge, atoms, enrichment dofs per node, r_c) of the discretisations in use: the named
# 8^3 and 32^3 workloads, and meshes of the batched workload between them
MESHES = {"8": (8, 2, 2, 0.25), "12": (12, 4, 3, 0.15), "16": (16, 6, 2, 0.15), "24": (24, 8, 3, 0.15),
          "32": (32, 8, 4, 0.15)}
N_LARGE, Q_LARGE, K_LARGE = 334272, 538, 282   # 64^3 workload: rows, widest [Psi P], nev + m0
N_MEDIUM, Q_MEDIUM = 47620, 149                 # 32^3 workload, nev = 64, m0 = 21


def listed():
    return [
        # steps 3/7 of the FP64 form on the smallest problem: a call of a few microseconds of work
        dict(name="spmm_fp64_8", kind="spmm", mesh="8", k=19, form="fp64"),
        # steps 3/7 of the mixed form on the 32^3 problem's block of nev + m0 columns
        dict(name="spmm_df64_32", kind="spmm", mesh="32", k=85, form="df64"),
        # step 6(a) of the mixed form: all 64 columns unconverged, as in most iterations
        dict(name="precond_f32_32", kind="precond", mesh="32", k=64, form="f32"),
        # step 6(b) of the mixed form: the localized columns of one iteration
        dict(name="minres_32", kind="minres", mesh="32", k=24, form="mixed"),
        # step 8 of the FP64 form, odd sizes
        dict(name="gram_fp64_24", kind="gram", n=20613, q=71, form="fp64"),
        # step 8 of the mixed form, 32^3 and 64^3 workloads
        dict(name="gram_df64_32", kind="gram", n=N_MEDIUM, q=Q_MEDIUM, form="df64"),
        dict(name="gram_df64_64", kind="gram", n=N_LARGE, q=Q_LARGE, form="df64"),
        # steps 10-11 of the mixed form, 64^3 workload
        dict(name="update_df64_64", kind="update", n=N_LARGE, q=Q_LARGE, k=K_LARGE, form="df64"),
        # step 9, 32^3 and 64^3 workloads (FP64 in both forms)
        dict(name="rr_32", kind="rr", q=Q_MEDIUM, k=85),
        dict(name="rr_64", kind="rr", q=Q_LARGE, k=K_LARGE),
        # one SCF step on a resident session: new H values on the pattern, then a mixed solve
        dict(name="scf_step_32", kind="scf", mesh="32", nev=64, m0=21, form="mixed"),
        # a new problem end to end with the default options: create (ordering, factor) and solve
        dict(name="new_problem_16", kind="new", mesh="16", nev=32, m0=-1, form="fp64"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spmm", "spmm", "precond", "minres", "gram", "gram", "update", "update", "rr", "rr", "scf"])
    if kind in ("spmm", "precond", "minres"):
        mesh = rng.choice(sorted(MESHES))
        k = _logint(rng, 1, {"spmm": 300, "precond": 128, "minres": 64}[kind])
        form = {"spmm": rng.choice(["fp64", "df64", "df64"]), "precond": rng.choice(["f32", "f32", "fp64"]),
                "minres": rng.choice(["mixed", "fp64"])}[kind]
        return dict(kind=kind, mesh=mesh, k=k, form=form)
    if kind in ("gram", "update"):
        form = rng.choice(["df64", "df64", "fp64"])
        q = _logint(rng, 16, Q_LARGE)
        n = _logint(rng, 646, N_LARGE)
        if form == "fp64":   # the FP64 form is used on the smaller problems
            n = min(n, int(2e9 / (q * q)))
        if kind == "gram":
            return dict(kind=kind, n=n, q=q, form=form)
        return dict(kind=kind, n=n, q=q, k=max(1, min(q, int(q * rng.uniform(0.5, 1.0)))), form=form)
    if kind == "rr":
        q = _logint(rng, 8, Q_LARGE)
        return dict(kind=kind, q=q, k=max(1, min(q, int(q * rng.uniform(0.5, 1.0)))))
    return dict(kind="scf", mesh="8", nev=rng.randint(6, 24), m0=-1, form=rng.choice(["mixed", "fp64"]))


# ---- what a program keeps: the problem and its session ----------------------------------------

@functools.lru_cache(maxsize=None)
def _problem(mesh):
    n_el, atoms, enr, rc = MESHES[mesh]
    return pufe.generate(n_el, atoms, enr, rc, 1)


@functools.lru_cache(maxsize=3)
def _session(mesh, form, m0=-1):
    precision = hbsd.PRECISION_FP64 if form == "fp64" else hbsd.PRECISION_MIXED
    return hbsd.Session.from_problem(_problem(mesh), precision=precision, m0=m0)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + 17)


def _block(n, k, dtype=torch.float64):
    """An n x k row-major device block with the leading dimension the library asks for."""
    mult = 4 if dtype == torch.float32 else 2
    return torch.zeros(n, (k + mult - 1) // mult * mult, dtype=dtype, device="cuda")[:, :k]


def _normal(n, k, g, dtype=torch.float64):
    t = _block(n, k, dtype)
    t.copy_(torch.randn(n, k, generator=g, dtype=dtype, device="cuda"))
    return t


def _row_scale(n, g):
    """diag(S)^{-1/2} of an enriched basis: most rows at one size, a third spread over many decades."""
    u = torch.rand(n, 1, generator=g, dtype=torch.float64, device="cuda")
    v = torch.rand(n, 1, generator=g, dtype=torch.float64, device="cuda")
    return torch.where(u < 0.3, 10.0 ** (2.5 + 10.0 * v), torch.full_like(v, 300.0))


def _col_scale(q, g):
    """Psi columns of one size, then P columns of very different sizes."""
    s = torch.ones(q, dtype=torch.float64, device="cuda")
    h = (q + 1) // 2
    s[h:] = 10.0 ** (-4.0 + 5.0 * torch.rand(q - h, generator=g, dtype=torch.float64, device="cuda"))
    return s


def _gram_blocks(case, seed):
    g, n, q = _gen(seed), case["n"], case["q"]
    d, c = _row_scale(n, g), _col_scale(q, g)
    Z, ZH, ZS = (_normal(n, q, g) for _ in range(3))
    ZS += 0.5 * Z
    ZH += 2.0 * Z
    Z *= d * c
    ZH *= c / d
    ZS *= c / d
    return Z, ZH, ZS


def _update_blocks(case, seed):
    g, n, q, k = _gen(seed), case["n"], case["q"], case["k"]
    Z = _normal(n, q, g)
    Z *= _row_scale(n, g)
    W = torch.randn(q, k, generator=g, dtype=torch.float64, device="cuda")
    W = torch.linalg.qr(W)[0].contiguous()   # orthonormal columns: repeated updates stay bounded
    return Z, W


def _pencil(case, seed):
    """Reduced matrices of [Psi P]: a spectrum without clusters (each vector is then determined), and
    columns of very different norms."""
    g, q = _gen(seed), case["q"]
    lam = torch.cumsum(0.5 + torch.rand(q, generator=g, dtype=torch.float64, device="cuda"), 0)
    G = torch.randn(q, q, generator=g, dtype=torch.float64, device="cuda") * (0.3 / math.sqrt(q))
    G += torch.eye(q, dtype=torch.float64, device="cuda")
    G *= _col_scale(q, g)
    HR, SR = G.T @ (lam[:, None] * G), G.T @ G
    sign = torch.randn(q, generator=g, dtype=torch.float64, device="cuda")
    return (0.5 * (HR + HR.T)).contiguous(), (0.5 * (SR + SR.T)).contiguous(), sign


@functools.lru_cache(maxsize=None)
def _noise_step(mesh):
    """Change of H under 1% noise on the potential (an SCF-style follow-up of the same problem)."""
    n_el, atoms, enr, rc = MESHES[mesh]
    return pufe.generate(n_el, atoms, enr, rc, 1, v_noise=0.01).h_val - _problem(mesh).h_val


def _h_values(mesh, seed):
    return _problem(mesh).h_val + np.random.default_rng(seed).uniform(0.2, 1.0) * _noise_step(mesh)


def _minres_inputs(case, seed):
    s, p, k = _session(case["mesh"], case["form"]), _problem(case["mesh"]), case["k"]
    g = _gen(seed)
    d = torch.from_numpy(s.dscale()).cuda()[:, None]
    R = _normal(p.n, k, g)
    R /= d
    P0 = _block(p.n, k)
    s.precond_apply(R, P0)   # the start that step 6(a) hands to step 6(b)
    e = 0.1 + 2.0 * torch.rand(k, generator=g, dtype=torch.float64, device="cuda")
    return s, R, P0, e


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "case": case}
    if kind == "spmm":
        s, n = _session(case["mesh"], "mixed"), _problem(case["mesh"]).n
        X = _normal(n, case["k"], _gen(seed))
        X *= torch.from_numpy(s.dscale()).cuda()[:, None]
        st.update(s=s, X=X, HX=_block(n, case["k"]), SX=_block(n, case["k"]))
    elif kind == "precond":
        s, n = _session(case["mesh"], "mixed"), _problem(case["mesh"]).n
        dt = torch.float32 if case["form"] == "f32" else torch.float64
        R = _normal(n, case["k"], _gen(seed), dt)
        if case["form"] == "fp64":
            R /= torch.from_numpy(s.dscale()).cuda()[:, None]
        P = _block(n, case["k"], dt)
        if case["form"] == "f32":
            s.precond_apply_f32(R, P)   # the FP32 panels are made with the session's first use
        st.update(s=s, R=R, P=P)
    elif kind == "minres":
        s, R, P0, e = _minres_inputs(case, seed)
        st.update(s=s, R=R, P0=P0, e=e, P=_block(R.shape[0], case["k"]),
                  steps=torch.zeros(case["k"], dtype=torch.int32, device="cuda"))
    elif kind == "gram":
        Z, ZH, ZS = _gram_blocks(case, seed)
        q = case["q"]
        st.update(Z=Z, ZH=ZH, ZS=ZS, HR=torch.zeros(q, q, dtype=torch.float64, device="cuda"),
                  SR=torch.zeros(q, q, dtype=torch.float64, device="cuda"))
    elif kind == "update":
        Z, W = _update_blocks(case, seed)
        st.update(Z=Z, W=W)
    elif kind == "rr":
        HR, SR, sign = _pencil(case, seed)
        st.update(HR=HR, SR=SR, sign=sign, theta=torch.zeros(case["k"], dtype=torch.float64, device="cuda"),
                  W=torch.zeros(case["q"], case["k"], dtype=torch.float64, device="cuda"),
                  info=torch.zeros(2, dtype=torch.int32, device="cuda"))
    elif kind == "scf":
        p = _problem(case["mesh"])
        s = _session(case["mesh"], case["form"], case["m0"])
        w = case["nev"] + s.m0(case["nev"])
        st.update(s=s, h=_h_values(case["mesh"], seed), X0=np.random.default_rng(seed).standard_normal((p.n, w)))
    elif kind == "new":
        p = _problem(case["mesh"])
        m0 = case["m0"] if case["m0"] >= 0 else max(3, -(-case["nev"] // 10))
        X0 = np.random.default_rng(seed).standard_normal((p.n, case["nev"] + m0))
        st.update(p=p, h=_h_values(case["mesh"], seed), X0=X0)
    else:
        raise ValueError(kind)
    return st


def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "spmm":
        (st["s"].spmm_pair_df64 if case["form"] == "df64" else st["s"].spmm_pair)(st["X"], st["HX"], st["SX"])
        return st["HX"], st["SX"]
    if kind == "precond":
        (st["s"].precond_apply_f32 if case["form"] == "f32" else st["s"].precond_apply)(st["R"], st["P"])
        return st["P"]
    if kind == "minres":
        st["P"].copy_(st["P0"])   # refined in place
        st["s"].minres(st["R"], st["e"], st["P"], 0.25, 20, st["steps"])
        return st["P"], st["steps"]
    if kind == "gram":
        (hbsd.gram_df64 if case["form"] == "df64" else hbsd.gram)(st["Z"], st["ZH"], st["ZS"], st["HR"], st["SR"])
        return st["HR"], st["SR"]
    if kind == "update":
        (hbsd.update_df64 if case["form"] == "df64" else hbsd.update)(st["Z"], st["W"], case["k"])
        return st["Z"]
    if kind == "rr":
        hbsd.rayleigh_ritz(st["HR"], st["SR"], case["k"], st["theta"], st["W"], st["info"])
        # an eigenvector's sign is free: fix it by its product with a given vector
        return st["theta"], st["W"] * torch.sign(st["sign"] @ st["W"])
    if kind == "scf":
        st["s"].update_H(st["h"])
        return st["s"].solve(case["nev"], TOL, X0=st["X0"], want_vectors=False)[0]
    p = st["p"]
    precision = hbsd.PRECISION_FP64 if case["form"] == "fp64" else hbsd.PRECISION_MIXED
    s = hbsd.Session(p.n, p.row_ptr, p.col_idx, st["h"], p.s_val, p.dof_node, p.grid, p.eps_bar, precision=precision,
                     m0=case["m0"])
    lam = s.solve(case["nev"], TOL, X0=st["X0"], want_vectors=False)[0]
    s.close()
    return lam


# ---- work and exact results ---------------------------------------------------------------------

def _factor_nnz(n, nnz):
    """Entries of the sparse factor: the fill measured on the 32^3 and 64^3 workloads."""
    return 16.5 * (n / 47620.0) ** 0.35 * nnz


def work(case):
    kind = case["kind"]
    if kind in ("spmm", "precond", "minres", "scf", "new"):
        p = _problem(case["mesh"])
        n, nnz = p.n, p.nnz
        nl = _factor_nnz(n, nnz)
    if kind == "spmm":
        return {"bytes": 20.0 * nnz + 24.0 * n * case["k"], "flops": 4.0 * nnz * case["k"]}
    if kind == "precond":
        b = 4 if case["form"] == "f32" else 8
        return {"bytes": b * (nl + 2.0 * n * case["k"]), "flops": 4.0 * nl * case["k"]}
    if kind == "minres":   # 20 steps at most; two products per stored entry and about 12 n per step
        return {"bytes": 20.0 * nnz + 24.0 * n * case["k"], "flops": 20 * case["k"] * (4.0 * nnz + 24.0 * n)}
    if kind == "gram":
        n, q = case["n"], case["q"]
        return {"bytes": 24.0 * n * q + 16.0 * q * q, "flops": (2.0 if case["form"] == "df64" else 4.0) * n * q * (q + 1)}
    if kind == "update":
        n, q, k = case["n"], case["q"], case["k"]
        return {"bytes": 8.0 * n * (q + k) + 8.0 * q * k, "flops": 2.0 * n * q * k}
    if kind == "rr":
        q, k = case["q"], case["k"]
        return {"bytes": 16.0 * q * q + 8.0 * q * k, "flops": 5.0 * q ** 3 + 4.0 * q * q * k}
    # a whole solve: 20 outer iterations of products, factor solves, Gram and update
    m = case["nev"]
    w = m + (case["m0"] if case["m0"] >= 0 else max(3, -(-m // 10)))
    q = w + m
    it = 4.0 * nnz * m + 4.0 * nl * m + 2.0 * n * q * q + 2.0 * n * q * w + 10.0 * q ** 3
    return {"bytes": 16.0 * nnz + 8.0 * n * w + 20 * (4.0 * nl + 24.0 * n * q), "flops": 20 * it}


def _csr(p, v):
    return torch.sparse_csr_tensor(torch.from_numpy(p.row_ptr), torch.from_numpy(p.col_idx.astype(np.int64)),
                                   torch.from_numpy(v), size=(p.n, p.n)).cuda()


def _dense_pair(p, h):
    rows = np.repeat(np.arange(p.n), np.diff(p.row_ptr))
    H, S = np.zeros((p.n, p.n)), np.zeros((p.n, p.n))
    H[rows, p.col_idx], S[rows, p.col_idx] = h, p.s_val
    return torch.from_numpy(H), torch.from_numpy(S)


def _eig(H, S):
    """Generalised eigenpairs by scaled Cholesky, ascending."""
    d = S.diagonal().rsqrt()
    L = torch.linalg.cholesky(d[:, None] * S * d)
    T = torch.linalg.solve_triangular(L, d[:, None] * H * d, upper=False)
    C = torch.linalg.solve_triangular(L, T.T.contiguous(), upper=False)
    lam, Q = torch.linalg.eigh(0.5 * (C + C.T))
    return lam, d[:, None] * torch.linalg.solve_triangular(L.T.contiguous(), Q, upper=True)


def exact(case, seed):
    kind = case["kind"]
    if kind == "spmm":
        p, s = _problem(case["mesh"]), _session(case["mesh"], "mixed")
        X = prepare(case, seed)["X"].contiguous()
        return _csr(p, p.h_val - s.sigma0 * p.s_val) @ X, _csr(p, p.s_val) @ X
    if kind == "precond" and case["mesh"] == "8" and case["form"] == "fp64":
        p = _problem("8")
        H, S = _dense_pair(p, p.h_val)
        return -torch.linalg.solve(H - p.eps_bar * S, prepare(case, seed)["R"].cpu())
    if kind == "gram":
        Z, ZH, ZS = _gram_blocks(case, seed)
        A, B = Z.T @ ZH, Z.T @ ZS
        if case["form"] == "df64":   # the entries a <= b, mirrored
            return torch.triu(A) + torch.triu(A, 1).T, torch.triu(B) + torch.triu(B, 1).T
        return 0.5 * (A + A.T), 0.5 * (B + B.T)
    if kind == "update":
        Z, W = _update_blocks(case, seed)
        out = Z.clone()
        out[:, :case["k"]] = Z @ W
        return out
    if kind == "rr":
        HR, SR, sign = _pencil(case, seed)
        lam, X = _eig(HR, SR)
        lam, X = lam[:case["k"]], X[:, :case["k"]]
        return lam, X * torch.sign(sign @ X)
    if kind == "scf" and case["mesh"] == "8":
        p = _problem("8")
        return _eig(*_dense_pair(p, _h_values(case["mesh"], seed)))[0][:case["nev"]].numpy()
    return None   # a factor solve, MINRES or a solve of thousands of unknowns
