"""Performance cases: what programs built on this library spend their time in.

A case is a dict of plain values; ``family`` says which public entry points it
goes through:

* ``apply``   one operator application, ``DiracOp.apply`` / ``apply_normal``
* ``solve``   one multi-RHS Krylov solve, ``DiracOp.solve``
* ``batch``   independent solves of different shapes, ``solve_batched``
* ``action``  a differentiable pseudofermion action, forward and backward
* ``md``      one fermion step of molecular dynamics: new links into an
              operator, chi = D psi, the link force

Sizes are those of the tests, the benchmark and the paper's tables.  Links are
exp(i eps sum_k a_k lambda_k), sources complex Gaussian; both are drawn on the
GPU from the seed alone.  ``exact`` restates the operators in torch complex128
from the equations (no library code).
"""
import math

import numpy as np
import torch

from paper_2112_14640_gb300 import dirac as D
from paper_2112_14640_gb300 import inputs as I
from paper_2112_14640_gb300.autograd import PseudofermionAction

DEVICE = "cuda"
KINDS = {"wilson": D.WILSON, "brillouin": D.BRILLOUIN, "staggered": D.STAGGERED,
         "wlap": D.WLAP, "blap": D.BLAP, "wsuv": D.WSUV, "bsuv": D.BSUV}
PRECS = {"f64": D.F64, "f32": D.F32, "bf16": D.BF16, "f16": D.F16}
BYTES = {"f64": 8, "f32": 4, "bf16": 2, "f16": 2}
COLOUR_ONLY = ("staggered", "wsuv", "bsuv")
USES_W = ("brillouin", "blap", "bsuv")
BC = (1, 1, 1, -1)


# ------------------------------------------------------------------- the cases
def _dims(nx, ny, nz, nt):
    return {"nx": nx, "ny": ny, "nz": nz, "nt": nt}


def _apply(name, kind, dims, nv, prec="f32", nc=3, layout="inner", op="D", m0=0.1, csw=0.0, links="native",
           tune=False):
    return {"name": name, "family": "apply", "kind": kind, "prec": prec, **_dims(*dims), "nc": nc, "nv": nv,
            "layout": layout, "op": op, "m0": m0, "csw": csw, "links": links, "tune": tune, "eps": 0.4}


def _solve(name, kind, dims, nv, method, prec, inner, m0, tol, layout="inner", mode="reliable", links="native",
           eps=0.4):
    return {"name": name, "family": "solve", "kind": kind, **_dims(*dims), "nc": 3, "nv": nv, "method": method,
            "prec": prec, "inner": inner, "mode": mode, "links": links, "m0": m0, "tol": tol, "layout": layout,
            "eps": eps}


def listed():
    small, bench, large = (8, 8, 8, 8), (16, 16, 16, 32), (32, 32, 32, 64)
    return [
        # the smallest call: one FP64 vector on 4^4, as interactive checks and tiny test systems make it
        _apply("wilson_4x4_f64", "wilson", (4, 4, 4, 4), 1, prec="f64", layout="outer"),
        # the benchmark's operators on its lattice, tuned as a long-running program tunes them
        _apply("wilson_nv12", "wilson", bench, 12, tune=True),
        _apply("brillouin_nv12", "brillouin", bench, 12, tune=True),
        # production volume: nothing fits the L2 cache
        _apply("staggered_large", "staggered", large, 12, m0=0.05, tune=True),
        # the Brillouin Laplacian, the operator of smearing and eigenmode work
        _apply("blap_nv12", "blap", bench, 12, tune=True),
        # the paper's full Wilson operator (clover term) on an odd-sized lattice with an odd number of
        # right-hand sides in the paper's own vector order, untuned, daggered
        _apply("wilson_clover_ragged", "wilson", (18, 14, 11, 25), 7, layout="outer", op="Ddag", csw=1.0),
        # the colour sweep's N_c = 4 column: D^dag D as solvers and eigensolvers apply it
        _apply("wilson_nc4_normal", "wilson", (16, 16, 16, 32), 24, nc=4, op="normal", tune=True),
        # a small FP32 propagator solve: launches and host round trips count
        _solve("cg_staggered_8", "staggered", small, 3, "cg", "f32", "f32", 0.1, 1e-5, layout="outer"),
        # the mixed-precision solve of the benchmark's precision study (16-bit sloppy vectors, FP32 sloppy
        # links, FP64 solution) on its apply lattice, at a mass where the 16-bit iteration carries it through
        _solve("cg_mixed_f16", "staggered", bench, 12, "cg", "f64", "f16", 0.2, 1e-10, mode="adaptive",
               links="f32"),
        # a batch of independent propagator solves of uneven shape (the batched-solve workload)
        {"name": "batch_mixed_shapes", "family": "batch", "prec": "f32", "tol": 1e-5, "eps": 0.4,
         "solves": "wilson 8 8 8 8 5 0.1; staggered 12 12 12 12 17 0.1; wilson 12 12 12 12 2 0.1; "
                   "staggered 8 8 8 8 1 0.1; wilson 8 8 8 8 24 0.1; staggered 8 8 8 8 11 0.1; "
                   "wilson 16 16 16 32 3 0.1; staggered 16 16 16 32 8 0.1"},
        # differentiable pseudofermion action (the differentiation workload): S, dS/dU, dS/dphi
        {"name": "action_wilson", "family": "action", "kind": "wilson", "prec": "f32", **_dims(*bench), "nc": 3,
         "nv": 4, "m0": 0.2, "tol": 1e-6, "eps": 0.4},
        # one molecular-dynamics fermion step with the Brillouin operator: links change every step
        {"name": "md_brillouin", "family": "md", "kind": "brillouin", "prec": "f32", **_dims(*bench), "nc": 3,
         "nv": 4, "m0": 0.1, "layout": "outer", "eps": 0.4},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _extents(rng, lo, hi, vmax, even):
    while True:
        d = [_log_int(rng, lo, hi) for _ in range(3)] + [_log_int(rng, lo, 2 * hi)]
        if even:
            d = [x + (x & 1) for x in d]
        if math.prod(d) <= vmax:
            return d


def draw(rng):
    """One more case of the same ranges: every family, kind, precision, layout and option the listed ones stand for."""
    family = rng.choice(["apply"] * 6 + ["solve", "solve", "batch", "action", "md", "md"])
    if family == "apply":
        kind = rng.choice(["wilson", "wilson", "staggered", "staggered", "brillouin", "brillouin", "wlap", "blap",
                           "wsuv", "bsuv"])
        dirac = kind in ("wilson", "staggered", "brillouin")
        prec = rng.choice(["f32"] * 4 + ["f64"] + (["bf16", "f16"] if dirac else []))
        nc = rng.choice([3] * 6 + [1, 2, 4] + ([5, 6, 8] if prec in ("f32", "f64") else []))
        w = kind in USES_W
        vmax = (131072 if nc <= 3 else 20000) if w else (800000 if nc <= 3 else 131072)
        if prec == "f64":
            vmax //= 4
        d = _extents(rng, 3, 32, vmax, kind == "staggered")
        nv = _log_int(rng, 1, 24)
        c = _apply("", kind, d, nv, prec=prec, nc=nc, layout=rng.choice(["inner", "outer"]),
                   op=rng.choice(["D", "D", "Ddag", "normal"]), m0=0.05 if kind == "staggered" else 0.1,
                   csw=rng.choice([0.0, 0.0, 1.0]) if kind in ("wilson", "brillouin") else 0.0,
                   links=rng.choice(["native", "f32"]) if prec in ("bf16", "f16") else "native",
                   tune=rng.random() < 0.3 and math.prod(d) * nv < 2000000)
    elif family == "solve":
        kind = rng.choice(["wilson", "staggered", "staggered", "brillouin"])
        method, prec, inner = rng.choice([("cg", "f32", "f32"), ("cg", "f64", "f32"), ("cg", "f64", "f16"),
                                          ("cg", "f64", "f64"), ("bicgstab", "f64", "f32")])
        if method == "bicgstab" and kind == "staggered":
            kind = "wilson"
        d = _extents(rng, 4, 16, 2500 if prec == inner == "f64" else (12000 if kind == "brillouin" else 50000),
                     kind == "staggered")
        c = _solve("", kind, d, _log_int(rng, 1, 12), method, prec, inner, 0.2, 1e-5 if prec == "f32" else 1e-9,
                   layout=rng.choice(["inner", "outer"]),
                   mode=rng.choice(["reliable", "adaptive"]) if method == "cg" else "restart",
                   links="f32" if inner == "f16" else "native")
    elif family == "batch":
        solves = []
        for _ in range(rng.randint(2, 10)):
            kind = rng.choice(["wilson", "staggered"])
            d = rng.choice([(8, 8, 8, 8), (8, 8, 8, 8), (12, 12, 12, 12), (6, 10, 8, 12), (16, 16, 16, 16)])
            solves.append("%s %d %d %d %d %d 0.1" % ((kind,) + d + (rng.randint(1, 16),)))
        c = {"family": "batch", "prec": "f32", "tol": 1e-5, "eps": 0.4, "solves": "; ".join(solves)}
    elif family == "action":
        kind = rng.choice(["wilson", "staggered"])
        d = _extents(rng, 4, 12, 16000, kind == "staggered")
        c = {"family": "action", "kind": kind, "prec": "f32", **_dims(*d), "nc": 3, "nv": _log_int(rng, 1, 6),
             "m0": 0.3, "tol": 1e-6 if kind == "wilson" else 1e-5, "eps": 0.4}   # what FP32 reaches
    else:
        kind = rng.choice(["wilson", "staggered", "brillouin", "brillouin"])
        prec = rng.choice(["f32", "f32", "f64"])
        nc = rng.choice([3, 3, 3, 2, 4])
        d = _extents(rng, 3, 20, 131072 if prec == "f32" and nc <= 3 else 20000, kind == "staggered")
        c = {"family": "md", "kind": kind, "prec": prec, **_dims(*d), "nc": nc, "nv": _log_int(rng, 1, 8),
             "m0": 0.1, "layout": rng.choice(["inner", "outer"]), "eps": 0.4}
    c.pop("name", None)
    return c


# ------------------------------------------------------------------- inputs
def _generator(seed, stream):
    return torch.Generator(device=DEVICE).manual_seed(1000003 * int(seed) + stream)


def _mm(A, B):
    """A B for (..., n, n) fields, as n elementwise products (small n)."""
    out = A[..., :, 0, None] * B[..., None, 0, :]
    for k in range(1, A.shape[-1]):
        out = out + A[..., :, k, None] * B[..., None, k, :]
    return out


def _gauge(dims, nc, eps, gen):
    """Random SU(N_c) links (Nt, Nz, Ny, Nx, 4, Nc, Nc), complex128: exp(i eps sum_k a_k lambda_k)."""
    nx, ny, nz, nt = dims
    shape = (nt, nz, ny, nx, 4)
    if nc == 1:
        a = torch.randn(shape, dtype=torch.float64, device=DEVICE, generator=gen)
        return torch.polar(torch.ones_like(a), eps * a)[..., None, None].contiguous()
    gm = torch.from_numpy(I.gell_mann(nc)).to(DEVICE).reshape(nc * nc - 1, nc * nc)
    a = torch.randn(shape + (nc * nc - 1,), dtype=torch.float64, device=DEVICE, generator=gen)
    # X = i eps H / 2^6: |X| < 0.2, twelve Taylor terms leave less than 1e-16
    X = ((1j * eps / 64.0) * (a.to(torch.complex128) @ gm)).reshape(shape + (nc, nc))
    del a
    one = torch.eye(nc, dtype=torch.complex128, device=DEVICE)
    E = one + X / 12.0
    for k in range(11, 0, -1):
        E = one + _mm(X, E) / k
    for _ in range(6):
        E = _mm(E, E)
    return E.contiguous()


def _source(dims, nc, nv, colour_only, gen, dtype=torch.float64):
    """Gaussian source, site-outer order, Re and Im ~ N(0, 1)."""
    nx, ny, nz, nt = dims
    shape = (nt, nz, ny, nx, nc, nv) if colour_only else (nt, nz, ny, nx, nc, 4, nv)
    return torch.view_as_complex(torch.randn(shape + (2,), dtype=dtype, device=DEVICE, generator=gen))


def _rounded(v, prec):
    """A complex128 tensor holding what storage in ``prec`` keeps of v."""
    if prec == "f64":
        return v
    if prec == "f32":
        return v.to(torch.complex64).to(torch.complex128)
    dt = torch.bfloat16 if prec == "bf16" else torch.float16
    r = torch.view_as_real(v.to(torch.complex64)).to(dt).to(torch.float64)
    return torch.view_as_complex(r.contiguous())


def _shape(case):
    return (case["nx"], case["ny"], case["nz"], case["nt"])


def _layout(case):
    return D.SITE_INNER if case.get("layout") == "inner" else D.SITE_OUTER


def _fields(case, seed):
    dims = _shape(case)
    U = _gauge(dims, case["nc"], case["eps"], _generator(seed, 1))
    # sources are drawn in the operator's own precision
    dt = torch.float64 if case["prec"] == "f64" else torch.float32
    b = _source(dims, case["nc"], case["nv"], case["kind"] in COLOUR_ONLY, _generator(seed, 2), dt)
    return U, b


def _batch_spec(case):
    out = []
    for s in case["solves"].split(";"):
        f = s.split()
        out.append((f[0], tuple(int(v) for v in f[1:5]), int(f[5]), float(f[6])))
    return out


def _batch_fields(case, seed):
    for i, (kind, dims, nv, m0) in enumerate(_batch_spec(case)):
        U = _gauge(dims, 3, case["eps"], _generator(seed, 10 + 2 * i))
        yield kind, dims, nv, m0, U, _source(dims, 3, nv, kind in COLOUR_ONLY, _generator(seed, 11 + 2 * i),
                                             torch.float32)


# ------------------------------------------------------------------- prepare / run
def prepare(case, seed):
    fam = case["family"]
    if fam == "batch":
        ops, bs, m0s = [], [], []
        for kind, dims, nv, m0, U, b in _batch_fields(case, seed):
            op = D.DiracOp(KINDS[kind], U, nv, BC, PRECS[case["prec"]])
            ops.append(op)
            bs.append(op.to_prec(op.from_site_outer(b)))
            m0s.append(m0)
        return {"case": case, "ops": ops, "bs": bs, "m0s": m0s}
    U, b = _fields(case, seed)
    if fam == "action":
        act = PseudofermionAction(case["m0"], BC, prec=PRECS[case["prec"]], tol=case["tol"], kind=KINDS[case["kind"]])
        return {"case": case, "act": act, "U": U.requires_grad_(True), "phi": b.requires_grad_(True)}
    links = D.LINKS_F32 if fam == "apply" and case["links"] == "f32" else D.LINKS_NATIVE
    op = D.DiracOp(KINDS[case["kind"]], U, case["nv"], BC, PRECS[case["prec"]], layout=_layout(case),
                   link_storage=links)
    st = {"case": case, "op": op, "x": op.to_prec(op.from_site_outer(b))}
    if fam == "apply":
        if case["csw"]:
            op.set_clover(case["csw"], U)
        if case["tune"]:
            op.autotune(case["m0"])
        st["out"] = op.new_vector()
    elif fam == "md":
        st["U"] = U
    return st


def run(state):
    case = state["case"]
    fam = case["family"]
    if fam == "apply":
        op, m0 = state["op"], case["m0"]
        if case["op"] == "normal":
            return op.apply_normal(state["x"], state["out"], m0=m0)
        return op.apply(state["x"], state["out"], m0=m0, dagger=case["op"] == "Ddag")
    if fam == "solve":
        mode = {"reliable": D.MIXED_RELIABLE, "adaptive": D.MIXED_ADAPTIVE, "restart": D.MIXED_RESTART}[case["mode"]]
        x, _ = state["op"].solve(state["x"], m0=case["m0"], tol=case["tol"], maxit=20000,
                                 solver=D.BICGSTAB if case["method"] == "bicgstab" else D.CG_NORMAL,
                                 inner_prec=PRECS[case["inner"]], mixed_mode=mode,
                                 sloppy_links=D.LINKS_F32 if case["links"] == "f32" else D.LINKS_NATIVE)
        return x
    if fam == "batch":
        xs, _, _ = D.solve_batched(state["ops"], state["bs"], m0s=state["m0s"], solver=D.CG_NORMAL, tol=case["tol"],
                                   maxit=20000)
        return xs
    if fam == "action":
        S = state["act"](state["U"], state["phi"])
        gU, gphi = torch.autograd.grad(S, (state["U"], state["phi"]))
        return {"S": S.detach(), "gU": gU, "gphi": gphi}
    op = state["op"]   # md
    op.update_links(state["U"])
    chi = op.apply(state["x"], m0=case["m0"])
    return {"chi": chi, "force": op.force(state["x"], chi, D.FORCE_TA)}


# ------------------------------------------------------------------- work
def _flops_per_site(kind, nc):
    """Flops per site and RHS of one apply (App. E of the paper)."""
    n = nc
    return {"wilson": 128 * n * n + 72 * n, "brillouin": 2560 * n * n + 2376 * n, "staggered": 64 * n * n + 2 * n,
            "wlap": 256 * n * n + 8 * n, "blap": 2560 * n * n + 648 * n, "wsuv": 64 * n * n + 2 * n,
            "bsuv": 640 * n * n + 162 * n}[kind]


def _vec_bytes(kind, V, nc, nv, eb):
    return V * nc * (1 if kind in COLOUR_ONLY else 4) * nv * 2 * eb


def _link_bytes(kind, V, nc, eb):
    return V * (80 if kind in USES_W else 4) * nc * nc * 2 * eb


# Krylov iterations these solves take (masses and tolerances of the cases above)
_ITERS = {("wilson", "f32"): 35, ("staggered", "f32"): 130, ("brillouin", "f32"): 10,
          ("wilson", "f64"): 50, ("staggered", "f64"): 140, ("brillouin", "f64"): 17}


def _solve_work(kind, V, nc, nv, eb, iters):
    """One D^dag D per iteration; x, r and p read and written, q written and read."""
    vec, links = _vec_bytes(kind, V, nc, nv, eb), _link_bytes(kind, V, nc, eb)
    return {"bytes": iters * (8 * vec + 2 * links), "flops": iters * 2 * V * nv * _flops_per_site(kind, nc)}


def work(case):
    fam = case["family"]
    if fam == "batch":
        parts = [_solve_work(kind, math.prod(dims), 3, nv, 4, _ITERS[kind, "f32"])
                 for kind, dims, nv, _ in _batch_spec(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    kind, V, nc, nv = case["kind"], math.prod(_shape(case)), case["nc"], case["nv"]
    eb = BYTES[case["prec"]]
    flops = V * nv * _flops_per_site(kind, nc)
    vec = _vec_bytes(kind, V, nc, nv, eb)
    if fam == "apply":
        lb = 4 if case["links"] == "f32" else eb
        clov = V * 4 * nc * nc * 2 * lb if case["csw"] else 0
        if case["csw"]:
            flops += V * nv * 64 * nc * nc
        return {"bytes": 2 * vec + _link_bytes(kind, V, nc, lb) + clov,
                "flops": flops * (2 if case["op"] == "normal" else 1)}
    if fam == "solve":
        ib = BYTES[case["inner"]]
        return _solve_work(kind, V, nc, nv, ib, _ITERS[kind, case["prec"]])
    if fam == "action":   # the forward and the adjoint solve
        w = _solve_work(kind, V, nc, nv, eb, 2 * _ITERS[kind, "f32"])
        return {"bytes": w["bytes"] + 2 * V * 4 * nc * nc * 16, "flops": w["flops"]}
    # md: links in (complex128), D psi, the force out; flops of D, and 36 N_c^2 per link and RHS for the force
    ops = flops + V * nv * 4 * 36 * nc * nc
    if kind in USES_W:
        # every W link from 216 colour products forward, twice that backward, and M_s per offset and RHS
        ops += V * 3 * 216 * 8 * nc ** 3 + V * nv * 80 * 32 * nc * nc
    return {"bytes": V * 4 * nc * nc * 16 + 2 * vec + V * 4 * nc * nc * 2 * eb, "flops": ops}


def tolerance(case):
    """About four times what another order of sums, or of the solver's roundings, was seen to give."""
    fam = case["family"]
    if fam == "apply":
        # one stencil: link and vector rounding at the storage precision
        return {"rel": {"f64": 2e-15, "f32": 1e-6, "bf16": 1e-2, "f16": 2e-3}[case["prec"]],
                "max": {"f64": 1e-13, "f32": 1e-5, "bf16": 6e-2, "f16": 1e-2}[case["prec"]]}
    if fam == "md":
        return {"rel": 1e-14 if case["prec"] == "f64" else 2e-6, "max": 1e-12 if case["prec"] == "f64" else 1e-4}
    if fam == "action":
        return {"rel": 10 * case["tol"], "max": 500 * case["tol"]}
    # solves stop at a relative residual of tol: the solution is uncertain by tol times the root of the condition number
    return {"rel": 30 * case["tol"], "max": 1000 * case["tol"]}


# ------------------------------------------------------------------- exact
_G = np.zeros((4, 4, 4), np.complex128)   # gamma matrices, chiral basis (App. A)
_G[0][0, 3], _G[0][1, 2], _G[0][2, 1], _G[0][3, 0] = -1j, -1j, 1j, 1j
_G[1][0, 3], _G[1][1, 2], _G[1][2, 1], _G[1][3, 0] = -1, 1, 1, -1
_G[2][0, 2], _G[2][1, 3], _G[2][2, 0], _G[2][3, 1] = -1j, 1j, 1j, -1j
_G[3][0, 2], _G[3][1, 3], _G[3][2, 0], _G[3][3, 1] = 1, 1, 1, 1
_RHO = [None, 64 / 432, 16 / 432, 4 / 432, 1 / 432]
_LAM = [-240 / 64, 8 / 64, 4 / 64, 2 / 64, 1 / 64]


def _at(v, s):
    """v(n + s) for an offset s = (sx, sy, sz, st); the site axes lead, t first."""
    ax = [3 - mu for mu in range(4) if s[mu]]
    return torch.roll(v, [-s[mu] for mu in range(4) if s[mu]], ax) if ax else v


def _unit(mu, sign):
    return tuple(sign if nu == mu else 0 for nu in range(4))


def _dagm(M):
    return M.conj().transpose(-1, -2)


def _colour(M, v):
    """(M v)(n): an N_c x N_c field times the colour index of a vector field."""
    flat = v.reshape(v.shape[:5] + (-1,))
    return torch.matmul(M, flat).reshape(v.shape)


def _spin(G, v):
    return torch.einsum("st,...tv->...sv", torch.as_tensor(G, device=v.device), v)


class _Exact:
    """One operator in torch complex128, site-outer order."""

    def __init__(self, kind, U, csw=0.0):
        self.kind = kind
        Up = U.clone()
        for mu in range(4):   # boundary phases on the links that leave the lattice
            if BC[mu] != 1:
                sel = [slice(None)] * 4
                sel[3 - mu] = -1
                Up[tuple(sel) + (mu,)] = BC[mu] * Up[tuple(sel) + (mu,)]
        self.U = Up
        self.W = self._w_links() if kind in USES_W else None
        self.C = self._clover(U, csw) if csw else None

    def hop(self, mu, sign):
        """V_{sign mu}(n): U_mu(n), or U_mu(n - mu)^dag."""
        L = self.U[..., mu, :, :]
        return L if sign > 0 else _dagm(_at(L, _unit(mu, -1)))

    def _w_links(self):
        """W_s(n): the average over the k! orders of the hops to n + s, grouped by the last hop."""
        nc = self.U.shape[-1]
        one = torch.eye(nc, dtype=self.U.dtype, device=self.U.device).expand(self.U.shape[:4] + (nc, nc))
        hops = {(mu, sg): self.hop(mu, sg) for mu in range(4) for sg in (1, -1)}
        W = {(0, 0, 0, 0): one}
        offs = [tuple(int(c) - 1 for c in np.base_repr(i + 81, 3)[1:]) for i in range(81)]
        for s in sorted(offs, key=lambda s: sum(map(abs, s))):
            k = sum(map(abs, s))
            if k:
                acc = 0
                for mu in range(4):
                    if s[mu]:
                        prev = tuple(0 if nu == mu else s[nu] for nu in range(4))
                        acc = acc + _mm(W[prev], _at(hops[mu, s[mu]], prev))
                W[s] = acc / k
        return W

    def _clover(self, V, csw):
        """C(n) = -(c_SW/2) sum_{mu<nu} sigma_mu,nu F_mu,nu(n) as (spin matrix, colour field) pairs."""
        def link(mu, sign, s):
            L = V[..., mu, :, :]
            return _at(L, s) if sign > 0 else _dagm(_at(L, tuple(a + b for a, b in zip(s, _unit(mu, -1)))))

        out = []
        for mu in range(4):
            for nu in range(mu + 1, 4):
                Q = 0
                for (a, sa, b, sb) in ((mu, 1, nu, 1), (nu, 1, mu, -1), (mu, -1, nu, -1), (nu, -1, mu, 1)):
                    z, ea, eb = (0, 0, 0, 0), _unit(a, sa), _unit(b, sb)
                    eab = tuple(p + q for p, q in zip(ea, eb))
                    Q = Q + _mm(_mm(link(a, sa, z), link(b, sb, ea)), _mm(link(a, -sa, eab), link(b, -sb, eb)))
                sigma = 0.5j * (_G[mu] @ _G[nu] - _G[nu] @ _G[mu])
                out.append((-0.5 * csw * sigma, (Q - _dagm(Q)) / 8j))
        return out

    def _eta(self, mu):
        nt, nz, ny, nx = self.U.shape[:4]
        x = [torch.arange(n, device=self.U.device) for n in (nx, ny, nz, nt)]
        e = torch.zeros(nt, nz, ny, nx, dtype=torch.long, device=self.U.device)
        for nu in range(mu):
            e = e + (x[nu] + 1).reshape([-1 if ax == 3 - nu else 1 for ax in range(4)])
        return (1 - 2 * (e % 2)).to(torch.float64)

    def apply(self, v, m, dagger=False):
        k = self.kind
        if dagger and k in ("wilson", "brillouin"):
            g5 = torch.tensor([1.0, 1, -1, -1], dtype=torch.float64, device=v.device)[:, None]
            return g5 * self.apply(g5 * v, m)
        if k == "staggered":
            out = m * v
            for mu in range(4):
                eta = (0.5 if not dagger else -0.5) * self._eta(mu)[..., None, None]
                for sg in (1, -1):
                    out = out + (sg * eta) * _colour(self.hop(mu, sg), _at(v, _unit(mu, sg)))
            return out
        if k in ("wlap", "wsuv"):
            out = (4 + 0.5 * m * m) * v
            for mu in range(4):
                for sg in (1, -1):
                    out = out - 0.5 * _colour(self.hop(mu, sg), _at(v, _unit(mu, sg)))
            return out
        if k in ("blap", "bsuv"):
            out = (0.5 * m * m - 0.5 * _LAM[0]) * v
            for s, W in self.W.items():
                n = sum(map(abs, s))
                if n:
                    out = out - (0.5 * _LAM[n]) * _colour(W, _at(v, s))
            return out
        if k == "wilson":
            out = (4 + m) * v
            for mu in range(4):
                for sg in (1, -1):
                    h = _colour(self.hop(mu, sg), _at(v, _unit(mu, sg)))
                    out = out - 0.5 * _spin(np.eye(4) - sg * _G[mu], h)
        else:
            out = (m - 0.5 * _LAM[0]) * v
            for s, W in self.W.items():
                n = sum(map(abs, s))
                if n:
                    S = _RHO[n] * sum(s[mu] * _G[mu] for mu in range(4)) - 0.5 * _LAM[n] * np.eye(4)
                    out = out + _spin(S, _colour(W, _at(v, s)))
        if self.C is not None:
            for sigma, F in self.C:
                out = out + _spin(sigma, _colour(F, v))
        return out

    def normal(self, v, m):
        if self.kind in ("wlap", "blap", "wsuv", "bsuv"):   # apply_normal: A applied twice
            return self.apply(self.apply(v, m), m)
        return self.apply(self.apply(v, m), m, dagger=True)

    def solve(self, rhs, m, tol=1e-12, maxit=3000):
        """CG on D^dag D x = rhs, one recurrence per right-hand side."""
        dims = tuple(range(rhs.dim() - 1))
        dot = lambda a, b: (a.conj() * b).sum(dims).real  # noqa: E731
        x, r, p = torch.zeros_like(rhs), rhs.clone(), rhs.clone()
        rr, stop = dot(r, r), tol * tol * dot(rhs, rhs)
        for _ in range(maxit):
            if bool((rr <= stop).all()):
                break
            q = self.normal(p, m)
            a = rr / dot(p, q)
            x += a * p
            r -= a * q
            new = dot(r, r)
            p = r + (new / rr) * p
            rr = new
        return x


def _to_layout(v, case):
    """A site-outer result in the operator's own vector order (and as real pairs for 16-bit storage)."""
    if case.get("layout") == "inner":
        n = v.dim()
        v = v.permute(*range(4, n - 1), 0, 1, 2, 3, n - 1)
    return torch.view_as_real(v.contiguous()) if case["prec"] in ("bf16", "f16") else v.contiguous()


def _exact_gradient(kind, U, psi, chi, m):
    """G with dS = Re sum conj(G) dU for dS = -2 Re <chi, dD psi>, by automatic differentiation."""
    Ug = U.detach().clone().requires_grad_(True)
    with torch.enable_grad():
        L = -2.0 * (chi.conj() * _Exact(kind, Ug).apply(psi, m)).sum().real
        G, = torch.autograd.grad(L, Ug)
    return G


@torch.no_grad()
def exact(case, seed):
    fam = case["family"]
    if fam == "batch":
        out = []
        for kind, dims, nv, m0, U, b in _batch_fields(case, seed):
            E, b = _Exact(kind, U), b.to(torch.complex128)
            small = math.prod(dims) * nv <= 131072
            out.append(E.solve(E.apply(b, m0, dagger=True), m0) if small else None)
        return out
    U, b = _fields(case, seed)
    kind, m0 = case["kind"], case["m0"]
    V = math.prod(_shape(case))
    b = _rounded(b.to(torch.complex128), case["prec"])
    if fam == "apply":
        if V * case["nv"] * case["nc"] ** 2 * (10 if kind in USES_W else 1) > 4e8:
            return None
        E = _Exact(kind, U, case["csw"])
        v = E.normal(b, m0) if case["op"] == "normal" else E.apply(b, m0, dagger=case["op"] == "Ddag")
        return _to_layout(v, case)
    if fam == "solve":
        if V * case["nv"] * (20 if kind == "brillouin" else 4 if kind == "wilson" else 1) > 2e6:
            return None
        E = _Exact(kind, U)
        return _to_layout(E.solve(E.apply(b, m0, dagger=True), m0, tol=1e-13), case)
    if fam == "action":
        E = _Exact(kind, U)
        psi = E.solve(b, m0)
        S = (b.conj() * psi).sum().real
        return {"S": S, "gU": _exact_gradient(kind, U, psi, E.apply(psi, m0), m0), "gphi": 2 * psi}
    chi = _Exact(kind, U).apply(b, m0)
    G = _exact_gradient(kind, U, b, chi, m0)
    M = _mm(U, _dagm(G))   # traceless anti-hermitian part of U G^dag
    A = 0.5 * (M - _dagm(M))
    tr = A.diagonal(dim1=-2, dim2=-1).sum(-1) / case["nc"]
    F = A - tr[..., None, None] * torch.eye(case["nc"], dtype=A.dtype, device=A.device)
    return {"chi": _to_layout(chi, case), "force": F}
