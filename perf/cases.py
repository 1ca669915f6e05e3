"""What is timed of this library: calls that its users make, over the range of
sizes, forms, precisions and directions that they make them in.

A program that uses the library keeps one context for the process and creates
an operator for each matrix or gauge field; `prepare` does both and puts the
sources on the GPU, `run` makes one call of a public entry point.

Inputs are drawn on the GPU from the seed alone: links U = exp(i eps H), H a
random traceless Hermitian matrix; complex Gaussian sources; log-spaced shifts
(the recipes of paper_1102_2143_gb300/inputs.py). `exact` restates the
operators and the solves in plain torch, in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1102_2143_gb300 as msc
from paper_1102_2143_gb300 import autograd

DEV = "cuda"
C128 = torch.complex128

# The FP64 true residual that the solves are asked for (tighter than the
# default 1e-10, so that two correct solutions agree to about 1e-10).
TOL = 1e-11


def listed():
    return [
        # The smallest call: A x on a 4^4 lattice inside somebody's own inner
        # loop, queued without waiting; launches and latency are all of it.
        dict(name="apply_queued_4x4", kind="apply", form="queued", L0=4, L1=4, L2=4, L3=4, nc=3, mass=0.1, eps=0.5),
        # An ordinary A x on a lattice whose extents all differ.
        dict(name="apply_10x6x14x18", kind="apply", form="stencil", L0=10, L1=6, L2=14, L3=18, nc=3, mass=0.05, eps=0.7),
        # The largest lattice of the benchmark: A x at 32^4, FP64 (a check of
        # somebody's own solution, one step of somebody's own solver).
        dict(name="apply_32x4", kind="apply", form="stencil", L0=32, L1=32, L2=32, L3=32, nc=3, mass=0.01, eps=0.9),
        # The generic matrix: A x with the 24^4 operator exported as block-CSR.
        dict(name="apply_bsr_24x4", kind="apply", form="bsr", L0=24, L1=24, L2=24, L3=24, nc=3, mass=0.05, eps=0.8),
        # The smallest solve: 4^4, 8 shifts (the correctness workload).
        dict(name="solve_4x4_8shifts", kind="solve", form="stencil", precision="mixed", L0=4, L1=4, L2=4, L3=4, nc=3,
             mass=0.1, eps=0.5, nrhs=1, S=8, lo=1e-3, hi=1.0, tol=TOL),
        # The plain FP64 solve, SU(2), uneven extents, two sources.
        dict(name="solve_fp64_su2", kind="solve", form="stencil", precision="fp64", L0=12, L1=10, L2=14, L3=16, nc=2,
             mass=0.1, eps=0.6, nrhs=2, S=6, lo=1e-3, hi=1.0, tol=TOL),
        # The headline: 24^4 as block-CSR, 15 shifts, one source.
        dict(name="solve_bsr_24x4_15shifts", kind="solve", form="bsr", precision="mixed", L0=24, L1=24, L2=24, L3=24, nc=3,
             mass=0.05, eps=0.8, nrhs=1, S=15, lo=1e-4, hi=10.0, tol=TOL),
        # The largest solve: eight sources x 20 shifts through the stencil
        # (the largest workload's recipe at 24^4 and a heavier mass, so that a
        # pass stays below a second or two).
        dict(name="solve_24x4_8rhs_20shifts", kind="solve", form="stencil", precision="mixed", L0=24, L1=24, L2=24, L3=24,
             nc=3, mass=0.05, eps=0.9, nrhs=8, S=20, lo=1e-4, hi=10.0, tol=TOL),
        # The paper's own test: 2-D Poisson, 15 shifts, generic 1 x 1 blocks.
        dict(name="solve_poisson_1000", kind="poisson", precision="fp64", N=1000, S=15, lo=1e-3, hi=10.0, tol=TOL),
        # Many uneven small systems in one batched call, 4 sources each.
        dict(name="batch_16_uneven", kind="batch", count=16, nrhs=4, Lmax=12, tol=TOL),
        # A non-Hermitian family: the multi-mass staggered Dirac operator by
        # BiCGStab-M.
        dict(name="dirac_16x4_8masses", kind="dirac", L0=16, L1=16, L2=16, L3=16, nc=3, mass=0.2, eps=0.6, nrhs=1, S=8,
             lo=1e-3, hi=1.0, tol=TOL),
        # Forward and backward: the rational action and its gradients with
        # respect to the source and the links, through torch.autograd.
        dict(name="quadform_16x4_12shifts", kind="quadform", L0=16, L1=16, L2=16, L3=16, nc=3, mass=0.05, eps=0.7, S=12,
             lo=1e-4, hi=5.0, tol=TOL),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _extents(rng, vmax, lo=4):
    """Four even extents whose volume is spread over its logarithm, the
    extents themselves uneven."""
    v = _log(rng, lo ** 4, vmax)
    ext = []
    for k in range(4, 0, -1):
        e = v ** (1.0 / k) * (math.exp(rng.uniform(-0.35, 0.35)) if k > 1 else 1.0)
        e = max(lo, 2 * int(e / 2))
        ext.append(e)
        v = max(1.0, v / e)
    while ext[0] * ext[1] * ext[2] * ext[3] > vmax:
        ext[ext.index(max(ext))] -= 2
    return dict(L0=ext[0], L1=ext[1], L2=ext[2], L3=ext[3])


def draw(rng):
    kind = rng.choice(["apply", "apply", "solve", "solve", "poisson", "batch", "dirac", "quadform"])
    nc = rng.choice([2, 3, 3])
    phys = dict(nc=nc, mass=round(rng.uniform(0.05, 0.2), 4), eps=round(rng.uniform(0.4, 0.9), 3))
    if kind == "apply":
        form = rng.choice(["queued", "stencil", "bsr"])
        vmax = {"queued": 349525, "stencil": 32 ** 4, "bsr": 24 ** 4}[form]
        return dict(kind=kind, form=form, **_extents(rng, vmax), **phys)
    if kind == "solve":
        form = rng.choice(["stencil", "stencil", "even", "odd", "bsr"])
        precision = rng.choice(["mixed", "mixed", "fp64"])
        vmax = 24 ** 4 if precision == "mixed" else 16 ** 4
        ext = _extents(rng, vmax)
        v = ext["L0"] * ext["L1"] * ext["L2"] * ext["L3"]
        most = max(1, min(8, 8 * 24 ** 4 // (4 * v))) if form != "bsr" else 2
        return dict(kind=kind, form=form, precision=precision, nrhs=rng.randint(1, most), S=rng.randint(1, 20),
                    lo=1e-3, hi=rng.choice([1.0, 10.0]), tol=TOL, **ext, **phys)
    if kind == "poisson":
        return dict(kind=kind, precision=rng.choice(["mixed", "fp64"]), N=int(_log(rng, 60, 1000)), S=rng.randint(2, 15),
                    lo=1e-3, hi=10.0, tol=TOL)
    if kind == "batch":
        return dict(kind=kind, count=int(_log(rng, 3, 16)), nrhs=rng.randint(1, 4), Lmax=rng.choice([6, 8, 10, 12]), tol=TOL)
    if kind == "dirac":
        phys["mass"] = round(rng.uniform(0.15, 0.4), 4)
        return dict(kind=kind, nrhs=rng.randint(1, 2), S=rng.randint(1, 10), lo=1e-3, hi=1.0, tol=TOL,
                    **_extents(rng, 16 ** 4), **phys)
    return dict(kind=kind, S=rng.randint(2, 12), lo=1e-3, hi=5.0, tol=TOL, **_extents(rng, 16 ** 4), **phys)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------

def _gen(seed, k=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000 * int(seed) + k)
    return g


def _gauss(g, *shape):
    """Complex Gaussian, real and imaginary parts ~ N(0, 1/2)."""
    return torch.complex(torch.randn(shape, generator=g, device=DEV, dtype=torch.float64),
                         torch.randn(shape, generator=g, device=DEV, dtype=torch.float64)) * math.sqrt(0.5)


def _links(g, V, nc, eps):
    """U = exp(i eps H) for 4 V links, H = (G + G^dag)/2 - tr/nc: a Taylor
    series of the argument halved three times, squared back (to rounding)."""
    out = torch.empty(4 * V, nc, nc, device=DEV, dtype=C128)
    eye = torch.eye(nc, device=DEV, dtype=C128)
    step = 1 << 19
    for lo in range(0, 4 * V, step):
        G = _gauss(g, min(step, 4 * V - lo), nc, nc)
        H = 0.5 * (G + G.mH)
        H = H - (torch.diagonal(H, dim1=1, dim2=2).sum(1) / nc)[:, None, None] * eye
        X = (1j * eps / 8) * H
        U = eye + X / 14
        for k in range(13, 0, -1):
            U = eye + _mm(X, U) / k
        for _ in range(3):
            U = _mm(U, U)
        out[lo:lo + len(U)] = U
    return out.reshape(4, V, nc, nc)


def _mm(a, b):
    return (a[:, :, :, None] * b[:, None, :, :]).sum(2)


def _dims(c):
    return (c["L0"], c["L1"], c["L2"], c["L3"])


def _vol(c):
    return c["L0"] * c["L1"] * c["L2"] * c["L3"]


def _shifts(c):
    if c["S"] == 1:
        return np.array([c["lo"]])
    return np.logspace(math.log10(c["lo"]), math.log10(c["hi"]), c["S"])


def _parity_sites(dims, p):
    x = torch.arange(math.prod(dims), device=DEV)
    s, r = torch.zeros_like(x), x
    for L in dims:
        s, r = s + r % L, torch.div(r, L, rounding_mode="floor")
    return torch.nonzero(s % 2 == p).reshape(-1)


def _staggered_inputs(c, seed):
    g = _gen(seed)
    V = _vol(c)
    U = _links(g, V, c["nc"], c["eps"])
    m = V // 2 if c.get("form") in ("even", "odd") else V
    b = _gauss(g, c.get("nrhs", 1), m * c["nc"])
    return U, b


def _batch_sizes(c):
    """The batch's problems: sizes that depend on the case alone."""
    r = np.random.Generator(np.random.PCG64(17 + c["count"]))
    for _ in range(c["count"]):
        L = int(r.choice([v for v in (4, 6, 8, 10, 12) if v <= c["Lmax"]]))
        yield dict(L0=L, L1=L, L2=L, L3=L, nc=int(r.choice([2, 3])), mass=float(r.uniform(0.05, 0.2)), eps=0.6,
                   S=int(r.integers(4, 21)), lo=1e-4, hi=1.0)


def _batch_inputs(c, seed):
    g = _gen(seed)
    return [(q, _links(g, _vol(q), q["nc"], q["eps"]), _gauss(g, c["nrhs"], _vol(q) * q["nc"])) for q in _batch_sizes(c)]


def _hops(dims):
    """Per direction: sites one hop forward and back, and eta / 2."""
    V = math.prod(dims)
    x = torch.arange(V, device=DEV)
    out, stride, par = [], 1, torch.zeros_like(x)
    for L in dims:
        c = torch.div(x, stride, rounding_mode="floor") % L
        out.append((torch.where(c == L - 1, x - (L - 1) * stride, x + stride),
                    torch.where(c == 0, x + (L - 1) * stride, x - stride), 0.5 - (par % 2).double()))
        stride, par = stride * L, par + c
    return out


def _dirac_bsr(U, dims, nc, mass):
    """m + D as block-CSR: 9 blocks a row (columns may repeat on extent 2)."""
    V = math.prod(dims)
    cols, blks = [torch.arange(V, device=DEV)], [(mass * torch.eye(nc, device=DEV, dtype=C128)).expand(V, nc, nc)]
    for mu, (f, b, eta) in enumerate(_hops(dims)):
        cols += [f, b]
        blks += [eta[:, None, None] * U[mu], -eta[:, None, None] * U[mu][b].mH]
    return (torch.arange(V + 1, device=DEV, dtype=torch.int64) * 9,
            torch.stack(cols, 1).to(torch.int32).reshape(-1).contiguous(),
            torch.stack(blks, 1).reshape(-1, nc, nc).resolve_conj().contiguous())


# ----------------------------------------------------------------------------
# the library's side
# ----------------------------------------------------------------------------

class _Op:
    """An operator handle, destroyed with the state that holds it."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        try:
            msc.msc_op_destroy(self.h)
        except Exception:
            pass


_CTX = None


def _ctx():
    """The process's context, ordered against torch's current stream."""
    global _CTX
    if _CTX is None:
        _CTX = msc.msc_create(0, torch.cuda.current_stream())
    return _CTX


def _staggered_op(c, U):
    return _Op(msc.msc_op_staggered(_ctx(), c["nc"], _dims(c), U, c["mass"]))


def _exported(op):
    nbr, nnzb, bd = msc.msc_op_bsr_size(op.h)
    rp = torch.empty(nbr + 1, dtype=torch.int64, device=DEV)
    ci = torch.empty(nnzb, dtype=torch.int32, device=DEV)
    va = torch.empty((nnzb, bd, bd), dtype=C128, device=DEV)
    msc.msc_staggered_export_bsr(_ctx(), op.h, rp, ci, va)
    return _Op(msc.msc_op_bsr(_ctx(), nbr, bd, rp, ci, va))


def prepare(case, seed):
    c = dict(case)
    k = c["kind"]
    torch.cuda.set_device(0)
    if k == "batch":
        return dict(c=c, items=[(_staggered_op(q, U), b, _shifts(q)) for q, U, b in _batch_inputs(c, seed)])
    if k == "poisson":
        N = c["N"]
        rp, ci, va = (torch.from_numpy(a).to(DEV) for a in msc.inputs.poisson_5pt_bsr(N))
        return dict(c=c, op=_Op(msc.msc_op_bsr(_ctx(), N * N, 1, rp, ci, va)), b=_gauss(_gen(seed), 1, N * N),
                    sigma=_shifts(c))
    U, b = _staggered_inputs(c, seed)
    if k == "quadform":
        sig = _shifts(c)
        return dict(c=c, phi=b[0].clone().requires_grad_(True), U=U.requires_grad_(True), sigma=sig,
                    w=sig ** 0.5 / c["S"])
    if k == "dirac":
        rp, ci, va = _dirac_bsr(U, _dims(c), c["nc"], c["mass"])
        return dict(c=c, op=_Op(msc.msc_op_bsr(_ctx(), _vol(c), c["nc"], rp, ci, va)), b=b, sigma=_shifts(c))
    op = _staggered_op(c, U)
    if c["form"] == "bsr":
        op = _exported(op)
    s = dict(c=c, op=op, b=b)
    if k == "apply":
        s["x"], s["out"] = b[0], torch.empty_like(b[0])
    else:
        s["sigma"] = _shifts(c)
    return s


def run(state):
    c = state["c"]
    k = c["kind"]
    if k == "apply":
        if c["form"] == "queued":
            msc.msc_op_apply_noalloc(state["op"].h, 0.01, state["x"], state["out"], torch.cuda.current_stream())
        else:
            msc.msc_op_apply(_ctx(), state["op"].h, 0.01, state["x"], state["out"], msc.MSC_FP64)
        return state["out"]
    if k == "batch":
        xs, _, _ = msc.solve_batched(_ctx(), [(op.h, b, sig) for op, b, sig in state["items"]], tol=c["tol"])
        return xs
    if k == "dirac":
        x, _ = msc.solve_nonherm(_ctx(), state["op"].h, state["b"], state["sigma"], tol=c["tol"])
        return list(x)
    if k == "quadform":
        phi, U = state["phi"], state["U"]
        phi.grad = U.grad = None
        v = autograd.quad_form(phi, U, state["sigma"], state["w"], _dims(c), c["nc"], c["mass"], tol=c["tol"])
        v.backward()
        return v.detach(), phi.grad, U.grad
    prec = msc.MSC_FP64 if c["precision"] == "fp64" else msc.MSC_MIXED
    if c.get("form") in ("even", "odd"):
        x, _ = msc.solve_parity(_ctx(), state["op"].h, int(c["form"] == "odd"), state["b"], state["sigma"], tol=c["tol"],
                                precision=prec)
    else:
        x, _ = msc.solve(_ctx(), state["op"].h, state["b"], state["sigma"], tol=c["tol"], precision=prec)
    return list(x)


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------

def _iterations(lmax, lmin, tol):
    """CG's iterations to a relative residual of tol on [lmin, lmax]."""
    return max(1.0, 0.5 * math.sqrt(lmax / lmin) * math.log(2.0 / tol))


def _solve_work(n, op_bytes, op_flops, nrhs, sigma, d0, lmax, tol, applies=1):
    it = [_iterations(lmax + s, d0 + s, tol) for s in sigma]
    flops = nrhs * (applies * max(it) * (op_flops + 16 * n) + 12.0 * n * sum(it))
    return {"bytes": op_bytes + 16.0 * n * nrhs * (1 + len(sigma)), "flops": flops}


def work(case):
    """Bytes: links or matrix and source once in, results once out. Flops:
    the operator's, times the iterations that CG needs at this condition, and
    the axpys of every shift until it has converged."""
    c = case
    if c["kind"] == "batch":
        ws = [work(dict(q, kind="solve", form="stencil", nrhs=c["nrhs"], tol=c["tol"])) for q in _batch_sizes(c)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    if c["kind"] == "poisson":
        n = c["N"] ** 2
        return _solve_work(n, n * 5 * 20.0, n * 5 * 8.0, 1, _shifts(c), 2 * (math.pi / (c["N"] + 1)) ** 2, 8.0, c["tol"])
    V, nc = _vol(c), c["nc"]
    half = 0.5 if c.get("form") in ("even", "odd") else 1.0
    n = V * nc * half
    links = 4.0 * V * nc * nc * 16
    hop = 8.0 * nc * nc          # flops of one complex nc x nc times vector
    if c["kind"] == "dirac":
        lo = c["mass"] + c["lo"]
        return _solve_work(n, 9.0 * V * (nc * nc * 16 + 4), 9 * V * hop, c["nrhs"], _shifts(c), lo * lo, 8.0, c["tol"], 2)
    if c.get("form") == "bsr":
        op_bytes, op_flops = 33.0 * V * (nc * nc * 16 + 4), 33 * V * hop
    else:
        op_bytes, op_flops = links, 16 * V * hop * half
    if c["kind"] == "apply":
        return {"bytes": op_bytes + 32.0 * n, "flops": op_flops + 8 * n}
    w = _solve_work(n, op_bytes, op_flops, c.get("nrhs", 1), _shifts(c), c["mass"] ** 2, 8.0, c["tol"])
    if c["kind"] == "quadform":
        w["bytes"] = 2 * links + 32.0 * n
        w["flops"] += c["S"] * (8 * V * hop + 4 * V * nc * nc * 16)
    return w


# ----------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ----------------------------------------------------------------------------

class _D:
    """D of the staggered operator on vectors [k][V * nc]."""

    def __init__(self, U, dims, nc):
        self.h, self.nc, self.V = _hops(dims), nc, math.prod(dims)
        self.f = [e[:, None, None] * U[mu] for mu, (_, _, e) in enumerate(self.h)]
        self.b = [-e[:, None, None] * U[mu][b].mH.resolve_conj() for mu, (_, b, e) in enumerate(self.h)]

    def __call__(self, x):
        v = x.reshape(-1, self.V, self.nc)
        y = torch.zeros_like(v)
        for mu, (f, b, _) in enumerate(self.h):
            for to, M in ((f, self.f[mu]), (b, self.b[mu])):
                w = v[:, to]
                for a in range(self.nc):
                    y += w[:, :, a, None] * M[None, :, :, a]
        return y.reshape(x.shape)


def _cgm(A, b, sigma, tol=3e-15):
    """Multi-shift CG for every source of b [k][n]: x [k][S][n]. Shifts above
    the first follow from the first's residual polynomial."""
    k, n = b.shape
    S = len(sigma)
    base = int(np.argmin(sigma))
    rel = torch.tensor(sigma - sigma[base], device=DEV)[None, :]
    x = torch.zeros(k, S, n, device=DEV, dtype=C128)
    ps = b[:, None, :].expand(k, S, n).clone()
    r, p = b.clone(), b.clone()
    one = torch.ones(k, S, device=DEV, dtype=torch.float64)
    z, zp = one.clone(), one.clone()
    R = (r.real ** 2 + r.imag ** 2).sum(1)
    R0, ap, bp = R.clone(), torch.ones_like(R), torch.zeros_like(R)
    for it in range(20000):
        q = A(p) + sigma[base] * p
        a = R / (p.real * q.real + p.imag * q.imag).sum(1)
        den = a[:, None] * bp[:, None] * (zp - z) + zp * ap[:, None] * (1 + rel * a[:, None])
        zn = z * zp * ap[:, None] / den
        zn = torch.where(zn.abs() < 1e-150, torch.zeros_like(zn), zn)
        zr = torch.where(z == 0, torch.zeros_like(z), zn / torch.where(z == 0, one, z))
        x += (a[:, None] * zr)[:, :, None] * ps
        r = r - a[:, None] * q
        Rn = (r.real ** 2 + r.imag ** 2).sum(1)
        be = Rn / R
        ps = zn[:, :, None] * r[:, None, :] + (be[:, None] * zr * zr)[:, :, None] * ps
        p = r + be[:, None] * p
        zp, z, R, ap, bp = torch.where(z == 0, one, z), zn, Rn, a, be
        if it % 10 == 9 and bool((R <= tol * tol * R0).all()):
            break
    return x


def _cost(n, k, S, it):
    """Seconds that _cgm would take, generously."""
    return it * (2e-3 + k * n * (60 + 20 * S) * 1e-12 * 16)


def exact(case, seed):
    c = dict(case)
    k = c["kind"]
    if k == "batch":
        out = []
        for q, U, b in _batch_inputs(c, seed):
            D = _D(U, _dims(q), q["nc"])
            out.append(_cgm(lambda v, D=D, q=q: q["mass"] ** 2 * v - D(D(v)), b, _shifts(q)))
        return out
    if k == "poisson":
        N = c["N"]

        def lap(v):
            u = v.reshape(-1, N, N)
            y = 4 * u
            y[:, 1:] -= u[:, :-1]
            y[:, :-1] -= u[:, 1:]
            y[:, :, 1:] -= u[:, :, :-1]
            y[:, :, :-1] -= u[:, :, 1:]
            return y.reshape(v.shape)
        return list(_cgm(lap, _gauss(_gen(seed), 1, N * N), _shifts(c)))
    U, b = _staggered_inputs(c, seed)
    dims, nc, m = _dims(c), c["nc"], c["mass"]
    D = _D(U, dims, nc)

    def A(v):
        return m * m * v - D(D(v))
    if k == "apply":
        return (A(b) + 0.01 * b)[0]
    sig = _shifts(c)
    V = _vol(c)
    if k == "dirac":
        x = _cgm(lambda v: -D(D(v)), b, (m + sig) ** 2)
        ms = torch.tensor(m + sig, device=DEV)[None, :, None]
        return list(ms * x - torch.stack([D(xk) for xk in x]))
    if k == "quadform":
        x = _cgm(A, b, sig)[0]
        w = torch.tensor(sig ** 0.5 / c["S"], device=DEV)
        val = (w[:, None] * (b.conj() * x).real).sum()
        y = D(x).reshape(-1, V, nc)
        xs = x.reshape(-1, V, nc)
        dU = torch.zeros(4, V, nc, nc, device=DEV, dtype=C128)
        for mu, (f, _, e) in enumerate(D.h):
            for s in range(len(sig)):
                t = xs[s][:, :, None] * y[s][f].conj()[:, None, :] - y[s][:, :, None] * xs[s][f].conj()[:, None, :]
                dU[mu] += (2 * w[s] * e)[:, None, None] * t
        return val, 2 * (w[:, None] * x).sum(0), dU
    if c["form"] in ("even", "odd"):
        at = _parity_sites(dims, int(c["form"] == "odd"))
        full = torch.zeros(b.shape[0], V, nc, device=DEV, dtype=C128)
        full[:, at] = b.reshape(b.shape[0], -1, nc)
        b = full.reshape(b.shape[0], -1)
    out, left = [], 12.0
    for r in range(b.shape[0]):        # the sources that fit the time
        left -= _cost(V * nc, 1, len(sig), _iterations(8.0, m * m + min(sig), 1e-15))
        if left < 0:
            out.append(None)
            continue
        x = _cgm(A, b[r:r + 1], sig)[0]
        if c["form"] in ("even", "odd"):
            x = x.reshape(len(sig), V, nc)[:, at].reshape(len(sig), -1)
        out.append(x)
    return out if any(v is not None for v in out) else None
