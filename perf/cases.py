"""The work a user of this framework has it do: builds of M (first and repeated), the
adjoint of the frozen pattern, products with M and preconditioned solves.

Matrices are the framework's own synthetic problems: upwind convection-diffusion stencils
in 2-D and 3-D (regular, small least-squares problems) and random matrices with power-law
rows (a few dense rows, long uneven least-squares problems), with the parameters of its
configurations, tests and benchmark.
"""
import math

import numpy as np
import torch

from paper_1503_04500_gb300 import autograd, inputs, rsai

DEVICE = "cuda"

# Algorithmic work per column of M, from rsai_get_stats on the listed sizes (QR + solve +
# residual flops, entries of M): stencils at eps = 0.3 and 0.15, power law at c = 5, l_max = 8.
FLOPS_PER_COLUMN = {"2d": 4.8e3, "3d": 2.4e4, "tight": 2.1e5, "power": 3.7e8, "power_small": 4.2e7, "mixed": 8.5e7}
ENTRIES_PER_COLUMN = {"2d": 10, "3d": 15.7, "tight": 30, "power": 92, "power_small": 76, "mixed": 59}
# Entries per column of the caller's own buffers for M (its size depends on the values of A)
ROOM_PER_COLUMN = {"2d": 40, "3d": 40, "tight": 100, "power": 200, "power_small": 200, "mixed": 200}


def _kind(case):
    """The key of a case in the tables above."""
    if case["matrix"] == "power":
        return "power" if case["n"] > 4000 else "power_small"
    return "tight" if case["matrix"] != "mixed" and case["eps"] < 0.3 else case["matrix"]


def listed():
    return [
        # the smallest call: the 20 x 20 problem, built once in FP64 (latency, launches, host set-up)
        {"name": "build_2d_small_fp64", "what": "build", "matrix": "2d", "N": 20, "precision": "fp64",
         "drop": "fixed", "eps": 0.3, "c": 3, "l_max": 10},
        # the benchmark's problem, a first build of a new matrix in FP32 with refinement
        {"name": "build_3d_fp32", "what": "build", "matrix": "3d", "N": 64, "precision": "fp32_refine",
         "drop": "fixed", "eps": 0.3, "c": 3, "l_max": 10},
        # the same problem in FP64, rebuilt on its structure with new coefficients (a time step)
        {"name": "rebuild_3d_fp64", "what": "rebuild", "matrix": "3d", "N": 64, "precision": "fp64",
         "drop": "fixed", "eps": 0.3, "c": 3, "l_max": 10},
        # a 2-D problem rebuilt with new coefficients in FP32 with refinement
        {"name": "rebuild_2d_fp32", "what": "rebuild", "matrix": "2d", "N": 256, "precision": "fp32_refine",
         "drop": "fixed", "eps": 0.3, "c": 3, "l_max": 10},
        # a better preconditioner: small eps, many loops, the paper's adaptive drop; an odd size
        {"name": "build_3d_tight_fp32", "what": "build", "matrix": "3d", "N": 33, "precision": "fp32_refine",
         "drop": "adaptive", "eps": 0.15, "c": 3, "l_max": 15},
        # row-irregular matrix (circuit, power grid): hundreds of columns per problem
        {"name": "build_power_fp32", "what": "build", "matrix": "power", "n": 12000, "precision": "fp32_refine",
         "drop": "fixed", "eps": 0.4, "c": 5, "l_max": 8},
        # the same kind in FP64, small and of odd size
        {"name": "build_power_fp64", "what": "build", "matrix": "power", "n": 1111, "precision": "fp64",
         "drop": "fixed", "eps": 0.4, "c": 5, "l_max": 8},
        # many small systems of both kinds at once, with the gradient of a loss: one training pass
        {"name": "batch_grad_fp32", "what": "batch", "matrix": "mixed", "members": 8, "nmin": 600, "nmax": 2400,
         "precision": "fp32_refine", "drop": "fixed", "eps": 0.3, "c": 3, "l_max": 10},
        # differentiable refit of the 256 x 256 parametric problem, forward and backward
        {"name": "grad_2d_fp32", "what": "grad", "matrix": "2d", "N": 256, "precision": "fp32_refine",
         "drop": "fixed", "eps": 0.3, "c": 3, "l_max": 10},
        # the same in 3-D and FP64
        {"name": "grad_3d_fp64", "what": "grad", "matrix": "3d", "N": 40, "precision": "fp64",
         "drop": "fixed", "eps": 0.3, "c": 3, "l_max": 10},
        # M in use: one application y = M x ...
        {"name": "apply_3d", "what": "apply", "matrix": "3d", "N": 64, "precision": "fp32_refine",
         "drop": "fixed", "eps": 0.3, "c": 3, "l_max": 10},
        # ... and a whole preconditioned BiCGStab solve to 1e-8
        {"name": "solve_3d", "what": "solve", "matrix": "3d", "N": 64, "precision": "fp32_refine",
         "drop": "fixed", "eps": 0.3, "c": 3, "l_max": 10},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["build", "build", "rebuild", "grad", "solve", "apply", "power", "batch"])
    precision = rng.choice(["fp32_refine", "fp64"])
    case = {"what": what, "precision": precision, "drop": "fixed", "eps": 0.3, "c": 3, "l_max": 10}
    if what == "power":
        top = 9000 if precision == "fp32_refine" else 1100
        case.update(what="build", matrix="power", n=_log_int(rng, 500, top), eps=0.4, c=5, l_max=8)
    elif what == "batch":
        lo = _log_int(rng, 200, 600)
        case.update(matrix="mixed", members=rng.randrange(2, 9), nmin=lo, nmax=lo * rng.randrange(2, 4),
                    precision="fp32_refine")
    else:
        dim = rng.choice(["2d", "3d"])
        case.update(matrix=dim, N=_log_int(rng, 12, 400) if dim == "2d" else _log_int(rng, 6, 60),
                    drop=rng.choice(["fixed", "adaptive"]))
        if what == "build" and rng.random() < 0.5:
            case.update(N=min(case["N"], 150 if dim == "2d" else 30), eps=round(rng.uniform(0.15, 0.3), 3), l_max=15)
    return case


# ---------------------------------------------------------------------------
# inputs


class _Rng:
    """Two generators of one seed: numpy's for a few scalars, torch's on the device for vectors."""

    def __init__(self, seed, device):
        self.host = np.random.default_rng(seed)
        self.dev = torch.Generator(device=device).manual_seed(seed)
        self.device = device

    def normal(self, n):
        return torch.randn(n, generator=self.dev, dtype=torch.float64, device=self.device)


def _beta(rng, dim, N):
    """A random flow direction at cell Peclet number 5 (the benchmark's)."""
    d = rng.uniform(0.2, 1.0, dim) * rng.choice([-1.0, 1.0], dim)
    return 2.0 * 5.0 * (N + 1) * d / np.abs(d).max()


def _stencil(dim, N, beta, device):
    """Upwind convection-diffusion on an N^dim grid (-Laplace + beta . grad, zero boundary),
    in CSR and CSC, built on the device: the problem of inputs.convdiff2d / convdiff3d."""
    h = 1.0 / (N + 1)
    n = N**dim
    idx = torch.arange(n, device=device)
    offs, coef, ok = [], [], []
    for a in list(range(dim))[::-1]:  # lower neighbours, farthest first
        offs.append(-(N**a))
        coef.append(-1.0 / h**2 - max(float(beta[a]), 0.0) / h)
        ok.append((idx // N**a) % N > 0)
    offs.append(0)
    coef.append(2.0 * dim / h**2 + float(np.abs(beta).sum()) / h)
    ok.append(torch.ones(n, dtype=torch.bool, device=device))
    for a in range(dim):
        offs.append(N**a)
        coef.append(-1.0 / h**2 - max(-float(beta[a]), 0.0) / h)
        ok.append((idx // N**a) % N < N - 1)
    off = torch.tensor(offs, device=device)
    cof = torch.tensor(coef, dtype=torch.float64, device=device)
    ok = torch.stack(ok, 1)
    ptr = torch.zeros(n + 1, dtype=torch.int64, device=device)
    ptr[1:] = ok.sum(1).cumsum(0)
    nbr = (idx[:, None] + off)[ok].to(torch.int32)
    val = cof.expand(n, -1)[ok].contiguous()
    # column j holds A(j + o, j): the coefficient of offset -o
    cval = cof.flip(0).expand(n, -1)[ok].contiguous()
    return rsai.DeviceMatrix(n, int(val.numel()), ptr, nbr, val, ptr.clone(), nbr.clone(), cval)


def _power(n, rng, device):
    """inputs.powerlaw's matrix of n rows: its structure, and the seed's values on it."""
    H = inputs.powerlaw(n, seed=1503 + n)
    row = np.repeat(np.arange(n), np.diff(H.row_ptr))
    val = rng.host.standard_normal(H.nnz)
    val[row == H.col_idx] = 0.0
    diag = 1.1 * np.bincount(row, weights=np.abs(val), minlength=n) * rng.host.choice([-1.0, 1.0], n)
    val[row == H.col_idx] = diag
    return rsai.DeviceMatrix.from_host(H.with_values(val), device=device)


def _matrix(case, rng, device=None):
    device = device or DEVICE
    if case["matrix"] == "power":
        return _power(case["n"], rng, device)
    dim = 2 if case["matrix"] == "2d" else 3
    return _stencil(dim, case["N"], _beta(rng.host, dim, case["N"]), device)


def _members(case, rng, device=None):
    """Half power law, a quarter each 2-D and 3-D stencils, sizes spread over [nmin, nmax]."""
    device = device or DEVICE
    out = []
    for b in range(case["members"]):
        n = round(case["nmin"] + (case["nmax"] - case["nmin"]) * ((0.35 + 0.618034 * b) % 1.0))
        if b % 2 == 0:
            out.append(_power(n, rng, device))
        else:
            dim = 2 if b % 4 == 1 else 3
            N = round(n ** (1.0 / dim))
            out.append(_stencil(dim, N, _beta(rng.host, dim, N), device))
    return out


def _keywords(case):
    return dict(c=case["c"], l_max=case["l_max"], eps=case["eps"], drop=case["drop"], tol=1e-3,
                precision=case["precision"])


def prepare(case, seed):
    rng = _Rng(seed, DEVICE)
    kw = _keywords(case)
    what = case["what"]
    state = {"what": what, "kw": kw}

    def room(n):
        most = n * ROOM_PER_COLUMN[_kind(case)]
        state["col_idx"] = torch.zeros(most, dtype=torch.int32, device=DEVICE)
        state["val_M"] = torch.zeros(most, dtype=torch.float64, device=DEVICE)

    if what == "batch":
        state["members"] = _members(case, rng)
        room(sum(A.n for A in state["members"]))
        state["A_val"] = torch.cat([A.val for A in state["members"]])
        state["g_rho2"] = rng.normal(sum(A.n for A in state["members"]))
        return state
    A = _matrix(case, rng)
    state["A"] = A
    room(A.n)
    if what == "build":
        return state
    state["h"] = h = rsai.build(A, **kw)
    if what == "rebuild":
        state["val"] = _matrix(case, rng).val  # another flow on the same grid
    elif what == "grad":
        state["A_val"] = A.val.clone().requires_grad_(True)
        state["g_M"] = rng.normal(h.stats()["nnz_M"])
        state["g_rho2"] = rng.normal(A.n)
    else:
        state["x"] = rng.normal(A.n)
    return state


# ---------------------------------------------------------------------------
# one pass


def _keep(buffer, values):
    """Values into the caller's own buffer, which has room for more."""
    buffer[: values.numel()] = values
    return buffer


def _built(h, state):
    """M and its columns' residuals, read out as a program does that keeps M in its own buffers."""
    rho, loops, flags = h.columns()
    row_ptr, col_idx, val = h.M()
    state["M_val"] = val
    return {"row_ptr": row_ptr, "col_idx": _keep(state["col_idx"], col_idx), "val": _keep(state["val_M"], val),
            "rho": rho, "loops": loops, "flags": flags}


def run(state):
    what = state["what"]
    if what == "build":
        return _built(rsai.build(state["A"], **state["kw"]), state)
    if what == "rebuild":
        h = state["h"]
        h.set_values(state["val"])
        h.rebuild()
        return _built(h, state)
    if what == "batch":
        h = rsai.build_batch(state["members"], **state["kw"])
        out = _built(h, state)
        # loss = sum_k g_k ||r_k||^2 + |M|^2 / 2
        out["grad"] = h.backward(state["A_val"], state["M_val"], state["g_rho2"])
        return out
    if what == "grad":
        M_val, rho2 = autograd.frozen_rsai(state["A_val"], state["h"])
        (grad,) = torch.autograd.grad((M_val, rho2), state["A_val"], (state["g_M"], state["g_rho2"]))
        return {"val": _keep(state["val_M"], M_val.detach()), "rho2": rho2.detach(), "grad": grad}
    if what == "apply":
        return state["h"].apply(state["x"])
    x, iters, relres, status = rsai.bicgstab(state["A"], state["h"], state["x"])
    return {"x": x, "iters": iters, "status": status}


# ---------------------------------------------------------------------------
# what a pass cannot do without


def work(case):
    kind = _kind(case)
    if kind == "mixed":
        n = case["members"] * 0.5 * (case["nmin"] + case["nmax"])
    else:
        n = case["n"] if case["matrix"] == "power" else case["N"] ** (2 if case["matrix"] == "2d" else 3)
    nnz = n * {"2d": 5, "3d": 7, "power": 7.8, "mixed": 7}[case["matrix"]]
    entries, flops = n * ENTRIES_PER_COLUMN[kind], n * FLOPS_PER_COLUMN[kind]
    matrix, m_csr = 2 * (12.0 * nnz + 8 * n), 12.0 * entries + 8 * n
    what = case["what"]
    if what == "apply":
        return {"bytes": m_csr + 16.0 * n, "flops": 2.0 * entries}
    if what == "solve":  # about 15 iterations of two products with A and two with M, once each from memory
        return {"bytes": 12.0 * nnz + 8 * n + m_csr + 16.0 * n, "flops": 15 * 4.0 * (nnz + entries)}
    if what == "grad":  # values in, M and rho out; M's and rho's gradients in, A's gradient out
        return {"bytes": matrix + 12.0 * entries + 16.0 * entries + 24.0 * n + 8.0 * nnz, "flops": flops}
    out = m_csr + 16.0 * n
    if what == "batch":
        return {"bytes": matrix + out + 16.0 * nnz, "flops": 1.25 * flops}
    return {"bytes": matrix + out, "flops": flops}


# ---------------------------------------------------------------------------
# the same results in 64 bits, in plain torch: every column of M at once, in padded arrays


def _ell(ptr, idx, val, n):
    """Rows of a compressed matrix as padded [n + 1, W] arrays (index n = padding)."""
    length = ptr[1:] - ptr[:-1]
    W = int(length.max())
    at = ptr[:-1, None] + torch.arange(W, device=ptr.device)
    have = torch.arange(W, device=ptr.device) < length[:, None]
    at = torch.where(have, at, 0)
    i = torch.full((n + 1, W), n, dtype=torch.int64, device=ptr.device)
    v = torch.zeros((n + 1, W), dtype=torch.float64, device=ptr.device)
    e = torch.full((n + 1, W), -1, dtype=torch.int64, device=ptr.device)
    i[:n] = torch.where(have, idx[at].long(), n)
    v[:n] = torch.where(have, val[at], 0.0)
    e[:n] = torch.where(have, at, -1)
    return i, v, e


def _sorted_set(x, pad):
    """Rows of x as sorted sets, padded on the right and cut to the widest."""
    x = x.sort(1).values
    x[:, 1:] = torch.where(x[:, 1:] == x[:, :-1], pad, x[:, 1:])
    x = x.sort(1).values
    return x[:, : max(1, int((x < pad).sum(1).max()))].contiguous()


class _Exact:
    """RSAI(tol) in 64 bits: Algorithm 1 with the drop rule of Eq. 4.3, batched over columns."""

    def __init__(self, A, case):
        self.A, self.n, self.case = A, A.n, case
        self.rc, self.rv, _ = _ell(A.row_ptr, A.col_idx, A.val, A.n)
        self.cr, self.cv, self.ce = _ell(A.col_ptr, A.row_idx, A.cval, A.n)
        self.norm1 = float(self.cv.abs().sum(1).max())

    def gather(self, k, J):
        """I (with k) and B = A(I, J), padded with zero rows and columns."""
        m, P = J.shape
        rows, vals = self.cr[J].reshape(m, -1), self.cv[J].reshape(m, -1)
        I = _sorted_set(torch.cat([rows, k[:, None]], 1), self.n)
        at = torch.searchsorted(I, rows).clamp_(max=I.shape[1] - 1)
        col = torch.arange(P, device=J.device).repeat_interleave(self.cr.shape[1])
        B = torch.zeros(m, I.shape[1] * P, dtype=torch.float64, device=J.device)
        B.scatter_add_(1, at * P + col, vals)
        return I, B.view(m, I.shape[1], P)

    @staticmethod
    def factor(B, rhs):
        """Householder QR of every B applied to rhs (in place); returns R."""
        B = B.clone()
        for j in range(min(B.shape[2], B.shape[1])):
            v = B[:, j:, j].clone()
            s = v.square().sum(1).sqrt()
            v[:, 0] += torch.where(v[:, 0] >= 0, s, -s)
            vv = v.square().sum(1)
            f = torch.where(vv > 0, 2.0 / torch.where(vv > 0, vv, 1.0), 0.0)
            B[:, j:, j:] -= (f[:, None] * v)[:, :, None] * (v[:, None, :] @ B[:, j:, j:])
            rhs[:, j:] -= (f * (v * rhs[:, j:]).sum(1))[:, None] * v
        P = B.shape[2]
        if B.shape[1] < P:
            B = torch.cat([B, B.new_zeros(B.shape[0], P - B.shape[1], P)], 1)
        return B[:, :P].triu()

    @staticmethod
    def triangular(R, b, lower):
        """R x = b or R^T x = b; padded columns (zero diagonal) give 0."""
        d = torch.diagonal(R, dim1=1, dim2=2)
        R = R + torch.diag_embed((d == 0).double())
        x = torch.linalg.solve_triangular(R.mT if lower else R, b[:, :, None], upper=not lower)[:, :, 0]
        return torch.where(d == 0, 0.0, x)

    def solve(self, k, J):
        I, B = self.gather(k, J)
        e = (I == k[:, None]).double()
        b = e.clone()
        R = self.factor(B, b)
        P = J.shape[1]
        b = torch.cat([b, b.new_zeros(b.shape[0], max(0, P - b.shape[1]))], 1)[:, :P]
        m = self.triangular(R, b, False)
        return m, I, (B @ m[:, :, None])[:, :, 0] - e, B, R

    def solve_drop(self, k, J):
        c = self.case
        m, I, r, _, _ = self.solve(k, J)
        valid = J < self.n
        p = valid.sum(1)
        tau = c["eps"] / (p * self.norm1) if c["drop"] == "adaptive" else torch.full_like(r[:, 0], 1e-3 / self.norm1)
        keep = valid & (m.abs() > tau[:, None])
        none = ~keep.any(1)
        keep[none, torch.where(valid, m.abs(), -1.0).argmax(1)[none]] = True
        again = keep.sum(1) < p
        if not again.any():
            return J, m, I, r
        J = torch.where(keep, J, self.n).sort(1).values
        a = again.nonzero()[:, 0]
        J2 = J[a][:, : int((J[a] < self.n).sum(1).max())].contiguous()
        m2, I2, r2, _, _ = self.solve(k[a], J2)
        m[a], I[a], r[a] = 0.0, self.n, 0.0
        m[a, : J2.shape[1]] = m2
        I[a[:, None], torch.arange(I2.shape[1], device=k.device)] = I2
        r[a[:, None], torch.arange(I2.shape[1], device=k.device)] = r2
        return J, m, I, r

    def columns(self, k):
        """(J, m, rho, loops) of the columns k, padded."""
        c, n, dev = self.case["c"], self.n, k.device
        total, done = k.numel(), []
        own = torch.arange(total, device=dev)
        J, m, I, r = self.solve_drop(k, k[:, None].clone())
        used = torch.full((total, 1), n, dtype=torch.int64, device=dev)
        loops = torch.zeros(total, dtype=torch.int64, device=dev)
        while own.numel():
            rho = r.square().sum(1).sqrt()
            a = r.abs()
            band = 1e-12 * a.max(1, keepdim=True).values
            cand = (a > band) & (I < n) & ~(I[:, :, None] == used[:, None, :]).any(2)
            go = (rho > self.case["eps"]) & (loops < self.case["l_max"]) & cand.any(1)
            if not go.all():
                s = ~go
                done.append((own[s], J[s], m[s], rho[s], loops[s]))
                own, k, J, m, I, r, used, loops, a, band, cand = (
                    t[go] for t in (own, k, J, m, I, r, used, loops, a, band, cand))
            if not own.numel():
                break
            top = torch.where(cand, a, -1.0)
            v = top.topk(min(c, top.shape[1]), 1).values[:, -1:]
            few = cand.sum(1, keepdim=True) <= c
            above = cand & (a > v + band)
            tie = cand & (a >= v - band) & (a <= v + band)
            sel = torch.where(few, cand, above | (tie & (tie.cumsum(1) <= c - above.sum(1, keepdim=True))))
            rows = torch.where(sel, I, n)
            rows = rows.sort(1).values[:, : int(sel.sum(1).max())]
            used = torch.cat([used, rows], 1)
            loops = loops + 1
            new = _sorted_set(torch.cat([J, self.rc[rows].reshape(own.numel(), -1)], 1), n)
            grown = (new < n).sum(1) > (J < n).sum(1)
            if grown.any():
                g = grown.nonzero()[:, 0]
                Jg, mg, Ig, rg = self.solve_drop(k[g], new[g])

                def put(old, part, fill):
                    w = max(old.shape[1], part.shape[1])
                    out = torch.full((old.shape[0], w), fill, dtype=old.dtype, device=dev)
                    out[:, : old.shape[1]] = old
                    out[g] = fill
                    out[g[:, None], torch.arange(part.shape[1], device=dev)] = part
                    return out

                J, m, I, r = put(J, Jg, n), put(m, mg, 0.0), put(I, Ig, n), put(r, rg, 0.0)
        return done

    def chunks(self, size=16384):
        for k0 in range(0, self.n, size):
            yield torch.arange(k0, min(self.n, k0 + size), device=self.rc.device)

    def build(self):
        """M (row_ptr, col_idx, val), rho, loops and, per column, its padded J."""
        n, dev = self.n, self.rc.device
        rho = torch.zeros(n, dtype=torch.float64, device=dev)
        loops = torch.zeros(n, dtype=torch.int32, device=dev)
        rows, cols, vals, self.J = [], [], [], []
        for k in self.chunks():
            for own, J, m, rh, lo in self.columns(k):
                kk = k[own]
                rho[kk], loops[kk] = rh, lo.to(torch.int32)
                have = J < n
                rows.append(J[have])
                cols.append(kk[:, None].expand_as(J)[have])
                vals.append(m[have])
                self.J.append((kk, J[:, : max(1, int(have.sum(1).max()))].contiguous()))
        rows, cols, vals = torch.cat(rows), torch.cat(cols), torch.cat(vals)
        self.key, order = (rows * n + cols).sort()
        ptr = torch.zeros(n + 1, dtype=torch.int64, device=dev)
        ptr[1:] = torch.bincount(rows, minlength=n).cumsum(0)
        return ptr, cols[order].to(torch.int32), vals[order], rho, loops

    def grad(self, g_M, g_rho2):
        """d(<g_M, M> + <g_rho2, rho^2>) / d(values of A, CSR order) on the built pattern."""
        n, A = self.n, self.A
        rows = torch.repeat_interleave(torch.arange(n, device=self.rc.device), A.row_ptr[1:] - A.row_ptr[:-1])
        key = rows * n + A.col_idx.long()
        out = torch.zeros(A.nnz, dtype=torch.float64, device=self.rc.device)
        for kk, J in self.J:
            for k, J in zip(kk.split(16384), J.split(16384)):
                m, I, r, B, R = self.solve(k, J)
                have = J < n
                at = torch.searchsorted(self.key, torch.where(have, J, 0) * n + k[:, None]).clamp_(max=self.key.numel() - 1)
                G = torch.where(have, g_M[at], 0.0)
                z = self.triangular(R, self.triangular(R, G, True), False)
                w = (B @ z[:, :, None])[:, :, 0]
                alpha = 2.0 * g_rho2[k][:, None] * m - z
                D = r[:, :, None] * alpha[:, None, :] - w[:, :, None] * m[:, None, :]
                # entries (i, j) of column j of A, at the position of i in I
                i = self.cr[J]
                pos = torch.searchsorted(I, i.reshape(k.numel(), -1)).clamp_(max=I.shape[1] - 1).view(i.shape)
                d = torch.gather(D.transpose(1, 2), 2, pos)
                ok = i < n
                e = torch.searchsorted(key, (i * n + J[:, :, None])[ok])
                out.index_add_(0, e, d[ok])
        return out


def _spmv(ptr, idx, val, x):
    row = torch.repeat_interleave(torch.arange(ptr.numel() - 1, device=x.device), ptr[1:] - ptr[:-1])
    return torch.zeros(ptr.numel() - 1, dtype=torch.float64, device=x.device).index_add_(0, row, val * x[idx.long()])


def exact(case, seed, device=None):
    """What run returns, from plain 64-bit torch; None for the power-law and mixed cases, whose
    thousands of problems of hundreds of columns would take minutes this way."""
    if case["matrix"] in ("power", "mixed"):
        return None
    device = device or DEVICE
    rng = _Rng(seed, device)
    A = _matrix(case, rng, device)
    what = case["what"]
    if what == "rebuild":
        A = _matrix(case, rng, device)
    E = _Exact(A, case)
    ptr, idx, val, rho, loops = E.build()

    def room(v):
        return torch.cat([v, v.new_zeros(A.n * ROOM_PER_COLUMN[_kind(case)] - v.numel())])

    if what in ("build", "rebuild"):
        return {"row_ptr": ptr, "col_idx": room(idx), "val": room(val), "rho": rho, "loops": loops, "flags": None}
    if what == "grad":
        g_M = rng.normal(int(val.numel()))
        g_rho2 = rng.normal(A.n)
        return {"val": room(val), "rho2": rho.square(), "grad": E.grad(g_M, g_rho2)}
    b = rng.normal(A.n)
    if what == "apply":
        return _spmv(ptr, idx, val, b)
    # the solution itself: the solve stops at a residual of 1e-8, so run's x is near it only to
    # that; no value to hold x to
    return None
