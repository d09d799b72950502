"""Performance cases of the dual-system solver: what a user has it do, through its public entry points.

A case is one program step around a handle (``D3M`` or ``D3MBatch``), on one of the domain grids
this repository uses:

* ``step``  -- factor K, then solve K X = B with refinement (a new frequency or new material: K changes
  every time, so the factorization counts on every pass);
* ``solve`` -- solve only, against a factorization the program keeps (many excitations of one structure);
* ``grad``  -- factor, solve, adjoint solve, dJ/deps per domain and dJ/dK on the stored pattern (one
  gradient evaluation of an inverse-design loop);
* ``batch`` -- many uneven systems held in one batched handle, factored and solved together (a frequency
  sweep, or a population of designs).

K is assembled as in the repository's workloads: M_i = G_i G_i^T - k^2 I + i tau I per domain, added into
the blocks of its interfaces, with G complex normal, cols = rows = unknowns of the domain's interfaces.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2002_05026_gb300 import D3M, D3MBatch, d3m_order_grid_nd
from paper_2002_05026_gb300._abi import d3m_analyze

DEVICE = "cuda"


# ------------------------------------------------------------------------------ the cases
def _case(kind, nx, ny, nz, m, nrhs, precision, k2, tau, ragged=False, host=False, pivot=False, count=1):
    return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "m": m, "nrhs": nrhs, "precision": precision, "k2": k2,
            "tau": tau, "ragged": ragged, "host": host, "pivot": pivot, "count": count}


def listed():
    return [
        # the smallest system one factors and solves: four interfaces, one right-hand side; launches and
        # waits are all of it (the repository's grid2x2_m64)
        dict(_case("step", 2, 2, 1, 64, 1, "bf16x3", 1.0, 0.1), name="tiny_2x2_m64"),
        # the ordinary planar problem with the default engine (grid8x8_m512): a long chain of separators
        dict(_case("step", 8, 8, 1, 512, 8, "bf16x3", 2.0, 0.05), name="planar_8x8_m512"),
        # the largest: a 3-D grid with 32 right-hand sides on the TF32 engine (grid6x6x6_m512's recipe at a
        # size of which three fit on one card)
        dict(_case("step", 5, 5, 4, 512, 32, "tf32", 4.0, 0.02), name="cube_5x5x4_m512_tf32"),
        # interfaces of uneven and odd sizes (a real mesh), 3-D, default engine, an odd number of columns
        dict(_case("step", 3, 3, 3, 300, 11, "bf16x3", 2.0, 0.05, ragged=True), name="ragged_3x3x3"),
        # many excitations against one kept factorization: solves without a factorization
        dict(_case("solve", 5, 5, 3, 256, 32, "bf16x3", 2.0, 0.05), name="resolve_5x5x3_m256"),
        # one gradient evaluation of an inverse-design loop (adjoint8x8_m256)
        dict(_case("grad", 8, 8, 1, 256, 1, "bf16x3", 2.0, 0.05), name="gradient_8x8_m256"),
        # a batch of uneven instances (batch256's recipe, 64 of them), default engine
        dict(_case("batch", 0, 0, 0, 256, 4, "bf16x3", 0.0, 0.0, count=64), name="batch64_bf16x3"),
        # a batch of small interfaces only, on the engine the autotuner has for them
        dict(_case("batch", 0, 0, 0, 64, 4, "simt32", 0.0, 0.0, count=32), name="batch32_m64_simt32"),
        # the plain FP64 path at an ordinary size (grid4x4_m512)
        dict(_case("step", 4, 4, 1, 512, 8, "fp64", 2.0, 0.05), name="fp64_4x4_m512"),
        # the plain FP64 path, small and odd
        dict(_case("step", 3, 3, 1, 100, 3, "fp64", 1.0, 0.1), name="fp64_3x3_m100"),
        # end to end from page-locked host memory: K and B up, X back (grid4x4_m512)
        dict(_case("step", 4, 4, 1, 512, 8, "bf16x3", 2.0, 0.05, host=True), name="host_4x4_m512"),
        # pivoting inside the diagonal tiles (FP64), on a K with vanishing diagonal entries
        dict(_case("step", 3, 3, 1, 64, 2, "fp64", 1.0, 0.1, pivot=True), name="pivot_3x3_m64"),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    k2, tau = round(rng.uniform(1.0, 4.0), 3), round(rng.uniform(0.02, 0.2), 3)

    def engine(*names):
        # the TF32 engine is for systems whose unpivoted factor its 11 bits can carry: away from small k^2
        p = rng.choice(names)
        return p, (round(3.0 + k2 / 4.0, 3) if p == "tf32" else k2)

    kind = rng.choice(["planar", "planar", "cube", "solve", "grad", "batch", "simt32", "fp64", "host", "pivot"])
    if kind in ("planar", "host"):
        p, k = engine("bf16x3", "bf16x3", "tf32")
        return _case("step", rng.randint(2, 8), rng.randint(2, 8), 1, logint(48, 512), logint(1, 32), p, k, tau,
                     ragged=rng.random() < 0.4, host=kind == "host")
    if kind == "cube":
        p, k = engine("bf16x3", "tf32", "tf32")
        return _case("step", rng.randint(2, 4), rng.randint(2, 4), rng.randint(2, 4), logint(64, 512), logint(4, 32),
                     p, k, tau, ragged=rng.random() < 0.3)
    if kind == "solve":
        p, k = engine("bf16x3", "tf32", "fp64")
        return _case("solve", rng.randint(2, 5), rng.randint(2, 5), rng.randint(1, 3), logint(64, 384), logint(1, 32),
                     p, k, tau, ragged=rng.random() < 0.3)
    if kind == "grad":
        return _case("grad", rng.randint(2, 8), rng.randint(2, 8), 1, logint(64, 320), logint(1, 8), "bf16x3", k2, tau)
    if kind == "batch":
        return _case("batch", 0, 0, 0, 256, logint(1, 8), "bf16x3", 0.0, 0.0, count=rng.randint(8, 64))
    if kind == "simt32":
        return _case("batch", 0, 0, 0, 64, logint(1, 8), "simt32", 0.0, 0.0, count=rng.randint(8, 64))
    if kind == "fp64":
        return _case("step", rng.randint(2, 4), rng.randint(2, 4), 1, logint(32, 512), logint(1, 16), "fp64", k2, tau,
                     ragged=rng.random() < 0.4)
    # interfaces of one tile: the pivoting is confined to diagonal tiles
    return _case("step", rng.randint(2, 4), rng.randint(2, 4), 1, logint(16, 64), logint(1, 8),
                 rng.choice(["fp64", "simt32"]), k2, tau, pivot=True)


# ------------------------------------------------------------------------------ grids
def _interfaces(nx, ny, nz):
    """(domain, neighbour) of every interface: domain order, then axis x, y, z."""
    out = []
    for ix in range(nx):
        for iy in range(ny):
            for iz in range(nz):
                d = (ix * ny + iy) * nz + iz
                if ix + 1 < nx:
                    out.append((d, d + ny * nz))
                if iy + 1 < ny:
                    out.append((d, d + nz))
                if iz + 1 < nz:
                    out.append((d, d + 1))
    return out


def _domains(nx, ny, nz):
    lists = [[] for _ in range(nx * ny * nz)]
    for f, (d, e) in enumerate(_interfaces(nx, ny, nz)):
        lists[d].append(f)
        lists[e].append(f)
    return [sorted(l) for l in lists]


class _System:
    """Grid, block sizes and stored lower pattern of one K."""

    def __init__(self, nx, ny, nz, m, k2, tau, ragged=False, zeros=False):
        self.grid, self.k2, self.tau, self.zeros = (nx, ny, nz), k2, tau, zeros
        self.dom = _domains(nx, ny, nz)
        nf = len(_interfaces(nx, ny, nz))
        if ragged:   # sizes between a quarter of m and m, the same for every seed: the mesh is the program's
            g = np.random.RandomState(nf * 1009 + m)
            self.size = [int(v) for v in g.randint(max(1, m // 4), m + 1, nf)]
        else:
            self.size = [m] * nf
        cols = [{g} for g in range(nf)]
        for I in self.dom:
            for a in I:
                for b in I:
                    if a >= b:
                        cols[b].add(a)
        self.rows = [sorted(c) for c in cols]
        self.colptr = np.concatenate([[0], np.cumsum([len(r) for r in self.rows])]).astype(np.int64)
        self.rowidx = np.concatenate(self.rows).astype(np.int32)
        self.off, o = {}, 0
        for g in range(nf):
            for f in self.rows[g]:
                self.off[(f, g)] = o
                o += self.size[f] * self.size[g]
        self.nvals, self.n = o, sum(self.size)
        self.start = np.concatenate([[0], np.cumsum(self.size)]).astype(np.int64)

    def values(self, gen, out):
        """Fills `out` (complex128, nvals) with K's lower blocks, column-major each."""
        out.zero_()
        for I in self.dom:
            r = sum(self.size[f] for f in I)
            if r == 0:
                continue
            G = torch.randn(r, r, generator=gen, device=DEVICE, dtype=torch.complex64)
            M = (G @ G.T).to(torch.complex128) / r   # E|G|^2 = 1: entries (N + iN) / sqrt(2 r)
            M = (M + M.T) / 2
            M.diagonal().add_(complex(-self.k2, self.tau))
            at = np.concatenate([[0], np.cumsum([self.size[f] for f in I])])
            for b, g in enumerate(I):
                for a in range(b, len(I)):
                    f = I[a]
                    sub = M[at[a]:at[a + 1], at[b]:at[b + 1]]
                    out[self.off[(f, g)]:self.off[(f, g)] + sub.numel()].view(self.size[g], self.size[f]).add_(sub.T)
        if self.zeros:    # one unknown in 16 has a vanishing diagonal: unpivoted elimination meets a zero pivot
            for f, mf in enumerate(self.size):
                o = self.off[(f, f)]
                out[o:o + mf * mf].view(mf, mf).diagonal()[::16].zero_()

    def block(self, K, f, g):
        """Stored block (f, g), f >= g, as a matrix (a view)."""
        o = self.off[(f, g)]
        return K[o:o + self.size[f] * self.size[g]].view(self.size[g], self.size[f]).T

    def handle_args(self):
        return dict(blk_size=np.asarray(self.size, dtype=np.int32), perm=d3m_order_grid_nd(*self.grid))

    def flops(self, nrhs):
        d = d3m_analyze(self.colptr, self.rowidx, perm=d3m_order_grid_nd(*self.grid),
                        blk_size=np.asarray(self.size, dtype=np.int32))
        return d["factor_flops"], d["solve_flops_per_rhs"] * nrhs


def _systems(case):
    if case["kind"] != "batch":
        return [_System(case["nx"], case["ny"], case["nz"], case["m"], case["k2"], case["tau"], case["ragged"],
                        zeros=case["pivot"])]
    # uneven instances: grid {2x2, 3x3, 4x4, 6x6}, m {64, 128, 256} up to the case's, k^2 ~ U(1, 4), tau ~ U(0.01, 0.2)
    g = np.random.RandomState(20260105)
    ms = [m for m in (64, 128, 256) if m <= case["m"]]
    out = []
    for _ in range(case["count"]):
        a = (2, 3, 4, 6)[g.randint(4)]
        out.append(_System(a, a, 1, ms[g.randint(len(ms))], 1.0 + 3.0 * g.rand(), 0.01 + 0.19 * g.rand()))
    return out


def _inputs(case, seed):
    """Systems, K (complex128, all stored blocks) and the right-hand sides as (nrhs, n), on the GPU."""
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(int(seed) % (1 << 62))
    sys_ = _systems(case)
    K = torch.empty(sum(s.nvals for s in sys_), dtype=torch.complex128, device=DEVICE)
    o = 0
    for s in sys_:
        s.values(gen, K[o:o + s.nvals])
        o += s.nvals
    n = sum(s.n for s in sys_)
    B = torch.randn(case["nrhs"], n, generator=gen, device=DEVICE, dtype=torch.complex128)
    C = None
    if case["kind"] == "grad":   # an objective on one interface
        s = sys_[0]
        f = len(s.size) // 2
        C = torch.zeros_like(B)
        C[:, s.start[f]:s.start[f + 1]] = torch.randn(case["nrhs"], s.size[f], generator=gen, device=DEVICE,
                                                      dtype=torch.complex128)
    return sys_, K, B, C


# ------------------------------------------------------------------------------ prepare and run
class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.case = case
    st.sys, st.K, B, C = _inputs(case, seed)
    st.X = None
    kw = dict(precision=case["precision"], max_nrhs=case["nrhs"])
    if case["kind"] == "batch":
        st.h = D3MBatch([(s.colptr, s.rowidx, s.size[0]) for s in st.sys],
                        [d3m_order_grid_nd(*s.grid) for s in st.sys], **kw)
    else:
        s = st.sys[0]
        st.h = D3M(s.colptr, s.rowidx, pivot=case["pivot"], **s.handle_args(), **kw)
    if case["host"]:
        st.K, B = st.K.cpu().pin_memory(), B.cpu().pin_memory()
        st.X = torch.empty_like(B).pin_memory()
    st.B, st.C = B.T, None if C is None else C.T
    if case["kind"] == "solve":
        st.h.factor(st.K)
        st.h.info()          # the program looks at the factorization's status before it goes on
    return st


def run(st):
    case = st.case
    if case["kind"] == "solve":
        return {"X": st.h.solve(st.B)}
    st.h.factor(st.K)
    X = st.h.solve(st.B, X=st.X)
    if case["kind"] != "grad":
        return {"X": X}
    lam = st.h.adjoint(st.C)
    s = st.sys[0]
    return {"X": X, "lam": lam, "deps": st.h.grad_eps(lam, X, s.dom, s.k2), "dK": st.h.grad_pattern(lam, X, s.nvals)}


# ------------------------------------------------------------------------------ work and exact values
def work(case):
    sys_ = _systems(case)
    nvals, n = sum(s.nvals for s in sys_), sum(s.n for s in sys_)
    fl = [s.flops(case["nrhs"]) for s in sys_]
    factor, solve = sum(f for f, _ in fl), sum(q for _, q in fl)
    vec = 16.0 * n * case["nrhs"]
    if case["kind"] == "solve":
        return {"bytes": 16.0 * nvals + 2 * vec, "flops": solve}
    if case["kind"] == "grad":
        return {"bytes": 32.0 * nvals + 4 * vec, "flops": factor + 2 * solve + 16.0 * nvals * case["nrhs"]}
    return {"bytes": 16.0 * nvals + 2 * vec, "flops": factor + solve}


def _eliminate(s, K, rhs):
    """K^{-1} rhs by block elimination in 64 bits (pivoted LU of every diagonal block), rhs (n, k)."""
    N = len(s.size)
    A = {(f, g): s.block(K, f, g).clone() for (f, g) in s.off}
    nb = [set() for _ in range(N)]
    for f, g in A:
        if f != g:
            nb[f].add(g)
            nb[g].add(f)
    x = [rhs[s.start[f]:s.start[f + 1]].clone() for f in range(N)]
    left, done = set(range(N)), []

    def get(f, g):   # block (f, g) of the symmetric matrix
        return A[(f, g)] if f >= g else A[(g, f)].T

    while left:      # the block with the fewest neighbours first
        k = min(left, key=lambda f: (len(nb[f] & left), f))
        left.discard(k)
        nk = sorted(nb[k] & left)
        lu = torch.linalg.lu_factor(A[(k, k)])
        if nk:
            T = torch.cat([get(f, k) for f in nk])                                  # A_ik
            W = torch.linalg.lu_solve(*lu, torch.cat([T.T, x[k]], dim=1))            # A_kk^{-1} [A_ki | x_k]
            U = T @ W
            at = np.concatenate([[0], np.cumsum([s.size[f] for f in nk])])
            for a, f in enumerate(nk):
                for b, g in enumerate(nk[:a + 1]):
                    u = U[at[a]:at[a + 1], at[b]:at[b + 1]]
                    A[(f, g)] = A[(f, g)] - u if (f, g) in A else -u
                    if f != g:
                        nb[f].add(g)
                        nb[g].add(f)
                x[f] = x[f] - U[at[a]:at[a + 1], at[-1]:]
            done.append((k, nk, W[:, :at[-1]].clone(), W[:, at[-1]:].clone()))
        else:
            done.append((k, nk, None, torch.linalg.lu_solve(*lu, x[k])))
    for k, nk, W, xk in reversed(done):
        x[k] = xk if W is None else xk - W @ torch.cat([x[f] for f in nk])
    return torch.cat(x)


def exact(case, seed):
    if work(case)["flops"] > 6e12:   # over about 20 seconds in 64 bits
        return None
    sys_, K, B, C = _inputs(case, seed)
    out, o, r = [], 0, 0
    for s in sys_:
        rhs = B[:, r:r + s.n].T
        if C is not None:
            rhs = torch.cat([rhs, C.T], dim=1)
        out.append(_eliminate(s, K[o:o + s.nvals], rhs))
        o += s.nvals
        r += s.n
    Z = torch.cat(out)
    X = Z[:, :case["nrhs"]]
    if case["kind"] != "grad":
        return {"X": X.cpu() if case["host"] else X}
    s, lam = sys_[0], Z[:, case["nrhs"]:]
    part = [(lam[s.start[f]:s.start[f + 1]] * X[s.start[f]:s.start[f + 1]]).sum() for f in range(len(s.size))]
    deps = np.array([float(s.k2 * sum(part[f].real for f in I)) for I in s.dom])
    dK = torch.empty_like(K)
    for (f, g), at in s.off.items():
        lf, lg = (lam[s.start[q]:s.start[q + 1]] for q in (f, g))
        xf, xg = (X[s.start[q]:s.start[q + 1]] for q in (f, g))
        D = -(lf @ xg.T) if f == g else -(lf @ xg.T + xf @ lg.T)
        dK[at:at + D.numel()] = D.T.reshape(-1)
    return {"X": X, "lam": lam, "deps": deps, "dK": dK}
