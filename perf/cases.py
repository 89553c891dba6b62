"""The work that users of this library have it do, as cases to be timed and compared.

One pass goes through the public calls of ``paper_1402_2585_gb300.binding`` on
device buffers.  Sizes, actions, blockings and storage precisions are those of
the workloads in ``synthetic.configs`` and of the tests.  ``exact`` restates
the operators in 64-bit torch arithmetic, independent of the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1402_2585_gb300 import binding as hd

DEV = "cuda"
PREC = {"f64": hd.F64, "f32": hd.F32, "f16": hd.F16, "bf16": hd.BF16, "df64": hd.DF64}
DTYPE = {"f64": torch.float64, "df64": torch.float64, "f32": torch.float32, "f16": torch.float16,
         "bf16": torch.bfloat16}
REAL_BYTES = {"f64": 8, "df64": 8, "f32": 4, "f16": 2, "bf16": 2}
M5 = 1.8


def listed():
    return [
        # the tiny FP64 lattice that a program starts with: launches and latency count
        dict(name="mpc_f64_8x8x8x8_ls8", kind="mpc", dims="8x8x8x8", Ls=8, moebius=False, mass=0.01, prec="f64",
             antiperiodic=False),
        # one H in the precisions that a solve applies it in: outer iteration (FP32),
        # preconditioner (FP16), true residual (double-float)
        dict(name="h_f32_16x16x16x16_ls16", kind="h", dims="16x16x16x16", Ls=16, moebius=False, mass=0.005,
             prec="f32", antiperiodic=False),
        dict(name="h_f16_24x24x24x48_ls16", kind="h", dims="24x24x24x48", Ls=16, moebius=True, mass=0.002,
             prec="f16", antiperiodic=False),
        dict(name="h_f32_32x32x32x64_ls16", kind="h", dims="32x32x32x64", Ls=16, moebius=True, mass=0.001,
             prec="f32", antiperiodic=False),
        dict(name="h_df64_16x16x16x16_ls16", kind="h", dims="16x16x16x16", Ls=16, moebius=True, mass=0.005,
             prec="df64", antiperiodic=True),
        # source preparation and reconstruction around every solve (FP64)
        dict(name="schur_16x16x16x16_ls16", kind="schur", dims="16x16x16x16", Ls=16, moebius=True, mass=0.005,
             antiperiodic=True),
        # the deflation projector P R on the fine lattice, 16-bit subspace
        dict(name="project_f16_24x24x24x48_n32", kind="project", dims="24x24x24x48", Ls=16, nvec=32, prec="f16"),
        # the little Dirac stencil for the 12 spin-colour sources of one propagator
        # (16-bit operator), and its high-mode preconditioner with the Nvec of the
        # three-level workload
        dict(name="coarse_f16_24x24x24x48_n32_r12", kind="coarse", dims="24x24x24x48", nvec=32, nrhs=12, prec="f16"),
        dict(name="qtrunc_16x16x16x32_n40_r4", kind="qtrunc", dims="16x16x16x32", nvec=40, nrhs=4, prec="f32",
             order=8),
        # whole solves: plain CG on the tiny lattice, HDCG for one source, HDCG for a
        # batch with the 16-bit preconditioner
        dict(name="solve_cg_8x8x8x8_ls8", kind="solve", dims="8x8x8x8", Ls=8, moebius=False, mass=0.01, alg="cg",
             sloppy="f32", nvec=0, nrhs=1, coarse="none"),
        dict(name="solve_hdcg_16x16x16x16_n24", kind="solve", dims="16x16x16x16", Ls=16, moebius=False, mass=0.005,
             alg="adef2", sloppy="f32", nvec=24, nrhs=1, coarse="f32"),
        dict(name="solve_hdcg_16x16x16x16_f16_r4", kind="solve", dims="16x16x16x16", Ls=16, moebius=True, mass=0.01,
             alg="adef2", sloppy="f16", nvec=24, nrhs=4, coarse="f32"),
    ]


def _draw_dims(rng, lo, hi, step, cap):
    """Four extents, multiples of `step`, volume spread over its logarithm up to `cap`."""
    target = math.exp(rng.uniform(math.log(lo ** 4), math.log(cap)))
    while True:
        d = [step * max(1, round(rng.uniform(lo, hi) / step)) for _ in range(4)]
        v = d[0] * d[1] * d[2] * d[3]
        if 0.6 * target <= v <= min(cap, 1.7 * target):
            return "x".join(str(x) for x in d)


def draw(rng):
    kind = rng.choice(["mpc", "h", "h", "h", "schur", "project", "coarse", "qtrunc", "solve"])
    mob, mass = rng.random() < 0.6, rng.choice([0.001, 0.002, 0.005, 0.01])
    apbc = rng.random() < 0.3
    if kind in ("mpc", "h"):
        return dict(kind=kind, dims=_draw_dims(rng, 4, 40, 2, 24 * 24 * 24 * 48), Ls=rng.choice([4, 8, 16, 16, 32]),
                    moebius=mob, mass=mass, prec=rng.choice(["f64", "df64", "f32", "f32", "f16", "f16", "bf16"]),
                    antiperiodic=apbc)
    if kind == "schur":
        return dict(kind=kind, dims=_draw_dims(rng, 4, 24, 2, 16 ** 4), Ls=rng.choice([4, 8, 16]), moebius=mob,
                    mass=mass, antiperiodic=apbc)
    if kind == "project":
        return dict(kind=kind, dims=_draw_dims(rng, 8, 28, 4, 16 ** 3 * 32), Ls=rng.choice([4, 8, 16]),
                    nvec=rng.randint(5, 40), prec=rng.choice(["f32", "f16"]))
    if kind in ("coarse", "qtrunc"):
        c = dict(kind=kind, dims=_draw_dims(rng, 12, 28, 4, 16 ** 3 * 32), nvec=rng.randint(5, 48),
                 nrhs=rng.randint(1, 16), prec=rng.choice(["f32", "f16"]))
        if kind == "qtrunc":
            c["order"] = rng.choice([8, 16])
        return c
    return dict(kind=kind, dims=_draw_dims(rng, 8, 16, 4, 12 ** 4), Ls=rng.choice([8, 16]), moebius=mob, mass=0.01,
                alg="adef2", sloppy=rng.choice(["f32", "f16"]), nvec=rng.randint(12, 24), nrhs=rng.choice([1, 1, 3]),
                coarse=rng.choice(["f32", "f16"]))


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _dims(case):
    return tuple(int(x) for x in case["dims"].split("x"))


def _gen(seed, k):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 1009 + k)
    return g


def _normal(shape, g, dtype=torch.float64):
    """Complex Gaussian with E|z|^2 = 1 as a real tensor with a trailing [re, im]."""
    return (torch.randn(*shape, 2, device=DEV, dtype=torch.float32, generator=g) * math.sqrt(0.5)).to(dtype)


def _gauge(dims, seed, eps=0.4):
    """Random SU(3) links near 1 + i eps H, H Hermitian Gaussian, rows reunitarised."""
    n = 4 * int(np.prod(dims))
    w = torch.view_as_complex(_normal((n, 3, 3), _gen(seed, 1)))
    h = 0.5 * (w + w.conj().transpose(1, 2))
    u = torch.eye(3, device=DEV, dtype=torch.complex128) + 1j * eps * h
    r0 = u[:, 0]
    r0 = r0 / torch.linalg.vector_norm(r0, dim=-1, keepdim=True)
    r1 = u[:, 1]
    r1 = r1 - (r0.conj() * r1).sum(-1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=-1, keepdim=True)
    r2 = torch.linalg.cross(r0, r1).conj()
    return torch.stack([r0, r1, r2], 1).reshape(-1, 4, 3, 3).contiguous()


def _action(case):
    return (M5, 1.5, 0.5, case["mass"]) if case["moebius"] else (M5, 1.0, 0.0, case["mass"])


def _sites(dims, Ls):
    return int(np.prod(dims)) // 2 * Ls


def _coarse_operator(cd, nvec, seed, prec):
    """Hermitian positive little Dirac operator [Vc][81][n][n]: couplings fall by a
    decade per block hop, as between blocks of a deflation subspace, the self block
    dominates; every entry is representable in the storage precision."""
    vc = int(np.prod(cd))
    nb, hops, mate, stored = _coarse_tables(cd)
    g = _gen(seed, 3)
    A = torch.zeros(vc, 81, nvec, nvec, device=DEV, dtype=torch.complex128)
    for l in range(81):
        if not stored[l]:
            continue
        m = mate[l]
        if m < l:
            A[:, l] = A[nb[:, l], m].conj().transpose(1, 2)
            continue
        b = torch.view_as_complex(_normal((vc, nvec, nvec), g)) * (0.3 / math.sqrt(nvec) * 10.0 ** -hops[l])
        if m == l:    # the self block, or an offset that is its own inverse on an extent of 2
            b = b.to(torch.complex64).to(torch.complex128)
            b = 0.5 * (b + b[nb[:, l]].conj().transpose(1, 2))
        A[:, l] = b
        if l == 40:
            A[:, l] += torch.eye(nvec, device=DEV, dtype=torch.complex128)
    r = torch.view_as_real(A)
    return torch.view_as_complex(r.to(DTYPE[prec]).to(torch.float64))


def _coarse_tables(cd):
    """Neighbour of every coarse site per offset, block hops and the opposite offset
    (among the stored ones) of the 81 offsets, and which offsets are stored."""
    v = int(np.prod(cd))
    x, r = [], np.arange(v)
    for L in cd:
        x.append(r % L)
        r = r // L
    nb, hops, mate, stored = np.zeros((v, 81), dtype=np.int64), [], [], []
    for l in range(81):
        d = [l // 3 ** mu % 3 - 1 for mu in range(4)]
        idx, mul, m = 0, 1, 0
        for mu, L in enumerate(cd):
            idx = idx + ((x[mu] + d[mu]) % L) * mul
            mul *= L
            m += 3 ** mu * ((d[mu] if L == 2 else -d[mu]) + 1)
        nb[:, l] = idx
        hops.append(sum(abs(q) for q in d))
        mate.append(m)
        stored.append(all(L >= 3 or (q >= 0 if L == 2 else q == 0) for q, L in zip(d, cd)))
    return torch.from_numpy(nb).to(DEV), hops, mate, stored


def _coarse_vectors(case, seed):
    vc = int(np.prod(_dims(case))) // 256
    return torch.view_as_complex(_normal((case["nrhs"], vc, case["nvec"]), _gen(seed, 4)))


def _interval(case):
    """Chebyshev interval around the spectrum of the nine kept blocks."""
    return 0.05, 2.2


class State:
    pass


def _subspace_vectors(case, seed, Ls):
    n4 = int(np.prod(_dims(case))) // 2
    return _normal((case["nvec"], n4, Ls, 4, 3), _gen(seed, 5))


def _field(case, seed, k):
    return _normal((int(np.prod(_dims(case))) // 2, case["Ls"], 4, 3), _gen(seed, k), DTYPE[case.get("prec", "f64")])


def prepare(case, seed):
    s = State()
    s.case = case
    kind, dims = case["kind"], _dims(case)
    if kind in ("mpc", "h", "schur", "solve"):
        # solves run on a stream of their own, operator calls on the current one
        s.stream = torch.cuda.Stream() if kind == "solve" else None
        s.h = hd.Hdcg(dims, case["Ls"], case.get("antiperiodic", False),
                      s.stream.cuda_stream if s.stream else None)
        s.h.set_dwf(*_action(case))
        U = _gauge(dims, seed)
        torch.cuda.synchronize()
        s.h.set_gauge(U)
        del U
    if kind in ("mpc", "h"):
        s.inp, s.prec = _field(case, seed, 2), PREC[case["prec"]]
        s.out = torch.empty_like(s.inp)
        s.out2 = torch.empty_like(s.inp) if kind == "mpc" else None
    elif kind == "schur":
        s.eta_e, s.eta_o = _field(case, seed, 2), _field(case, seed, 6)
        s.psi_o = _field(case, seed, 7)
        s.b, s.psi_e = torch.empty_like(s.eta_o), torch.empty_like(s.eta_e)
    elif kind == "project":
        s.h = hd.Hdcg(dims, case["Ls"])
        phi = _subspace_vectors(case, seed, case["Ls"])
        torch.cuda.synchronize()
        s.h.set_subspace((4, 4, 4, 4), phi, PREC[case["prec"]])
        del phi
        s.inp, s.prec = _field(case, seed, 2), PREC[case["prec"]]
        s.out = torch.empty_like(s.inp)
        s.c = torch.empty(int(np.prod(dims)) // 256, case["nvec"], device=DEV, dtype=torch.complex128)
    elif kind in ("coarse", "qtrunc"):
        # the stencil alone: the shortest fifth dimension carries the blocking
        s.h = hd.Hdcg(dims, 2)
        phi = _subspace_vectors(case, seed, 2)
        torch.cuda.synchronize()
        s.h.set_subspace((4, 4, 4, 4), phi, PREC[case["prec"]])
        del phi
        A = _coarse_operator(tuple(d // 4 for d in dims), case["nvec"], seed, case["prec"])
        torch.cuda.synchronize()
        s.h.set_coarse(A, PREC[case["prec"]])
        del A
        if kind == "qtrunc":
            s.h.set_coarse_preconditioner(case["order"], *_interval(case))
        s.x = _coarse_vectors(case, seed)
        s.y = torch.empty_like(s.x)
    else:
        if case["alg"] == "adef2":
            s.h.build_subspace((4, 4, 4, 4), case["nvec"], PREC["f16" if case["sloppy"] == "f16" else "f32"],
                               inv_steps=2, inv_tol=1e-2, inv_maxiter=100, seed=seed + 11)
            s.h.build_coarse(PREC[case["coarse"]])
        s.b = torch.view_as_complex(_normal((case["nrhs"], int(np.prod(dims)) // 2, case["Ls"], 4, 3), _gen(seed, 2)))
        s.x = torch.empty_like(s.b)
        s.par = s.h.default_params(algorithm=hd.ALG_ADEF2 if case["alg"] == "adef2" else hd.ALG_CG,
                                   outer_prec=hd.F32, sloppy_prec=PREC[case["sloppy"]])
        torch.cuda.synchronize()
    return s


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "h":
        s.h.apply_mdagm(s.inp, s.out, s.prec)
        return s.out
    if kind == "mpc":
        s.h.apply_mpc(s.inp, s.out, False, s.prec)
        s.h.apply_mpc(s.out, s.out2, True, s.prec)
        return [s.out, s.out2]
    if kind == "schur":
        s.h.prep_source(s.eta_e, s.eta_o, s.b)
        s.h.reconstruct(s.eta_e, s.psi_o, s.psi_e)
        return [s.b, s.psi_e]
    if kind == "project":
        s.h.restrict(s.inp, s.prec, s.c)
        s.h.prolong(s.c, s.out, s.prec)
        return s.out
    if kind == "coarse":
        s.h.coarse_apply_multi(s.x, s.y, case["nrhs"])
        return s.y.to(torch.complex64)      # an FP32 computation: kept in FP32
    if kind == "qtrunc":
        s.h.coarse_precondition(s.x, s.y, case["nrhs"])
        return s.y.to(torch.complex64)
    s.h.solve(s.b, s.x, 1e-8, s.par, case["nrhs"])
    return s.x.to(torch.complex64)          # propagators are kept in single precision


def work(case):
    kind, dims = case["kind"], _dims(case)
    v = int(np.prod(dims))
    if kind in ("mpc", "h", "schur", "solve"):
        n5 = _sites(dims, case["Ls"])
        rb = REAL_BYTES[case.get("prec", "f64")]
        hflops = 7248 if case["moebius"] else 6528          # per 5D site of one H at Ls 16
        field, links = 24.0 * n5 * rb, 72.0 * v * rb
        if kind == "h":
            return {"bytes": 2 * field + links, "flops": float(hflops) * n5}
        if kind == "mpc":
            return {"bytes": 3 * field + links, "flops": float(hflops) * n5}
        if kind == "schur":
            return {"bytes": 6 * field + links, "flops": 1.0 * hflops * n5}
        # a solve: every outer iteration applies H once in FP32 and, in HDCG, eight
        # times in the preconditioner; 20 (HDCG) or 200 (CG) iterations as a scale
        r = case["nrhs"]
        sb = REAL_BYTES[case["sloppy"]]
        if case["alg"] == "cg":
            return {"bytes": 200.0 * (7 * 24 * 4 * n5 * r + 72 * 4 * v), "flops": 200.0 * hflops * n5 * r}
        outer = 7 * 24 * 4 * n5 * r + 72 * 4 * v + 8 * (7 * 24 * sb * n5 * r + 72 * sb * v) \
            + 2 * 24 * case["nvec"] * sb * n5
        return {"bytes": 20.0 * outer, "flops": 20.0 * 9 * hflops * n5 * r}
    n, vc = case["nvec"], v // 256
    rb = REAL_BYTES[case["prec"]]
    if kind == "project":
        n5 = _sites(dims, case["Ls"])
        return {"bytes": 2 * 24.0 * n5 * rb * (n + 1), "flops": 2 * 96.0 * n * n5}
    r = case["nrhs"]
    blocks = 81 if kind == "coarse" else 9
    passes = 1 if kind == "coarse" else case["order"] - 1
    return {"bytes": 2.0 * rb * blocks * vc * n * n + 32.0 * vc * n * r, "flops": 8.0 * passes * blocks * vc * n * n * r}


# ----------------------------------------------------------------------------
# the same results in 64 bits
# ----------------------------------------------------------------------------
class _Dwf:
    """The red-black domain-wall operator in complex double."""

    def __init__(self, case, seed):
        dims, Ls = _dims(case), case["Ls"]
        m5, b, c, mass = _action(case)
        self.Ls = Ls
        self.P = []                                      # P_s per chirality: + down shift, - up shift
        for up in (False, True):
            p = np.zeros((Ls, Ls))
            for s in range(Ls):
                t = s + 1 if up else s - 1
                p[s, t % Ls] = 1.0 if 0 <= t < Ls else -mass
            self.P.append(p)
        one = np.eye(Ls)
        al, be = b * (4 - m5) + 1, c * (4 - m5) - 1
        self.K = [torch.from_numpy(b * one + c * p).to(DEV) for p in self.P]
        self.M = [torch.from_numpy(al * one + be * p).to(DEV) for p in self.P]
        self.Minv = [torch.from_numpy(np.linalg.inv(al * one + be * p)).to(DEV) for p in self.P]
        U = _gauge(dims, seed)
        if case.get("antiperiodic", False):
            U = U.reshape(dims[3], -1, 4, 3, 3)
            U[-1, :, 3] *= -1
            U = U.reshape(-1, 4, 3, 3)
        self.U = U
        self.tab = []
        v = int(np.prod(dims))
        lex = np.arange(v)
        x = [lex % dims[0], lex // dims[0] % dims[1], lex // (dims[0] * dims[1]) % dims[2],
             lex // (dims[0] * dims[1] * dims[2])]
        par = (x[0] + x[1] + x[2] + x[3]) % 2
        for p in range(2):
            sel = np.nonzero(par == p)[0]
            sel = sel[np.argsort(sel >> 1, kind="stable")]
            fw, bw = [], []
            for mu in range(4):
                for step, to in ((1, fw), (-1, bw)):
                    y = [q[sel].copy() for q in x]
                    y[mu] = (y[mu] + step) % dims[mu]
                    to.append(torch.from_numpy(y[0] + dims[0] * (y[1] + dims[1] * (y[2] + dims[2] * y[3]))).to(DEV))
            self.tab.append((torch.from_numpy(sel).to(DEV), fw, bw))

    GAMMA = []
    for _a, _b in (([[0, -1j], [-1j, 0]], [[0, 1j], [1j, 0]]), ([[0, -1], [1, 0]], [[0, 1], [-1, 0]]),
                   ([[-1j, 0], [0, 1j]], [[1j, 0], [0, -1j]]), ([[1, 0], [0, 1]], [[1, 0], [0, 1]])):
        _g = np.zeros((4, 4), dtype=np.complex128)
        _g[:2, 2:], _g[2:, :2] = _a, _b
        GAMMA.append(_g)

    def s_op(self, mats, f, dag=False):
        """An operator of the fifth dimension, one matrix per chirality."""
        out = torch.empty_like(f)
        r, o = torch.view_as_real(f), torch.view_as_real(out)
        for k, sl in enumerate((slice(0, 2), slice(2, 4))):
            m = mats[k].t() if dag else mats[k]
            o[:, :, sl] = torch.einsum("st,ntabc->nsabc", m, r[:, :, sl])
        return out

    def hop(self, f, out_par, dag=False):
        """Dh (or its adjoint) onto parity out_par."""
        sel, fw, bw = self.tab[out_par]
        out = torch.zeros_like(f)
        for mu in range(4):
            for forward in (True, False):
                nb = fw[mu] if forward else bw[mu]
                sign = -1.0 if forward != dag else 1.0
                u = self.U[sel, mu] if forward else self.U[nb, mu].conj().transpose(1, 2)
                proj = torch.from_numpy(np.eye(4) + sign * self.GAMMA[mu]).to(DEV)
                g = f[nb >> 1]
                n = g.shape[0]
                g = torch.matmul(u[:, None], g.reshape(n, self.Ls * 4, 3).transpose(1, 2)[:, None])[:, 0]
                g = g.transpose(1, 2).reshape(n, self.Ls, 4, 3)
                out += torch.einsum("ab,nsbc->nsac", proj, g)
        return out

    def mpc(self, f):
        t = self.s_op(self.Minv, self.hop(self.s_op(self.K, f), 0))
        return self.s_op(self.M, f) - 0.25 * self.hop(self.s_op(self.K, t), 1)

    def mpc_dag(self, f):
        t = self.s_op(self.Minv, self.s_op(self.K, self.hop(f, 0, True), True), True)
        return self.s_op(self.M, f, True) - 0.25 * self.s_op(self.K, self.hop(t, 1, True), True)


def _real(z):
    return torch.view_as_real(z.contiguous())


def exact(case, seed):
    kind, dims = case["kind"], _dims(case)
    if kind in ("mpc", "h", "schur"):
        D = _Dwf(case, seed)
        if kind == "schur":
            e, o, psi = (torch.view_as_complex(_field(case, seed, k)) for k in (2, 6, 7))
            b = D.mpc_dag(o + 0.5 * D.hop(D.s_op(D.K, D.s_op(D.Minv, e)), 1))
            return [_real(b), _real(D.s_op(D.Minv, e + 0.5 * D.hop(D.s_op(D.K, psi), 0)))]
        f = torch.view_as_complex(_field(case, seed, 2).double())
        m = D.mpc(f)
        h = D.mpc_dag(m)
        return _real(h) if kind == "h" else [_real(m), _real(h)]
    if kind == "project":
        # Phi (Phi^dag Phi)^-1 Phi^dag v, block by block
        n4, n = int(np.prod(dims)) // 2, case["nvec"]
        lex = 2 * np.arange(n4)
        t = [lex // dims[0] % dims[1], lex // (dims[0] * dims[1]) % dims[2], lex // (dims[0] * dims[1] * dims[2])]
        x0 = lex % dims[0] + (1 + t[0] + t[1] + t[2]) % 2
        blk = np.zeros(n4, dtype=np.int64)
        for q, L in zip(reversed([x0] + t), reversed(dims)):
            blk = blk * (L // 4) + q // 4
        order = torch.from_numpy(np.argsort(blk, kind="stable")).to(DEV).reshape(-1, 128)
        phi = torch.view_as_complex(_subspace_vectors(case, seed, case["Ls"])).reshape(n, n4, -1)
        v = torch.view_as_complex(_field(case, seed, 2).double()).reshape(n4, -1)
        out = torch.empty_like(v)
        for at in order.split(128):
            p = phi[:, at].reshape(n, at.shape[0], -1).transpose(0, 1)       # [blocks][n][sites]
            w = v[at].reshape(at.shape[0], -1, 1)
            c = torch.linalg.solve(p.conj() @ p.transpose(1, 2), p.conj() @ w)
            out[at] = (p.transpose(1, 2) @ c).reshape(*at.shape, -1)
        return _real(out.reshape(n4, case["Ls"], 4, 3))
    if kind in ("coarse", "qtrunc"):
        cd = tuple(d // 4 for d in dims)
        A = _coarse_operator(cd, case["nvec"], seed, case["prec"])
        nb, hops, _, stored = _coarse_tables(cd)
        x = _coarse_vectors(case, seed)

        def apply(f, most):
            y = torch.zeros_like(f)
            for l in range(81):
                if stored[l] and hops[l] <= most:
                    y += torch.einsum("ajk,rak->raj", A[:, l], f[:, nb[:, l]])
            return y

        if kind == "coarse":
            return apply(x, 4)
        lo, hi = _interval(case)
        theta, delta = 0.5 * (hi + lo), 0.5 * (hi - lo)
        y, r, d, rho = torch.zeros_like(x), x.clone(), x / theta, delta / theta
        for k in range(case["order"]):
            y = y + d
            if k + 1 == case["order"]:
                return y
            r = r - apply(d, 1)
            new = 1.0 / (2 * theta / delta - rho)
            d, rho = new * rho * d + 2 * new / delta * r, new
    if case["alg"] != "cg":
        return None                   # the same equation in 64 bits takes minutes on these lattices
    D = _Dwf(case, seed)
    b = torch.view_as_complex(_normal((case["nrhs"], int(np.prod(dims)) // 2, case["Ls"], 4, 3), _gen(seed, 2)))
    xs = []
    for k in range(case["nrhs"]):
        x, r = torch.zeros_like(b[k]), b[k].clone()
        p, rr = r.clone(), float(torch.linalg.vector_norm(r)) ** 2
        stop = 1e-24 * rr
        for _ in range(2000):
            w = D.mpc_dag(D.mpc(p))
            al = rr / float((p.conj() * w).sum().real)
            x += al * p
            r -= al * w
            new = float(torch.linalg.vector_norm(r)) ** 2
            if new <= stop:
                break
            p, rr = r + new / rr * p, new
        xs.append(x)
    return torch.stack(xs)
