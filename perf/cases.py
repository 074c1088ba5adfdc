"""Measured workloads of the quasi-particle fRG framework: what a user has it do.

Five kinds of pass, each through the calls of the public binding:

  rhs    one one-loop right-hand side dV/dLambda of a given vertex (qpfrg_rhs)
  sigma  the weights Z of a vertex and, with a frequency grid, Sigma(k_F, w)
         (qpfrg_selfenergy)
  step   one RK4 step of the temperature flow with Z feedback, from a state
         image in pinned host memory (qpfrg_set_state, qpfrg_step,
         qpfrg_read_state)
  gstep  the same for the interaction flow with the self-energy ODE and the
         Katanin factor (the flows of the Fig. 4 comparison)
  sweep  a batch of complete flows over (U, T_end, N_p) (qpfrg_flow_batch)

The mixed precisions compute to 32-bit accuracy in the FP64 buffers of the C
ABI; their results are taken as float32, those of the FP64 path as float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2005_00827_gb300 import api

PREC = {"fp64": api.QPFRG_FP64, "mixed": api.QPFRG_MIXED, "tc": api.QPFRG_MIXED_TC}
ETA = 0.02
DLNT = math.log(0.98)
DG = 0.05


# --- the cases ---------------------------------------------------------------
def _rhs(prec, N, nt, nr, T, U=2.0, sym=True, shells=1, tp=0.0, **more):
    return dict(kind="rhs", prec=prec, N=N, nt=nt, nr=nr, T=T, U=U, sym=sym, shells=shells, tp=tp, **more)


def _sigma(prec, N, nt, nr, T, U=2.0, n_omega=0, sym=True, **more):
    return dict(kind="sigma", prec=prec, N=N, nt=nt, nr=nr, T=T, U=U, n_omega=n_omega, sym=sym, shells=1, tp=0.0, **more)


def listed():
    return [
        # the smallest configuration (16 patches, 8 x 8 points) in the default
        # precision: parameter scans and tests, where launches count
        _rhs("fp64", 16, 8, 8, 0.3, name="rhs_np16_fp64"),
        # the ordinary size (48 patches) in the default precision
        _rhs("fp64", 48, 16, 16, 0.1, U=3.0, name="rhs_np48_fp64"),
        # the same in mixed precision
        _rhs("mixed", 48, 16, 16, 0.1, U=3.0, name="rhs_np48_mixed"),
        # the production size on the tensor cores, a vertex with the lattice
        # symmetry as every flow has it
        _rhs("tc", 96, 32, 32, 0.1, U=2.5, name="rhs_np96_tc"),
        # a vertex without the lattice symmetry on a ragged grid with t'
        _rhs("tc", 60, 10, 14, 0.15, sym=False, tp=-0.1, name="rhs_np60_tc_general"),
        # energy shells: 32 angular sections x 7 shells = 224 patches
        _rhs("tc", 224, 8, 8, 0.2, shells=7, name="rhs_np224_shell_tc"),
        # Z of a given vertex in the default precision, smallest configuration
        _sigma("fp64", 16, 8, 8, 0.3, name="z_np16_fp64"),
        # Z of a given vertex at the ordinary size
        _sigma("mixed", 48, 16, 16, 0.2, U=3.0, name="z_np48_mixed"),
        # Sigma(k_F, w) on 512 frequencies (spectral functions)
        _sigma("mixed", 48, 16, 16, 0.2, U=3.0, n_omega=512, name="sigma_np48_mixed"),
        # a step of the Z-feedback flow on the fine 32 x 32 grid
        dict(kind="step", prec="tc", N=48, nt=32, nr=32, T=0.3, U=3.0, sym=True, shells=1, tp=0.0, name="step_np48_tc"),
        # a step of the Katanin-corrected interaction flow, 48 angular patches
        dict(kind="gstep", prec="mixed", N=48, nt=8, nr=8, T=0.15, U=1.0, g=1.0, sym=True, shells=1, tp=0.0,
             name="gstep_np48_mixed"),
        # a sweep of flows over two patch counts
        dict(kind="sweep", prec="tc", flows=24, na=48, nb=96, nt=16, nr=16, name="sweep_24"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid(rng, lo, hi):
    # angular counts of any parity, radial ones even (the framework's rule)
    return int(round(_log(rng, lo, hi))), 2 * int(round(_log(rng, lo, hi) / 2))


def draw(rng):
    kind = rng.choice(["rhs", "rhs", "rhs", "rhs", "shell", "sigma", "sigma", "step", "gstep", "sweep"])
    if kind == "sweep":
        na = 4 * rng.randint(5, 12)
        return dict(kind="sweep", prec="tc", flows=rng.randint(4, 24), na=na, nb=na + 4 * rng.randint(1, 9),
                    nt=4 * rng.randint(2, 4), nr=rng.choice([8, 12, 16]))
    T, U = round(_log(rng, 0.05, 0.8), 4), round(rng.uniform(1.0, 3.0), 3)
    tp = rng.choice([0.0, 0.0, 0.0, -0.1, -0.2])
    if kind == "shell":
        shells = rng.choice([3, 5, 7])
        n = rng.choice([4, 6, 8])
        return _rhs(rng.choice(["fp64", "mixed", "tc"]), shells * 4 * rng.randint(2, 4), n, n, T, U, shells=shells)
    if kind == "rhs":
        prec = rng.choice(["fp64", "mixed", "tc"])
        N = 4 * int(round(_log(rng, 8, 64) / 4)) if prec != "tc" else 4 * int(round(_log(rng, 16, 96) / 4))
        nt, nr = _grid(rng, 4, 32)
        return _rhs(prec, N, nt, nr, T, U, sym=rng.random() < 0.7, tp=tp)
    if kind == "sigma":
        prec = rng.choice(["fp64", "mixed", "mixed", "tc"])
        N = 4 * int(round(_log(rng, 8, 20 if prec == "fp64" else 56) / 4))
        nt, nr = _grid(rng, 4, 8 if prec == "fp64" else 16)
        return _sigma(prec, N, nt, nr, T, U, n_omega=rng.choice([0, rng.randint(100, 1024)]), sym=rng.random() < 0.7)
    prec = rng.choice(["mixed", "tc"])
    N = 4 * int(round(_log(rng, 16, 48) / 4))
    if kind == "gstep":
        nt, nr = _grid(rng, 4, 8)
        return dict(kind="gstep", prec=prec, N=N, nt=nt, nr=nr, T=round(rng.uniform(0.1, 0.4), 4), U=1.0,
                    g=round(rng.uniform(0.4, 1.4), 3), sym=True, shells=1, tp=tp)
    nt, nr = _grid(rng, 8, 32)
    return dict(kind="step", prec=prec, N=N, nt=nt, nr=nr, T=T, U=U, sym=True, shells=1, tp=tp)


def work(case):
    if case["kind"] == "sweep":
        b = f = 0.0
        for N in (case["na"], case["nb"]):
            # flows of one size share the loop tables of a stage; ln(1 / 0.25) / 0.0202 steps
            n, stages = case["flows"] / 2, 4 * 68
            f += stages * (2.0 * N ** 3 * case["nt"] * case["nr"] / 8 * 20 + n * 8.0 * N ** 5 / 8)
            b += n * stages * 16.0 * N ** 3
        return {"bytes": b, "flops": f}
    N, P = case["N"], case["nt"] * case["nr"]
    M, fold = float(N * P), 8.0 if case["sym"] else 1.0
    rhs = (2.0 * N * N * M * 20 + 8.0 * N ** 5) / fold        # loop kernels and contractions
    pairs = M * M * N / fold * 40                             # self-energy pairs
    state = 8.0 * (N ** 3 + N)
    if case["kind"] == "rhs":
        return {"bytes": 2 * state, "flops": rhs}
    if case["kind"] == "sigma":
        return {"bytes": state + 16.0 * N * case["n_omega"] + 8.0 * N, "flops": pairs * (2 if case["n_omega"] else 1)}
    if case["kind"] == "step":
        return {"bytes": 2 * state, "flops": 4 * rhs + pairs}
    return {"bytes": 2 * state + 32.0 * N, "flops": 4 * (rhs + pairs)}


# --- inputs ------------------------------------------------------------------
def _c4v(N, shells):
    """The 8 patch permutations of the square lattice's point group."""
    Na = N // shells
    w, s = np.divmod(np.arange(N), shells)
    return [((sg * w + m * Na // 4) % Na) * shells + s for m in range(4) for sg in (1, -1)]


def _vertex(case, seed):
    """A coupling of the size that a flow at moderate coupling has: U plus
    fluctuations of half of U, with the lattice symmetry unless asked otherwise,
    and weights Z near 0.9 with the anisotropy of the Fermi surface."""
    N, U, rng = case["N"], case["U"], np.random.default_rng(seed)
    V = U + 0.5 * U * (2.0 * rng.random((N, N, N)) - 1.0)
    Z = 0.85 + 0.1 * rng.random(N)
    if case["sym"]:
        maps = _c4v(N, case["shells"])
        V = sum(V[np.ix_(g, g, g)] for g in maps) / 8.0
        Z = sum(Z[g] for g in maps) / 8.0
    return V, Z


def _sweep_specs(case, seed):
    """Flows that end before strong coupling: U in [1, 2], T_end in [0.2, 0.35]."""
    rng = np.random.default_rng(seed)
    u, t = rng.random(case["flows"]), rng.random(case["flows"])
    return [(case["na"] if i % 2 == 0 else case["nb"], 1.0 + u[i], 1.0, 0.2 * 1.75 ** t[i]) for i in range(case["flows"])]


def _gflow_state(case, seed):
    """Chord slopes of Sigma and Sigma' as a g-flow builds them up (Z near 0.95)."""
    rng = np.random.default_rng(seed + 1)
    N = case["N"]
    s1, s2 = -0.05 - 0.02 * rng.random(N), -0.05 - 0.02 * rng.random(N)
    maps = _c4v(N, 1)
    return np.concatenate([sum(s1[g] for g in maps) / 8.0, sum(s2[g] for g in maps) / 8.0])


def prepare(case, seed):
    if case["kind"] == "sweep":
        o = api.qpfrg_default_options()
        o.precision = PREC[case["prec"]]
        return dict(case=case, options=o, specs=_sweep_specs(case, seed), lattice=api.qpfrg_lattice(1.0, 0.0, 0.0),
                    grid=api.qpfrg_fine_grid(case["nt"], case["nr"], api.QPFRG_GRID_WEDGE, 1, 0.0))
    N = case["N"]
    opts = dict(precision=PREC[case["prec"]], eta=ETA)
    regulator, lam = api.QPFRG_REG_TEMPERATURE, case["T"]
    if case["kind"] == "sigma" and case["n_omega"]:
        opts.update(n_omega=case["n_omega"], omega_min=-4.0, omega_max=4.0)
    if case["kind"] == "step":
        opts.update(z_feedback=1, step=DLNT, lambda_end=0.01, stop_abs_v=1e6)
    if case["kind"] == "gstep":
        regulator, lam = api.QPFRG_REG_INTERACTION, case["g"]
        opts.update(z_feedback=1, sigma_ode=1, katanin=1, step=DG, lambda_end=10.0, T_fixed=case["T"], eta=0.05,
                    stop_abs_v=1e6)
    ctx = api.Context(N, case["nt"], case["nr"], U=case["U"], lambda0=lam, tp=case["tp"], regulator=regulator,
                      mode=api.QPFRG_GRID_SHELL if case["shells"] > 1 else api.QPFRG_GRID_WEDGE, n_shell=case["shells"], **opts)
    V, Z = _vertex(case, seed)
    st = dict(case=case, ctx=ctx)
    new = lambda *n: torch.zeros(*n, dtype=torch.float64, device="cuda")  # noqa: E731
    if case["kind"] in ("step", "gstep"):
        # a checkpoint of the flow in pinned memory: its 64-byte header, then the state
        head = api.qpfrg_get_state(ctx.h)[:64]
        parts = [V.ravel(), Z] + ([_gflow_state(case, seed)] if case["kind"] == "gstep" else [])
        image = np.concatenate([np.frombuffer(head, dtype=np.uint8), np.concatenate(parts).view(np.uint8)])
        st.update(image=torch.from_numpy(image).pin_memory(), V=new(N, N, N), Z=new(N))
        if case["kind"] == "gstep":
            st.update(slopes=new(2, N), zka=new(3 * N + 1))
        return st
    st.update(V=torch.from_numpy(V).cuda(), Z=torch.from_numpy(Z).cuda())
    if case["kind"] == "rhs":
        st.update(dV=new(N, N, N))
    else:
        st.update(Z_out=new(N))
        if case["n_omega"]:
            st.update(re=new(N, case["n_omega"]), im=new(N, case["n_omega"]))
    return st


# --- one pass ----------------------------------------------------------------
def _taken(case, x):
    return x if case["prec"] == "fp64" else x.float()


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "sweep":
        r = api.qpfrg_flow_batch(st["lattice"], st["grid"], api.QPFRG_REG_TEMPERATURE, st["options"], st["specs"],
                                 torch.cuda.current_stream().cuda_stream)
        return dict(ended=np.array([x["status"] == "REACHED_END" for x in r], dtype=np.int32),
                    steps=np.array([x["steps"] for x in r], dtype=np.int32),
                    lam=np.array([x["lam"] for x in r], dtype=np.float32),
                    max_abs_v=np.array([x["max_abs_v"] for x in r], dtype=np.float32))
    h = st["ctx"].h
    if kind == "rhs":
        api.qpfrg_rhs(h, case["T"], st["V"], st["Z"], st["dV"])
        return _taken(case, st["dV"])
    if kind == "sigma":
        api.qpfrg_selfenergy(h, case["T"], st["V"], st["Z"], st.get("re"), st.get("im"), st["Z_out"])
        out = dict(Z=_taken(case, st["Z_out"]))
        if case["n_omega"]:
            out.update(re=_taken(case, st["re"]), im=_taken(case, st["im"]))
        return out
    api.qpfrg_set_state_from(h, st["image"])
    api.qpfrg_step(h, 1)
    api.qpfrg_read_state(h, st["V"], st["Z"])
    out = dict(V=_taken(case, st["V"]), Z=_taken(case, st["Z"]))
    if kind == "gstep":
        api.qpfrg_read_sigma_flow(h, st["slopes"], None, st["zka"])
        out.update(slopes=_taken(case, st["slopes"]), zka=_taken(case, st["zka"]))
    return out


# --- the same in 64 bits, plain torch ----------------------------------------
class _Plain:
    """The patch geometry and the sums of the method in FP64 (t = 1, mu = 0)."""

    def __init__(self, case, eta):
        self.N, self.ns, self.tp, self.eta = case["N"], case["shells"], case["tp"], eta
        self.nt, self.nr = case["nt"], case["nr"]
        self.Na, self.P = self.N // self.ns, self.nt * self.nr
        self.M = self.N * self.P
        self.dth = 2 * math.pi / self.Na
        self.D = 2 * max(abs(self._xi(0, 0)), abs(self._xi(math.pi, math.pi)), abs(self._xi(math.pi, 0))) / self.ns
        kf, pts, w = [], [], []
        for wd in range(self.Na):
            th0 = self.dth * wd
            for sh in range(self.ns):
                r = self._level(th0, (sh - self.ns // 2) * self.D)
                kf.append((r * math.cos(th0), r * math.sin(th0)))
                for a in range(self.nt):
                    th = float(np.longdouble(th0) + np.longdouble((a + 0.5) / self.nt - 0.5) * np.longdouble(self.dth))
                    for r0, r1 in self._cells(th, sh):
                        r = 0.5 * (r0 + r1)
                        pts.append((r * math.cos(th), r * math.sin(th)))
                        w.append(0.5 * (r1 * r1 - r0 * r0) * (self.dth / self.nt) / (4 * math.pi ** 2))
        dev = lambda x: torch.tensor(x, dtype=torch.float64, device="cuda")  # noqa: E731
        self.kf, self.p, self.w = dev(kf), dev(pts), dev(w)
        self.pa = torch.arange(self.M, device="cuda") // self.P
        self.x = self.xi(self.p[:, 0], self.p[:, 1])

    def _xi(self, kx, ky):
        cx, cy = math.cos(kx), math.cos(ky)
        return -2.0 * (cx + cy) - 4.0 * self.tp * cx * cy

    def xi(self, kx, ky):
        cx, cy = torch.cos(kx), torch.cos(ky)
        return -2.0 * (cx + cy) - 4.0 * self.tp * cx * cy

    def _edge(self, th):
        return math.pi / max(abs(math.cos(th)), abs(math.sin(th)))

    def _level(self, th, eps):
        c, s, lo, hi = math.cos(th), math.sin(th), 0.0, self._edge(th)
        if self._xi(hi * c, hi * s) < eps:
            return hi
        if self._xi(0.0, 0.0) >= eps:
            return 0.0
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            if mid == lo or mid == hi:
                break
            if self._xi(mid * c, mid * s) < eps:
                lo = mid
            else:
                hi = mid
        return 0.5 * (lo + hi)

    def _cells(self, th, sh):
        nr, nh, mid = self.nr, self.nr // 2, self.ns // 2
        lo = 0.0 if sh == 0 else self._level(th, (sh - 0.5 * self.ns) * self.D)
        hi = self._edge(th) if sh == self.ns - 1 else self._level(th, (sh + 1 - 0.5 * self.ns) * self.D)
        if sh != mid:
            return [(lo + (hi - lo) * i / nr, lo + (hi - lo) * (i + 1) / nr) for i in range(nr)]
        rf = self._level(th, 0.0)
        return [(lo + (rf - lo) * i / nh, lo + (rf - lo) * (i + 1) / nh) for i in range(nh)] + \
               [(rf + (hi - rf) * i / nh, rf + (hi - rf) * (i + 1) / nh) for i in range(nh)]

    def patch(self, kx, ky):
        tau = 2 * math.pi
        x, y = kx - tau * torch.round(kx / tau), ky - tau * torch.round(ky / tau)
        wd = torch.floor(torch.atan2(y, x) / self.dth + 0.5).long() % self.Na
        if self.ns == 1:
            return wd
        cx, cy = torch.cos(x), torch.cos(y)
        xi = -2.0 * (cx + cy) - 4.0 * self.tp * cx * cy
        return wd * self.ns + torch.clamp(torch.floor(xi / self.D + 0.5 * self.ns).long(), 0, self.ns - 1)

    # loop kernels: T-flow dD/dT, g-flow D, D(a, b) = (f(a) - f(b)) / (a - b)
    def _loop(self, pp, xp, xq, T, gflow):
        xb = -xq if pp else xq
        den, mid = xp - xb, 0.5 * (xp + xb)
        near = den.abs() < 1e-5 * T
        den = torch.where(near, torch.ones_like(den), den)
        if gflow:
            f, fc = torch.sigmoid, lambda v: torch.sigmoid(v)  # noqa: E731
            fa, fb = f(-xp / T), f(-xb / T)
            ca, cb = fc(xp / T), fc(xb / T)
            num = torch.where((xp < 0) & (xb < 0), cb - ca, fa - fb)
            at = -torch.sigmoid(mid / T) * torch.sigmoid(-mid / T) / T
        else:
            g = lambda v: v / (T * T) * torch.sigmoid(v / T) * torch.sigmoid(-v / T)  # noqa: E731
            num = g(xp) - g(xb)
            at = torch.sigmoid(mid / T) * torch.sigmoid(-mid / T) / T * (1 / T - mid * torch.tanh(mid / (2 * T)) / (T * T))
        v = torch.where(near, at, num / den)
        return -v if pp else v

    def rhs(self, T, V, Z, g=None, K=None):
        """dV / dT of (V, Z) (g given: dV / dg at fixed T with Katanin factors K)."""
        N = self.N
        NN = N * N
        out = torch.zeros(N, N, N, dtype=torch.float64, device="cuda")
        if g is None:
            lines = Z[:, None] * Z[None, :]
        else:
            kz = K * Z
            lines = g * Z[:, None] * Z[None, :] * (kz[:, None] + kz[None, :])
        chunk = max(1, (1 << 25) // self.M)
        i_of, l_of = torch.arange(NN, device="cuda") // N, torch.arange(NN, device="cuda") % N
        Vpp, Vcr = V.reshape(NN, N), V.reshape(N, NN).T
        Vd1, Vd2 = V.permute(2, 0, 1).reshape(NN, N), V.permute(2, 1, 0).reshape(NN, N)  # V[b,n,a], V[n,b,a]
        for pp in (True, False):
            for q0 in range(0, NN, chunk):
                Q = torch.arange(q0, min(NN, q0 + chunk), device="cuda")
                u, v = i_of[Q], l_of[Q]
                K2 = self.kf[u] + self.kf[v] if pp else self.kf[u] - self.kf[v]
                if pp:
                    qx, qy = K2[:, :1] - self.p[None, :, 0], K2[:, 1:] - self.p[None, :, 1]
                else:
                    qx, qy = self.p[None, :, 0] + K2[:, :1], self.p[None, :, 1] + K2[:, 1:]
                L = self.w * self._loop(pp, self.x[None, :].expand_as(qx), self.xi(qx, qy), T, g is not None)
                at = (torch.arange(len(Q), device="cuda")[:, None] * NN + self.pa[None, :] * N + self.patch(qx, qy)).reshape(-1)
                B = torch.zeros(len(Q) * NN, dtype=torch.float64, device="cuda").index_add_(0, at, L.reshape(-1))
                B = B.view(-1, N, N) * lines
                if pp:     # rows (i, j)
                    out.view(NN, N)[Q] -= (B * V[u, v][:, :, None]).reshape(-1, NN) @ Vpp
                else:      # crossed rows (l, j); direct rows (i, l)
                    out[:, v, u] -= ((B * V[:, v, u].T[:, None, :]).reshape(-1, NN) @ Vcr).T
                    via, vai = V[u, :, v], V[:, u, v].T
                    r = (B * (2 * via - vai)[:, :, None]).reshape(-1, NN) @ Vd1 - (B * via[:, :, None]).reshape(-1, NN) @ Vd2
                    out[u, :, v] += r
        return out

    def pairs(self, targets, T, V, Z, K=None, moments=None):
        """Chord slopes of the two-loop term at the targets or, with moments =
        (count, e_min, h, nbins), the pole weights' moments per bin of width h."""
        N, M, P = self.N, self.M, self.P
        f, fc = torch.sigmoid(-self.x / T), torch.sigmoid(self.x / T)
        wz = self.w * Z[self.pa]
        xj = self.xi(self.kf[:, 0], self.kf[:, 1])
        step = max(1, min(P, (1 << 25) // M))
        slopes = []
        for j in targets:
            acc = torch.zeros((), dtype=torch.float64, device="cuda")
            if moments:
                nm, e_min, h, nb = moments
                acc = torch.zeros(nm, nb, dtype=torch.float64, device="cuda")
            for p0 in range(0, M, step):
                p = slice(p0, min(M, p0 + step))
                a = self.pa[p]
                rx = (self.kf[j, 0] + self.p[p, :1]) - self.p[None, :, 0]
                ry = (self.kf[j, 1] + self.p[p, 1:]) - self.p[None, :, 1]
                xr, c = self.xi(rx, ry), self.patch(rx, ry)
                fr, fcr = torch.sigmoid(-xr / T), torch.sigmoid(xr / T)
                vab, vac = V[j][a][:, self.pa], torch.gather(V[j][a], 1, c)
                amp = (2 * vab - vac) * vab * (f[p, None] * fc * fcr + fc[p, None] * f * fr) * wz[p, None] * wz * Z[c]
                if K is not None:
                    za, zb, zc = Z[a][:, None], Z[self.pa][None, :], Z[c]
                    ka, kb, kc = (K * Z)[a][:, None], (K * Z)[self.pa][None, :], (K * Z)[c]
                    amp = amp * (ka * (zb + zc) + kb * (za + zc) + kc * (za + zb)) / 6
                E = self.x + xr - self.x[p, None]
                if moments:
                    b = ((E - e_min) / h).floor().clamp(0, nb - 1)
                    d, b = E - (e_min + (b + 0.5) * h), b.long().reshape(-1)
                    for m in range(nm):
                        acc[m].index_add_(0, b, amp.reshape(-1))
                        amp = amp * d
                else:
                    d, e2 = xj[j] - E, self.eta ** 2
                    dp, dm = d + 2 * T, d - 2 * T
                    acc = acc + (amp * (e2 - dp * dm) / ((dp * dp + e2) * (dm * dm + e2))).sum()
            slopes.append(acc)
        return torch.stack(slopes)

    def z(self, T, V, Z):
        return 1 / (1 - self.pairs(range(self.N), T, V, Z))

    def sigma(self, T, V, Z, omega, sym):
        """Sigma on the grid from moments 0..7 in bins of eta / 16 (1e-12 of a pole)."""
        N, h = self.N, self.eta / 16
        top = 3 * (4 + 4 * abs(self.tp))
        nb, nm = int(2 * top / h) + 2, 8
        # a symmetric vertex needs the irreducible patches and the zone-edge ones
        # (where the diagonals are patch centres: no momentum on a wedge boundary)
        q = N // 4
        fold = sym and N % 8 == 0 and self.nt % 2 == 0
        rep = [min(j % q, q - j % q) if fold and j % q else j for j in range(N)]
        need = sorted(set(rep))
        H = self.pairs(need, T, V, Z, moments=(nm, -top, h, nb))
        E = -top + (torch.arange(nb, dtype=torch.float64, device="cuda") + 0.5) * h
        out = torch.zeros(len(need), len(omega), dtype=torch.complex128, device="cuda")
        for m0 in range(0, len(omega), 64):
            u = 1 / (torch.tensor(omega[m0:m0 + 64], device="cuda")[:, None] + 1j * self.eta - E)
            g = u.clone()
            for n in range(nm):
                out[:, m0:m0 + 64] += H[:, n].to(torch.complex128) @ g.T
                g = g * u
        S = out[torch.tensor([need.index(r) for r in rep], device="cuda")]
        return S.real.contiguous(), S.imag.contiguous()


def _rk4(f, y, h):
    add = lambda a, s, b: [u + s * v for u, v in zip(a, b)]  # noqa: E731
    k1 = f(0.0, y)
    k2 = f(0.5, add(y, 0.5 * h, k1))
    k3 = f(0.5, add(y, 0.5 * h, k2))
    k4 = f(1.0, add(y, h, k3))
    return [u + h / 6 * (a + 2 * b + 2 * c + d) for u, a, b, c, d in zip(y, k1, k2, k3, k4)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        return None
    N, M = case["N"], case["N"] * case["nt"] * case["nr"]
    calls = {"rhs": 0, "sigma": 1 + bool(case.get("n_omega")), "step": 1, "gstep": 4}[kind]
    if calls * N * float(M) ** 2 > 2.2e10 or 2.0 * N * N * M > 4e9:
        return None      # minutes of FP64 pairs
    V, Z = (torch.from_numpy(x).cuda() for x in _vertex(case, seed))
    T = case["T"]
    P = _Plain(case, 0.05 if kind == "gstep" else ETA)
    if kind == "rhs":
        return P.rhs(T, V, Z)
    if kind == "sigma":
        out = dict(Z=P.z(T, V, Z))
        if case["n_omega"]:
            out["re"], out["im"] = P.sigma(T, V, Z, np.linspace(-4.0, 4.0, case["n_omega"]), case["sym"])
        return out
    if kind == "step":
        Zs = P.z(T, V, Z)
        f = lambda c, y: [T * math.exp(c * DLNT) * P.rhs(T * math.exp(c * DLNT), y[0], Zs)]  # noqa: E731
        return dict(V=_rk4(f, [V], DLNT)[0], Z=Zs)
    g0 = case["g"]

    def zka(g, s1, s2):
        z = 1 / (1 - g * s1)
        return z, 1 + g * g * s2, 2 * z * (s1 + g * s2)

    def slope(c, y):
        g = g0 + c * DG
        z, k, a = zka(g, y[1], y[2])
        return [P.rhs(T, y[0], z, g, k), y[2], a.mean() * y[2] + 6 * g * P.pairs(range(N), T, y[0], z, k)]

    s = torch.from_numpy(_gflow_state(case, seed)).cuda()
    V, s1, s2 = _rk4(slope, [V, s[:N], s[N:]], DG)
    z, k, a = zka(g0 + DG, s1, s2)
    return dict(V=V, Z=z, slopes=torch.stack([s1, s2]), zka=torch.cat([z, k, a, a.mean()[None]]))
