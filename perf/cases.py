"""Performance cases of the reactive-mixture lattice Boltzmann library.

Each case is one pass through the public Solver calls that a simulation is
made of: time steps (in the three precisions, with periodic and with
ghost-node x faces, one lattice or a batch, constant or mixture-averaged
transport), whole short runs, the reported fields, the heat-release
objective with its sensitivities, and the gradient through time.

  listed()            the cases, each with a comment on what it stands for
  draw(rng)           one more case of the same ranges
  prepare(case, seed) a solver holding an initial state made from the seed
  run(state)          one pass, and its outputs
  work(case)          bytes and floating-point operations of one pass
  exact(case, seed)   the outputs in 64 bits from the method's formulas,
                      written out in plain torch below

Mechanisms and lattices come from workload/ (the seeded three-gas and
nine-species inputs); the initial fields are formed here, on the device.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import workload as w
from paper_2101_01702_gb300 import lbm

PRECISIONS = {"fp64": lbm.LBM_FP64, "mixed": lbm.LBM_MIXED, "mixed_fast": lbm.LBM_MIXED_FAST}
ALL_FIELDS = (lbm.LBM_F_RHO_A | lbm.LBM_F_RHOU | lbm.LBM_F_RHOE | lbm.LBM_F_T | lbm.LBM_F_P | lbm.LBM_F_Y
              | lbm.LBM_F_J_A | lbm.LBM_F_RHO_DOT | lbm.LBM_F_HRR)
DEV = "cuda"


def _case(name, op, problem, nx, ny, nz, precision, steps=0, transport="constant", flames=0):
    c = {"op": op, "problem": problem, "nx": nx, "ny": ny, "nz": nz, "precision": precision, "steps": steps,
         "transport": transport, "flames": flames}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest problem anyone runs: three gases on 1024 nodes, double,
        # fields in, a few steps, fields out; launches and latency count
        _case("gases_64x4x4_fp64", "whole", "gases", 64, 4, 4, "fp64", steps=20),
        # a short flame tube with ghost-node faces, as in parameter scans
        _case("tube_512x4x4_mixed", "step", "tube", 512, 4, 4, "mixed", steps=10),
        # the flame-speed tube in double, the mode of validation runs
        _case("tube_4096x4x4_fp64", "step", "tube", 4096, 4, 4, "fp64", steps=4),
        # the expanding flame in double at a size of everyday use
        _case("sphere_128_fp64", "step", "sphere", 128, 128, 128, "fp64", steps=1),
        # the expanding flame at production size in the production precision
        _case("sphere_256_mixed", "step", "sphere", 256, 256, 256, "mixed", steps=1),
        # the same in the fast mixed precision
        _case("sphere_160_mixed_fast", "step", "sphere", 160, 160, 160, "mixed_fast", steps=1),
        # a ragged box (no dimension a multiple of a warp or a block) with
        # mixture-averaged transport
        _case("box_131x97x73_transport", "step", "sphere", 131, 97, 73, "mixed", steps=1, transport="mixture"),
        # 48 flames of ragged lengths side by side, replayed from a graph
        _case("flames48_graph_mixed", "graph", "flames", 0, 4, 4, "mixed", steps=2, flames=48),
        # a whole short run on a mid-sized box: initial fields in, a few
        # steps, every reported field out
        _case("run_72x60x44_fp64", "whole", "sphere", 72, 60, 44, "fp64", steps=4),
        # the reported fields of a production state (output of a running job)
        _case("moments_160_mixed", "moments", "sphere", 160, 160, 160, "mixed"),
        # the heat release with its sensitivities at a state
        _case("heat_release_128_mixed", "heat_release", "sphere", 128, 128, 128, "mixed"),
        # gradients of the time-integrated heat release, forward and reverse
        # sweep with checkpoints, on the periodic flame tube
        _case("gradient_512x4x4_fp64", "gradient", "ring", 512, 4, 4, "fp64", steps=24),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, nodes):
    """Three dimensions of at least 4, of about the given product, within a factor of four of a cube."""
    a = nodes ** (1.0 / 3.0)
    nx = max(4, int(a * math.exp(rng.uniform(-0.7, 0.7))))
    ny = max(4, int(math.sqrt(nodes / nx) * math.exp(rng.uniform(-0.3, 0.3))))
    return nx, ny, max(4, int(nodes / (nx * ny)))


def draw(rng):
    kind = rng.choice(["gases", "tube", "tube", "sphere", "sphere", "sphere", "flames", "whole", "moments",
                       "heat_release", "gradient"])
    precision = rng.choice(["fp64", "mixed", "mixed", "mixed_fast"])
    most = {"fp64": 2.0e6, "mixed": 1.4e7, "mixed_fast": 1.4e7}[precision]
    if kind == "gases":
        return _case("", "whole", "gases", _log_int(rng, 24, 400), rng.randint(4, 9), rng.randint(4, 9), "fp64",
                     steps=rng.randint(4, 20))
    if kind == "tube":
        return _case("", rng.choice(["step", "graph"]), "tube", _log_int(rng, 200, 8000), rng.randint(4, 7), 4,
                     precision, steps=rng.randint(1, 5))
    if kind == "sphere":
        return _case("", "step", "sphere", *_box(rng, _log_int(rng, 8e3, most)), precision, steps=1,
                     transport=rng.choice(["constant", "constant", "mixture"]))
    if kind == "flames":
        return _case("", "graph", "flames", 0, 4, 4, precision, steps=rng.randint(1, 3), flames=rng.randint(3, 40))
    if kind == "whole":
        return _case("", "whole", "sphere", *_box(rng, _log_int(rng, 8e3, 3e5)), "fp64", steps=rng.randint(1, 5))
    if kind == "moments":
        return _case("", "moments", "sphere", *_box(rng, _log_int(rng, 8e3, 6e6)), precision)
    if kind == "heat_release":
        return _case("", "heat_release", "sphere", *_box(rng, _log_int(rng, 8e3, 3e6)), precision)
    return _case("", "gradient", "ring", _log_int(rng, 40, 600), 4, 4, "fp64", steps=rng.randint(5, 24))


# ---------------------------------------------------------------------------
# Problems: lattice, tables and initial fields from the seed
# ---------------------------------------------------------------------------
def _lengths(case):
    """Lengths of a batch's flames: as drawn for the 48-flame batch, the first of them."""
    return [int(v) for v in w.batched_flames_lengths(count=48)[0][:case["flames"]]]


def _lattice(case):
    if case["problem"] == "flames":
        seg = _lengths(case)
        return w.LatticeSpec(sum(seg), case["ny"], case["nz"], 1, seg_nx=seg)
    return w.LatticeSpec(case["nx"], case["ny"], case["nz"], 1 if case["problem"] == "tube" else 0)


def _tables(case):
    sp, mech = w.mech3() if case["problem"] == "gases" else w.mech9()
    if case["transport"] == "mixture":
        X = np.maximum([0.296, 0.148, 0, 0, 0, 0, 0, 0, 0.556], 1e-12)
        sp = w.with_mixture_transport(sp, X, mech.P0, 300.0)
    return sp, mech


def _phi_mixture(phi):
    """Unburnt H2/O2/N2 mole fractions 2 phi : 1 : 3.76; phi a number or a tensor."""
    phi = torch.as_tensor(phi, dtype=torch.float64, device=DEV)
    X = torch.full((9,) + phi.shape, 1e-12, dtype=torch.float64, device=DEV)
    tot = 2.0 * phi + 4.76
    X[0], X[1], X[8] = 2.0 * phi / tot, 1.0 / tot, 3.76 / tot
    return X / X.sum(0)


def _fields(case, lat, sp, mech, seed):
    """Initial mole fractions X [M, N], temperature T [N] and pressure, on the device."""
    gen = torch.Generator(device=DEV).manual_seed(seed)

    def uniform(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(shape, generator=gen, dtype=torch.float64, device=DEV)

    N, nx, ny = lat.n_nodes, lat.nx, lat.ny
    # a little water and radicals, so that the chain reactions run from the first step
    radicals = torch.tensor([0.0, 0.0, 0.02, 2e-3, 2e-3, 4e-3, 1e-4, 1e-4, 0.0], dtype=torch.float64,
                            device=DEV)[:, None]
    n = torch.arange(N, device=DEV)
    x, y, z = n % nx, (n // nx) % ny, n // (nx * ny)
    kind = case["problem"]
    if kind == "gases":
        # hot slab across an eighth of the box, +-1e-3 composition noise
        X = torch.tensor([0.3, 0.5, 0.2], dtype=torch.float64, device=DEV)[:, None] + uniform(-1e-3, 1e-3, 3, N)
        T = torch.where((16 * x >= 7 * nx) & (16 * x < 9 * nx), 4.0, 1.0).to(torch.float64)
        P = sp.r_lat / float(np.dot([0.3, 0.5, 0.2], sp.W))
        return X / X.sum(0), T, P
    if kind in ("tube", "ring", "flames"):
        # unburnt gas at 300 K, the rightmost fifth of each flame at its slab temperature
        seg = lat.seg_nx or [nx]
        K = len(seg)
        L = torch.tensor(seg, device=DEV)
        k = torch.repeat_interleave(torch.arange(K, device=DEV), L)[x]
        x0 = (L.cumsum(0) - L)[k]
        phi, Ts = uniform(0.5, 3.0, K), uniform(1400.0, 1600.0, K)
        X = _phi_mixture(phi)[:, k]
        if kind == "ring":
            X = (X + radicals) / (1.0 + radicals.sum())
        T = torch.where(x - x0 >= torch.round(0.8 * L[k].double()).long(), Ts[k], 300.0)
        return X.contiguous(), T, mech.P0
    # the expanding flame: phi = 1 with +-1e-3 noise on the species present and
    # a hot kernel at 2000 K
    X = _phi_mixture(torch.ones(1))[:, :1].expand(9, N) + radicals
    for s in (0, 1, 8):
        X[s] += uniform(-1e-3, 1e-3, N)
    r2 = (x - nx // 2) ** 2 + (y - ny // 2) ** 2 + (z - lat.nz // 2) ** 2
    hot = r2 < max(3.0, min(nx, ny, lat.nz) * (20.0 / 256.0)) ** 2
    T = torch.where(hot, 2000.0, 300.0).to(torch.float64)
    return (X / X.sum(0)).contiguous(), T, mech.P0


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _views(buf, M, N, precision):
    """The populations of a state buffer: sets, directions, nodes (layout of include/lbm.h)."""
    if precision == "fp64":
        return {"populations": buf.view(torch.float64).view(M + 1, 27, N)}
    nb = (M * 27 * N * 4 + 15) // 16 * 16
    mov = buf[:M * 27 * N * 4].view(torch.float32).view(M, 27, N)
    dbl = buf[nb:].view(torch.float64)
    # the float block's rest slot is not used: rest populations are the first doubles
    return {"moving_a": mov[:, :13], "moving_b": mov[:, 14:], "rest": dbl[:M * N].view(M, N),
            "energy": dbl[M * N:(M + 27) * N].view(27, N)}


def prepare(case, seed):
    lat = _lattice(case)
    sp, mech = _tables(case)
    X, T, P = _fields(case, lat, sp, mech, seed)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream() if case["op"] == "graph" else None
    s = lbm.Solver(lat, sp, mech, PRECISIONS[case["precision"]], stream=stream)
    s.init(X, T, None, P)
    views = {b.data_ptr(): _views(b, s.M, s.N, case["precision"]) for b in s.pop}
    keep = (X, T, P) if case["op"] in ("whole", "gradient") else None
    return {"case": case, "solver": s, "views": views, "T": s.macro[:s.N], "fields": keep}


def _state(st):
    """The current state: the buffer that holds it, and the temperature row."""
    return {**st["views"][lbm.lbm_state_buffer(st["solver"].ctx)], "T": st["T"]}


def run(state):
    c, s = state["case"], state["solver"]
    op = c["op"]
    if op == "step":
        s.step(c["steps"])
        return _state(state)
    if op == "graph":
        s.step_graph(c["steps"])
        return _state(state)
    if op == "moments":
        return s.moments(ALL_FIELDS, device=True)
    if op == "heat_release":
        J, dA, dT, drho = s.heat_release(device=True)
        return {"J": J, "dlogA": dA, "dT": dT, "drho": drho}
    X, T, P = state["fields"]
    s.init(X, T, None, P)
    if op == "whole":
        s.step(c["steps"])
        return s.moments(ALL_FIELDS, device=True)
    J, dA, dT0, _ = s.heat_release_gradient(c["steps"], checkpoint_every=8)
    return {"J": J, "dlogA": dA, "dT0": dT0}


# ---------------------------------------------------------------------------
# Bytes and operations
# ---------------------------------------------------------------------------
def work(case):
    M, R = (3, 1) if case["problem"] == "gases" else (9, 21)
    N = _lattice(case).n_nodes
    state = N * ((M + 1) * 27 * 8 if case["precision"] == "fp64" else M * 26 * 4 + (M + 27) * 8)
    # a node's operations: moments, temperature and thermodynamics, the
    # Stefan-Maxwell solve, the rates, the collisions with their cross terms
    moments = 60 * (M + 1)
    node = 100 + 40 * M + moments
    solve = 2 * (M ** 3 / 3 + 6 * M * M) / 2
    rates = 40 * M + 40 * R
    collide = 27 * (2 * M * (M - 1) + 14 * M)
    step = {"bytes": 2 * state, "flops": N * (node + solve + rates + collide)}
    fields = 8 * N * (5 * M + 3 + 4 + M)
    op, k = case["op"], case["steps"]
    if op in ("step", "graph"):
        return {m: k * v for m, v in step.items()}
    if op == "moments":
        return {"bytes": state + 8 * N + fields, "flops": N * (node + rates)}
    if op == "heat_release":
        return {"bytes": state + 8 * N * (M + 2), "flops": N * (node + 2 * rates + 20 * R)}
    if op == "whole":
        return {"bytes": 8 * N * (M + 1) + 2 * state + (k - 1) * step["bytes"] + fields,
                "flops": N * 27 * 6 * (M + 1) + k * step["flops"] + N * (node + rates)}
    # the gradient: every step forward and its transpose (about twice a step)
    return {"bytes": 8 * N * (M + 1) + k * (2 * step["bytes"] + 2 * state), "flops": 3 * k * step["flops"]}


# ---------------------------------------------------------------------------
# The method in 64 bits, in plain torch (fields are [.., N], N = nz ny nx)
# ---------------------------------------------------------------------------
_C = [(i % 3 - 1, (i // 3) % 3 - 1, i // 9 - 1) for i in range(27)]


class _Method:
    def __init__(self, lat, sp, mech, log_A=None):
        def t(a):
            return torch.tensor(np.asarray(a, dtype=np.float64), device=DEV)

        self.lat, self.sp, self.mech, self.M = lat, sp, mech, sp.M
        self.W, self.Ra = t(sp.W), t(sp.r_lat / sp.W)
        self.c = t(_C).T                                                  # [3, 27]
        self.w = t([math.prod((2 / 3 if v == 0 else 1 / 6) for v in c) for c in _C])
        self.log_A = t(mech.log_A) if log_A is None else log_A
        self.A = t([[0.0 if a == b else 1.0 / (sp.W[a] * sp.W[b] * sp.D[a][b]) for b in range(sp.M)]
                    for a in range(sp.M)])
        # U_a(T) = sum_k u[a][k] T^k
        u = np.zeros((sp.M, 6))
        for a in range(sp.M):
            R = sp.r_lat / sp.W[a]
            if sp.thermo == 0:
                u[a, 1] = (sp.cp_R[a] - 1.0) * R
                u[a, 0] = sp.h_form[a] - R * sp.T0 - u[a, 1] * sp.T0
            else:
                p = sp.poly7[a]
                u[a] = R * np.array([p[5], p[0] - 1.0, p[1] / 2, p[2] / 3, p[3] / 4, p[4] / 5])
        self.u = t(u)
        seg = lat.seg_nx or [lat.nx]
        ends = np.cumsum(seg)
        self.x0, self.x1 = torch.tensor(ends - seg, device=DEV), torch.tensor(ends - 1, device=DEV)
        lo, hi = np.repeat(ends - seg, seg), np.repeat(ends - 1, seg)
        x = np.arange(lat.nx)
        self.shift = {}
        for c in (-1, 0, 1):
            xn = (x + c) % lat.nx if lat.bc_x == 0 else np.clip(x + c, lo, hi)
            self.shift[c] = torch.tensor(xn, device=DEV)

    # lattice -----------------------------------------------------------
    def grid(self, f):
        return f.reshape(f.shape[:-1] + (self.lat.nz, self.lat.ny, self.lat.nx))

    def grad(self, f):
        """(1/theta) sum_i w_i c_i f(x + c_i), axis by axis: [3, .., N]."""
        g = self.grid(f)
        xp, xm = g.index_select(-1, self.shift[1]), g.index_select(-1, self.shift[-1])
        sx, dx = (4 * g + xp + xm) / 6, (xp - xm) / 6

        def axis(v, d):
            p, m = torch.roll(v, -1, d), torch.roll(v, 1, d)
            return (4 * v + p + m) / 6, (p - m) / 6

        sy_sx, dy_sx = axis(sx, -2)
        sy_dx, _ = axis(dx, -2)
        out = [axis(sy_dx, -3)[0], axis(dy_sx, -3)[0], axis(sy_sx, -3)[1]]
        return 3.0 * torch.stack([v.reshape(f.shape) for v in out])

    def pull(self, F, T_start):
        """s_i(x) = s_i(x - c_i) of every set; equilibrium ghost nodes beyond non-periodic x faces."""
        lat, sides = self.lat, None
        if lat.bc_x == 1:
            sides = []
            for left, xb in ((True, self.x0), (False, self.x1)):
                b = [self.grid(f)[..., xb].reshape(27, -1) for f in F]
                rho_a, u, T = self.node_state(b, self.grid(T_start)[..., xb].reshape(-1))[:3]
                eq = self.equilibria(rho_a, torch.zeros_like(u) if left else u, T)
                sides.append([e.reshape(27, lat.nz, lat.ny, -1) for e in eq])
        out = []
        for s in range(len(F)):
            g, rows = self.grid(F[s]), []
            for i, (cx, cy, cz) in enumerate(_C):
                v = torch.roll(g[i], (cz, cy, cx), (0, 1, 2))
                if sides is not None and cx != 0:
                    k, xb = (0, self.x0) if cx > 0 else (1, self.x1)
                    v[..., xb] = torch.roll(sides[k][s][i], (cz, cy), (0, 1))
                rows.append(v.reshape(-1))
            out.append(torch.stack(rows))
            F[s] = None if not torch.is_grad_enabled() else F[s]
        return out

    # thermodynamics ----------------------------------------------------
    @staticmethod
    def poly(u, T):
        r = u[5]
        for k in range(4, -1, -1):
            r = r * T + u[k]
        return r

    @staticmethod
    def dpoly(u, T):
        r = 5 * u[5]
        for k in range(4, 0, -1):
            r = r * T + k * u[k]
        return r

    def temperature(self, Y, e, T):
        eu = self.u.T @ Y
        with torch.no_grad():
            for _ in range(12):
                T = T - (self.poly(eu, T) - e) / self.dpoly(eu, T)
        T = T.detach()
        return T - (self.poly(eu, T) - e) / self.dpoly(eu, T)          # carries the derivatives

    def enthalpy(self, T):
        return self.poly(self.u.T[:, :, None], T) + self.Ra[:, None] * T

    def product_form(self, rho, v, zeta):
        """rho Psi_cx Psi_cy Psi_cz for the 27 directions: [27, N]."""
        ax = []
        for d in range(3):
            s = v[d] * v[d] + zeta
            ax.append(torch.stack([(s - v[d]) / 2, 1.0 - s, (s + v[d]) / 2]))
        return ((rho * ax[2])[:, None, None] * ax[1][None, :, None] * ax[0][None, None, :]).reshape(27, -1)

    def energy_set(self, rhoE, q, Rm):
        """The energy populations with moments rhoE, q [3], Rm [3, 3]."""
        c, second = self.c, 0.0
        for a in range(3):
            for b in range(3):
                cc = c[a] * c[b] - (1.0 / 3.0 if a == b else 0.0)
                second = second + cc[:, None] * (Rm[a][b] - (rhoE / 3.0 if a == b else 0.0))
        first = c.T @ q
        return self.w[:, None] * (rhoE + 3.0 * first + 4.5 * second)

    def energy_moments(self, rho, u, P, Hk):
        Rm = [[Hk * (rho * u[a] * u[b] + (P if a == b else 0.0)) + P * u[a] * u[b] for b in range(3)]
              for a in range(3)]
        return Hk * rho * u, Rm

    def equilibria(self, rho_a, u, T):
        rho = rho_a.sum(0)
        Y = rho_a / rho
        Rm = self.sp.r_lat * (Y / self.W[:, None]).sum(0)
        usq = (u * u).sum(0)
        out = [self.product_form(rho_a[s], u, self.Ra[s] * T) for s in range(self.M - 1)]
        out.append(self.product_form(rho, u, Rm * T))
        U, H = (Y * self.poly(self.u.T[:, :, None], T)).sum(0), (Y * self.enthalpy(T)).sum(0)
        q, R2 = self.energy_moments(rho, u, rho * Rm * T, H + usq / 2)
        out.append(self.energy_set(rho * (U + usq / 2), q, R2))
        return out

    def initial(self, X, T, P):
        m = (X * self.W[:, None]).sum(0)
        rho = P / (self.sp.r_lat / m * T)
        return self.equilibria(rho * X * self.W[:, None] / m, torch.zeros((3,) + T.shape, device=DEV).double(), T)

    # a node's state ------------------------------------------------------
    def node_state(self, F, T_start):
        M = self.M
        rho_s = [F[s].sum(0) for s in range(M)]
        rho = rho_s[M - 1]
        rho_a = torch.stack(rho_s[:M - 1] + [rho - sum(rho_s[:M - 1])])
        j = self.c @ F[M - 1]
        u = j / rho
        rhoE = F[M].sum(0)
        T = self.temperature(rho_a / rho, rhoE / rho - (u * u).sum(0) / 2, T_start)
        return rho_a, u, T, rho, j, rhoE

    def rates(self, rho_a, T):
        """Production rates [M, N] (Eq. (sumRhoDot))."""
        sp, me, M = self.sp, self.mech, self.M
        conc = rho_a / self.W[:, None]
        H = self.enthalpy(T) / (self.Ra[:, None] * T)
        if sp.thermo == 0:
            S = torch.tensor(sp.cp_R, device=DEV)[:, None] * torch.log(T / sp.T0)
        else:
            p = torch.tensor(sp.poly7.T, device=DEV)[:, :, None]
            S = p[0] * torch.log(T) + T * (p[1] + T * (p[2] / 2 + T * (p[3] / 3 + T * p[4] / 4))) + p[6]
        g = H - S
        dot = [0.0] * M
        lnT = torch.log(T / me.T_ref)
        for k in range(me.R):
            ln_kf = self.log_A[k] + float(me.b[k]) * lnT - float(me.theta[k]) / T
            kf = torch.exp(ln_kf)
            cM = None
            if me.rtype[k] != 0:
                cM = sum(float(me.eff[k, a]) * conc[a] for a in range(M))
            if me.rtype[k] == 2:
                k0 = torch.exp(float(me.low[k, 0]) + float(me.low[k, 1]) * lnT - float(me.low[k, 2]) / T)
                Pr = k0 * cM / kf
                kf = kf * Pr / (1.0 + Pr)
            qf, dn = kf, 0
            for a in range(M):
                for _ in range(int(me.nu_f[k, a])):
                    qf = qf * conc[a]
            q = qf
            if me.reversible[k]:
                dG = 0.0
                for a in range(M):
                    d = int(me.nu_r[k, a]) - int(me.nu_f[k, a])
                    if d:
                        dG, dn = dG + d * g[a], dn + d
                qr = kf * torch.exp(dG) * (me.P0 / (sp.r_lat * T)) ** (-dn)
                for a in range(M):
                    for _ in range(int(me.nu_r[k, a])):
                        qr = qr * conc[a]
                q = qf - qr
            if me.rtype[k] == 1:
                q = q * cM
            for a in range(M):
                d = int(me.nu_r[k, a]) - int(me.nu_f[k, a])
                if d:
                    dot[a] = dot[a] + (float(self.sp.W[a]) * d) * q
        return torch.stack([v if torch.is_tensor(v) else torch.zeros_like(T) for v in dot])

    def heat_release(self, rho_a, T):
        return -(self.enthalpy(T) * self.rates(rho_a, T)).sum(0)

    def relaxation(self, Y, Rm, T, P):
        """1/omega - 1/2, 1/omega_1 - 1/2, and the factor of the binary diffusivities."""
        sp = self.sp
        if not sp.transport:
            nup = sp.nu / (Rm * T) if sp.visc_model == 0 else torch.full_like(T, sp.nu)
            return nup, nup / sp.Pr, 1.0
        X = Y / self.W[:, None] / (Y / self.W[:, None]).sum(0)
        mu = [float(sp.mu0[a]) * (T / sp.T_tr) ** float(sp.mu_exp[a]) for a in range(self.M)]
        num = ls = lr = 0.0
        cv = self.dpoly(self.u.T[:, :, None], T)
        for a in range(self.M):
            den = 0.0
            for b in range(self.M):
                r = 1.0 + torch.sqrt(mu[a] / mu[b]) * float(sp.W[b] / sp.W[a]) ** 0.25
                den = den + X[b] * r * r / math.sqrt(8.0 * (1.0 + float(sp.W[a] / sp.W[b])))
            lam = mu[a] * (cv[a] + 2.25 * float(self.Ra[a]))
            num, ls, lr = num + X[a] * mu[a] / den, ls + X[a] * lam, lr + X[a] / lam
        Cp = (Y * cv).sum(0) + Rm
        return num / P, 0.5 * (ls + 1.0 / lr) / (P * Cp), (T / sp.T_tr) ** sp.D_exp * sp.P_tr / P

    def diffusion(self, Y, u, ua, kappa):
        """Diffusion velocities [M, 3, N] of Eq. (transform1), and 1/tau_a [M, N]."""
        M = self.M
        B = [[None] * M for _ in range(M)]
        ita = kappa * (self.A @ Y)
        for a in range(M):
            for b in range(M):
                B[a][b] = 1.0 + ita[a] / 2 if a == b else -0.5 * float(self.A[a, b]) * kappa * Y[b]
        r = [ua[a] - u for a in range(M)]
        for k in range(M):
            for a in range(k + 1, M):
                f = B[a][k] / B[k][k]
                for b in range(k + 1, M):
                    B[a][b] = B[a][b] - f * B[k][b]
                r[a] = r[a] - f * r[k]
        x = [None] * M
        for a in range(M - 1, -1, -1):
            x[a] = (r[a] - sum((B[a][b] * x[b] for b in range(a + 1, M)), torch.zeros_like(u))) / B[a][a]
        return torch.stack(x), ita

    # one step ------------------------------------------------------------
    def moments(self, Pl, T_start):
        """The state of the pulled sets Pl: rho_a, u, T, rho, j, rhoE, j_a."""
        rho_a, u, T, rho, j, rhoE = self.node_state(Pl, T_start)
        ja = [self.c @ Pl[s] for s in range(self.M - 1)]
        return rho_a, u, T, rho, j, rhoE, torch.stack(ja + [j - sum(ja)])

    def record(self, Pl, T_start):
        sp, M = self.sp, self.M
        rho_a, u, T, rho, j, rhoE, ja = self.moments(Pl, T_start)
        Y = rho_a / rho
        inv_m = (Y / self.W[:, None]).sum(0)
        Rm = sp.r_lat * inv_m
        P = rho * Rm * T
        nup, nup1, dfac = self.relaxation(Y, Rm, T, P)
        kappa = sp.r_lat * T / inv_m / dfac
        ua = [ja[a] / rho_a[a] for a in range(M)]
        du, ita = self.diffusion(Y, u, ua, kappa)
        return rho_a, u, T, rho, rhoE, Y, Rm, P, nup, nup1, kappa, du, ita

    def step(self, F, T_start):
        M, Pl = self.M, self.pull(F, T_start)
        rho_a, u, T, rho, rhoE, Y, Rm, P, nup, nup1, kappa, du, ita = self.record(Pl, T_start)
        om, om1 = 1.0 / (0.5 + nup), 1.0 / (0.5 + nup1)
        beta = ita / (2.0 + ita)
        X = [None] * 3
        for a in range(3):
            G = nup * self.grad(rho * u[a] * (1.0 - 3.0 * Rm * T) - rho * u[a] ** 3)[a]
            X[a] = -self.grad(G)[a]
        dot = self.rates(rho_a, T)
        out = []
        eq = [self.product_form(torch.ones_like(T), u, self.Ra[b] * T) for b in range(M)]
        D = [rho_a[b] * (eq[b] - self.product_form(torch.ones_like(T), u + du[b], self.Ra[b] * T)) for b in range(M)]
        for a in range(M - 1):
            cross = 0.0
            for b in range(M):
                if b != a:
                    cross = cross + float(self.A[a, b]) * D[b]
            cross = cross * (kappa * Y[a])
            f = Pl[a]
            out.append(f + 2.0 * beta[a] * (rho_a[a] * eq[a] - f) + (beta[a] - 1.0) * cross + dot[a] * eq[a])
        del D, eq
        f = Pl[M - 1]
        axis = ((self.c * self.c).sum(0) == 1).double()
        fm = f + om * (self.product_form(rho, u, Rm * T) - f) + (axis * 0.5)[:, None] * (self.c.T @ torch.stack(X))
        # energy set
        c, g = self.c, Pl[M]
        H_a = self.enthalpy(T)
        Hk = (Y * H_a).sum(0) + (u * u).sum(0) / 2
        qeq, Req = self.energy_moments(rho, u, P, Hk)
        q = c @ g
        HgY = (H_a * self.grad(Y)).sum(1)
        dq = []
        for d in range(3):
            uP = sum(u[a] * (((c[a] * c[d]) @ f) - rho * u[a] * u[d] - (P if a == d else 0.0)) for a in range(3))
            dq.append((om - om1) * (q[d] - uP - qeq[d]) + om1 * rho * (H_a * Y * du[:, d]).sum(0)
                      + 0.5 * (2.0 - om1) * P * HgY[d])
        geq = self.energy_set(rhoE, qeq, Req)
        gn = g + om * (geq - g) + 3.0 * self.w[:, None] * (c.T @ torch.stack(dq))
        return out + [fm, gn], T


def _references(m, X, T, P):
    """Rest states from which the mixed modes store deviations: float32 [M, 27]."""
    mean_W = (X * m.W[:, None]).sum(0)
    rho = P * mean_W / (m.sp.r_lat * T)
    rho_a = rho * X * m.W[:, None] / mean_W
    inv_m = sum(float(rho_a[a].mean()) / float(rho.mean()) / float(m.W[a]) for a in range(m.M))
    ref = torch.zeros((m.M, 27), dtype=torch.float64, device=DEV)
    for s in range(m.M):
        last = s == m.M - 1
        zeta = (m.sp.r_lat * inv_m if last else float(m.Ra[s])) * float(T.mean())
        low = float(rho.min()) if last else float(rho_a[s].min())
        for i, c in enumerate(_C):
            ref[s, i] = low * math.prod(1.0 - zeta if v == 0 else 0.5 * zeta for v in c)
    return ref.float().double()


def exact(case, seed):
    lat = _lattice(case)
    sp, mech = _tables(case)
    X, T, P = _fields(case, lat, sp, mech, seed)
    op, k = case["op"], case["steps"]
    if op == "gradient":
        log_A = torch.tensor(mech.log_A, device=DEV, requires_grad=True)
        T0 = T.clone().requires_grad_(True)
        m = _Method(lat, sp, mech, log_A)
        return _exact_gradient(m, X, T0, P, k, log_A)
    m = _Method(lat, sp, mech)
    if op == "heat_release":
        return _exact_heat_release(m, X, T, P)
    with torch.no_grad():
        ref = _references(m, X, T, P) if case["precision"] != "fp64" else None
        F = m.initial(X, T, P)
        del X
        for _ in range(k):
            F, T = m.step(F, T)
        if op in ("step", "graph"):
            if ref is None:
                return {"populations": torch.stack(F), "T": T}
            mov = torch.stack([F[s] - ref[s][:, None] for s in range(m.M)])
            return {"moving_a": mov[:, :13], "moving_b": mov[:, 14:],
                    "rest": torch.stack([F[s][13] for s in range(m.M)]), "energy": F[m.M], "T": T}
        rho_a, u, T, rho, j, rhoE, ja = m.moments(m.pull(F, T), T)
        Y = rho_a / rho
        return {"rho_a": rho_a, "rhou": j, "rhoE": rhoE, "T": T,
                "P": rho * sp.r_lat * (Y / m.W[:, None]).sum(0) * T, "Y": Y, "j_a": ja,
                "rho_dot": m.rates(rho_a, T), "hrr": m.heat_release(rho_a, T)}


def _exact_heat_release(m, X, T, P):
    with torch.no_grad():
        rho_a, u, T = m.node_state(m.pull(m.initial(X, T, P), T), T)[:3]
    log_A = m.log_A.clone().requires_grad_(True)
    m.log_A = log_A
    rho_a, T = rho_a.detach().requires_grad_(True), T.detach().requires_grad_(True)
    J = m.heat_release(rho_a, T).sum()
    dA, dT, drho = torch.autograd.grad(J, (log_A, T, rho_a))
    return {"J": float(J.detach()), "dlogA": dA.cpu().numpy(), "dT": dT, "drho": drho}


def _exact_gradient(m, X, T0, P, steps, log_A):
    """J = sum over steps and nodes of the heat release at the state each collision sees, by autograd."""
    F, T, J = m.initial(X, T0, P), T0.detach(), 0.0
    for _ in range(steps):
        rho_a, _, Tn = m.node_state(m.pull(F, T), T)[:3]
        J = J + m.heat_release(rho_a, Tn).sum()
        F, T = m.step(F, T)
        T = T.detach()
    dA, dT0 = torch.autograd.grad(J, (log_A, T0))
    return {"J": float(J.detach()), "dlogA": dA.cpu().numpy(), "dT0": dT0}
