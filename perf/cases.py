"""Performance cases of the DG solver: what a user's program has it do,
through the package's public entry points.

Kinds:
  step       one pass of a time loop on the bound state: the CFL time step, an
             SSP-RK3 step and what the loop does beside it ("loop"):
             "step"    cfl_dt, step (the accuracy and shock-tube runs);
             "bench"   cfl_dt, driven step, isothermal energy reset (bench.py);
             "driven"  cfl_dt, driven step, diagnostics, energy reset with its
                       dissipated energy (the turbulence run driver);
  rhs        R(y) of the bound state into the caller's buffer (dg_rhs);
  analysis   velocity power spectrum and density PDF of the bound state;
  indicator  one full-batch training step of the troubled-cell indicator
             (forward, backward, Adam).

Outputs: FP64 runs return the state (or R) itself; FP32-mixed runs return the
state as the single-precision snapshot a program would store (the mixed
path's increments are accurate to single precision). exact() gives the same
in 64 bits with plain torch: dense quadrature instead of the library's
sum-factorised kernels.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1602_09079_gb300 as dg
from paper_1602_09079_gb300 import roofline
from paper_1602_09079_gb300.forcing import OUDriving, half_space_modes

GAMMA = 5.0 / 3.0
HIDDEN = 64  # width of the indicator's hidden layers
EPS = 1e-12  # the library's default positivity floors


def _step(name, n, order, precision, flow, loop, flux="hllc", gamma=GAMMA, courant=0.3):
    return {"name": name, "kind": "step", "nx": n[0], "ny": n[1], "nz": n[2], "order": order, "precision": precision,
            "flow": flow, "loop": loop, "flux": flux, "gamma": gamma, "courant": courant}


def listed():
    return [
        # the smallest run of the accuracy configurations: latency and launches
        _step("wave_8_o2_fp64", (8, 8, 8), 2, "fp64", "wave", "step"),
        # the convergence sweep at its largest size and highest order
        _step("wave_64_o4_fp64", (64, 64, 64), 4, "fp64", "wave", "step"),
        # the driven-turbulence benchmark in plain FP64 (the default precision)
        _step("bench_128_o3_fp64", (128, 128, 128), 3, "fp64", "turbulence", "bench"),
        # the driven-turbulence benchmark in FP32-mixed precision (headline)
        _step("bench_128_o3_mixed", (128, 128, 128), 3, "mixed", "turbulence", "bench"),
        # the same at the highest order, on a mesh three states of which fit
        _step("bench_160_o4_mixed", (160, 160, 160), 4, "mixed", "turbulence", "bench"),
        # second order, the cheapest scheme for the same memory, ragged box
        _step("bench_100x90x84_o2_mixed", (100, 90, 84), 2, "mixed", "turbulence", "bench"),
        # the turbulence run driver's default: 64^3, order 3, gamma 1.01,
        # diagnostics and dissipated energy every step
        _step("driven_64_o3_mixed", (64, 64, 64), 3, "mixed", "turbulence", "driven", gamma=1.01),
        # shock tube with a random plane normal: the positivity limiter at work
        _step("sod_128_o3_mixed", (128, 128, 128), 3, "mixed", "sod", "step", courant=0.15),
        # the exact Riemann solver in place of HLLC, odd sizes
        _step("exact_flux_65x63x61_o3_mixed", (65, 63, 61), 3, "mixed", "turbulence", "step", flux="exact"),
        # one right-hand side of a small ragged mesh (a caller's own integrator)
        {"name": "rhs_33x32x31_o3_fp64", "kind": "rhs", "nx": 33, "ny": 32, "nz": 31, "order": 3, "precision": "fp64",
         "flow": "turbulence", "flux": "hllc", "gamma": GAMMA},
        # end-of-run analysis on 4^3 samples per cell
        {"name": "analysis_64_o3_sub4", "kind": "analysis", "nx": 64, "ny": 64, "nz": 64, "order": 3, "sub": 4,
         "flow": "turbulence", "gamma": GAMMA},
        # indicator training: a full batch of captured rows
        {"name": "indicator_262144_o3", "kind": "indicator", "rows": 262144, "order": 3},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case: sizes over the whole range (over their logarithm), odd
    ones and unequal axes among them."""
    kind = rng.choices(["step", "rhs", "analysis", "indicator"], [8, 2, 1, 1])[0]
    if kind == "analysis":
        sub = rng.randint(1, 4)
        n = _log_int(rng, 8, 64)
        return {"kind": kind, "nx": n, "ny": n, "nz": n, "order": rng.randint(2, 4), "sub": sub,
                "flow": "turbulence", "gamma": rng.choice([GAMMA, 1.01])}
    if kind == "indicator":
        return {"kind": kind, "rows": _log_int(rng, 1000, 262144), "order": rng.randint(2, 4)}
    # R itself is wanted by a caller's own integrator, in full precision
    precision = "fp64" if kind == "rhs" else rng.choice(["fp64", "mixed"])
    order = rng.choice([1, 2, 3, 3, 4])
    # FP64 runs stay below the largest listed one (128^3 at order 3)
    top = {"mixed": 128, "fp64": 96 if order < 4 else 64}[precision]
    n = [_log_int(rng, 6, top) for _ in range(3)]
    if kind == "rhs":
        return {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "order": order, "precision": precision,
                "flow": rng.choice(["turbulence", "wave"]), "flux": "hllc", "gamma": GAMMA}
    loop = rng.choice(["step", "bench", "driven"])
    flow = rng.choice(["wave", "turbulence", "sod"]) if loop == "step" else "turbulence"
    gamma = 1.01 if loop == "driven" and rng.random() < 0.5 else GAMMA
    c = _step("", n, order, precision, flow, loop, gamma=gamma, courant=0.15 if flow == "sod" else 0.3)
    del c["name"]
    if loop == "step" and flow == "turbulence" and precision == "mixed":
        c["flux"] = rng.choice(["hllc", "exact"])
    return c


# ------------------------------------------------------------------- inputs

def _modes(k):
    """Mode exponents: total degree ascending, then u, then v descending."""
    return [(u, v, d - u - v) for d in range(k + 1) for u in range(d, -1, -1) for v in range(d - u, -1, -1)]


def _legendre(k, x):
    """[k+1][len(x)]: sqrt(2u+1) P_u(x) and its derivative, FP64 on the GPU."""
    c = [np.polynomial.legendre.Legendre.basis(u) for u in range(k + 1)]
    p = np.array([math.sqrt(2 * u + 1) * c[u](x) for u in range(k + 1)])
    d = np.array([math.sqrt(2 * u + 1) * c[u].deriv()(x) if u else np.zeros(len(x)) for u in range(k + 1)])
    return torch.from_numpy(p).cuda(), torch.from_numpy(d).cuda()


def _coordinates(case, x):
    """Per axis, the physical coordinates of the points x of every cell."""
    return [((torch.arange(n, dtype=torch.float64)[:, None] + 0.5 + 0.5 * torch.from_numpy(x)) / n).reshape(-1).cuda()
            for n in (case["nx"], case["ny"], case["nz"])]


def _fourier(nv, amp, X, Y, Z):
    """sum_j Re((amp_j0 + i amp_j1) exp(2 pi i n_j . x)) on the tensor grid
    [Z][Y][X], from one-dimensional exponentials."""
    a = torch.complex(torch.from_numpy(amp[:, 0]).cuda(), torch.from_numpy(amp[:, 1]).cuda())
    e = [torch.exp(2j * math.pi * torch.from_numpy(nv[:, d].astype(np.float64)).cuda()[:, None] * c[None, :])
         for d, c in enumerate((X, Y, Z))]
    xy = (a[:, None, None] * e[1][:, :, None] * e[0][:, None, :]).reshape(len(nv), -1)
    return (e[2].real.T @ xy.real - e[2].imag.T @ xy.imag).reshape(len(Z), len(Y), len(X))


def _conserved(rho, v, p, gamma):
    return [rho, rho * v[0], rho * v[1], rho * v[2],
            p / (gamma - 1.0) + 0.5 * rho * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2])]


def _flow(case, seed):
    """The initial condition fn(X, Y, Z) -> 5 conserved fields on [Z][Y][X]."""
    rng = np.random.default_rng(seed)
    gamma = case["gamma"]
    if case["flow"] == "wave":  # smooth advected density wave along the diagonal
        phase, amp = rng.uniform(0, 1), rng.uniform(0.1, 0.3)

        def fn(X, Y, Z):
            s = X[None, None, :] + Y[None, :, None] + Z[:, None, None] + phase
            rho = 1.0 + amp * torch.sin(2 * math.pi * s)
            one = torch.ones_like(rho)
            return _conserved(rho, (one, one, one), one, gamma)
    elif case["flow"] == "sod":  # two states divided by planes of a random normal
        nrm = rng.standard_normal(3)
        nrm /= np.linalg.norm(nrm)
        off = rng.uniform(0, 1)

        def fn(X, Y, Z):
            s = (nrm[0] * (X - 0.5)[None, None, :] + nrm[1] * (Y - 0.5)[None, :, None]
                 + nrm[2] * (Z - 0.5)[:, None, None] + off) % 1.0
            left = s < 0.5
            rho, p = torch.where(left, 1.0, 0.125).double(), torch.where(left, 1.0, 0.1).double()
            zero = torch.zeros_like(rho)
            return _conserved(rho, (zero, zero, zero), p, gamma)
    else:  # subsonic turbulence: solenoidal velocity at rms Mach 0.3 over the
        # large scales and a few per cent of density variation, p = rho / gamma
        nv = half_space_modes(1.0, 3.0)
        amp = rng.standard_normal((len(nv), 2, 3)) * (np.linalg.norm(nv, axis=1) ** -1.5)[:, None, None]
        nn = nv / np.linalg.norm(nv, axis=1, keepdims=True)
        amp -= np.einsum("jpd,jd->jp", amp, nn)[:, :, None] * nn[:, None, :]
        amp *= 0.3 / math.sqrt(0.5 * np.sum(amp ** 2))
        damp = 0.02 * rng.standard_normal((len(nv), 2)) / math.sqrt(len(nv))

        def fn(X, Y, Z):
            rho = torch.exp(_fourier(nv, damp, X, Y, Z))
            v = [_fourier(nv, amp[:, :, d], X, Y, Z) for d in range(3)]
            return _conserved(rho, v, rho / gamma, gamma)
    return fn


def _initial(case, seed):
    """Coefficients of the projected initial condition, canonical layout
    [nz][ny][nx][5][N]: w_l = 1/8 sum_q f(x_q) phi_l(x_q) omega_q."""
    k, fn = case["order"] - 1, _flow(case, seed)
    nx, ny, nz, q = case["nx"], case["ny"], case["nz"], k + 1
    x, w = np.polynomial.legendre.leggauss(q)
    pw = _legendre(k, x)[0] * torch.from_numpy(w).cuda() * 0.5
    X, Y, Z = _coordinates(case, x)
    modes = _modes(k)
    out = torch.empty((nz, ny, nx, 5, len(modes)), dtype=torch.float64, device="cuda")
    slab = max(1, min(nz, (1 << 24) // (nx * ny * q ** 3)))
    for z in range(0, nz, slab):
        e = min(nz, z + slab)
        for i, f in enumerate(fn(X, Y, Z[z * q:e * q])):
            f = f.reshape(e - z, q, ny, q, nx, q) @ pw.T
            f = torch.einsum("zaybxu,vb,wa->zyxuvw", f, pw, pw)
            for l, (u, v, ww) in enumerate(modes):
                out[z:e, :, :, i, l] = f[..., u, v, ww]
    return out


def _driving(case, seed):
    """(wave vectors, amplitudes) of the Ornstein-Uhlenbeck driving after one
    update, scaled as for rms Mach 0.3."""
    nv = half_space_modes(1.0, 2.0)
    z = np.random.default_rng(seed + 1).standard_normal((2, len(nv), 6))
    t_s = 1.0 / 0.6
    d = OUDriving(nv, t_s, 0.1 * t_s, 0.3 ** 2 * 2 * math.pi * 1.5, z[0])
    d.update(z[1])
    return d.nvec, d.ahat()


def _indicator_inputs(case, seed):
    """Feature rows, labels and FP32 parameters of the indicator. Rows are
    the size of captured ones: modes and neighbour differences well below
    one, a tenth of the cells troubled."""
    nf, F, npar, work = dg.dg_indicator_sizes(case["order"])
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    X = 0.3 * torch.randn(case["rows"], F, device="cuda", generator=g)
    X[:, nf:] = 0
    y = (torch.rand(case["rows"], device="cuda", generator=g) < 0.1).float()
    rng = np.random.default_rng(seed)
    a, b = math.sqrt(6.0 / F), math.sqrt(6.0 / HIDDEN)
    P = np.concatenate([rng.uniform(-a, a, HIDDEN * F), rng.uniform(-0.1, 0.1, HIDDEN),
                        rng.uniform(-b, b, HIDDEN * HIDDEN), rng.uniform(-0.1, 0.1, HIDDEN),
                        rng.uniform(-b, b, HIDDEN), [0.0]])
    return X.to(torch.bfloat16), y, torch.from_numpy(P.astype(np.float32)).cuda(), npar, work


def prepare(case, seed):
    if case["kind"] == "indicator":
        X, y, P, npar, work = _indicator_inputs(case, seed)
        f32 = {"dtype": torch.float32, "device": "cuda"}
        return {"case": case, "X": X, "y": y, "P": P, "m": torch.zeros_like(P), "v": torch.zeros_like(P),
                "G": torch.zeros(npar + 1, **f32), "logits": torch.empty(len(y), **f32), "npar": npar,
                "work": torch.empty(work, dtype=torch.uint8, device="cuda"), "step": 0,
                "stream": torch.cuda.current_stream().cuda_stream}
    driven = case.get("loop") in ("bench", "driven")
    s = dg.Solver((case["nx"], case["ny"], case["nz"]), case["order"], case["gamma"], forcing=driven)
    st = {"case": case, "solver": s}
    if case["kind"] != "analysis":
        s.set_precision(dg.DG_PREC_MIXED if case["precision"] == "mixed" else dg.DG_PREC_FP64)
        s.set_flux(dg.DG_FLUX_EXACT if case["flux"] == "exact" else dg.DG_FLUX_HLLC)
    s.set_state(_initial(case, seed))
    if driven:
        s.set_forcing(*_driving(case, seed))
    if case["kind"] == "step":
        s.limit()  # a running loop's state is limited
    if case["kind"] == "rhs":
        st["R"] = torch.empty_like(s.y)
    return st


def run(state):
    case = state["case"]
    if case["kind"] == "indicator":
        o, n, s = case["order"], len(state["y"]), state["stream"]
        state["step"] += 1
        dg.dg_indicator_forward(o, state["X"], n, state["P"], state["logits"], s)
        dg.dg_indicator_backward(o, state["X"], state["y"], n, 9.0, state["P"], state["G"], state["work"],
                                 state["work"].numel(), s)
        dg.dg_indicator_adam(state["P"], state["m"], state["v"], state["G"], state["npar"], 3e-3, 0.9, 0.999, 1e-8,
                             state["step"], s)
        return {"logits": state["logits"], "gradients_and_loss": state["G"]}
    s = state["solver"]
    if case["kind"] == "analysis":
        return {"spectrum": s.velocity_spectrum(case["sub"]), "pdf": s.density_pdf(case["sub"], -0.5, 0.5, 100)}
    if case["kind"] == "rhs":
        dg.dg_rhs(s.ctx, None, state["R"])
        return {"R": state["R"]}
    dt = s.cfl_dt(case["courant"])
    s.step(dt)
    out = {"dt": dt}
    if case["loop"] == "driven":
        mach, kinetic, power = s.diagnostics()
        out["diagnostics"] = [float(mach), float(kinetic), float(power)]
    if case["loop"] != "step":
        # c_iso^2 = p / rho of the initial state; the dissipated energy is a
        # difference of nearly equal sums: the run's budget, not an output
        s.energy_reset(math.sqrt(1.0 / case["gamma"]), 1.0, want_dissipated=case["loop"] == "driven")
    out["state"] = s.y.float() if case["precision"] == "mixed" else s.y
    return out


def work(case):
    """Bytes and flops of one pass that the method cannot do without: state
    in and out of each RK stage in FP64, sum-factorised quadrature."""
    if case["kind"] == "indicator":
        F = dg.dg_indicator_sizes(case["order"])[1]
        mac = F * HIDDEN + HIDDEN * HIDDEN + HIDDEN
        return {"bytes": case["rows"] * (2 * F + 8), "flops": 2 * case["rows"] * (2 * mac + 2 * HIDDEN * HIDDEN)}
    k, nc = case["order"] - 1, case["nx"] * case["ny"] * case["nz"]
    N = len(_modes(k))
    if case["kind"] == "analysis":
        M3 = nc * case["sub"] ** 3
        # one real transform per velocity component; density and the shells
        return {"bytes": nc * 4 * N * 8, "flops": M3 * (8 * N + 3 * 2.5 * math.log2(max(2, M3)) + 10)}
    forced = case.get("loop") in ("bench", "driven")
    if case["kind"] == "rhs":
        return {"bytes": nc * 2 * 5 * N * 8, "flops": nc * roofline.stage_flops(k, False)}
    byts, flops = roofline.step_min_bytes(k) + 40, 3 * roofline.stage_flops(k, forced)
    if forced:  # energy reset: rho, m and the mean energy in, energy out
        byts += (4 * N + 1 + N) * 8
        flops += 2 * (4 * N + N) * (k + 1) ** 2
    if case["loop"] == "driven":  # diagnostics: means, momentum against the driving
        byts += (2 + 3 * N) * 8
        flops += 6 * N * (k + 1)
    return {"bytes": nc * byts, "flops": nc * flops}


# ------------------------------------------------------------- 64-bit values

class _Dense:
    """The DG method in plain torch FP64, dense quadrature; state
    [5][N][nz][ny][nx]."""

    def __init__(self, case):
        self.case, self.k = case, case["order"] - 1
        self.g = case["gamma"]
        k, self.q = self.k, self.k + 1
        self.n = (case["nx"], case["ny"], case["nz"])
        x, w = np.polynomial.legendre.leggauss(self.q)
        self.x = x
        m = 2 if k <= 1 else 3
        gll = np.array([-1.0, 1.0] if m == 2 else [-1.0, 0.0, 1.0])
        self.cfl_factor = min(1.0 / (2 * k + 1), (1.0 if m == 2 else 1.0 / 3.0) / 2)
        w = torch.from_numpy(w).cuda()
        om = (w[:, None, None] * w[None, :, None] * w[None, None, :]).reshape(-1, 1)

        def table(px, py, pz):  # [points][N], x fastest
            return torch.stack([torch.einsum("a,b,c->cba", px[u], py[v], pz[ww]).reshape(-1)
                                for u, v, ww in _modes(k)], dim=1)

        p, d = _legendre(k, x)
        end = [_legendre(k, np.array([e]))[0] for e in (-1.0, 1.0)]
        self.phi = table(p, p, p)
        self.dphi = [table(*[d if a == b else p for b in range(3)]) * om / 4 for a in range(3)]
        self.phiw = self.phi * om / 8
        w2 = (w[:, None] * w[None, :]).reshape(-1, 1) / 4
        self.face = [[table(*[end[e] if a == b else p for b in range(3)]) for e in (0, 1)] for a in range(3)]
        self.facew = [[f * w2 for f in fs] for fs in self.face]
        lob = _legendre(k, gll)[0]
        self.S = torch.cat([table(*[lob if a == b else p for b in range(3)]) for a in range(3)])
        self.field = None

    def set_forcing(self, nv, ahat):
        """a(x) at the volume points, [3][q][nz][ny][nx]."""
        q, (nx, ny, nz) = self.q, self.n
        X, Y, Z = _coordinates(self.case, self.x)
        f = [_fourier(nv, np.stack([ahat[:, d], ahat[:, 3 + d]], 1), X, Y, Z) for d in range(3)]
        self.field = torch.stack([a.reshape(nz, q, ny, q, nx, q).permute(1, 3, 5, 0, 2, 4).reshape(q ** 3, nz, ny, nx)
                                  for a in f])

    def pressure(self, U):
        return (self.g - 1) * (U[4] - 0.5 * (U[1] * U[1] + U[2] * U[2] + U[3] * U[3]) / U[0])

    def euler(self, U, p, d):
        v = U[1 + d] / U[0]
        F = [U[i] * v for i in range(4)] + [(U[4] + p) * v]
        F[1 + d] = F[1 + d] + p
        return F

    def hllc(self, L, R, d):
        """HLLC with Einfeldt's wave speeds from Roe averages."""
        g = self.g
        pL, pR = self.pressure(L), self.pressure(R)
        uL, uR = L[1 + d] / L[0], R[1 + d] / R[0]
        cL, cR = (torch.sqrt(g * p / U[0]) for p, U in ((pL, L), (pR, R)))
        sL, sR = torch.sqrt(L[0]), torch.sqrt(R[0])
        v = [(L[1 + a] / sL + R[1 + a] / sR) / (sL + sR) for a in range(3)]
        H = ((L[4] + pL) / sL + (R[4] + pR) / sR) / (sL + sR)
        c = torch.sqrt((g - 1) * (H - 0.5 * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2])))
        SL, SR = torch.minimum(uL - cL, v[d] - c), torch.maximum(uR + cR, v[d] + c)
        aL, aR = L[0] * (SL - uL), R[0] * (SR - uR)
        Ss = (pR - pL + uL * aL - uR * aR) / (aL - aR)
        left = Ss >= 0

        def pick(a, b):
            return torch.where(left, a, b)

        U = [pick(a, b) for a, b in zip(L, R)]
        p, S, u, ak = pick(pL, pR), pick(SL, SR), pick(uL, uR), pick(aL, aR)
        chi = ak / (S - Ss)
        star = [chi] + [chi * U[1 + a] / U[0] for a in range(3)]
        star[1 + d] = chi * Ss
        star.append(chi * (U[4] / U[0] + (Ss - u) * Ss) + (Ss - u) * p / (S - Ss))
        FL, FR = self.euler(L, pL, d), self.euler(R, pR, d)
        out = []
        for i in range(5):
            f = pick(FL[i], FR[i]) + S * (star[i] - U[i])
            out.append(torch.where(SL >= 0, FL[i], torch.where(SR <= 0, FR[i], f)))
        return out

    def godunov(self, L, R, d):
        """Flux of the exact Riemann solution at x/t = 0 (no vacuum)."""
        g = self.g
        z = (g - 1) / (2 * g)
        side = []
        for U in (L, R):
            p = self.pressure(U)
            side.append((U[0], U[1 + d] / U[0], p, torch.sqrt(g * p / U[0])))
        du = side[1][1] - side[0][1]

        def jump(ps, k):
            rho, u, p, c = k
            q = torch.sqrt(2 / ((g + 1) * rho) / (ps + (g - 1) / (g + 1) * p))
            shock, r = ps > p, (ps / p) ** z
            f = torch.where(shock, (ps - p) * q, 2 * c / (g - 1) * (r - 1))
            df = torch.where(shock, q * (1 - 0.5 * (ps - p) / (ps + (g - 1) / (g + 1) * p)), c * r / (g * ps))
            return f, df

        ps = ((side[0][3] + side[1][3] - 0.5 * (g - 1) * du)
              / (side[0][3] * side[0][2] ** -z + side[1][3] * side[1][2] ** -z)) ** (1 / z)
        for _ in range(12):
            (fL, dL), (fR, dR) = jump(ps, side[0]), jump(ps, side[1])
            ps = torch.clamp(ps - (fL + fR + du) / (dL + dR), min=1e-14)
        fL, fR = jump(ps, side[0])[0], jump(ps, side[1])[0]
        us = 0.5 * (side[0][1] + side[1][1] + fR - fL)
        left = us >= 0
        rho, u, p, c = (torch.where(left, a, b) for a, b in zip(*side))
        sg = torch.where(left, 1.0, -1.0).double()
        ratio = ps / p
        g6 = (g - 1) / (g + 1)
        shock = ps > p
        speed = u - sg * c * torch.sqrt((g + 1) / (2 * g) * ratio + z)
        head, tail = u - sg * c, us - sg * c * ratio ** z
        cf = torch.clamp(2 / (g + 1) * (c + sg * 0.5 * (g - 1) * u), min=0)
        ahead = torch.where(shock, sg * speed >= 0, sg * head >= 0)
        star = shock | (sg * tail < 0)
        rs = torch.where(shock, rho * (ratio + g6) / (g6 * ratio + 1), rho * ratio ** (1 / g))
        W = [torch.where(ahead, a, torch.where(star, b, f)) for a, b, f in (
            (rho, rs, rho * (cf / c) ** (2 / (g - 1))), (u, us, sg * cf), (p, ps, p * (cf / c) ** (2 * g / (g - 1))))]
        v = [torch.where(left, L[1 + a] / L[0], R[1 + a] / R[0]) for a in range(3)]
        v[d] = W[1]
        U = _conserved(W[0], v, W[2], g)
        return self.euler(U, W[2], d)

    def dwdt(self, W):
        """-R(W), in slabs of z planes with one halo plane each."""
        nx, ny, nz = self.n
        flux = self.godunov if self.case["flux"] == "exact" else self.hllc
        out = torch.empty_like(W)
        slab = max(1, min(nz, (1 << 21) // (nx * ny * self.q ** 3) + 1))
        at = (4, 3, 2)  # dimension of x, y, z in [5][N][z][y][x]
        for z in range(0, nz, slab):
            e = min(nz, z + slab)
            own = W[:, :, z:e]
            U = torch.einsum("ql,ilzyx->iqzyx", self.phi, own)
            p = self.pressure(U)
            acc = torch.zeros_like(own)
            for d in range(3):
                F = torch.stack(self.euler(U, p, d))
                acc += torch.einsum("ql,iqzyx->ilzyx", self.dphi[d], F) * self.n[d]
            if self.field is not None:
                a = self.field[:, :, z:e]
                src = torch.stack([torch.zeros_like(p), U[0] * a[0], U[0] * a[1], U[0] * a[2],
                                   U[1] * a[0] + U[2] * a[1] + U[3] * a[2]])
                acc += torch.einsum("ql,iqzyx->ilzyx", self.phiw, src)
            del U, p
            for d in range(3):
                if d < 2:
                    lo, hi = own, torch.roll(own, 1, at[d])
                else:
                    pl = [(j % nz) for j in range(z - 1, e + 1)]
                    ext = W[:, :, pl]
                    lo, hi = ext[:, :, 1:], ext[:, :, :-1]
                R = torch.einsum("ql,ilzyx->iqzyx", self.face[d][0], lo)
                L = torch.einsum("ql,ilzyx->iqzyx", self.face[d][1], hi)
                F = torch.stack(flux(L, R, d))
                low = F if d < 2 else F[:, :, :-1]
                high = torch.roll(F, -1, at[d]) if d < 2 else F[:, :, 1:]
                acc += (torch.einsum("ql,iqzyx->ilzyx", self.facew[d][0], low)
                        - torch.einsum("ql,iqzyx->ilzyx", self.facew[d][1], high)) * self.n[d]
            out[:, :, z:e] = acc
        return out

    def limit(self, W):
        """Zhang-Shu positivity limiter on the GLL x Gauss point set."""
        if self.k == 0:
            return W
        big = self.S.abs().amax(0)[1:]
        dev = torch.einsum("l,ilzyx->izyx", big, W[:, 1:].abs())
        mean = W[:, 0]
        rlo = mean[0] - dev[0]
        kin = 0.5 * ((mean[1:4].abs() + dev[1:4]) ** 2).sum(0) / rlo
        bad = ~((rlo > 1e-9) & (mean[4] - dev[4] - kin > 1e-9))
        idx = bad.reshape(-1).nonzero()[:, 0]
        flat = W.reshape(5, W.shape[1], -1)
        for c in idx.split(1 << 17):
            w = flat[:, :, c]
            rho = torch.einsum("ql,lc->qc", self.S, w[0])
            th1 = torch.clamp((w[0, 0] - EPS) / (w[0, 0] - rho.amin(0)), max=1.0)
            w[0, 1:] *= torch.where(rho.amin(0) < EPS, th1, 1.0)
            U = torch.einsum("ql,ilc->iqc", self.S, w)
            D = U - w[:, :1]
            neg = self.pressure(U) < EPS
            tau = torch.ones_like(rho)
            for _ in range(40):  # Newton from tau = 1, monotone (concave pressure)
                s = w[:, :1] + tau * D
                m2, md = (s[1:4] ** 2).sum(0), (s[1:4] * D[1:4]).sum(0)
                f = (self.g - 1) * (s[4] - 0.5 * m2 / s[0]) - EPS
                fp = (self.g - 1) * (D[4] - md / s[0] + 0.5 * m2 * D[0] / s[0] ** 2)
                tau = torch.where(neg, torch.minimum(tau, torch.clamp(tau - f / fp, min=0.0)), tau)
            w[:, 1:] *= torch.where(neg, tau, 1.0).amin(0)
            flat[:, :, c] = w
        return flat.reshape(W.shape)

    def cfl_dt(self, W):
        U = W[:, 0]
        c = torch.sqrt(self.g * self.pressure(U) / U[0])
        s = sum((U[1 + d].abs() / U[0] + c) * self.n[d] for d in range(3))
        return self.case["courant"] * self.cfl_factor / float(s.max())

    def step(self, W, dt):
        Y = self.limit(W + dt * self.dwdt(W))
        Y = self.limit(0.75 * W + 0.25 * (Y + dt * self.dwdt(Y)))
        return self.limit(W / 3 + 2.0 / 3 * (Y + dt * self.dwdt(Y)))

    def diagnostics(self, W):
        U, nc = W[:, 0], self.n[0] * self.n[1] * self.n[2]
        m2 = U[1] ** 2 + U[2] ** 2 + U[3] ** 2
        mach = torch.sqrt((m2 / U[0] / (self.g * self.pressure(U))).mean())
        P = 0.0
        for z in range(self.n[2]):
            m = torch.einsum("ql,ilyx->iqyx", self.phi, W[1:4, :, z])
            P += float((self.phiw[:, 0][:, None, None] * (m * self.field[:, :, z]).sum(0)).sum())
        return [float(mach), float((0.5 * m2 / U[0]).mean()), P / nc]

    def energy_reset(self, W, c_iso):
        W = W.clone()
        for z in range(self.n[2]):
            U = torch.einsum("ql,ilyx->iqyx", self.phi, W[:4, :, z])
            E = (0.5 * (U[1] ** 2 + U[2] ** 2 + U[3] ** 2) / U[0]
                 + U[0] * (c_iso * c_iso / (self.g - 1) * U[0] ** (self.g - 1)))
            W[4, :, z] = torch.einsum("ql,qyx->lyx", self.phiw, E)
        return self.limit(W)


def _exact_indicator(case, seed):
    """Logits, gradients and loss of the class-weighted cross entropy at the
    given parameters, FP64 throughout."""
    X, y, P, npar, _ = _indicator_inputs(case, seed)
    X, y, P = X.double(), y.double(), P.double().requires_grad_()
    F, H = X.shape[1], HIDDEN
    W1, b1, W2, b2, w3, b3 = P.split([H * F, H, H * H, H, H, 1])
    h = torch.relu(X @ W1.view(H, F).T + b1)
    h = torch.relu(h @ W2.view(H, H).T + b2)
    z = h @ w3 + b3
    loss = (9.0 * y * torch.nn.functional.softplus(-z) + (1 - y) * torch.nn.functional.softplus(z)).mean()
    loss.backward()
    return {"logits": z.detach(), "gradients_and_loss": torch.cat([P.grad, loss.detach()[None]])}


def _exact_analysis(case, W):
    n, sub, k = case["nx"], case["sub"], case["order"] - 1
    M = n * sub
    x = -1.0 + (2.0 * np.arange(sub) + 1.0) / sub
    p = _legendre(k, x)[0]

    def sample(w):  # [N][z][y][x] -> [M][M][M]
        s = 0.0
        for l, (u, v, ww) in enumerate(_modes(k)):
            s = s + torch.einsum("zyx,c,b,a->zcybxa", w[l], p[ww], p[v], p[u])
        return s.reshape(M, M, M)

    rho = sample(W[0])
    f = np.fft.fftfreq(M, 1.0 / M)
    h = np.arange(M // 2 + 1)
    f, h = torch.from_numpy(f).cuda(), torch.from_numpy(h).double().cuda()
    shell = torch.floor(torch.sqrt(f[:, None, None] ** 2 + f[None, :, None] ** 2 + h ** 2) + 0.5).long()
    twice = torch.where((h == 0) | (2 * h == M), 1.0, 2.0).double()
    nb = int(math.floor(math.sqrt(3.0) * M / 2.0)) + 2
    bins = torch.zeros(nb, dtype=torch.float64, device="cuda")
    for d in range(3):
        a = torch.fft.rfftn(sample(W[1 + d]) / rho)
        e = (a.real ** 2 + a.imag ** 2) * twice / float(M) ** 6
        bins += torch.bincount(shell.reshape(-1), e.reshape(-1), nb)[:nb]
    s = torch.log(rho)
    j = torch.clamp(torch.floor((s + 0.5) * 100).long(), max=99) + 1
    j = torch.where(s < -0.5, 0, torch.where(s >= 0.5, 101, j))
    return {"spectrum": bins, "pdf": torch.bincount(j.reshape(-1), minlength=102)}


def exact(case, seed):
    if case["kind"] == "indicator":
        return _exact_indicator(case, seed)
    W = _initial(case, seed).permute(3, 4, 0, 1, 2).contiguous()
    if case["kind"] == "analysis":
        return _exact_analysis(case, W)
    D = _Dense(case)
    if case["kind"] == "rhs":
        return {"R": -D.dwdt(W).reshape(-1)}
    if case["loop"] != "step":
        D.set_forcing(*_driving(case, seed))
    W = D.limit(W)
    dt = D.cfl_dt(W)
    out = {"dt": dt}
    W = D.step(W, dt)
    if case["loop"] == "driven":
        out["diagnostics"] = D.diagnostics(W)
    if case["loop"] != "step":
        W = D.energy_reset(W, math.sqrt(1.0 / case["gamma"]))
    out["state"] = W.reshape(-1)
    return out
