"""Workloads of the VL+CT ideal-MHD library whose speed is tracked.

Every case runs through the package's public entry points: ``Sim.run``,
``Sim.evolve``, ``mhd_run_host``, ``Sim.adjoint_step``,
``Sim.adjoint_step_cfl`` and ``autograd.rollout``.  ``listed()`` names the
workloads of this repository's configurations, tests and benchmark;
``draw()`` gives more of the same ranges (any grid shape, reconstruction and
precision).  ``exact()`` is the same method in plain torch float64, its
derivatives by torch's own autograd.
"""
from __future__ import annotations

import math

import torch
from torch.utils.checkpoint import checkpoint

from paper_2402_05240_gb300 import autograd as mhd_autograd
from paper_2402_05240_gb300 import mhd

GAMMA = 5.0 / 3.0
FLOOR = 1e-20  # Sim's default density and pressure floors
GHOST = 8      # ghost cells of exact()'s outflow boundaries (a step reaches 5 cells)

# Floating-point operations per cell that one step executes (predictor and
# corrector Riemann solvers, edge fields, updates, primitives: 2400; the three
# reconstructions on top).
STEP_FLOPS = {"pcm": 2400, "plm_prim": 2700, "plmc": 3300, "ppmc": 4200}


def listed():
    return [
        # parity and convergence studies: the 32^3 fast magnetosonic wave, ten steps
        {"name": "wave32_fp64", "kind": "run", "init": "wave", "nx": 32, "ny": 32, "nz": 32, "recon": "plmc",
         "precision": "fp64", "steps": 10, "cfl": 0.4},
        # small parameter scans and test problems: every launch is short
        {"name": "box64_fp32", "kind": "run", "init": "turbulent", "nx": 64, "ny": 64, "nz": 64, "recon": "ppmc",
         "precision": "fp32_bulk", "steps": 10, "cfl": 0.3},
        # a Riemann problem along x with outflow boundaries, advanced in time
        {"name": "tube_fp64", "kind": "evolve", "init": "tube", "nx": 512, "ny": 16, "nz": 16, "recon": "ppmc",
         "precision": "fp64", "steps": 20, "cfl": 0.4},
        # an ordinary turbulent box in the default precision and reconstruction
        {"name": "box256_fp64", "kind": "run", "init": "turbulent", "nx": 256, "ny": 256, "nz": 256, "recon": "plmc",
         "precision": "fp64", "steps": 2, "cfl": 0.3},
        # the benchmark workload in its three precisions
        {"name": "box512_fp64", "kind": "run", "init": "turbulent", "nx": 512, "ny": 512, "nz": 512, "recon": "ppmc",
         "precision": "fp64", "steps": 1, "cfl": 0.3},
        {"name": "box512_df", "kind": "run", "init": "turbulent", "nx": 512, "ny": 512, "nz": 512, "recon": "ppmc",
         "precision": "fp64_df", "steps": 2, "cfl": 0.3},
        {"name": "box512_fp32", "kind": "run", "init": "turbulent", "nx": 512, "ny": 512, "nz": 512, "recon": "ppmc",
         "precision": "fp32_bulk", "steps": 2, "cfl": 0.3},
        # the slow-wave throughput problem on an odd grid (no row a multiple of a warp)
        {"name": "slow459_df", "kind": "run", "init": "slow_wave", "nx": 459, "ny": 459, "nz": 459, "recon": "plmc",
         "precision": "fp64_df", "steps": 1, "cfl": 0.4},
        # a box that starts and ends in host memory, five steps between the copies
        {"name": "host256_df", "kind": "host", "init": "turbulent", "nx": 256, "ny": 256, "nz": 256, "recon": "plmc",
         "precision": "fp64_df", "steps": 5, "cfl": 0.3},
        # gradients: one reverse step at fixed dt, one through the CFL dt, and
        # a checkpointed rollout through torch's autograd
        {"name": "adjoint128_fp64", "kind": "adjoint", "init": "perturbed", "nx": 128, "ny": 128, "nz": 128,
         "recon": "ppmc", "precision": "fp64", "steps": 1, "cfl": 0.3},
        {"name": "adjoint256_fp32", "kind": "adjoint_cfl", "init": "perturbed", "nx": 256, "ny": 256, "nz": 256,
         "recon": "ppmc", "precision": "fp32_bulk", "steps": 1, "cfl": 0.3},
        {"name": "rollout64_df", "kind": "rollout", "init": "perturbed", "nx": 64, "ny": 64, "nz": 64, "recon": "plmc",
         "precision": "fp64_df", "steps": 4, "cfl": 0.3},
    ]


def draw(rng):
    kind = rng.choice(["run"] * 6 + ["evolve", "host", "adjoint", "adjoint", "adjoint_cfl", "rollout"])
    precision = rng.choice(["fp64", "fp64", "fp64_df", "fp32_bulk"])
    recon = rng.choice(["plmc", "ppmc", "plmc", "ppmc", "pcm"] + (["plm_prim"] if kind in ("run", "host") else []))
    steps = 1 if kind in ("adjoint", "adjoint_cfl") else rng.randint(2, 4) if kind == "rollout" else rng.randint(1, 10)
    # cells so that a case stays below the largest listed one (about 0.8 s)
    ns = {"fp64": 6.5, "fp64_df": 1.8, "fp32_bulk": 0.5}[precision] * steps
    ns *= {"adjoint": 6, "adjoint_cfl": 6, "rollout": 7, "evolve": 2, "host": 3}.get(kind, 1)
    cap = min(6e8 / ns, 1.2e8 if kind == "run" else 1.2e7)
    if kind == "evolve":
        cap = min(cap, 2e6)
    cells = math.exp(rng.uniform(math.log(700.0), math.log(cap)))
    side = cells ** (1.0 / 3.0)
    n = [max(6, int(round(side * math.exp(rng.uniform(-0.4, 0.4))))) for _ in range(2)]
    n.append(max(6, int(round(cells / (n[0] * n[1])))))
    init = {"run": rng.choice(["turbulent", "turbulent", "wave", "slow_wave"]), "evolve": "tube",
            "host": "turbulent"}.get(kind, "perturbed")
    return {"kind": kind, "init": init, "nx": n[0], "ny": n[1], "nz": n[2], "recon": recon, "precision": precision,
            "steps": steps, "cfl": rng.choice([0.3, 0.4])}


# ---- inputs ------------------------------------------------------------------
def _centres(case):
    out = []
    for a, n in enumerate((case["nx"], case["ny"], case["nz"])):
        x = (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n
        out.append(x.view([-1 if d == 2 - a else 1 for d in range(3)]))
    return out


def _noise(case, gen, kmax=16):
    """Gaussian noise with a k^-2 shell spectrum over 1 <= |k| <= kmax, rms 1."""
    shape = (case["nz"], case["ny"], case["nx"])
    f = torch.fft.rfftn(torch.randn(shape, generator=gen, dtype=torch.float64, device="cuda"))
    kz = torch.fft.fftfreq(shape[0], 1.0 / shape[0], dtype=torch.float64, device="cuda")[:, None, None]
    ky = torch.fft.fftfreq(shape[1], 1.0 / shape[1], dtype=torch.float64, device="cuda")[None, :, None]
    kx = torch.fft.rfftfreq(shape[2], 1.0 / shape[2], dtype=torch.float64, device="cuda")[None, None, :]
    k2 = kx * kx + ky * ky + kz * kz
    f *= torch.where((k2 >= 1) & (k2 <= kmax * kmax), 1.0 / torch.clamp(k2, min=1.0), torch.zeros_like(k2))
    x = torch.fft.irfftn(f, s=shape)
    return x / x.square().mean().sqrt()


def _cell_field(B):
    return [0.5 * (B[a] + torch.roll(B[a], 1, dims=2 - a)) for a in range(3)]


def _assemble(rho, v, p, B):
    """Conserved state [8, nz, ny, nx] of density, velocity, pressure and face fields."""
    shape = torch.broadcast_shapes(*(x.shape for x in [rho, p, *v, *B]))
    B = [b.expand(shape) for b in B]
    U = torch.empty((8,) + tuple(shape), dtype=torch.float64, device="cuda")
    U[0] = rho
    U[4] = p / (GAMMA - 1.0)
    for a, b in enumerate(_cell_field(B)):
        U[1 + a] = rho * v[a]
        U[5 + a] = B[a]
        U[4] += 0.5 * rho * v[a] * v[a] + 0.5 * b * b
    return U


def _turbulent(case, gen, perturbed):
    """Mach-1 velocity noise on a mean field plus the discrete curl of a
    random edge potential (div B = 0 to round-off); perturbed: smooth density
    and pressure variations, as the gradient tests use."""
    n = (case["nx"], case["ny"], case["nz"])
    v = [_noise(case, gen) for _ in range(3)]
    s = (sum(x.square().mean() for x in v) / GAMMA).sqrt()  # rms |v| = c_s
    v = [x / s for x in v]
    A = [_noise(case, gen) for _ in range(3)]
    B = []
    for a in range(3):
        b, c = (a + 1) % 3, (a + 2) % 3
        B.append((A[c] - torch.roll(A[c], 1, dims=2 - b)) * n[b] - (A[b] - torch.roll(A[b], 1, dims=2 - c)) * n[c])
    del A
    s = sum(x.square().mean() for x in _cell_field(B)).sqrt() / 0.1
    B = [x / s for x in B]
    B[0] = B[0] + 0.5
    rho = p = torch.ones((1, 1, 1), dtype=torch.float64, device="cuda")
    if perturbed:
        x, y, z = _centres(case)
        t = 2 * math.pi
        rho = 1 + 0.2 * torch.sin(t * (x + 0.1)) * torch.cos(t * (y + 0.3)) * torch.cos(t * (z + 0.2))
        p = 1 + 0.2 * torch.cos(t * (x + 0.2)) * torch.sin(t * (z + 0.4)) * torch.cos(t * (y + 0.1))
    return _assemble(rho, v, p, B)


def _wave(case, gen, slow):
    """A small-amplitude velocity and pressure wave (phase and amplitude from
    the seed) along x on the linear-wave backgrounds of the system tests."""
    x = _centres(case)[0]
    u = torch.rand(2, generator=gen, dtype=torch.float64, device="cuda")
    s = (1e-6 * (1 + u[0])) * torch.sin(2 * math.pi * (x + u[1]))
    one = torch.ones((case["nz"], case["ny"], case["nx"]), dtype=torch.float64, device="cuda")
    by, bz = (1.5, 0.0) if slow else (math.sqrt(2.0), 0.5)
    return _assemble(one * (1 + s), [0.5 * s, -0.3 * s, 0.2 * s], one * (1 / GAMMA + s),
                     [one, by + 0.4 * s * one, bz + 0.2 * s * one])


def _tube(case, gen):
    """A shock tube (the Brio-Wu states) with seeded cell-to-cell variations of 1e-3."""
    x = _centres(case)[0]
    shape = (case["nz"], case["ny"], case["nx"])
    left = (x < 0.5).double()
    r = [1 + 1e-3 * torch.randn(shape, generator=gen, dtype=torch.float64, device="cuda") for _ in range(2)]
    zero, one = torch.zeros(shape, dtype=torch.float64, device="cuda"), torch.ones(shape, dtype=torch.float64, device="cuda")
    return _assemble((left + 0.125 * (1 - left)) * r[0], [zero, zero, zero], (left + 0.1 * (1 - left)) * r[1],
                     [0.75 * one, (2 * left - 1) * one, zero])


def _initial(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    if case["init"] in ("turbulent", "perturbed"):
        return _turbulent(case, gen, case["init"] == "perturbed"), gen
    if case["init"] == "tube":
        return _tube(case, gen), gen
    return _wave(case, gen, case["init"] == "slow_wave"), gen


def _cotangent(case, gen):
    return torch.randn((8, case["nz"], case["ny"], case["nx"]), generator=gen, dtype=torch.float64, device="cuda")


def _fixed_dt(case):
    # well inside the CFL limit of the perturbed boxes (|v| + c_f up to about 6)
    return 0.05 / max(case["nx"], case["ny"], case["nz"])


def prepare(case, seed):
    U, gen = _initial(case, seed)
    bc = ("outflow", "periodic", "periodic") if case["init"] == "tube" else ("periodic",) * 3
    sim = mhd.Sim(case["nx"], case["ny"], case["nz"], gamma=GAMMA, cfl=case["cfl"], recon=case["recon"],
                  precision=case["precision"], bc=bc)
    state = {"case": case, "sim": sim, "U": U}
    kind = case["kind"]
    if kind == "run":
        state["dts"] = torch.zeros(case["steps"], dtype=torch.float64, device="cuda")
    elif kind == "evolve":
        state["U0"] = U
        state["U"] = U.clone()
    elif kind == "host":
        state["U"] = mhd.host_buffer(*U.shape)
        state["U"].copy_(U)
    else:
        state["g"] = _cotangent(case, gen)
    return state


def run(state):
    case, sim, U, kind = state["case"], state["sim"], state["U"], state["case"]["kind"]
    if kind == "run":  # a stretch of a simulation: the state advances in place
        sim.run(U, case["steps"], state["dts"])
        return {"U": U, "dts": state["dts"]}
    if kind == "evolve":  # a run from its initial state
        U.copy_(state["U0"])
        t, n = sim.evolve(U, 1.0, case["steps"])
        return {"U": U, "t": t, "n": n}
    if kind == "host":
        mhd.mhd_run_host(sim.ctx, U, case["steps"])
        return {"U": U}
    if kind == "adjoint":
        return {"gU": sim.adjoint_step(U, _fixed_dt(case), state["g"])}
    if kind == "adjoint_cfl":
        gU, dt, g_dt = sim.adjoint_step_cfl(U, state["g"])
        return {"gU": gU, "dt": dt, "g_dt": g_dt}
    U0 = U.detach().requires_grad_(True)
    out = mhd_autograd.rollout(sim, U0, case["steps"], checkpoint_every=2, dt_grad=True)
    out.backward(state["g"])
    return {"U": out.detach(), "gU": U0.grad}


def work(case):
    """The state read once and written once per call (and, for gradients, its
    cotangent likewise; host copies move it twice more), and the method's
    arithmetic."""
    cells = case["nx"] * case["ny"] * case["nz"]
    kind, steps = case["kind"], case["steps"]
    flops = STEP_FLOPS[case["recon"]] * cells * steps
    if kind in ("adjoint", "adjoint_cfl"):  # the step recomputed, and its reverse (two to three times it)
        return {"bytes": 192 * cells, "flops": 3.5 * flops}
    if kind == "rollout":
        return {"bytes": 256 * cells, "flops": 4.5 * flops}
    return {"bytes": (256 if kind == "host" else 128) * cells, "flops": flops}


# ---- the method in plain torch float64 -----------------------------------------
# Cell p + s e_a of an array [..., nz, ny, nx] is at(x, a, s).
def at(x, a, s):
    return torch.roll(x, -s, dims=-1 - a)


def _safe(mask, x):
    return torch.where(mask, x, torch.ones_like(x))


def _primitives(U):
    rho = U[0].clamp(min=FLOOR)
    v = [U[1 + a] / rho for a in range(3)]
    B = [0.5 * (U[5 + a] + at(U[5 + a], a, -1)) for a in range(3)]
    ke = 0.5 * sum(U[1 + a] * v[a] for a in range(3))
    p = ((GAMMA - 1) * (U[4] - ke - 0.5 * sum(b * b for b in B))).clamp(min=FLOOR)
    return torch.stack([rho, *v, p, *B])


def _axis_vector(W, a):
    b, c = (a + 1) % 3, (a + 2) % 3
    return [W[0], W[1 + a], W[1 + b], W[1 + c], W[4], W[5 + b], W[5 + c]]


def _rho_cf2(w, bn):
    gp, bt2 = GAMMA * w[4], w[5] ** 2 + w[6] ** 2
    d = gp - bn * bn - bt2
    return 0.5 * (gp + bn * bn + bt2 + torch.sqrt(d * d + 4 * gp * bt2))


def _cfl_dt(W, n, cfl):
    rates = []
    for a in range(3):
        w = _axis_vector(W, a)
        rates.append((w[1].abs() + torch.sqrt(_rho_cf2(w, W[5 + a]) / w[0])) * n[a])
    return cfl / torch.stack([r.max() for r in rates]).max()


def _flux_of(w, bn, e, pt):
    vb = w[1] * bn + w[2] * w[5] + w[3] * w[6]
    return [w[0] * w[1], w[0] * w[1] * w[1] + pt - bn * bn, w[0] * w[1] * w[2] - bn * w[5],
            w[0] * w[1] * w[3] - bn * w[6], (e + pt) * w[1] - bn * vb, w[5] * w[1] - bn * w[2],
            w[6] * w[1] - bn * w[3]]


def _hlld(L, R, bn, eps):
    """HLLD fluxes of left and right states (Miyoshi & Kusano 2005); the
    degenerate limits below eps times the star pressure."""
    cf = torch.maximum(torch.sqrt(_rho_cf2(L, bn) / L[0]), torch.sqrt(_rho_cf2(R, bn) / R[0]))
    SL, SR = torch.minimum(L[1], R[1]) - cf, torch.maximum(L[1], R[1]) + cf
    side = []
    for w in (L, R):
        mag = 0.5 * (bn * bn + w[5] ** 2 + w[6] ** 2)
        side.append((w[4] / (GAMMA - 1) + 0.5 * w[0] * (w[1] ** 2 + w[2] ** 2 + w[3] ** 2) + mag, w[4] + mag))
    rdL, rdR = L[0] * (SL - L[1]), R[0] * (SR - R[1])
    den = rdR - rdL
    SM = (rdR * R[1] - rdL * L[1] - side[1][1] + side[0][1]) / den
    pts = (rdR * side[0][1] - rdL * side[1][1] + rdL * rdR * (R[1] - L[1])) / den
    star = []
    for w, S, rd, (e, pt) in ((L, SL, rdL, side[0]), (R, SR, rdR, side[1])):
        r = rd / (S - SM)
        D = rd * (S - SM) - bn * bn
        ok = D.abs() >= eps * pts
        Ds = _safe(ok, D)
        t = bn * (SM - w[1]) / Ds
        q = (rd * (S - w[1]) - bn * bn) / Ds
        v, vv = (torch.where(ok, w[m] - w[m + 3] * t, w[m]) for m in (2, 3))
        by, bz = (torch.where(ok, w[m] * q, w[m]) for m in (5, 6))
        vb, vbs = w[1] * bn + w[2] * w[5] + w[3] * w[6], SM * bn + v * by + vv * bz
        es = ((S - w[1]) * e - pt * w[1] + pts * SM + bn * (vb - vbs)) / (S - SM)
        star.append((r, v, vv, by, bz, es, vbs))
    (rl, vl, wl, byl, bzl, _, _), (rr, vr, wr, byr, bzr, _, _) = star
    sl, sr, sg = torch.sqrt(_safe(rl > 0, rl)), torch.sqrt(_safe(rr > 0, rr)), torch.where(bn > 0, 1.0, -1.0)
    inv = 1 / (sl + sr)
    vd, wd = (sl * vl + sr * vr + (byr - byl) * sg) * inv, (sl * wl + sr * wr + (bzr - bzl) * sg) * inv
    byd = (sl * byr + sr * byl + sl * sr * (vr - vl) * sg) * inv
    bzd = (sl * bzr + sr * bzl + sl * sr * (wr - wl) * sg) * inv
    vbd = SM * bn + vd * byd + wd * bzd
    dbl = 0.5 * bn * bn >= eps * pts
    out = None
    for w, S, (e, pt), (r, v, vv, by, bz, es, vbs), s, sign in ((L, SL, side[0], star[0], sl, -1), (R, SR, side[1], star[1], sr, 1)):
        F = _flux_of(w, bn, e, pt)
        U0 = [w[0], w[0] * w[1], w[0] * w[2], w[0] * w[3], e, w[5], w[6]]
        U1 = [r, r * SM, r * v, r * vv, es, by, bz]
        U2 = [r, r * SM, r * vd, r * wd, es + sign * s * (vbs - vbd) * sg, byd, bzd]
        Sd = SM + sign * bn.abs() / s
        outer = SL >= 0 if sign < 0 else SR <= 0
        inner = dbl & ((Sd < 0) if sign < 0 else (Sd >= 0))
        f = []
        for q in range(7):
            one = F[q] + S * (U1[q] - U0[q])
            f.append(torch.where(outer, F[q], torch.where(inner, one + Sd * (U2[q] - U1[q]), one)))
        out = f if out is None else [torch.where((SL >= 0) | (~(SR <= 0) & (SM >= 0)), x, y) for x, y in zip(out, f)]
    return torch.stack(out)


def _eigen(w, bn):
    """Speeds and normalisation of the primitive eigenvectors (Stone et al. 2008)."""
    rho = w[0]
    a2, ca2, bt2 = GAMMA * w[4] / rho, bn * bn / rho, (w[5] ** 2 + w[6] ** 2) / rho
    D = a2 - ca2 - bt2
    arg = D * D + 4 * a2 * bt2
    split = arg > 0
    s = torch.where(split, torch.sqrt(_safe(split, arg)), torch.zeros_like(arg))
    cf = torch.sqrt(0.5 * (a2 + ca2 + bt2 + s))
    cs = torch.sqrt(a2) * bn.abs() / torch.sqrt(rho) / cf
    some = bt2 > 0
    bt = torch.sqrt(_safe(some, w[5] ** 2 + w[6] ** 2))
    b1, b2 = (torch.where(some, w[m] / bt, torch.full_like(bt, math.sqrt(0.5))) for m in (5, 6))
    big = torch.sqrt((_safe(split, s) + D.abs()) / (2 * _safe(split, s)))
    small = torch.where(some, torch.sqrt(a2) * bt / torch.sqrt(rho), torch.zeros_like(bt)) / (_safe(split, s) * big)
    af = torch.where(split, torch.where(D >= 0, big, small), torch.ones_like(s))
    al = torch.where(split, torch.where(D >= 0, small, big), torch.zeros_like(s))
    return rho, a2, cf, cs, af, al, b1, b2, torch.where(bn >= 0, 1.0, -1.0)


def _to_waves(E, d):
    rho, a2, cf, cs, af, al, b1, b2, sg = E
    a, sr = torch.sqrt(a2), torch.sqrt(rho)
    v, b = b1 * d[2] + b2 * d[3], (b1 * d[5] + b2 * d[6]) / sr
    tv, tb = b1 * d[3] - b2 * d[2], sg * (b1 * d[6] - b2 * d[5]) / sr
    fe, fv = af * d[4] / rho + al * a * b, al * cs * sg * v - af * cf * d[1]
    se, sv = al * d[4] / rho - af * a * b, -al * cs * d[1] - af * cf * sg * v
    n = 0.5 / a2
    return [n * (fe + fv), 0.5 * (tv + tb), n * (se + sv), d[0] - d[4] / a2, n * (se - sv), 0.5 * (tv - tb), n * (fe - fv)]


def _from_waves(E, q):
    rho, a2, cf, cs, af, al, b1, b2, sg = E
    a, sr = torch.sqrt(a2), torch.sqrt(rho)
    fp, fm, sp, sm, ap, am = q[0] + q[6], q[0] - q[6], q[2] + q[4], q[2] - q[4], q[1] + q[5], q[1] - q[5]
    comp = rho * (af * fp + al * sp)
    t = sg * (cs * al * fm - cf * af * sm)
    m = a * sr * (al * fp - af * sp)
    r = sg * sr * am
    return [comp + q[3], -cf * af * fm - cs * al * sm, b1 * t - b2 * ap, b2 * t + b1 * ap, a2 * comp, b1 * m - b2 * r,
            b2 * m + b1 * r]


def _least(x, *ys):
    """sgn(x) min(|x|, |y| ...) where all share a strict sign, else 0."""
    same = x != 0
    m = x.abs()
    for y in ys:
        same = same & (torch.sign(y) == torch.sign(x))
        m = torch.minimum(m, y.abs())
    return torch.where(same, torch.sign(x) * m, torch.zeros_like(x))


def _van_leer(l, r):
    ok = l * r > 0
    return torch.where(ok, 2 * l * r / _safe(ok, l + r), torch.zeros_like(l))


def _mean_limited(l, r, c, g):
    return torch.where(l * r > 0, torch.sign(c) * torch.minimum(torch.minimum(2 * l.abs(), 2 * r.abs()),
                                                                 torch.minimum(c.abs(), g.abs())), torch.zeros_like(l))


def _ppm(a, b, d, e):
    """Limited deviations of the two interface values from cell i, of the
    deviations of cells i-2, i-1, i+1, i+2."""
    C = 1.25
    lo, hi = 7 / 12 * b - (a + d) / 12, 7 / 12 * d - (b + e) / 12
    dm, d0, dp = a - 2 * b, b + d, e - 2 * d
    lo = torch.where((lo - b) * lo > 0, 0.5 * b - _least(3 * (b - 2 * lo), C * dm, C * d0) / 6, lo)
    hi = torch.where((d - hi) * hi < 0, 0.5 * d - _least(3 * (d - 2 * hi), C * d0, C * dp) / 6, hi)
    curv = 6 * (lo + hi)
    some = curv != 0
    r = torch.where(some, _least(curv, C * dm, C * d0, C * dp) / _safe(some, curv), torch.zeros_like(curv))
    peak = (lo * hi >= 0) | (b * d >= 0)
    lo2 = torch.where(peak, r * lo, torch.where(lo.abs() >= 2 * hi.abs(), -2 * hi, lo))
    hi2 = torch.where(peak, r * hi, torch.where(hi.abs() >= 2 * lo.abs(), -2 * lo, hi))
    return lo2, hi2


def _faces(W, a, recon):
    """States of every cell at its lower and upper face along a."""
    w = _axis_vector(W, a)
    if recon == "pcm":
        lo, hi = w, w
    elif recon == "ppmc":
        E = _eigen(w, W[5 + a])
        q = [_to_waves(E, [at(x, a, s) - x for x in w]) for s in (-2, -1, 1, 2)]
        lim = [_ppm(*x) for x in zip(*q)]
        lo = [x + y for x, y in zip(w, _from_waves(E, [m[0] for m in lim]))]
        hi = [x + y for x, y in zip(w, _from_waves(E, [m[1] for m in lim]))]
    else:
        l, r = [x - at(x, a, -1) for x in w], [at(x, a, 1) - x for x in w]
        g = [_van_leer(x, y) for x, y in zip(l, r)]
        if recon == "plmc":
            E = _eigen(w, W[5 + a])
            l, r, g = _to_waves(E, l), _to_waves(E, r), _to_waves(E, g)
        d = [_mean_limited(x, y, 0.5 * (x + y), z) for x, y, z in zip(l, r, g)]
        d = _from_waves(E, d) if recon == "plmc" else d
        lo, hi = [x - 0.5 * y for x, y in zip(w, d)], [x + 0.5 * y for x, y in zip(w, d)]
    floor = lambda s: [x.clamp(min=FLOOR) if m in (0, 4) else x for m, x in enumerate(s)]  # noqa: E731
    return floor(lo), floor(hi)


def _fluxes(W, Bn, a, recon, eps):
    lo, hi = _faces(W, a, recon)
    return _hlld(hi, [at(x, a, 1) for x in lo], Bn, eps)


def _upwind(m, lo, hi):
    return torch.where(m > 0, lo, torch.where(m < 0, hi, 0.5 * (lo + hi)))


def _edges(W, F):
    E = []
    for a in range(3):
        b, c = (a + 1) % 3, (a + 2) % 3
        ref = W[1 + c] * W[5 + b] - W[1 + b] * W[5 + c]
        rb, rc, rbc = at(ref, b, 1), at(ref, c, 1), at(at(ref, b, 1), c, 1)
        eb, ec = -F[b][5], F[c][6]
        ebc, ecb = at(eb, c, 1), at(ec, b, 1)
        slopes = _upwind(at(F[b][0], c, 1), ec - rc, ecb - rbc) + _upwind(F[b][0], ec - ref, ecb - rb)
        slopes = slopes + _upwind(at(F[c][0], b, 1), eb - rb, ebc - rbc) + _upwind(F[c][0], eb - ref, ebc - rc)
        E.append(0.25 * (eb + ebc + ec + ecb) + 0.25 * slopes)
    return E


def _updated(U, F, E, h, n):
    out = []
    for f in range(5):
        x = U[f]
        for a in range(3):
            q = F[a][f if f in (0, 4) else 1 + (f - 1 - a) % 3]
            x = x - h * n[a] * (q - at(q, a, -1))
        out.append(x)
    for a in range(3):
        b, c = (a + 1) % 3, (a + 2) % 3
        out.append(U[5 + a] - h * ((E[c] - at(E[c], b, -1)) * n[b] - (E[b] - at(E[b], c, -1)) * n[c]))
    return torch.stack(out)


def _step(U, dt, n, recon, eps):
    def fluxes(W, Bn, a, rc):
        if torch.is_grad_enabled():
            return checkpoint(_fluxes, W, Bn, a, rc, eps, use_reentrant=False)
        return _fluxes(W, Bn, a, rc, eps)

    W = _primitives(U)
    F = [fluxes(W, U[5 + a], a, "pcm") for a in range(3)]
    H = _updated(U, F, _edges(W, F), 0.5 * dt, n)
    W = _primitives(H)
    F = [fluxes(W, H[5 + a], a, recon) for a in range(3)]
    return _updated(U, F, _edges(W, F), dt, n)  # (no case comes near the floors)


def exact(case, seed):
    cells, kind, steps = case["nx"] * case["ny"] * case["nz"], case["kind"], case["steps"]
    if cells * steps > (6e6 if kind == "rollout" else 2.6e7 if kind.startswith("adjoint") else 1.3e8):
        return None
    U, gen = _initial(case, seed)
    n, recon = (case["nx"], case["ny"], case["nz"]), case["recon"]
    eps = 1e-4 if case["precision"] == "fp32_bulk" else 1e-8
    if kind in ("run", "host", "evolve"):
        ghosts = kind == "evolve"
        dts, t = [], 0.0
        with torch.no_grad():
            for _ in range(steps):
                if ghosts:  # outflow along x: zero-gradient ghost cells, filled once per step
                    U = torch.cat([U[..., :1].expand(*U.shape[:3], GHOST), U, U[..., -1:].expand(*U.shape[:3], GHOST)], -1)
                W = _primitives(U)
                dt = _cfl_dt(W[..., GHOST:-GHOST] if ghosts else W, n, case["cfl"])
                del W
                U = _step(U, dt, n, recon, eps)
                U = U[..., GHOST:-GHOST].contiguous() if ghosts else U
                dts.append(dt)
                t += float(dt)
        if kind == "run":
            return {"U": U, "dts": torch.stack(dts)}
        return {"U": U, "t": t, "n": None} if kind == "evolve" else {"U": U}
    g = _cotangent(case, gen)
    U.requires_grad_(True)
    if kind == "rollout":
        V = U
        for _ in range(steps):
            V = checkpoint(lambda X: _step(X, _cfl_dt(_primitives(X), n, case["cfl"]), n, recon, eps), V, use_reentrant=False)
        V.backward(g)
        return {"U": V.detach(), "gU": U.grad}
    if kind == "adjoint":
        _step(U, _fixed_dt(case), n, recon, eps).backward(g)
        return {"gU": U.grad}
    dt = _cfl_dt(_primitives(U), n, case["cfl"])
    d = dt.detach().requires_grad_(True)
    _step(U, d, n, recon, eps).backward(g)
    dt.backward(d.grad)
    return {"gU": U.grad, "dt": float(dt), "g_dt": float(d.grad)}
