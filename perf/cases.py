"""The work a user of the solver has it do, as timed cases through the package's public calls.

Kinds of case:
  dslash2   one fine Wilson apply in 2d (complex128, complex64 or half storage): the operator by itself, as a
            program with its own Krylov loop calls it
  dslash4   one SU(3) Wilson apply in 4d (complex64, complex128)
  sweep     one gauge configuration at one coupling: the adaptive setup at the lightest mass, a clone for each
            heavier mass and one source per mass solved by one launch (the headline workload of bench.py)
  small     the two-level FP64 workload: setup and one solve with the dense coarsest factorisation
  sources   many sources on hierarchies that are already set up, two configurations in one launch
  large     one source on one large lattice, hierarchy already set up
  su3       4d SU(3): setup of one configuration and a batch of sources (a propagator's columns)
  learned   one gradient of the near-null network (forward, loss, backward)
  normal    the conjugate gradient on the normal equations, preconditioned by multigrid

Solves ask for a relative residual of 1e-12, so that a solution is determined to far more digits than the way it
was reached: two solves of one system agree to 1e-10 whatever their rounding.

Gauge fields: U(1) links whose plaquette angles follow the quenched distribution of the coupling (in two
dimensions the plaquettes are independent up to the global constraint), in a random gauge; SU(3) links by the
recipe of the test suite (1 + 0.4 H projected to SU(3), four APE steps with alpha = 0.5).
"""
import math

import numpy as np
import torch

import paper_0707_4018_gb300 as mg

PRECISIONS = {"f64": mg.MG_FP64, "f32": mg.MG_FP32, "half": mg.MG_FP16}
# critical masses by coupling (256 x 256 fields of the test suite's table) and of the smeared SU(3) fields
M_CRIT = {3.0: -0.12420767671391457, 6.0: -0.06953918577037267, 10.0: -0.04629830091688258}
M_CRIT_SU3 = -0.028396369068779216
DELTAS = (0.02, 0.05, 0.1)  # masses above the critical one
TOL = 1e-12


def listed():
    return [
        # the smallest call: one apply on a lattice of a unit test or a coarse debugging run
        {"name": "dslash2-f64-48x36", "kind": "dslash2", "L0": 48, "L1": 36, "precision": "f64"},
        # the largest apply: the bandwidth point of bench.py
        {"name": "dslash2-f32-4096x4096", "kind": "dslash2", "L0": 4096, "L1": 4096, "precision": "f32"},
        # half storage, odd extents
        {"name": "dslash2-half-3071x2049", "kind": "dslash2", "L0": 3071, "L1": 2049, "precision": "half"},
        # the 4d apply of a mixed-precision cycle on the largest lattice of bench.py
        {"name": "dslash4-f32-32x32x32x64", "kind": "dslash4", "L0": 32, "L1": 32, "L2": 32, "L3": 64,
         "precision": "f32"},
        # the 4d apply of the FP64 outer loop and of true residuals
        {"name": "dslash4-f64-16x16x16x32", "kind": "dslash4", "L0": 16, "L1": 16, "L2": 16, "L3": 32,
         "precision": "f64"},
        # the FP64 parity workload: what a user checks a new field with
        {"name": "small-64x64-f64", "kind": "small", "L0": 64, "L1": 64, "beta": 6.0},
        # one coupling of the headline sweep: setup, clones, one solve per mass
        {"name": "sweep-256x256-f32", "kind": "sweep", "L0": 256, "L1": 256, "beta": 6.0, "precision": "f32"},
        # many sources on kept hierarchies of uneven sizes (the many-configuration workload)
        {"name": "sources-128+256-8rhs", "kind": "sources", "L0": 128, "L1": 256, "beta": 6.0, "nrhs": 8},
        # one source on a large lattice whose hierarchy is kept
        {"name": "large-1024x768-f32", "kind": "large", "L0": 1024, "L1": 768, "beta": 6.0, "precision": "f32"},
        # the 4d workload: setup and the twelve columns of a propagator
        {"name": "su3-16x16x16x32-12rhs", "kind": "su3", "L0": 16, "L1": 16, "L2": 16, "L3": 32, "nrhs": 12},
        # one training step's gradient at the training batch
        {"name": "learned-16x128x128", "kind": "learned", "L0": 128, "L1": 128, "fields": 16, "channels": 16},
        # the paper's own experiment: MG-CG on the normal equations, point source
        {"name": "normal-64x64", "kind": "normal", "L0": 64, "L1": 64, "beta": 6.0},
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def _mult(rng, lo, hi, step):
    return step * _log(rng, lo // step, hi // step)


def draw(rng):
    kind = rng.choice(["dslash2", "dslash4", "sweep", "small", "sources", "large", "su3", "learned", "normal"])
    beta = rng.choice([3.0, 6.0, 10.0])
    if kind == "dslash2":
        return {"kind": kind, "L0": _log(rng, 8, 4096), "L1": _log(rng, 8, 4096),
                "precision": rng.choice(["f64", "f32", "half"])}
    if kind == "dslash4":
        return {"kind": kind, "L0": _log(rng, 4, 32), "L1": _log(rng, 4, 32), "L2": _log(rng, 4, 32),
                "L3": _log(rng, 4, 64), "precision": rng.choice(["f32", "f64"])}
    if kind == "sweep":
        return {"kind": kind, "L0": _mult(rng, 64, 256, 16), "L1": _mult(rng, 64, 256, 16), "beta": beta,
                "precision": rng.choice(["f32", "f32", "f64", "half"])}
    if kind == "small":
        return {"kind": kind, "L0": _mult(rng, 16, 64, 4), "L1": _mult(rng, 16, 64, 4), "beta": beta}
    if kind == "sources":
        return {"kind": kind, "L0": _mult(rng, 64, 192, 16), "L1": _mult(rng, 144, 256, 16), "beta": beta,
                "nrhs": rng.randint(2, 8)}
    if kind == "large":
        return {"kind": kind, "L0": _mult(rng, 320, 1024, 32), "L1": _mult(rng, 320, 768, 32), "beta": beta,
                "precision": rng.choice(["f32", "half"])}
    if kind == "su3":
        return {"kind": kind, "L0": rng.choice([8, 12, 16]), "L1": rng.choice([8, 12, 16]),
                "L2": rng.choice([8, 12, 16]), "L3": _mult(rng, 8, 32, 4), "nrhs": rng.randint(1, 12)}
    if kind == "learned":
        return {"kind": kind, "L0": _mult(rng, 32, 128, 4), "L1": _mult(rng, 32, 128, 4), "fields": _log(rng, 1, 16),
                "channels": rng.randint(4, 16)}
    return {"kind": kind, "L0": _mult(rng, 32, 64, 4), "L1": _mult(rng, 32, 64, 4), "beta": beta}


# ---- inputs ------------------------------------------------------------------------------------------------

def _gen(seed, tag):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + tag) % (1 << 62))


def _gauss(seed, tag, shape, dtype=torch.complex128):
    """Independent N(0, 1) real and imaginary parts."""
    real = torch.float32 if dtype == torch.complex64 else torch.float64
    return torch.view_as_complex(torch.randn((*shape, 2), generator=_gen(seed, tag), device="cuda", dtype=real))


def _phases(seed, tag, shape, dtype):
    ang = torch.rand(shape, generator=_gen(seed, tag), device="cuda", dtype=torch.float64) * (2 * math.pi)
    return torch.polar(torch.ones_like(ang), ang).to(dtype)


def _u1_links(L0, L1, beta, seed, tag=0):
    """Thermal links U[x][mu], x = x0 + L0 x1: independent plaquettes, built in an axial gauge, then transformed."""
    rng = np.random.Generator(np.random.PCG64([int(seed), 77, tag]))
    P = torch.from_numpy(rng.vonmises(0.0, beta, (L1, L0))).cuda()
    P -= (P.sum() - 2 * math.pi * torch.round(P.sum() / (2 * math.pi))) / P.numel()
    hol = rng.uniform(0, 2 * math.pi, 2)
    t0 = torch.zeros((L1, L0), dtype=torch.float64, device="cuda")
    t1 = torch.zeros_like(t0)
    # P(x, y) = t0(x, y) + t1(x + 1, y) - t0(x, y + 1) - t1(x, y), t1 = 0 below the last row
    t0[0] = hol[0] / L0
    t0[1:] = t0[0] - torch.cumsum(P, 0)[:-1]
    step = P[-1] - t0[-1] + t0[0]  # t1(x + 1) - t1(x) in the last row
    t1[-1, 1:] = torch.cumsum(step, 0)[:-1]
    t1[-1] += hol[1]
    w = torch.rand((L1, L0), generator=_gen(seed, 100 + tag), device="cuda", dtype=torch.float64) * (2 * math.pi)
    th = torch.stack([t0 + w - torch.roll(w, -1, 1), t1 + w - torch.roll(w, -1, 0)], -1)
    return torch.polar(torch.ones_like(th), th).reshape(L0 * L1, 2).contiguous()


def _su3_project(M):
    a = M[..., 0, :]
    a = a / a.abs().square().sum(-1, keepdim=True).sqrt()
    b = M[..., 1, :]
    b = b - (a.conj() * b).sum(-1, keepdim=True) * a
    b = b / b.abs().square().sum(-1, keepdim=True).sqrt()
    return torch.stack([a, b, torch.linalg.cross(a, b).conj()], -2)


def _su3_links(dims, seed, smear):
    """U[mu] on the grid (L3, L2, L1, L0): 1 + 0.4 H projected to SU(3), then APE steps (alpha = 0.5)."""
    grid = tuple(reversed(dims))
    c = torch.randn((4, *grid, 8), generator=_gen(seed, 5), device="cuda", dtype=torch.float64) * (0.4 / math.sqrt(2))
    d8 = c[..., 7] / math.sqrt(3)
    M = torch.zeros((4, *grid, 3, 3), dtype=torch.complex128, device="cuda")
    M[..., 0, 0], M[..., 1, 1], M[..., 2, 2] = 1 + c[..., 2] + d8, 1 - c[..., 2] + d8, 1 - 2 * d8
    for i, j, k in ((0, 1, 0), (0, 2, 3), (1, 2, 5)):
        M[..., i, j] = torch.complex(c[..., k], -c[..., k + 1])
        M[..., j, i] = torch.complex(c[..., k], c[..., k + 1])
    U = _su3_project(M)
    for _ in range(smear):
        new = []
        for mu in range(4):
            S = torch.zeros_like(U[mu])
            for nu in range(4):
                if nu == mu:
                    continue
                un, um = U[nu], U[mu]
                up = torch.roll(um, -1, 3 - nu)          # U_mu(x + nu)
                right = torch.roll(un, -1, 3 - mu)       # U_nu(x + mu)
                S += un @ up @ right.mH
                low = un.mH @ um @ right                 # at x: U_nu(x)^+ U_mu(x) U_nu(x + mu)
                S += torch.roll(low, 1, 3 - nu)
            new.append(_su3_project(0.5 * U[mu] + (0.5 / 6) * S))
        U = torch.stack(new)
    return U


def _su3_flat(U):
    return U.permute(1, 2, 3, 4, 0, 5, 6).reshape(-1, 4, 3, 3).contiguous()


def _dims(case):
    return tuple(case[k] for k in ("L0", "L1", "L2", "L3") if k in case)


def _mass(case):
    return M_CRIT[case["beta"]] + DELTAS[0]


def _sweep_params(precision, **kw):
    return mg.mg_default_params(levels=3, blocks=[(4, 4), (2, 2)], Nv=[8, 8], precision=precision, coarsest_tol=0.2,
                                max_iter=3000, **kw)


def _net_weights(case, seed):
    """Weights [l][5][2 co][2 ci] of a network cin 8 -> channels -> channels -> channels -> 8, packed."""
    C = case["channels"]
    rng = np.random.Generator(np.random.PCG64([int(seed), 91]))
    out = []
    for ci, co in ((8, C), (C, C), (C, C), (C, 8)):
        w = rng.standard_normal((5, 2 * co, 2 * ci, 2)) / math.sqrt(10 * ci)
        out.append((w[..., 0] + 1j * w[..., 1]).astype(np.complex64))
    return out


def _net_target(case, seed):
    """Block-orthonormal columns on 4 x 4 blocks, [f][k][x][s]."""
    L0, L1, F = case["L0"], case["L1"], case["fields"]
    q = torch.linalg.qr(_gauss(seed, 31, (F, L1 // 4, L0 // 4, 32, 8)))[0]
    q = q.reshape(F, L1 // 4, L0 // 4, 4, 4, 2, 8)  # block y, block x, y, x, spin, column
    return q.permute(0, 6, 1, 3, 2, 4, 5).reshape(F, 8, L0 * L1, 2).contiguous()


def _net_seeds(case, seed):
    return [(int(seed) * 7919 + 13 * f + 1) % (1 << 40) for f in range(case["fields"])]


def prepare(case, seed):
    kind, dims = case["kind"], _dims(case)
    V = math.prod(dims)
    if kind in ("dslash2", "dslash4"):
        four = kind == "dslash4"
        prec = case["precision"]
        dt = torch.complex128 if prec == "f64" else torch.complex64
        U = _su3_flat(_su3_links(dims, seed, 0)).to(dt) if four else _phases(seed, 1, (V, 2), dt)
        psi = _gauss(seed, 2, (V, 4, 3) if four else (V, 2), dt)
        if prec == "half":
            Uh, ph = mg.half_links(V), mg.half_spinor(V)
            mg.mg_half_convert(2, U, Uh, V)
            mg.mg_half_convert(0, psi, ph, V)
            return {"case": case, "dims": dims, "U": Uh, "in": ph, "out": mg.half_spinor(V), "m": 0.01}
        return {"case": case, "dims": dims, "U": U, "in": psi, "out": torch.empty_like(psi), "m": 0.01}
    if kind == "sweep":
        chi = [_gauss(seed, 2 + i, (V, 2)) for i in range(len(DELTAS))]
        return {"case": case, "dims": dims, "U": _u1_links(*dims, case["beta"], seed), "chi": chi,
                "psi": [torch.empty_like(c) for c in chi],
                "params": _sweep_params(PRECISIONS[case["precision"]], gcr_restart=8)}
    if kind == "small":
        chi = _gauss(seed, 2, (V, 2))
        return {"case": case, "dims": dims, "U": _u1_links(*dims, case["beta"], seed), "chi": chi,
                "psi": torch.empty_like(chi), "params": mg.mg_default_params()}
    if kind == "sources":
        p = _sweep_params(mg.MG_FP32, max_rhs=case["nrhs"], gcr_restart=8)
        sizes = [(case["L0"], case["L0"]), (case["L1"], case["L1"])]
        U = [_u1_links(*s, case["beta"], seed, i) for i, s in enumerate(sizes)]
        chi = [_gauss(seed, 2 + i, (case["nrhs"], s[0] * s[1], 2)) for i, s in enumerate(sizes)]
        return {"case": case, "chi": chi, "psi": [torch.empty_like(c) for c in chi],
                "ctx": [mg.Context.setup(u, _mass(case), s, p) for u, s in zip(U, sizes)]}
    if kind == "large":
        chi = _gauss(seed, 2, (V, 2))
        ctx = mg.Context.setup(_u1_links(*dims, case["beta"], seed), _mass(case), dims,
                               _sweep_params(PRECISIONS[case["precision"]]))
        return {"case": case, "chi": chi, "psi": torch.empty_like(chi), "ctx": ctx}
    if kind == "su3":
        chi = _gauss(seed, 2, (case["nrhs"], V, 4, 3))
        p = mg.mg_default_params(levels=2, blocks=[(4, 4, 4, 4)], Nv=[24], precision=mg.MG_FP32, chiral_split=1,
                                 n_pass=1, nu_setup=400, coarsest_tol=0.3, coarsest_restart=64,
                                 coarsest_max_iter=128, gcr_restart=32, max_iter=300, max_rhs=case["nrhs"])
        return {"case": case, "dims": dims, "U": _su3_flat(_su3_links(dims, seed, 4)), "chi": chi,
                "psi": torch.empty_like(chi), "params": p}
    if kind == "learned":
        net = mg.NullNet(8, case["channels"], 8)
        net.set_weights(np.concatenate([w.reshape(-1) for w in _net_weights(case, seed)]))
        U = torch.stack([_u1_links(*dims, 6.0, seed, f) for f in range(case["fields"])])
        return {"case": case, "dims": dims, "net": net, "U": U, "target": _net_target(case, seed),
                "seeds": _net_seeds(case, seed)}
    p = mg.mg_default_params(levels=2, blocks=[(4, 4)], Nv=[8], n_pass=3, nu_setup=100)
    ctx = mg.CgContext.setup(_u1_links(*dims, case["beta"], seed), M_CRIT[case["beta"]] + DELTAS[1], dims, p)
    chi = _point_source(dims, seed)
    return {"case": case, "ctx": ctx, "chi": chi, "psi": torch.empty_like(chi)}


def _point_source(dims, seed):
    chi = torch.zeros((dims[0] * dims[1], 2), dtype=torch.complex128, device="cuda")
    chi[int(seed) * 37 % len(chi), 0] = 1.0
    return chi


# ---- one pass ----------------------------------------------------------------------------------------------

def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("dslash2", "dslash4"):
        if case["precision"] == "half":
            mg.mg_dslash_half(s["U"], s["in"], s["out"], s["m"], s["dims"])
            n = 8 * math.prod(s["dims"])
            return {"half": s["out"][:n].view(torch.float16), "norm": s["out"][n:].view(torch.float32)}
        mg.mg_dslash(s["U"], s["in"], s["out"], s["m"], s["dims"], PRECISIONS[case["precision"]])
        return s["out"]
    if kind == "sweep":
        m = [M_CRIT[case["beta"]] + d for d in DELTAS]
        ctx = mg.Context.setup(s["U"], m[0], s["dims"], s["params"])
        every = [ctx] + [ctx.clone(x) for x in m[1:]]
        mg.solve_multi(every, s["chi"], s["psi"], TOL)
        for c in every:
            c.close()
        return s["psi"]
    if kind == "small":
        ctx = mg.Context.setup(s["U"], _mass(case), s["dims"], s["params"])
        ctx.solve(s["chi"], s["psi"], TOL)
        ctx.close()
        return s["psi"]
    if kind == "sources":
        mg.solve_multi(s["ctx"], s["chi"], s["psi"], TOL, nrhs=[case["nrhs"]] * len(s["ctx"]))
        return s["psi"]
    if kind == "large":
        s["ctx"].solve(s["chi"], s["psi"], TOL)
        return s["psi"]
    if kind == "su3":
        ctx = mg.Context.setup(s["U"], M_CRIT_SU3 + DELTAS[0], s["dims"], s["params"])
        ctx.solve_batch(s["chi"], s["psi"], TOL)
        ctx.close()
        return [p for p in s["psi"]]
    if kind == "learned":
        loss, grad = s["net"].gradient(s["U"], s["dims"], s["seeds"], s["target"], (4, 4))
        return {"loss": loss, "grad": grad}
    s["ctx"].solve(s["chi"], s["psi"], 0.1 * TOL, max_iter=20000)
    return s["psi"]


# ---- what a pass cannot do without ---------------------------------------------------------------------------

def work(case):
    """Inputs read once and outputs written once; flops of the operators the method applies, where a solve counts
    as 30 multigrid cycles (four plus four smoothing steps, two residuals, transfers; coarse levels a third)."""
    kind, dims = case["kind"], _dims(case)
    V = math.prod(dims)
    if kind == "dslash2":
        return {"bytes": V * {"f64": 96, "f32": 48, "half": 32}[case["precision"]], "flops": 60 * V}
    if kind == "dslash4":
        return {"bytes": V * {"f64": 960, "f32": 480}[case["precision"]], "flops": 1368 * V}
    if kind == "learned":
        C, n = case["channels"], V * case["fields"]
        macs = 5 * 4 * (8 * C + C * C + C * C + C * 8)  # complex, forward; twice that again backward
        return {"bytes": n * (32 + 256), "flops": 3 * 8 * macs * n}
    if kind == "su3":
        n = case["nrhs"]
        per = 1368 + 2 * 8 * 48 * 6  # Wilson apply; restriction and prolongation
        return {"bytes": V * (576 + 2 * 192 * n), "flops": V * (24 * 400 * 1368 + n * 30 * (11 * 1368 + per))}
    if kind == "sources":
        V, n = case["L0"] ** 2 + case["L1"] ** 2, case["nrhs"]
        return {"bytes": V * (32 + 64 * n), "flops": V * n * 30 * 1200}
    n = len(DELTAS) if kind == "sweep" else 1
    setup = 8 * (8 * 60 + 4 * 1200) if kind in ("sweep", "small") else 0
    return {"bytes": V * (32 + 64 * n), "flops": V * (setup + n * 30 * 1200)}


# ---- the same results in 64 bits, in plain torch -----------------------------------------------------------------

def _wilson2(U, dims, m):
    """D and its adjoint on [v][x][s]; U complex128 [x][mu]."""
    L0, L1 = dims
    u = U.reshape(L1, L0, 2)
    u0, u1 = u[..., 0], u[..., 1]
    b0, b1 = torch.roll(u0, 1, 1).conj(), torch.roll(u1, 1, 0).conj()

    def apply(psi, sign):
        # sign +1: D; -1: its adjoint (gamma_5 D gamma_5 = the projectors exchanged)
        f = psi.reshape(-1, L1, L0, 2)
        a, b = f[..., 0], f[..., 1]
        out_a, out_b = (2 + m) * a, (2 + m) * b
        for fwd, back, ax, c in ((u0, b0, 2, 1.0), (u1, b1, 1, 1j)):
            # gamma_mu has [0][1] = conj(c), [1][0] = c
            for link, d, s in ((fwd, -1, sign), (back, 1, -sign)):
                pa, pb = link * torch.roll(a, d, ax), link * torch.roll(b, d, ax)
                cc = c.conjugate() if isinstance(c, complex) else c
                out_a = out_a - 0.5 * (pa - s * cc * pb)
                out_b = out_b - 0.5 * (pb - s * c * pa)
        return torch.stack([out_a, out_b], -1).reshape(psi.shape)

    return lambda p: apply(p, 1), lambda p: apply(p, -1)


# DeGrand-Rossi gamma_mu: row s has its one entry in column GAMMA[mu][s][0]
GAMMA = (((3, 1j), (2, 1j), (1, -1j), (0, -1j)), ((3, -1), (2, 1), (1, 1), (0, -1)),
         ((2, 1j), (3, -1j), (0, -1j), (1, 1j)), ((2, 1), (3, 1), (0, 1), (1, 1)))


def _wilson4(U, dims, m):
    """D and its adjoint on [x][s][c]; U[mu] complex128 on the grid (L3, L2, L1, L0)."""
    grid = tuple(reversed(dims))

    def apply(psi, sign):
        f = psi.reshape(*grid, 4, 3)
        out = (4 + m) * f
        for mu in range(4):
            cols = [e[0] for e in GAMMA[mu]]
            coef = torch.tensor([e[1] for e in GAMMA[mu]], dtype=psi.dtype, device=psi.device)[:, None]
            g = U[mu]
            n = torch.roll(f, -1, 3 - mu)
            n = n - sign * coef * n[..., cols, :]
            out = out - 0.5 * sum(g[..., None, :, b] * n[..., b, None] for b in range(3))
            n = f + sign * coef * f[..., cols, :]
            h = 0.5 * sum(g.conj()[..., None, b, :] * n[..., b, None] for b in range(3))
            out = out - torch.roll(h, 1, 3 - mu)
        return out.reshape(psi.shape)

    return lambda p: apply(p, 1), lambda p: apply(p, -1)


def _solve(ops, b):
    """x with D x = b for each leading vector: conjugate gradients on the normal equations, refined from the true
    residual until it stops falling."""
    D, Dd = ops
    n = b.shape[0]
    dot = lambda u, v: (u.conj() * v).real.reshape(n, -1).sum(1)  # noqa: E731
    wide = lambda a: a.reshape(n, *([1] * (b.dim() - 1)))  # noqa: E731
    x, best = torch.zeros_like(b), None
    for _ in range(12):
        r = b - D(x)
        rel = float((dot(r, r) / dot(b, b)).max().sqrt())
        if best is not None and rel > 0.3 * best[0]:
            if rel < best[0]:
                best = (rel, x)
            break
        best = (rel, x.clone())
        if rel < 2e-16:
            break
        s = Dd(r)
        e, p = torch.zeros_like(b), s.clone()
        s2 = s02 = dot(s, s)
        for it in range(20000):
            q = D(p)
            a = s2 / dot(q, q).clamp_min(1e-300)
            e += wide(a) * p
            r = r - wide(a) * q
            s = Dd(r)
            new = dot(s, s)
            p = s + wide(new / s2.clamp_min(1e-300)) * p
            s2 = new
            if it % 50 == 49 and bool((s2 < 1e-14 * s02).all()):
                break
        x = x + e
    return best[1]


def _philox(c, key):
    """Philox4x32-10 on four numpy uint64 arrays of 32-bit values."""
    mask, k0, k1 = np.uint64(0xFFFFFFFF), key & 0xFFFFFFFF, key >> 32
    for _ in range(10):
        p, q = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        sh = np.uint64(32)
        c = [(q >> sh) ^ c[1] ^ np.uint64(k0), q & mask, (p >> sh) ^ c[3] ^ np.uint64(k1), p & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _net_noise(n, key, channel):
    z = np.zeros(n, dtype=np.uint64)
    w = _philox([np.arange(n, dtype=np.uint64), z, z + np.uint64(channel), z + np.uint64(0x4E4E)], key)
    a = ((w[1] << np.uint64(32)) | w[0]) >> np.uint64(11)
    b = ((w[3] << np.uint64(32)) | w[2]) >> np.uint64(11)
    r = np.sqrt(-2 * np.log((a.astype(np.float64) + 1) * 2.0 ** -53))
    ang = 2 * math.pi * (b.astype(np.float64) * 2.0 ** -53)
    return r * np.cos(ang) + 1j * r * np.sin(ang)


def _bf16(z):
    """z with the rounding of bfloat16 storage (through which gradients pass unchanged)."""
    r = torch.view_as_real(z.detach().resolve_conj())
    return z + (torch.view_as_complex(r.float().bfloat16().double()) - z.detach())


def _net_exact(case, seed):
    L0, L1, F = case["L0"], case["L1"], case["fields"]
    W = [torch.from_numpy(w).cuda().to(torch.complex128).requires_grad_() for w in _net_weights(case, seed)]
    target = _net_target(case, seed)
    total = 0.0
    for f, key in enumerate(_net_seeds(case, seed)):
        u = _u1_links(L0, L1, 6.0, seed, f).to(torch.complex64).to(torch.complex128).reshape(L1, L0, 2, 1)
        u0, u1 = u[:, :, 0], u[:, :, 1]
        h = np.stack([_net_noise(2 * L0 * L1, key, c).reshape(L1, L0, 2) for c in range(8)], 2)
        h = _bf16(torch.from_numpy(h.reshape(L1, L0, 16)).cuda())
        for l, w in enumerate(W):
            T = (h, u0 * torch.roll(h, -1, 1), torch.roll(u0.conj() * h, 1, 1), u1 * torch.roll(h, -1, 0),
                 torch.roll(u1.conj() * h, 1, 0))
            a = sum(t @ w[d].T for d, t in enumerate(T))
            if l < 3:
                c = a.reshape(L1, L0, -1, 2)
                c = c / (1 + (c.real.square() + c.imag.square()).sum(-1, keepdim=True)).sqrt()
                h = _bf16(c.reshape(a.shape))
        rows = lambda t: t.reshape(L1 // 4, 4, L0 // 4, 4, 2, 8).permute(0, 2, 1, 3, 4, 5).reshape(-1, 32, 8)  # noqa: E731
        P = rows(a.reshape(L1, L0, 8, 2).permute(0, 1, 3, 2))
        Q = rows(target[f].to(torch.complex64).to(torch.complex128).permute(1, 2, 0).reshape(L1, L0, 2, 8))
        C = P.mH @ Q
        A = torch.linalg.solve(P.mH @ P, C)
        loss = (8 - (C.conj() * A).real.sum((1, 2))).mean() / 8 / F
        loss.backward()
        total += float(loss.detach())
    grad = torch.cat([w.grad.reshape(-1) for w in W]) / 2
    return {"loss": total, "grad": grad.resolve_conj().cpu().numpy()}


def exact(case, seed):
    kind, dims = case["kind"], _dims(case)
    V = math.prod(dims)
    if kind in ("dslash2", "dslash4"):
        prec = case["precision"]
        dt = torch.complex128 if prec == "f64" else torch.complex64
        if kind == "dslash4":
            U = _su3_links(dims, seed, 0).to(dt).to(torch.complex128)
            psi = _gauss(seed, 2, (V, 4, 3), dt).to(torch.complex128)
            return _wilson4(U, dims, 0.01)[0](psi)
        U = _phases(seed, 1, (V, 2), dt).to(torch.complex128)
        psi = _gauss(seed, 2, (V, 2), dt)
        if prec != "half":
            return _wilson2(U, dims, 0.01)[0](psi.to(torch.complex128))
        U = torch.view_as_complex(torch.view_as_real(U).half().double())
        norm = torch.view_as_real(psi).abs().reshape(V, 4).amax(1)
        q = (torch.view_as_real(psi).reshape(V, 4) / norm[:, None]).half().double() * norm[:, None].double()
        out = _wilson2(U, dims, 0.01)[0](torch.view_as_complex(q.reshape(V, 2, 2)))
        out = torch.view_as_real(out).reshape(V, 4)
        norm = out.abs().amax(1)
        return {"half": (out / norm[:, None]).reshape(-1), "norm": norm}
    if kind == "learned":
        return _net_exact(case, seed)
    if kind == "su3":
        # one column: all twelve would take minutes
        ops = _wilson4(_su3_links(dims, seed, 4), dims, M_CRIT_SU3 + DELTAS[0])
        chi = _gauss(seed, 2, (case["nrhs"], V, 4, 3))
        one = (lambda p: ops[0](p[0])[None], lambda p: ops[1](p[0])[None])
        return [_solve(one, chi[:1])[0]] + [None] * (case["nrhs"] - 1)
    if kind == "sources":
        out = []
        for i, L in enumerate((case["L0"], case["L1"])):
            ops = _wilson2(_u1_links(L, L, case["beta"], seed, i), (L, L), _mass(case))
            out.append(_solve(ops, _gauss(seed, 2 + i, (case["nrhs"], L * L, 2))))
        return out
    U = _u1_links(*dims, case["beta"], seed)
    if kind == "sweep":
        return [_solve(_wilson2(U, dims, M_CRIT[case["beta"]] + d), _gauss(seed, 2 + i, (1, V, 2)))[0]
                for i, d in enumerate(DELTAS)]
    if kind == "normal":
        return _solve(_wilson2(U, dims, M_CRIT[case["beta"]] + DELTAS[1]), _point_source(dims, seed)[None])[0]
    return _solve(_wilson2(U, dims, _mass(case)), _gauss(seed, 2, (1, V, 2)))[0]
