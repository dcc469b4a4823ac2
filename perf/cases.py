"""The workloads whose speed this repository follows, through its public calls.

A case is one call, or one short chain of calls, that a program using the
library makes over and over while it solves a non-LTE problem: a formal
solution for populations it holds on the GPU, MALI sweeps, a FAS V-cycle, a
lockstep cycle of a batch.  The handles are created with the library's own
launch shapes, as a program does that has not asked for autotuning.

``listed`` names the cases, ``draw`` gives others of the same ranges,
``prepare`` builds what a program has in hand (atmosphere, handle, populations
on the GPU), ``run`` is one pass and returns everything it computed, ``work``
counts what a pass cannot do without, and ``exact`` recomputes the same result
in plain 64-bit torch, independent of the library.

With the FP32 formal solution the results carry single precision, and a pass
hands them on as float32; with the FP64 one they stay float64.
"""
import math

import numpy as np
import torch

from paper_1701_01607_gb300 import mg3d as m
from paper_1701_01607_gb300 import synth

PREC = {"f64": m.MG3D_PREC_F64, "f32": m.MG3D_PREC_F32}
RAYS = 24
# Arithmetic of one unit (node x ray x frequency) that the method itself needs,
# exp and division counted as one operation each: the two-level atom shares the
# opacity and source interpolation over its frequencies and the step weights
# over mirror frequencies, a moving or multi-level one does not.
FLOPS_PER_UNIT = {"two": 21.0, "moving": 36.0, "six": 40.0}
# Multigrid schedule of the V-cycles: pre- and post-smoothing and the sweeps of
# the coarsest grid (the published three-level schedule).
NU1, NU2, NU3 = 2, 2, 32


def listed():
    return [
        # the smallest box the tests and examples use: one formal solution,
        # where launches and the chain of planes are all there is
        _case("formal 16x16x33 f64", "formal", "two", 16, 16, 33, 9, "f64"),
        # the benchmark box, one FP64 formal solution on device buffers
        _case("formal 64x64x129 f64", "formal", "two", 64, 64, 129, 9, "f64"),
        # the larger plane of the benchmark in mixed precision
        _case("formal 128x128x129 f32", "formal", "two", 128, 128, 129, 9, "f32"),
        # an odd box with its own frequency grid: MALI sweeps in FP64
        _case("mali 45x37x83 f64", "mali", "two", 45, 37, 83, 15, "f64", sweeps=3),
        # a wide line (more frequencies than one group holds), mixed precision
        _case("mali 96x80x161 f32", "mali", "two", 96, 80, 161, 21, "f32", sweeps=2),
        # the benchmark step: a three-grid V-cycle, FP64 throughout
        _case("vcycle 64x64x129 f64", "vcycle", "two", 64, 64, 129, 9, "f64", grids=3),
        # the same step with the FP32 formal solution
        _case("vcycle 64x64x129 f32", "vcycle", "two", 64, 64, 129, 9, "f32", grids=3),
        # a moving atmosphere (simulation snapshots): Doppler-shifted profiles
        _case("moving 48x48x97 f32", "mali", "two", 48, 48, 97, 17, "f32", sweeps=2,
              velocity=1.0),
        # partial redistribution of a resonance line
        _case("prd 32x32x65 f64", "mali", "two", 32, 32, 65, 17, "f64", sweeps=2, gamma=0.5),
        # the 6-level atom on a chromosphere, mixed precision, 120 frequencies
        _case("six 64x64x129 f32", "mali", "six", 64, 64, 129, 20, "f32", sweeps=1),
        # the 6-level atom in FP64 (converged references, strong scattering)
        _case("six 32x32x65 f64", "mali", "six", 32, 32, 65, 20, "f64", sweeps=1),
        # several atmospheres of uneven size and both atoms in lockstep
        _case("batch of 4 f32", "batch", "both", 32, 32, 33, 9, "f32", grids=3),
    ]


def _case(name, what, atom, nx, ny, nz, freq, prec, sweeps=1, grids=1, velocity=0.0, gamma=0.0):
    """freq: frequencies of the two-level line, or of each line of the 6-level
    atom (whose five continua take a fifth of that each)."""
    c = {"what": what, "atom": atom, "nx": nx, "ny": ny, "nz": nz, "freq": freq, "prec": prec,
         "sweeps": sweeps, "grids": grids, "velocity": velocity, "gamma": gamma}
    return dict(c, name=name) if name else c


def draw(rng):
    def size(lo, hi, multiple=1):
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        return max(multiple, int(round(v / multiple)) * multiple)

    def odd(lo, hi):
        return size(lo, hi) | 1

    prec = rng.choice(["f64", "f32"])
    big = 1.0 if prec == "f64" else 1.6
    kind = rng.choice(["formal", "mali", "vcycle", "moving", "prd", "six", "batch"])
    if kind in ("formal", "mali"):
        return _case(None, kind, "two", size(8, 64 * big), size(8, 64 * big), odd(17, 129),
                     rng.randint(3, 21 if prec == "f32" else 12), prec,
                     sweeps=rng.randint(1, 3) if kind == "mali" else 1)
    if kind == "vcycle":
        grids = rng.choice([2, 3])
        f = 2 ** (grids - 1)
        return _case(None, kind, "two", size(8, 48, f), size(8, 48, f), size(16, 96, f) + 1,
                     rng.randint(5, 12), prec, grids=grids)
    if kind == "moving":
        return _case(None, "mali", "two", size(8, 48), size(8, 48), odd(17, 97),
                     rng.randint(7, 19), prec, sweeps=rng.randint(1, 2),
                     velocity=rng.uniform(0.3, 1.5))
    if kind == "prd":
        return _case(None, "mali", "two", size(8, 40), size(8, 40), odd(17, 81),
                     rng.randint(7, 19), prec, sweeps=rng.randint(1, 2),
                     gamma=rng.uniform(0.2, 1.0))
    if kind == "six":
        return _case(None, "mali", "six", size(8, 32 * big), size(8, 32 * big),
                     odd(17, 65 * big), rng.choice([5, 10, 15, 20, 25]), prec)
    return _case(None, "batch", "both", size(16, 36, 4), size(16, 36, 4), size(16, 32, 4) + 1,
                 rng.randint(5, 12), prec, grids=3)


# ------------------------------------------------------------------- inputs

def _members(case):
    """(atom kind, nx, ny, nz, frequencies) of every atmosphere of the case."""
    nx, ny, nz, f = case["nx"], case["ny"], case["nz"], case["freq"]
    if case["what"] != "batch":
        return [(case["atom"], nx, ny, nz, f)]
    return [("two", nx, ny, nz, f), ("six", nx, ny, nz, 5),
            ("two", nx + 16, ny + 8, 2 * nz - 1, f), ("six", nx + 8, ny + 4, nz + 8, 5)]


def _inputs(case, seed):
    """[(kind, atmosphere, atom)] with the values these problems have: a
    stratified box from optically thin to thick with a log-normal density
    field, or a chromosphere with the 6-level atom."""
    out = []
    for i, (kind, nx, ny, nz, f) in enumerate(_members(case)):
        s = seed % 1000003 * 16 + i
        if kind == "two":
            wide = case["velocity"] > 0 or case["gamma"] > 0
            atom = synth.TwoLevelAtom(n_freq=f, x_max=5.0 if wide else 3.0,
                                      gamma_prd=case["gamma"])
            atm, atom = synth.stratified_two_level(nx, ny, nz, eps=1e-4, sigma=0.3, seed=s,
                                                   atom=atom, velocity=case["velocity"])
        else:
            atom = synth.hydrogen_like_atom(line_freq=f, cont_freq=max(1, f // 5), seed=2)
            atm = synth.chromosphere(nx, ny, nz, atom, seed=s)
        out.append((kind, atm, atom))
    return out


def _start(kind, atm, atom, seed):
    """Populations [levels, nz, ny, nx] on the GPU that a pass starts from: for
    the two-level atom an excitation that falls from LTE at the bottom to
    sqrt(eps) of it at the top, with node-to-node scatter; for the 6-level atom
    the LTE populations."""
    n_tot = torch.tensor(atm.n_tot, device="cuda")
    if kind == "six":
        saha = torch.tensor(atm.saha, device="cuda")
        saha[-1] = 1.0
        return (saha * (n_tot / saha.sum(0))).contiguous()
    g = torch.Generator(device="cuda").manual_seed(seed)
    depth = torch.linspace(0.0, 1.0, atm.nz, device="cuda", dtype=torch.float64)
    depart = (0.01 ** depth)[:, None, None] * torch.exp(
        0.1 * torch.randn(n_tot.shape, generator=g, device="cuda", dtype=torch.float64))
    ratio = atom.g_ratio * torch.exp(-atom.theta / torch.tensor(atm.T, device="cuda")) * depart
    return torch.stack([n_tot / (1.0 + ratio), n_tot * ratio / (1.0 + ratio)])


class _State:
    """Handles and device buffers of one case; the handles end with it."""

    def __init__(self, case, seed):
        m.load()
        self.case, self.handles, self.start, self.out, self.batch = case, [], [], [], None
        p = dict(n_grids=case["grids"], nu1=NU1, nu2=NU2, nu3=NU3, fs_prec=PREC[case["prec"]])
        for kind, atm, atom in _inputs(case, seed):
            create = m.mg3d_create if kind == "two" else m.mg3d_create_ml
            self.handles.append(create(atm, atom, **p))
            self.start.append(_start(kind, atm, atom, seed))
            self.out.append(torch.empty_like(self.start[-1]))
        if case["what"] == "batch":
            self.batch = m.mg3d_batch_create(self.handles)

    def __del__(self):
        try:
            torch.cuda.synchronize()
            if self.batch is not None:
                m.mg3d_batch_destroy(self.batch)
            for h in self.handles:
                m.mg3d_destroy(h)
        except Exception:   # the interpreter is going down
            pass


def prepare(case, seed):
    return _State(case, seed)


# --------------------------------------------------------------------- pass

def run(state):
    case, top = state.case, state.case["grids"]
    stream = torch.cuda.current_stream().cuda_stream
    single = case["prec"] == "f32"
    if case["gamma"] > 0:
        # the lagged mean intensity starts with the populations
        m.mg3d_init_zero_radiation(state.handles[0], top)
    else:
        for h, n in zip(state.handles, state.start):
            m.mg3d_set_populations_dev(h, top, n.data_ptr(), stream)
    if case["what"] == "formal":
        jeff, u = state.out[0][0], state.out[0][1]
        m.mg3d_formal_solve_dev(state.handles[0], top, PREC[case["prec"]], jeff.data_ptr(),
                                u.data_ptr(), stream)
        return {"jeff": jeff.float() if single else jeff, "u": u.float() if single else u}
    if case["what"] == "mali":
        change = m.mg3d_mali_sweep(state.handles[0], top, case["sweeps"])
    elif case["what"] == "vcycle":
        change = m.mg3d_fas_vcycle(state.handles[0], False)
    else:
        change = m.mg3d_batch_fas_vcycle(state.batch, len(state.handles), False)
    for h, n in zip(state.handles, state.out):
        m.mg3d_get_populations_dev(h, top, n.data_ptr(), stream)
    change = [float(c) for c in np.atleast_1d(change)]
    # level by level, so that a sparsely populated level is compared by itself
    return {"n": [(n.float() if single else n).unbind(0) for n in state.out], "change": change}


def work(case):
    """Bytes: the populations and the fields of the statistical equilibrium
    read once, the results written once.  Operations: the formal solutions of
    the pass, unit by unit."""
    total_b = total_f = 0.0
    for kind, nx, ny, nz, f in _members(case):
        nvox = nx * ny * nz
        levels = 2 if kind == "two" else 6
        freqs = f if kind == "two" else 5 * f + 5 * max(1, f // 5)
        fields = 0 if case["what"] == "formal" else 3 if kind == "two" else levels * levels + 8
        total_b += 8.0 * nvox * (2 * levels + fields)
        if case["what"] in ("formal", "mali"):
            solves = float(case["sweeps"])
        else:
            # formal solutions per grid (with the residual and the coarse
            # operator's), in units of the finest grid's
            solves = NU1 + 1 + NU2
            for k in range(1, case["grids"]):
                last = k == case["grids"] - 1
                solves += (1 + (NU3 if last else NU1 + 1 + NU2)) / 8.0 ** k
        per = FLOPS_PER_UNIT["moving" if case["velocity"] > 0 else kind]
        total_f += per * nvox * RAYS * freqs * solves
    return {"bytes": total_b, "flops": total_f}


# ---------------------------------------------------- the same in plain torch

def _directions():
    a = math.sqrt((4.0 - math.sqrt(6.4)) / 12.0)
    b = math.sqrt(1.0 - 2.0 * a * a)
    out = [(x * p[0], y * p[1], z * p[2]) for z in (1, -1) for y in (1, -1) for x in (1, -1)
           for p in ((b, a, a), (a, b, a), (a, a, b))]
    return torch.tensor(out, dtype=torch.float64, device="cuda")


def _weights(x):
    """e^-x, w0, w_up and u = 1 - w0 of the linear short characteristic."""
    ex = torch.exp(-x)
    big = x.clamp_min(0.05)
    u = -torch.expm1(-big) / big
    w0, wup = torch.zeros_like(x), torch.zeros_like(x)
    small = x.clamp_max(0.05)
    term = torch.ones_like(x)
    for k in range(1, 12):   # w0 = x/2 - x^2/6 + ..., w_up = x/2 - x^2/3 + ...
        term = term * small / k
        sign = 1.0 if k % 2 else -1.0
        w0 += sign * term / (k + 1)
        wup += sign * term * k / (k + 1)
    thin = x < 0.05
    w0 = torch.where(thin, w0, 1.0 - u)
    wup = torch.where(thin, wup, u - torch.exp(-big))
    return ex, w0, wup, 1.0 - w0


class _Grid:
    """One grid of a problem; fields are [nz, ny*nx], populations [N, nz, ny*nx]."""

    def __init__(self, nx, ny, nz, dx, dy, z, fields):
        self.nx, self.ny, self.nz, self.dx, self.dy, self.z = nx, ny, nz, dx, dy, z
        self.f = fields

    def coarser(self):
        f = {k: _restrict(v, self) for k, v in self.f.items()}
        return _Grid(self.nx // 2, self.ny // 2, (self.nz + 1) // 2, 2 * self.dx, 2 * self.dy,
                     self.z[::2], f)

    def sweep(self, chi, src, ibot, visit):
        """Every ray through the grid.  chi(k, rays), src(k, rays): [F, R or 1,
        ny*nx] of plane k; ibot [F, ny*nx]; visit(k, rays, part, I, w0, u) with
        part = I - w0 S, for 12 rays at a time."""
        mu = _directions()
        n = self.nx * self.ny
        x = torch.arange(self.nx, device="cuda")
        y = torch.arange(self.ny, device="cuda")
        for rays in (slice(0, 12), slice(12, 24)):
            d = mu[rays]
            up = rays.start == 0
            planes = list(range(self.nz)) if up else list(range(self.nz - 1, -1, -1))
            I = ibot[:, None, :].expand(-1, 12, n).contiguous() * (1.0 if up else 0.0)
            visit(planes[0], rays, I, I, torch.zeros_like(I), torch.ones_like(I))
            for kp, k in zip(planes, planes[1:]):
                s = abs(float(self.z[k] - self.z[kp])) / d[:, 2].abs()
                gx, gy = -s * d[:, 0] / self.dx, -s * d[:, 1] / self.dy
                fx, fy = gx.floor(), gy.floor()
                tx, ty = (gx - fx)[:, None], (gy - fy)[:, None]
                x0 = (x[None, :] + fx.long()[:, None]) % self.nx
                y0 = (y[None, :] + fy.long()[:, None]) % self.ny
                x1, y1 = (x0 + 1) % self.nx, (y0 + 1) % self.ny
                at = [(yy[:, :, None] * self.nx + xx[:, None, :]).reshape(12, n)
                      for yy in (y0, y1) for xx in (x0, x1)]
                wt = [(1 - tx) * (1 - ty), tx * (1 - ty), (1 - tx) * ty, tx * ty]

                def upwind(a):
                    if a.shape[1] == 1:
                        return sum(w * a[:, 0][:, i] for i, w in zip(at, wt))
                    return sum(w * a.gather(2, i.expand(a.shape[0], 12, n))
                               for i, w in zip(at, wt))

                S = src(k, rays)
                tau = 0.5 * s[:, None] * (upwind(chi(kp, rays)) + chi(k, rays))
                ex, w0, wup, u = _weights(tau)
                part = upwind(I) * ex + wup * upwind(src(kp, rays))
                I = part + w0 * S
                visit(k, rays, part, I, w0, u)


def _restrict(a, g):
    """Full weighting; on the two boundary planes only the plane itself."""
    s = a.shape[:-2]
    a = a.reshape(s + (g.nz, g.ny, g.nx))
    for dim in (-1, -2):
        a = 0.5 * a + 0.25 * (a.roll(1, dim) + a.roll(-1, dim))
    a = a[..., ::2, ::2]
    mid = 0.5 * a[..., 2:-2:2, :, :] + 0.25 * (a[..., 1:-3:2, :, :] + a[..., 3:-1:2, :, :])
    out = torch.cat([a[..., :1, :, :], mid, a[..., -1:, :, :]], dim=-3)
    return out.reshape(s + (out.shape[-3], -1))


def _prolong(a, coarse, fine):
    """Trilinear interpolation; linear in physical height."""
    s = a.shape[:-2]
    a = a.reshape(s + (coarse.nz, coarse.ny, coarse.nx))
    for dim in (-1, -2):
        nxt = 0.5 * (a + a.roll(-1, dim))
        a = torch.stack([a, nxt], dim=dim if dim == -1 else -2)
        a = a.flatten(-2) if dim == -1 else a.flatten(-3, -2)
    z = torch.tensor(fine.z, device="cuda")
    t = ((z[1::2] - z[:-2:2]) / (z[2::2] - z[:-2:2]))[:, None, None]
    between = (1 - t) * a[..., :-1, :, :] + t * a[..., 1:, :, :]
    out = torch.empty(s + (fine.nz, fine.ny, fine.nx), dtype=torch.float64, device="cuda")
    out[..., ::2, :, :], out[..., 1::2, :, :] = a, between
    return out.reshape(s + (fine.nz, -1))


class _TwoLevel:
    def __init__(self, atm, atom, grids):
        self.atom = atom
        x = torch.linspace(-1.0, 1.0, atom.n_freq, device="cuda", dtype=torch.float64)
        x = x * atom.x_max if atom.n_freq > 1 else x * 0.0
        w = torch.full_like(x, 1.0)
        if atom.n_freq > 1:
            w[0] = w[-1] = 0.5
        self.x, self.w = x, w
        self.phi = torch.exp(-x * x) / math.sqrt(math.pi)
        self.wphi = w * self.phi / (w * self.phi).sum()
        f = {k: torch.tensor(getattr(atm, k), device="cuda").reshape(atm.nz, -1)
             for k in ("T", "n_tot", "c_ul")}
        if atm.vel is not None:
            f["vel"] = torch.tensor(atm.vel, device="cuda").reshape(3, atm.nz, -1)
        self.grid = [_Grid(atm.nx, atm.ny, atm.nz, atm.dx, atm.dy, atm.z, f)]
        for _ in range(grids - 1):
            self.grid.append(self.grid[-1].coarser())
        for g in self.grid:
            g.jnu = torch.zeros((atom.n_freq,) + g.f["T"].shape, dtype=torch.float64,
                                device="cuda")
        if atom.gamma_prd > 0:
            ax = x.abs()
            R = 0.5 * torch.erfc(torch.maximum(ax[:, None], ax[None, :]))
            wq = self.wphi / self.phi
            c = torch.ones_like(x)
            for _ in range(200):
                c = torch.sqrt(c * self.phi / (R.T @ (wq * c)))
            self.redist = wq[:, None] * c[:, None] * R * c[None, :]

    def c_lu(self, g):
        return g.f["c_ul"] * self.atom.g_ratio * torch.exp(-self.atom.theta / g.f["T"])

    def prd_ratio(self, g):
        """Emission over absorption profile per frequency from the lagged field."""
        a = self.atom
        J = g.jnu.reshape(a.n_freq, -1)
        jbar = self.wphi @ J
        up = a.g_ratio * a.a_ul * jbar
        frad = up / (up + self.c_lu(g).reshape(-1))
        ratio = torch.where(jbar > 0, (self.redist.T @ J) / (self.phi[:, None] * jbar), 1.0)
        return (1.0 + a.gamma_prd * frad * (ratio - 1.0)).reshape(g.jnu.shape)

    def formal(self, g, n):
        a = self.atom
        diff = n[0] * a.g_ratio - n[1]
        chi0, S = a.kappa * diff, n[1] / diff
        F = a.n_freq
        ibot = (1.0 / torch.expm1(a.theta / g.f["T"][0])).expand(F, -1)
        jeff, U = torch.zeros_like(S), torch.zeros_like(S)
        wphi = self.wphi[:, None, None] / RAYS
        if "vel" in g.f:
            mu = _directions()

            def profile(k, rays):
                shift = torch.einsum("rc,cn->rn", mu[rays], g.f["vel"][:, k])
                return torch.exp(-(self.x[:, None, None] - shift) ** 2) / math.sqrt(math.pi)

            def chi(k, rays):
                return chi0[k] * profile(k, rays)

            def visit(k, rays, part, I, w0, u):
                w = self.w[:, None, None] * profile(k, rays)
                w = w / w.sum(0) / RAYS
                jeff[k] += (w * part).sum((0, 1))
                U[k] += (w * u).sum((0, 1))

            g.sweep(chi, lambda k, rays: S[k].expand(F, 1, -1), ibot, visit)
            return jeff, U
        rho = self.prd_ratio(g) if a.gamma_prd > 0 else torch.ones((F,) + S.shape, device="cuda",
                                                                   dtype=torch.float64)
        fresh = torch.zeros_like(g.jnu)

        def visit(k, rays, part, I, w0, u):
            jeff[k] += (wphi * part).sum((0, 1))
            U[k] += (wphi * (1.0 - w0 * rho[:, k][:, None] if a.gamma_prd > 0 else u)).sum((0, 1))
            fresh[:, k] += I.sum(1) / RAYS

        g.sweep(lambda k, rays: (self.phi[:, None] * chi0[k])[:, None],
                lambda k, rays: (rho[:, k] * S[k])[:, None], ibot, visit)
        g.jnu = fresh
        return jeff, U

    def matrix(self, g, n):
        jeff, U = self.formal(g, n)
        a = self.atom
        lu = a.g_ratio * a.a_ul * jeff + self.c_lu(g)
        ul = a.a_ul * U + a.a_ul * jeff + g.f["c_ul"]
        one = torch.ones_like(lu)
        return torch.stack([torch.stack([one, one], -1), torch.stack([-lu, ul], -1)], -2)

    def empty_start(self, g):
        lu, ul = self.c_lu(g), self.atom.a_ul + g.f["c_ul"]
        nu = g.f["n_tot"] * lu / (lu + ul)
        return torch.stack([g.f["n_tot"] - nu, nu])


class _SixLevel:
    def __init__(self, atm, atom, grids):
        self.atom = atom
        f = {k: torch.tensor(getattr(atm, k), device="cuda").reshape(atm.nz, -1)
             for k in ("T", "n_tot", "chi_c")}
        N = atom.n_levels
        f["c"] = torch.tensor(atm.c, device="cuda").reshape(N, N, atm.nz, -1)
        f["saha"] = torch.tensor(atm.saha, device="cuda").reshape(N, atm.nz, -1)
        self.grid = [_Grid(atm.nx, atm.ny, atm.nz, atm.dx, atm.dy, atm.z, f)]
        for _ in range(grids - 1):
            self.grid.append(self.grid[-1].coarser())

    def matrix(self, g, n):
        at, N = self.atom, self.atom.n_levels
        T = g.f["T"]
        P = g.f["c"].clone()
        P[range(N), range(N)] = 0.0
        for t in list(at.lines) + list(at.continua):
            line = hasattr(t, "upper")
            lo, up = t.lower, t.upper if line else N - 1
            F = t.n_freq
            v = np.linspace(-t.x_max, t.x_max, F) if line else np.linspace(1.0, t.y_max, F)
            w = np.full(F, v[1] - v[0] if F > 1 else 1.0)
            if F > 1:
                w[0] = w[-1] = 0.5 * w[0]
            v = torch.tensor(v, device="cuda")[:, None, None]
            w = torch.tensor(w, device="cuda")[:, None, None]

            def planck(rho):
                return rho ** 3 / torch.expm1(at.theta_ref * rho / T)

            if line:
                gr = float(at.g[up] / at.g[lo])
                d = torch.sqrt(T / at.t_ref)
                phi = torch.exp(-(v / d) ** 2) / (math.sqrt(math.pi) * d)
                wphi = w * phi / (w * phi).sum(0)
                chi_t = t.kappa * phi * (gr * n[lo] - n[up])
                eta_t = t.kappa * t.rho ** 3 * n[up] * phi
                B = planck(t.rho).expand(F, -1, -1)
            else:
                E = torch.exp(-at.theta_ref * t.rho * v / T)
                nG = n[up] * g.f["saha"][lo]
                chi_t = t.kappa * v ** -3 * (n[lo] - nG * E)
                eta_t = t.kappa * v ** -3 * nG * E * (t.rho * v) ** 3
                B = planck(t.rho * v)
            chi = chi_t + g.f["chi_c"]
            src, back = (eta_t + g.f["chi_c"] * B) / chi, g.f["chi_c"] * B / chi
            share = g.f["chi_c"] / chi
            J, U = torch.zeros_like(chi), torch.zeros_like(chi)

            def visit(k, rays, part, I, w0, u):
                J[:, k] += (part + w0 * back[:, k][:, None]).sum(1) / RAYS
                U[:, k] += (u + w0 * share[:, k][:, None]).sum(1) / RAYS

            g.sweep(lambda k, rays: chi[:, k][:, None], lambda k, rays: src[:, k][:, None],
                    B[:, 0], visit)
            if line:
                b_ul = t.a_ul / t.rho ** 3
                P[lo, up] += gr * b_ul * (wphi * J).sum(0)
                P[up, lo] += t.a_ul * (wphi * U).sum(0) + b_ul * (wphi * J).sum(0)
            else:
                q = t.beta * w * v ** -4
                P[lo, up] += (q * J).sum(0)
                P[up, lo] += g.f["saha"][lo] * (q * E * ((t.rho * v) ** 3 * U + J)).sum(0)
        M = -P.transpose(0, 1).clone()
        M[range(N), range(N)] = P.sum(1)
        M[0] = 1.0
        return M.permute(2, 3, 0, 1).contiguous()


def _solve(M, f):
    return torch.linalg.solve(M, f.permute(1, 2, 0)[..., None])[..., 0].permute(2, 0, 1)


def _sweeps(p, k, n, f, count):
    for _ in range(count):
        n = _solve(p.matrix(p.grid[k], n), f)
    return n


def _apply(p, k, n):
    return torch.einsum("znij,jzn->izn", p.matrix(p.grid[k], n), n)


def _vcycle(p, k, n, f):
    """FAS V-cycle from grid k (0: the finest) down to the last."""
    g, c = p.grid[k], p.grid[k + 1]
    n = _sweeps(p, k, n, f, NU1)
    r = f - _apply(p, k, n)
    before = _restrict(n, g)
    fc = _restrict(r, g) + _apply(p, k + 1, before)
    if k + 2 == len(p.grid):
        after = _sweeps(p, k + 1, before, fc, NU3)
    else:
        after = _vcycle(p, k + 1, before, fc)
    new = n * (1.0 + _prolong((after - before) / before, c, g))
    return _sweeps(p, k, torch.where(new <= 0.0, 0.1 * n, new), f, NU2)


def exact(case, seed):
    ns, change = [], []
    for kind, atm, atom in _inputs(case, seed):
        p = (_TwoLevel if kind == "two" else _SixLevel)(atm, atom, case["grids"])
        g = p.grid[0]
        shape = (-1, atm.nz, atm.ny, atm.nx)
        n0 = (p.empty_start(g) if case["gamma"] > 0 else
              _start(kind, atm, atom, seed).reshape(-1, atm.nz, atm.ny * atm.nx))
        if case["what"] == "formal":
            jeff, u = (a.reshape(shape[1:]) for a in p.formal(g, n0))
            return {"jeff": jeff, "u": u}
        f = torch.zeros_like(n0)
        f[0] = g.f["n_tot"]
        if case["what"] == "mali":
            n, last = n0, n0
            for _ in range(case["sweeps"]):
                last, n = n, _sweeps(p, 0, n, f, 1)
        else:
            n, last = _vcycle(p, 0, n0, f), n0
        change.append(float(((n - last).abs() / n.abs()).max()))
        ns.append(n.reshape(shape).unbind(0))
    return {"n": ns, "change": change}
