"""The work that a user of this solver has it do, as timed cases: implicit ohmic steps through the
public binding (paper_1009_0798_gb300/ohm.py) over uniform, ragged, refined and batched
hierarchies, in every precision mode, and the row-level calls that other programs build on.

A case is a dict of plain values.  kind:
  step      ohm_cn_step on one uniform periodic box (nx, ny, nz)
  eta_step  two consecutive ohm_cn_steps whose resistivity changes in between (the caller passes it)
  amr       ohm_cn_step on nested spheres of refinement about the centre of an n^3 box
  half      ohm_cn_step on the half-refined sinusoid box of Matsumoto (2011) Sec. 3.1
  batch     ohm_cn_step_batch on K independent n^3 boxes, replayed from CUDA graphs
  residual  ohm_op_residual (R = S - L B and its norms) on one uniform box
  vcycle    ohm_op_vcycle (one float64 multigrid cycle, the caller's own preconditioner)
A step starts from the same initial field on every pass (one device copy puts it back).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1009_0798_gb300 import ohm
from paper_1009_0798_gb300 import workloads as W

PRECISION = {"fp64": ohm.OHM_FP64, "mixed": ohm.OHM_MIXED, "ff": ohm.OHM_MIXED_FF}
# solver schedules: the library's defaults; the one the benchmark's 256^3 run uses; the one its
# batches and the solve service use
SCHEDULE = {
    "default": dict(),
    "default_fgmres": dict(krylov=6),
    "bench": dict(krylov=6, nu_pre=3, nu_post=2, n_coarse=2, omega=1.2, nu_coarse=(1, 0)),
    "service": dict(krylov=6, nu_pre=4, nu_post=4, n_coarse=4, omega=1.3, nu_coarse=(1, 1)),
}


def _step(name, dims, precision, schedule, eta, dtf, tol, kind="step"):
    return {"name": name, "kind": kind, "nx": dims[0], "ny": dims[1], "nz": dims[2], "precision": precision,
            "schedule": schedule, "eta": eta, "dtf": dtf, "tol": tol}


def listed():
    return [
        # the smallest call: the unit periodic box with constant resistivity (workloads.periodic_box_32),
        # library defaults: launches and read-backs decide
        _step("fp64_32", (32, 32, 32), "fp64", "default", "one", 10.0, 1e-10),
        # a small production run in mixed precision, the size of the paper's Sec. 3.3 box
        _step("mixed_64", (64, 64, 64), "mixed", "bench", "bump", 100.0, 1e-9),
        # the benchmark's box and schedule (resistive_bump_256): the largest
        _step("mixed_256", (256, 256, 256), "mixed", "bench", "bump", 100.0, 1e-9),
        # float-float outer residual, smooth two-decade resistivity
        _step("ff_128", (128, 128, 128), "ff", "bench", "lognormal", 50.0, 1e-9),
        # everything in float64 with the Krylov solver, for users who want no float32 anywhere
        _step("fp64_fgmres_128", (128, 128, 128), "fp64", "bench", "bump", 100.0, 1e-9),
        # a ragged box as the service admits it (edges any multiple of 8), resistivity following the
        # state: handed over anew with each of two steps
        _step("ragged_eta", (120, 104, 88), "mixed", "service", "lognormal", 30.0, 1e-9, "eta_step"),
        # three levels of refinement (workloads.nested_spheres_64)
        {"name": "amr_mixed_64", "kind": "amr", "n": 64, "levels": 3, "precision": "mixed", "schedule": "default_fgmres",
         "dtf": 100.0, "tol": 1e-9},
        # the paper's own refined test, backward Euler, float64 defaults
        {"name": "half_fp64", "kind": "half", "n": 16, "lam": 1.0, "precision": "fp64", "schedule": "default",
         "dt": 1e-4, "tol": 1e-10},
        # size classes of the 512-instance batch (workloads.batched_instances): an odd block count ...
        {"name": "batch_24x100", "kind": "batch", "n": 24, "K": 100, "precision": "mixed", "schedule": "service", "tol": 1e-9},
        # ... and the largest class
        {"name": "batch_64x28", "kind": "batch", "n": 64, "K": 28, "precision": "mixed", "schedule": "service", "tol": 1e-9},
        # residual of a given field, as a driver that checks another solver's answer calls it
        {"name": "residual_256", "kind": "residual", "nx": 256, "ny": 256, "nz": 256},
        # one float64 V-cycle as a preconditioner
        {"name": "vcycle_96", "kind": "vcycle", "nx": 96, "ny": 96, "nz": 96},
    ]


def _edge(rng, lo, hi):
    """A multiple of 8 in [lo, hi], spread over its logarithm."""
    return 8 * max(lo // 8, min(hi // 8, round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 8)))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "eta_step", "amr", "half", "batch", "batch", "residual", "vcycle"])
    if kind in ("step", "eta_step"):
        precision = rng.choice(["mixed", "mixed", "fp64", "ff"])
        hi = 112 if precision == "fp64" else 200
        cubic = rng.random() < 0.4
        n = _edge(rng, 16, hi)
        dims = (n, n, n) if cubic else (n, _edge(rng, 16, hi), _edge(rng, 16, hi))
        c = _step("", dims, precision, rng.choice(["bench", "service", "default_fgmres"]), rng.choice(["bump", "lognormal"]),
                  float(round(10 ** rng.uniform(1.0, 2.0), 2)), 1e-9, kind)
    elif kind == "amr":
        c = {"kind": kind, "n": 8 * rng.randint(4, 8), "levels": rng.randint(1, 3), "precision": rng.choice(["mixed", "fp64"]),
             "schedule": "default_fgmres", "dtf": float(round(10 ** rng.uniform(1.0, 2.0), 2)), "tol": 1e-9}
    elif kind == "half":
        c = {"kind": kind, "n": 8 * rng.randint(1, 4), "lam": rng.choice([0.5, 1.0]), "precision": rng.choice(["mixed", "fp64"]),
             "schedule": "default", "dt": float("%.3g" % (1e-4 * 10 ** rng.uniform(-0.5, 0.5))), "tol": 1e-10}
    elif kind == "batch":
        n = 8 * rng.randint(2, 8)
        K = max(1, min(200, int(2 ** rng.uniform(0, math.log2(8e6 / n ** 3)))))
        c = {"kind": kind, "n": n, "K": K, "precision": "mixed", "schedule": "service", "tol": 1e-9}
    else:
        hi = 256 if kind == "residual" else 160
        c = {"kind": kind, "nx": _edge(rng, 16, hi), "ny": _edge(rng, 16, hi), "nz": _edge(rng, 16, hi)}
    c.pop("name", None)
    return c


# ------------------------------------------------------------------------------- fields
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _dims(case):
    return (case["n"],) * 3 if "n" in case else (case["nx"], case["ny"], case["nz"])


def _to_blocks(dense, ijk):
    """[ncomp][nz][ny][nx] -> [nblocks][ncomp][8][8][8] in the order of the block list."""
    c, nz, ny, nx = dense.shape
    v = dense.reshape(c, nz // 8, 8, ny // 8, 8, nx // 8, 8).permute(1, 3, 5, 0, 2, 4, 6)
    return v[ijk[:, 2], ijk[:, 1], ijk[:, 0]].contiguous()


def _ijk(hier):
    return torch.from_numpy(np.ascontiguousarray(hier.blocks[:, 1:].astype(np.int64))).cuda()


def _random_field(dims, dx, gen):
    """Divergence-free random field of rms 1 with a k^-2 vector potential (workloads.random_potential_field)."""
    nx, ny, nz = dims
    kz, ky = (torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda") for n in (nz, ny))
    kx = torch.fft.rfftfreq(nx, 1.0 / nx, dtype=torch.float64, device="cuda")
    k2 = kz[:, None, None] ** 2 + ky[None, :, None] ** 2 + kx[None, None, :] ** 2
    amp = torch.where(k2 > 0, 1.0 / k2.clamp(min=1e-30), torch.zeros_like(k2))
    A = []
    for _ in range(3):
        z = torch.randn((2,) + tuple(k2.shape), dtype=torch.float64, device="cuda", generator=gen)
        A.append(torch.fft.irfftn(torch.complex(z[0], z[1]) * amp, s=(nz, ny, nx)))

    def d(f, ax):
        return (torch.roll(f, -1, ax) - torch.roll(f, 1, ax)) / (2.0 * dx)

    B = torch.stack([d(A[2], 1) - d(A[1], 0), d(A[0], 0) - d(A[2], 2), d(A[1], 2) - d(A[0], 1)])
    return B / B.square().sum(0).mean().sqrt()


def _eta(kind, dims, dx, gen):
    nx, ny, nz = dims
    if kind == "one":
        return torch.ones((nz, ny, nx), dtype=torch.float64, device="cuda")
    if kind == "bump":  # three decades about the centre (workloads.gaussian_bump_eta)
        x, y, z = ((torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * dx - 0.5 * n * dx for n in (nx, ny, nz))
        r2 = z[:, None, None] ** 2 + y[None, :, None] ** 2 + x[None, None, :] ** 2
        return 1e-3 * (1.0 + 999.0 * torch.exp(-r2 / (0.05 * max(dims) * dx) ** 2))
    # smooth two-decade lognormal field (workloads.smooth_lognormal_eta)
    noise = torch.randn((nz, ny, nx), dtype=torch.float64, device="cuda", generator=gen)
    kz, ky = (torch.fft.fftfreq(n, dtype=torch.float64, device="cuda") for n in (nz, ny))
    kx = torch.fft.rfftfreq(nx, dtype=torch.float64, device="cuda")
    k2 = kz[:, None, None] ** 2 + ky[None, :, None] ** 2 + kx[None, None, :] ** 2
    u = torch.fft.irfftn(torch.fft.rfftn(noise) * torch.exp(-2.0 * math.pi ** 2 * 4.0 * k2), s=(nz, ny, nx))
    u = (u - u.min()) / (u.max() - u.min())
    return 1e-3 * 10.0 ** (2.0 * u)


def _uniform_fields(case, seed):
    """Dense initial field, resistivities, step size and the hierarchy of a uniform case."""
    dims = _dims(case)
    dx = 1.0 / max(dims)
    gen = _gen(seed)
    eta = _eta(case.get("eta", "bump"), dims, dx, gen)
    etas = [eta]
    if case["kind"] == "eta_step":  # the second step's resistivity, up to 30% away
        etas.append(eta * (1.0 + 0.3 * _eta("lognormal", dims, dx, gen) / 0.1))
    emax = float(torch.stack([e.max() for e in etas]).max())
    dt = case.get("dtf", 100.0) * dx * dx / (6.0 * emax)
    B = _random_field(dims, dx, gen)
    if case.get("eta") == "one":  # a plane wave with a random field of rms 0.1 (workloads.periodic_box_32)
        x = 2.0 * math.pi * (torch.arange(dims[0], dtype=torch.float64, device="cuda") + 0.5) * dx
        B = 0.1 * B
        B[1] += torch.sin(x)
        B[2] += torch.cos(x)
    return B, etas, dt, dx


def _batch_fields(case, seed):
    n, K = case["n"], case["K"]
    gen = _gen(seed)
    B = torch.stack([_random_field((n, n, n), 1.0 / n, gen) for _ in range(K)])
    eta = torch.stack([_eta("lognormal", (n, n, n), 1.0 / n, gen) for _ in range(K)])
    f = torch.rand(K, dtype=torch.float64, device="cuda", generator=gen) * 90.0 + 10.0
    dt = f / (n * n) / (6.0 * eta.amax(dim=(1, 2, 3)))
    return B, eta, [float(v) for v in dt.cpu()]


def _centers(hier):
    """x, y, z of every cell, [nblocks][8][8][8] each."""
    b = torch.from_numpy(hier.blocks.astype(np.float64)).cuda()
    h = (hier.dx0 / 2.0 ** b[:, 0])[:, None]
    a = torch.arange(8, dtype=torch.float64, device="cuda") + 0.5
    x, y, z = ((b[:, 1 + d, None] * 8 + a) * h for d in range(3))
    full = (len(b), 8, 8, 8)
    return x[:, None, None, :].expand(full), y[:, None, :, None].expand(full), z[:, :, None, None].expand(full)


def _modes(x, y, z, ext, gen, amp):
    """A smooth random field of low Fourier modes (periodic in the box)."""
    out = []
    for _ in range(3):
        v = torch.zeros_like(x)
        for _ in range(6):
            k = torch.randint(-2, 3, (3,), device="cuda", generator=gen).to(torch.float64) * (2 * math.pi)
            p = torch.rand(2, dtype=torch.float64, device="cuda", generator=gen)
            v = v + p[0] * torch.sin(k[0] * x / ext[0] + k[1] * y / ext[1] + k[2] * z / ext[2] + 2 * math.pi * p[1])
        out.append(amp * v)
    return out


def _refined_fields(case, seed):
    gen = _gen(seed)
    n = case["n"]
    if case["kind"] == "half":  # workloads.sinusoid_half_refined
        h = W.refined(4 * n, 2 * n, n, 1.0 / (4 * n), [lambda lo, hi: hi[0] <= 0.5 + 1e-12])
        x, y, z = _centers(h)
        B = _modes(x, y, z, (1.0, 0.5, 0.25), gen, 0.1)
        B[2] = B[2] + torch.sin(2 * math.pi * (x + 2.0 * y))
        return h, torch.stack(B, 1).contiguous(), torch.ones_like(x).contiguous(), case["dt"]
    c = np.array([0.5, 0.5, 0.5])

    def sphere(r):
        return lambda lo, hi: float(np.sum((np.clip(c, lo, hi) - c) ** 2)) < r * r

    h = W.refined(n, n, n, 1.0 / n, [sphere(r) for r in (0.25, 0.125, 0.0625)[:case["levels"]]])
    x, y, z = _centers(h)
    X, Y, Z = x - 0.5, y - 0.5, z - 0.5
    rho = torch.sqrt(X * X + Y * Y)
    g = torch.exp(-((rho - 0.1) ** 2 + Z * Z) / 0.03 ** 2)
    amp = 0.03  # of the current ring: its field is then of order 1, like the uniform B_z
    m = _modes(x, y, z, (1.0, 1.0, 1.0), gen, 0.05)
    B = torch.stack([m[0] + amp * (X / 0.1) * (2.0 * Z / 0.03 ** 2) * g, m[1] + amp * (Y / 0.1) * (2.0 * Z / 0.03 ** 2) * g,
                     m[2] + 1.0 + amp * g / 0.1 * (2.0 - 2.0 * rho * (rho - 0.1) / 0.03 ** 2)], 1)
    r2 = X * X + Y * Y + Z * Z
    eta = torch.clamp(1e-3 * (1.0 + 0.05 ** 2 / r2.clamp(min=1e-300)), max=1.0)
    dxf = h.dx(h.nlevels - 1)
    return h, B.contiguous(), eta.contiguous(), case["dtf"] * dxf * dxf / 6.0


# ------------------------------------------------------------------------------- cases
def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "batch":
        n, K = case["n"], case["K"]
        B, eta, s["dt"] = _batch_fields(case, seed)
        hier = W.uniform(n, n, n, 1.0 / n)
        ijk = _ijk(hier)
        s["B0"] = torch.cat([_to_blocks(b, ijk) for b in B])
        s["stream"] = torch.cuda.Stream()
        s["h"] = ohm.ohm_create_hierarchy(hier.base_cells, hier.dx0, hier.blocks, precision=PRECISION[case["precision"]],
                                          n_instances=K, use_graphs=True, stream=s["stream"], **SCHEDULE[case["schedule"]])
        e = torch.cat([_to_blocks(v[None], ijk) for v in eta])
        torch.cuda.synchronize()
        ohm.ohm_set_eta(s["h"], e)
        s["B"] = torch.empty_like(s["B0"])
        torch.cuda.synchronize()
        return s
    if kind in ("amr", "half"):
        hier, s["B0"], eta, s["dt"] = _refined_fields(case, seed)
        s["h"] = ohm.ohm_create_hierarchy(hier.base_cells, hier.dx0, hier.blocks, lam=case.get("lam", 0.5),
                                          precision=PRECISION[case["precision"]], **SCHEDULE[case["schedule"]])
        ohm.ohm_set_eta(s["h"], eta)
        s["B"] = torch.empty_like(s["B0"])
        return s
    dims = _dims(case)
    hier = W.uniform(*dims, 1.0 / max(dims))
    ijk = _ijk(hier)
    B, etas, s["dt"], _ = _uniform_fields(case, seed)
    s["h"] = ohm.ohm_create_hierarchy(hier.base_cells, hier.dx0, hier.blocks,
                                      precision=PRECISION[case.get("precision", "fp64")],
                                      **SCHEDULE[case.get("schedule", "default")])
    s["eta"] = [_to_blocks(e[None], ijk) for e in etas]
    if kind != "eta_step":
        ohm.ohm_set_eta(s["h"], s["eta"][0])
    s["B0"] = _to_blocks(B, ijk)
    s["B"] = torch.empty_like(s["B0"])  # the step's field, or the row-level call's output
    if kind == "residual":
        s["S"] = _to_blocks(_random_field(dims, 1.0 / max(dims), _gen(seed + 7919)), ijk)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "residual":
        n = ohm.ohm_op_residual(s["h"], s["B0"], s["S"], s["dt"], s["B"])
        return {"R": s["B"], "l2_R": n["l2_R"], "max_abs": n["max_abs"]}
    if kind == "vcycle":
        ohm.ohm_op_vcycle(s["h"], s["B0"], s["dt"], s["B"])
        return {"e": s["B"]}
    if kind == "batch":
        with torch.cuda.stream(s["stream"]):
            s["B"].copy_(s["B0"])
        ohm.ohm_cn_step_batch(s["h"], s["B"], s["dt"], case["tol"])
        return {"B": s["B"]}
    s["B"].copy_(s["B0"])
    if kind == "eta_step":
        for e in s["eta"]:
            ohm.ohm_cn_step(s["h"], s["B"], e, s["dt"], case["tol"])
    else:
        ohm.ohm_cn_step(s["h"], s["B"], None, s["dt"], case["tol"])
    return {"B": s["B"]}


def _cells(case):
    if case["kind"] == "batch":
        return case["K"] * case["n"] ** 3
    if case["kind"] == "half":  # half of 4n x 2n x n, and that half refined (its covered cells are written too)
        return 8 * case["n"] ** 3 + 32 * case["n"] ** 3
    if case["kind"] == "amr":
        # base box and about 4/3 pi (r + half a block's diagonal)^3 of each refined sphere
        n, c = case["n"], float(case["n"] ** 3)
        for l in range(case["levels"]):
            c += min(4.2 * ((0.25 / 2 ** l + 4.0 / (n << l)) ** 3) * float((2 * n << l) ** 3), 8.0 * c)
        return int(c)
    return math.prod(_dims(case))


def work(case):
    """A step reads B and eta and writes B; a residual reads B, S and eta and writes R; a V-cycle reads R and
    eta and writes e.  Operations: the divergence of the fluxes (about 70 per cell) for each operator that
    the call cannot do without (S and the final R of a step)."""
    n = _cells(case)
    if case["kind"] == "residual":
        return {"bytes": 80.0 * n, "flops": 76.0 * n}
    steps = 2 if case["kind"] == "eta_step" else 1
    return {"bytes": 56.0 * n * steps, "flops": 152.0 * n * steps}


# ------------------------------------------------------------------------------- 64-bit values
def _div_flux(B, eta, dx):
    """div F of [K][3][nz][ny][nx] (Eqs. 4-11, 8): faces, then differences; periodic."""
    out = torch.zeros_like(B)
    dim = (4, 3, 2)  # tensor dimension of x, y, z in B; one less in eta

    for a in range(3):
        es = 0.5 * (eta + torch.roll(eta, -1, dim[a] - 1))
        Ba = B[:, a]
        pair = Ba + torch.roll(Ba, -1, dim[a] - 1)
        for b in range(3):
            if b == a:
                continue
            db, da = dim[b] - 1, dim[a] - 1
            t = (torch.roll(pair, -1, db) - torch.roll(pair, 1, db)) / (4.0 * dx)
            n = (torch.roll(B[:, b], -1, da) - B[:, b]) / dx
            F = es * (t - n)
            out[:, b] += (F - torch.roll(F, 1, da)) / dx
    return out


def _solve(b, eta, dt, dx, lam=0.5):
    """The theta step of [K][3][nz][ny][nx] fields: BiCGStab with the operator's diagonal, per instance."""
    k = dt.view(-1, 1, 1, 1, 1)
    L = lambda v: v + lam * k * _div_flux(v, eta, dx)  # noqa: E731
    dot = lambda u, v: (u * v).sum(dim=(1, 2, 3, 4), keepdim=True)  # noqa: E731
    sa = [0.5 * (2 * eta + torch.roll(eta, -1, d) + torch.roll(eta, 1, d)) for d in (3, 2, 1)]
    tot = sa[0] + sa[1] + sa[2]
    D = 1.0 + lam * k / (dx * dx) * torch.stack([tot - s for s in sa], 1)
    S = b - (1.0 - lam) * k * _div_flux(b, eta, dx)
    x = b.clone()
    goal = 1e-28 * dot(S, S)
    for _ in range(4):  # restarts from the true residual
        r = S - L(x)
        r0, p, v = r.clone(), torch.zeros_like(r), torch.zeros_like(r)
        rho = al = om = torch.ones_like(goal)
        for it in range(400):
            rho1 = dot(r0, r)
            be = rho1 / rho * (al / om)
            p = r + be * (p - om * v)
            ph = p / D
            v = L(ph)
            al = rho1 / dot(r0, v)
            s = r - al * v
            sh = s / D
            t = L(sh)
            tt = dot(t, t)
            om = dot(t, s) / tt.clamp(min=1e-300)
            live = dot(r, r) > goal
            x = x + torch.where(live, al, torch.zeros_like(al)) * ph + torch.where(live, om, torch.zeros_like(om)) * sh
            r = torch.where(live, s - om * t, r)
            rho = rho1
            if it % 5 == 4 and not bool(live.any()):
                break
        r = S - L(x)
        if bool((dot(r, r) <= 4 * goal).all()):
            break
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind in ("amr", "half", "vcycle"):  # coarse-fine rules and cycles: no plain 64-bit form
        return None
    if kind == "batch":
        n = case["n"]
        B, eta, dt = _batch_fields(case, seed)
        x = _solve(B, eta, torch.tensor(dt, dtype=torch.float64, device="cuda"), 1.0 / n)
        ijk = _ijk(W.uniform(n, n, n, 1.0 / n))
        return {"B": torch.cat([_to_blocks(v, ijk) for v in x])}
    dims = _dims(case)
    ijk = _ijk(W.uniform(*dims, 1.0 / max(dims)))
    B, etas, dt, dx = _uniform_fields(case, seed)
    if kind == "residual":
        S = _random_field(dims, dx, _gen(seed + 7919))
        R = S - B - 0.5 * dt * _div_flux(B[None], etas[0][None], dx)[0]
        return {"R": _to_blocks(R, ijk), "l2_R": float((R.square().sum() * dx ** 3).sqrt()), "max_abs": float(R.abs().max())}
    x, k = B[None], torch.tensor([dt], dtype=torch.float64, device="cuda")
    for e in etas:
        x = _solve(x, e[None], k, dx)
    return {"B": _to_blocks(x[0], ijk)}
