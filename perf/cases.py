"""Performance cases of the hydro library: the work a program has it do, through its public calls.

Each case is one call (or the few calls that belong together) on data a simulation would hold: a
uniform box, a set of AMR patches, oct groups, an oct level, the adjoint, magnetised gas, a coarse
step with its subcycled fine level.  Sizes come from the repository's configurations and
benchmark; ``draw`` spreads them over the ranges between.  ``exact`` computes the same outputs in
64-bit torch from the scheme's equations.

Fields are structure-of-arrays tensors (field, z, y, x).  Every case is seeded and built on the GPU.
"""
import math

import numpy as np
import torch

import paper_1412_0934_gb300 as hy

GAMMA, CFL, RHO_FLOOR, P_FLOOR = 5.0 / 3.0, 0.8, 1e-10, 1e-14
ALPHA = 0.4  # psi damping of the magnetised step
DEV = "cuda"
F64 = torch.float64


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # A small box stepped ten times as one captured run: the latency of a step, every step's
        # time step taken from the previous one's result on the device.
        dict(name="run_fp64_32", path="run", precision="fp64", limiter="minmod", nx=32, ny=32, nz=32, steps=10,
             gas="white", mach=0.3),
        # The headline: one FP64-accurate step of a large turbulent box.
        dict(name="step_df64_512", path="step", precision="df64", limiter="minmod", nx=512, ny=512, nz=512,
             gas="turbulent", mach=5.0),
        # The same gas in native double arithmetic, the reference the other precisions are held to.
        dict(name="step_fp64_256", path="step", precision="fp64", limiter="minmod", nx=256, ny=256, nz=256,
             gas="turbulent", mach=5.0),
        # A production-size single-precision turbulence box: MC slopes, very cold Mach-10 gas.
        dict(name="step_fp32_mc_512", path="step", precision="fp32", limiter="mc", nx=512, ny=512, nz=512,
             gas="turbulent", mach=10.0),
        # A whole AMR hierarchy's patches of uneven sizes and levels in one call.
        dict(name="patches_mixed_4096", path="patches", precision="mixed", limiter="minmod", npatch=4096,
             edges="8,16,24,32,48", parent=256),
        # One level of a small AMR run: a few small odd patches, FP64-accurate.
        dict(name="patches_df64_60", path="patches", precision="df64", limiter="minmod", npatch=60,
             edges="6,10,13,18,24", parent=96),
        # Oct groups gathered by a tree code into its 6^3 buffer.
        dict(name="octs_mixed_262144", path="octs", precision="mixed", limiter="minmod", groups=262144, parent=256),
        # A tree level after refinement: space-filling-curve order and neighbour table built, then
        # every oct stepped through the table.
        dict(name="octlevel_mixed_128", path="octlevel", precision="mixed", limiter="minmod", nx=128, ny=128, nz=128),
        # One reverse step of a gradient through a simulation.
        dict(name="adjoint_fp64_64", path="adjoint", precision="fp64", limiter="minmod", nx=64, ny=64, nz=64),
        # Magnetised gas, single precision.
        dict(name="mhd_fp32_256", path="mhd", precision="fp32", limiter="minmod", nx=256, ny=256, nz=256),
        # Parabolic reconstruction, FP64-accurate, on a box of odd sizes.
        dict(name="ppm_df64_191", path="step", precision="df64", limiter="ppm", nx=191, ny=203, nz=187,
             gas="turbulent", mach=3.0),
        # A coarse step with two fine substeps: ghosts from the coarse level and from siblings, flux
        # registers on both sides, refluxing and average-down.
        dict(name="amr_mixed_96", path="amr", precision="mixed", limiter="minmod", nx=96, ny=96, nz=96, edge=16,
             cover=0.3),
    ]


# Longest edge drawn for a box, by reconstruction and precision (a step of the largest costs no more
# than the headline's).
_MAX_EDGE = {("plm", "fp64"): 256, ("plm", "df64"): 400, ("plm", "fp32"): 512, ("plm", "mixed"): 512,
             ("ppm", "fp64"): 128, ("ppm", "df64"): 256, ("ppm", "fp32"): 384, ("ppm", "mixed"): 320,
             ("mhd", "fp64"): 160, ("mhd", "df64"): 208, ("mhd", "fp32"): 384, ("mhd", "mixed"): 352,
             ("adjoint", "fp64"): 96, ("adjoint", "fp32"): 192}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box_dims(rng, lo, hi):
    e = _log_int(rng, lo, hi)
    return {a: max(8, int(round(e * rng.uniform(0.6, 1.0)))) for a in ("nx", "ny", "nz")}


def draw(rng):
    path = rng.choice(["step", "step", "step", "patches", "patches", "run", "ppm", "mhd", "octs", "octlevel", "adjoint",
                       "amr"])
    prec = rng.choice(["fp64", "df64", "fp32", "mixed"])
    plm = rng.choice(["minmod", "mc"])
    if path in ("step", "ppm"):
        lim = "ppm" if path == "ppm" else plm
        return dict(path="step", precision=prec, limiter=lim, gas="turbulent", mach=round(rng.uniform(1.0, 5.0), 2),
                    **_box_dims(rng, 20, _MAX_EDGE[("ppm" if path == "ppm" else "plm", prec)]))
    if path == "run":
        return dict(path="run", precision=prec, limiter=plm, steps=rng.randint(2, 10), gas="white", mach=0.3,
                    **_box_dims(rng, 16, 96))
    if path == "patches":
        edges = sorted(_log_int(rng, 6, 48) for _ in range(4))
        mean = 1.5 * sum(e ** 3 for e in edges) / len(edges)
        budget = {"fp64": 12e6, "df64": 60e6, "fp32": 180e6, "mixed": 180e6}[prec]
        npatch = max(4, min(_log_int(rng, 8, 4096), int(budget / mean)))
        return dict(path="patches", precision=prec, limiter=plm, npatch=npatch, edges=",".join(map(str, edges)),
                    parent=rng.choice([96, 128, 256]))
    if path == "octs":
        return dict(path="octs", precision=prec, limiter=plm, groups=_log_int(rng, 500, 262144),
                    parent=rng.choice([64, 128, 256]))
    if path == "octlevel":
        return dict(path="octlevel", precision=rng.choice(["df64", "fp32", "mixed"]), limiter=plm,
                    **_box_dims(rng, 12, 128))
    if path == "adjoint":
        prec = rng.choice(["fp64", "fp32"])
        return dict(path="adjoint", precision=prec, limiter="minmod", **_box_dims(rng, 16, _MAX_EDGE[("adjoint", prec)]))
    if path == "mhd":
        return dict(path="mhd", precision=prec, limiter=plm, **_box_dims(rng, 24, _MAX_EDGE[("mhd", prec)]))
    edge = rng.choice([8, 12, 16, 24])
    blocks = [rng.randint(4, max(4, 224 // edge)) for _ in range(3)]
    return dict(path="amr", precision=rng.choice(["df64", "fp32", "mixed"]), limiter=plm, edge=edge,
                cover=round(rng.uniform(0.15, 0.5), 3), **{a: b * edge // 2 for a, b in zip(("nx", "ny", "nz"), blocks)})


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _randn(shape, gen):
    return torch.randn(shape, generator=gen, device=DEV, dtype=F64)


def _conserved(rho, v, p):
    return torch.stack([rho, rho * v[0], rho * v[1], rho * v[2],
                        p / (GAMMA - 1.0) + 0.5 * rho * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2])])


def _white_gas(shape, seed, mach=0.3, jitter=0.0):
    """Lognormal density (sigma 0.5), white velocities of `mach` per component, pressure 1 (or
    lognormal with sigma `jitter`)."""
    g = _gen(seed)
    rho = torch.exp(0.5 * _randn(shape, g) - 0.125)
    v = []
    for _ in range(3):
        c = _randn(shape, g) * (mach * math.sqrt(GAMMA))
        v.append(c - c.mean())
    p = torch.exp(jitter * _randn(shape, g) - 0.5 * jitter * jitter) if jitter else torch.ones_like(rho)
    return _conserved(rho, v, p)


def _turbulent_gas(shape, seed, mach, p_over_rho=1e-4):
    """Cold gas: lognormal density (sigma 1), velocities with a k^-4 power spectrum at rms Mach `mach`."""
    g = _gen(seed)
    nz, ny, nx = shape
    rho = torch.exp(_randn(shape, g) - 0.5)
    kz, ky = (torch.fft.fftfreq(n, device=DEV, dtype=F64) * n for n in (nz, ny))
    kx = torch.fft.rfftfreq(nx, device=DEV, dtype=F64) * nx
    k2 = kz[:, None, None] ** 2 + ky[None, :, None] ** 2 + kx[None, None, :] ** 2
    amp = torch.where(k2 > 0, 1.0 / k2.clamp_min(1e-30), torch.zeros_like(k2))
    del k2
    scale = mach * math.sqrt(GAMMA * p_over_rho / 3.0)
    v = []
    for _ in range(3):
        f = torch.fft.irfftn(torch.fft.rfftn(_randn(shape, g)).mul_(amp), s=shape)
        f -= f.mean()
        f *= scale / f.square().mean().sqrt()
        v.append(f)
    return _conserved(rho, v, p_over_rho * rho)


def _magnetised_gas(shape, seed):
    """Smooth periodic gas: each primitive field a sum of six random Fourier modes; sonic rms Mach 1,
    plasma beta 1, a small psi."""
    rng = np.random.default_rng(seed)
    ax = [(torch.arange(n, device=DEV, dtype=F64) + 0.5) * (2 * math.pi / n) for n in shape]

    def field():
        f = torch.zeros(shape, device=DEV, dtype=F64)
        for _ in range(6):
            k = rng.integers(0, 4, 3)
            k[int(rng.integers(0, 3))] += 1
            ph, a = float(rng.uniform(0, 2 * math.pi)), float(rng.normal())
            f += a * torch.sin(float(k[0]) * ax[2][None, None, :] + float(k[1]) * ax[1][None, :, None] +
                               float(k[2]) * ax[0][:, None, None] + ph)
        return f / f.square().mean().sqrt().clamp_min(1e-300)

    rho, p = 1.0 + 0.1 * field(), 1.0 + 0.1 * field()
    v = [math.sqrt(GAMMA / 3.0) * field() for _ in range(3)]
    B = [math.sqrt(2.0 / 3.0) * field() for _ in range(3)]
    psi = 0.01 * field()
    U = torch.stack([rho, rho * v[0], rho * v[1], rho * v[2], p / (GAMMA - 1.0), B[0], B[1], B[2], psi])
    U[4] += 0.5 * rho * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2) + 0.5 * (B[0] ** 2 + B[1] ** 2 + B[2] ** 2)
    return U


def _dtype(case):
    return torch.float32 if case["precision"] == "fp32" else F64


def _shape(case):
    return case["nz"], case["ny"], case["nx"]


def _box_gas(case, seed):
    if case["gas"] == "white":
        U = _white_gas(_shape(case), seed, case["mach"])
    else:
        U = _turbulent_gas(_shape(case), seed, case["mach"], 1e-5 if case["mach"] > 8 else 1e-4)
    return U.to(_dtype(case)).contiguous(), 1.0 / case["nx"]


def _wrap_pad(U, g):
    """Periodic box (..., z, y, x) with g ghost cells per side."""
    for d in (-1, -2, -3):
        n = U.shape[d]
        U = torch.cat([U.narrow(d, n - g, g), U, U.narrow(d, 0, g)], dim=d)
    return U


def _patch_layout(case, seed):
    """Patches as (nx, ny, nz, level, dx, ox, oy, oz): half cubes, half 2:1 boxes, levels 0-5
    (the case's own), at random origins."""
    shapes, rng = np.random.default_rng(case["npatch"]), np.random.default_rng(seed)
    edges = [int(e) for e in case["edges"].split(",")]
    rows = []
    for i in range(case["npatch"]):
        n = [int(shapes.choice(edges))] * 3
        if i % 2:
            n[int(shapes.integers(0, 3))] *= 2
        level = int(shapes.integers(0, 6))
        o = [int(rng.integers(0, case["parent"])) for _ in range(3)]
        rows.append((*n, level, 2.0 ** -level / 64.0, *o))
    return rows


def _patch_gas(case, seed):
    """The parent field padded by the longest patch, and each patch's ghosted window of it."""
    rows = _patch_layout(case, seed)
    U = _white_gas((case["parent"],) * 3, seed).to(_dtype(case))
    reach = max(max(r[:3]) for r in rows) + 2
    # origins stay below the parent's edge: two cells before it, the longest patch after it
    idx = torch.arange(-2, case["parent"] + reach, device=DEV) % case["parent"]
    U = U[:, idx][:, :, idx][:, :, :, idx].contiguous()

    def window(A, r, g=2):
        x, y, z = (r[5 + d] + 2 - g for d in range(3))
        return A[..., z:z + r[2] + 2 * g, y:y + r[1] + 2 * g, x:x + r[0] + 2 * g]

    return rows, U, window


def _offsets(rows, g):
    """Where each patch starts in a field's buffer (steps of 64 elements), and the buffer's size."""
    sizes = [-(-(r[0] + 2 * g) * (r[1] + 2 * g) * (r[2] + 2 * g) // 64) * 64 for r in rows]
    return np.concatenate([[0], np.cumsum(sizes)])


def _patch_view(flat, at, r, g):
    """Patch r of the buffers flat (5, size)."""
    shape = (r[2] + 2 * g, r[1] + 2 * g, r[0] + 2 * g)
    return flat[:, int(at):int(at) + math.prod(shape)].view(5, *shape)


def _oct_gas(case, seed):
    n = case["parent"]
    U = _white_gas((n, n, n), seed).to(_dtype(case))
    rng = np.random.default_rng(seed)
    o = torch.as_tensor(2 * rng.integers(0, n // 2, (case["groups"], 3)), device=DEV)
    r = torch.arange(-2, 4, device=DEV)
    x, y, z = ((o[:, d, None] + r) % n for d in range(3))
    flat = (z[:, :, None, None] * n + y[:, None, :, None]) * n + x[:, None, None, :]
    return torch.stack([u.reshape(-1)[flat] for u in U]), 1.0 / n


def _octlevel_gas(case, seed):
    """A periodic level of nx x ny x nz octs: its cells as a box, and the octs' positions."""
    X, Y, Z = case["nx"], case["ny"], case["nz"]
    U = _white_gas((2 * Z, 2 * Y, 2 * X), seed).to(_dtype(case))
    ax = [torch.arange(n, device=DEV, dtype=torch.int32) for n in (Z, Y, X)]
    z, y, x = torch.meshgrid(*ax, indexing="ij")
    return U, torch.stack([x, y, z], dim=-1).reshape(-1, 3).contiguous(), 1.0 / (2 * X)


def _to_octs(U):
    """Box (5, 2Z, 2Y, 2X) -> oct-major (5, octs, 8)."""
    _, Z, Y, X = U.shape
    return U.reshape(5, Z // 2, 2, Y // 2, 2, X // 2, 2).permute(0, 1, 3, 5, 2, 4, 6).reshape(5, -1, 8).contiguous()


def _amr_gas(case, seed):
    """Fine level over the whole domain, the coarse level as its mean, and the refined blocks (fine
    origins): the blocks where a smooth random field is largest, `cover` of them."""
    Z, Y, X = _shape(case)
    fine = _turbulent_gas((2 * Z, 2 * Y, 2 * X), seed, 0.8, 0.1).to(_dtype(case))
    coarse = fine.double().reshape(5, Z, 2, Y, 2, X, 2).mean(dim=(2, 4, 6)).to(_dtype(case)).contiguous()
    e = case["edge"]
    rng = np.random.default_rng(seed)
    bz, by, bx = (2 * n // e for n in (Z, Y, X))
    k, j, i = np.meshgrid(np.arange(bz), np.arange(by), np.arange(bx), indexing="ij")
    f = np.zeros((bz, by, bx))
    for _ in range(4):
        w = rng.integers(0, 3, 3)
        f += rng.normal() * np.sin(2 * np.pi * (w[0] * i / bx + w[1] * j / by + w[2] * k / bz) + rng.uniform(0, 6.3))
    f += 0.05 * rng.normal(size=f.shape)
    pick = np.sort(np.argsort(f, axis=None)[::-1][:max(1, int(case["cover"] * f.size))])
    origins = [(int(e * (b % bx)), int(e * (b // bx % by)), int(e * (b // (bx * by)))) for b in pick]
    return coarse, fine, origins, 1.0 / X


def _amr_dt(coarse, fine, dx):
    """(coarse dt, fine substep): the coarse CFL step, shortened to twice the fine level's."""
    dtc = torch.minimum(_cfl_dt(coarse, dx), 2.0 * _cfl_dt(fine, 0.5 * dx))
    return dtc, 0.5 * dtc


# ------------------------------------------------------------------ prepare
def prepare(case, seed):
    ctx = hy.hydro_init(gamma=GAMMA, cfl=CFL, rho_floor=RHO_FLOOR, p_floor=P_FLOOR, limiter=case["limiter"],
                        precision=case["precision"])
    s = dict(path=case["path"], ctx=ctx)
    path, dtype = case["path"], _dtype(case)
    if path == "step":
        U, dx = _box_gas(case, seed)
        out = torch.empty_like(U)
        s.update(U=U, res=list(out), a=hy.patch(U, 0, dx), b=hy.patch(out, 0, dx), dt=_cfl_dt(U, dx))
        s["dt_next"] = torch.empty(1, dtype=F64, device=DEV)
    elif path == "run":
        U, dx = _box_gas(case, seed)
        a, b = torch.empty_like(U), torch.empty_like(U)
        s.update(U=U, A=a, res=list(a if case["steps"] % 2 == 0 else b), a=hy.patch(a, 0, dx), b=hy.patch(b, 0, dx), steps=case["steps"])
        s["hist"] = torch.empty(case["steps"] + 1, dtype=F64, device=DEV)
    elif path == "patches":
        rows, U, window = _patch_gas(case, seed)
        at_in, at_out = _offsets(rows, 2), _offsets(rows, 0)
        fin, fout = (torch.zeros((5, int(at[-1])), dtype=dtype, device=DEV) for at in (at_in, at_out))
        speed = _speed(U)
        smax = torch.empty(len(rows), dtype=F64, device=DEV)
        ins, outs = [], []
        for p, r in enumerate(rows):
            A, B = _patch_view(fin, at_in[p], r, 2), _patch_view(fout, at_out[p], r, 0)
            A.copy_(window(U, r))
            ins.append(hy.patch(A, 2, r[4], r[3]))
            outs.append(hy.patch(B, 0, r[4], r[3]))
            torch.amax(window(speed, r, 0), dim=(0, 1, 2), out=smax[p])
        dt = CFL * torch.tensor([r[4] for r in rows], dtype=F64, device=DEV) / smax
        s.update(ins=ins, outs=outs, res=list(fout), dt=dt, dt_next=torch.empty_like(dt))
    elif path == "octs":
        G, dx = _oct_gas(case, seed)
        out = torch.empty((5, G.shape[1], 2, 2, 2), dtype=dtype, device=DEV)
        s.update(G=G, out=out, res=list(out), dx=dx, dt=_oct_dt(G, dx))
    elif path == "octlevel":
        U, pos, dx = _octlevel_gas(case, seed)
        V, n = _to_octs(U), pos.shape[0]
        out = torch.empty_like(V)
        s.update(V=V, out=out, res=list(out), pos=pos, dims=(case["nx"], case["ny"], case["nz"]), dx=dx,
                 order=torch.empty(n, dtype=torch.int32, device=DEV), dt=_cfl_dt(U, dx),
                 nbr=torch.empty((n, 27), dtype=torch.int32, device=DEV))
    elif path == "adjoint":
        U, lam, dx = _adjoint_inputs(case, seed)
        out = torch.empty_like(U)
        s.update(keep=(U, lam), res_lam=list(out), U=hy.patch(U, 0, dx), lam=hy.patch(lam, 0, dx), res=hy.patch(out, 0, dx),
                 dt=_cfl_dt(U, dx))
    elif path == "mhd":
        U = _magnetised_gas(_shape(case), seed).to(dtype).contiguous()
        dx = 1.0 / case["nx"]
        out = torch.empty_like(U)
        s.update(U=U, out=out, res=list(out), dx=dx, dt=CFL * dx / _mhd_speed_max(U),
                 dt_next=torch.empty(1, dtype=F64, device=DEV))
    else:
        coarse, fine, origins, dx = _amr_gas(case, seed)
        e, n = case["edge"], len(origins)
        A = torch.zeros((5, n, e + 4, e + 4, e + 4), dtype=dtype, device=DEV)
        for p, (x, y, z) in enumerate(origins):
            A[:, p, 2:-2, 2:-2, 2:-2] = fine[:, z:z + e, y:y + e, x:x + e]
        B, C, cout = torch.zeros_like(A), torch.zeros_like(A), torch.empty_like(coarse)
        dtc, dtf = _amr_dt(coarse, fine, dx)
        half = e // 2
        creg = torch.zeros((n, 5 * hy.register_size(half, half, half)), dtype=dtype, device=DEV)
        freg = torch.zeros((n, 5 * hy.register_size(e, e, e)), dtype=dtype, device=DEV)
        s.update(keep=(coarse, A, B), coarse=hy.patch(coarse, 0, dx), cout=hy.patch(cout, 0, dx),
                 fine=[[hy.patch(T[:, p], 2, 0.5 * dx, 1) for p in range(n)] for T in (A, B, C)], origins=origins,
                 boxes=[tuple(v // 2 for v in o) for o in origins], dims=[(half,) * 3] * n,
                 period=(2 * case["nx"], 2 * case["ny"], 2 * case["nz"]), creg=list(creg), freg=list(freg), dtc=dtc,
                 dtf=dtf.expand(n).contiguous(), res=dict(coarse=list(cout), fine=list(C), coarse_fluxes=creg, fine_fluxes=freg))
    return s


# ------------------------------------------------------------------ run
def run(s):
    ctx, path = s["ctx"], s["path"]
    if path == "step":
        hy.hydro_step(ctx, s["a"], s["b"], s["dt"], s["dt_next"])
        return dict(U=s["res"], dt=s["dt_next"])
    if path == "run":
        s["A"].copy_(s["U"])
        hy.hydro_run(ctx, s["a"], s["b"], s["steps"], s["hist"])
        return dict(U=s["res"], dt=s["hist"])
    if path == "patches":
        hy.hydro_step(ctx, s["ins"], s["outs"], s["dt"], s["dt_next"])
        return dict(U=s["res"], dt=s["dt_next"])
    if path == "octs":
        hy.hydro_step_octs(ctx, s["G"], s["out"], s["dx"], s["dt"])
        return dict(U=s["res"])
    if path == "octlevel":
        hy.hydro_octs_build(ctx, s["pos"], s["dims"], s["order"], s["nbr"])
        hy.hydro_step_octs_table(ctx, s["V"], s["out"], s["nbr"], s["order"], s["dx"], s["dt"])
        return dict(U=s["res"], order=s["order"], nbr=s["nbr"])
    if path == "adjoint":
        hy.hydro_adjoint_step(ctx, s["U"], s["dt"], s["lam"], s["res"])
        return dict(lam=s["res_lam"])
    if path == "mhd":
        hy.hydro_mhd_step(ctx, s["U"], s["out"], s["dx"], s["dt"], s["dt_next"])
        return dict(U=s["res"], dt=s["dt_next"])
    A, B, C = s["fine"]
    hy.hydro_level_fluxes(ctx, s["coarse"], s["boxes"], s["dims"], s["dtc"], s["creg"])
    hy.hydro_step(ctx, s["coarse"], s["cout"], s["dtc"])
    hy.hydro_fill_ghosts(ctx, s["coarse"], A, s["origins"])
    hy.hydro_exchange_ghosts(ctx, A, s["origins"], s["period"])
    hy.hydro_patch_fluxes(ctx, A, s["dtf"], s["freg"])
    hy.hydro_step(ctx, A, B, s["dtf"])
    hy.hydro_fill_ghosts_time(ctx, s["coarse"], s["cout"], 0.5, B, s["origins"])
    hy.hydro_exchange_ghosts(ctx, B, s["origins"], s["period"])
    hy.hydro_patch_fluxes(ctx, B, s["dtf"], s["freg"], accumulate=True)
    hy.hydro_step(ctx, B, C, s["dtf"])
    hy.hydro_reflux(ctx, s["cout"], s["boxes"], s["dims"], s["creg"], s["freg"])
    hy.hydro_average_down(ctx, s["cout"], C, s["origins"])
    return s["res"]


# ------------------------------------------------------------------ work
def work(case):
    """Bytes: the state read once and written once (a patch with its ghosts, an oct with the 80
    stencil cells its update depends on).  Flops of the scheme per cell: 375 for the PLM step, about
    620 with parabolas, 1500 for the magnetised step; a reverse step about three forward ones."""
    e = 4 if case["precision"] == "fp32" else 8
    path = case["path"]
    if path in ("step", "run"):
        n = case["nx"] * case["ny"] * case["nz"] * case.get("steps", 1)
        return dict(bytes=10 * e * n, flops=(620 if case["limiter"] == "ppm" else 375) * n)
    if path == "patches":
        rows = _patch_layout(case, 0)
        n = sum(r[0] * r[1] * r[2] for r in rows)
        return dict(bytes=5 * e * (n + sum((r[0] + 4) * (r[1] + 4) * (r[2] + 4) for r in rows)), flops=375 * n)
    if path == "octs":
        return dict(bytes=5 * e * 88 * case["groups"], flops=375 * 8 * case["groups"])
    if path == "octlevel":
        n = case["nx"] * case["ny"] * case["nz"]
        return dict(bytes=(80 * e + 12 + 4 + 108) * n, flops=375 * 8 * n)
    n = case["nx"] * case["ny"] * case["nz"]
    if path == "adjoint":
        return dict(bytes=15 * e * n, flops=3 * 375 * n)
    if path == "mhd":
        return dict(bytes=18 * e * n, flops=1500 * n)
    fine = 8 * n * case["cover"]
    return dict(bytes=10 * e * n + 20 * e * fine, flops=375 * (n + 2 * fine))


# ------------------------------------------------------------------ the scheme in 64 bits
def _prim(U):
    rho = torch.where(U[0] < RHO_FLOOR, torch.full_like(U[0], RHO_FLOOR), U[0])
    u, v, w = U[1] / rho, U[2] / rho, U[3] / rho
    p = (GAMMA - 1.0) * (U[4] - 0.5 * (U[1] * U[1] + U[2] * U[2] + U[3] * U[3]) / rho)
    return [rho, u, v, w, torch.where(p < P_FLOOR, torch.full_like(p, P_FLOOR), p)]


def _speed(U):
    q = _prim([u.double() for u in U])
    return q[1].abs() + q[2].abs() + q[3].abs() + 3.0 * torch.sqrt(GAMMA * q[4] / q[0])


def _cfl_dt(U, dx):
    """CFL time step of a periodic box (1-element tensor)."""
    m = torch.stack([_speed(U[:, z:z + 64]).max() for z in range(0, U.shape[1], 64)]).max()
    return (CFL * dx / m).reshape(1)


def _oct_dt(G, dx):
    return (CFL * dx / _speed(G[:, :, 2:4, 2:4, 2:4]).max()).reshape(1)


def _part(a, d, s, w):
    """The block of a shrunk by w cells per side in z, y and x, moved by s along axis d (0 x, 1 y, 2 z)."""
    for ax in range(3):
        n = a.shape[-1 - ax] - 2 * w
        a = a.narrow(-1 - ax, w + (s if ax == d else 0), n)
    return a


def _face_part(a, d, s):
    """Of a block with one ring cell per side: cells s .. n + s along axis d (n interior cells there),
    interior across it."""
    for ax in range(3):
        n = a.shape[-1 - ax] - 2
        a = a.narrow(-1 - ax, s, n + 1) if ax == d else a.narrow(-1 - ax, 1, n)
    return a


def _slope(a, b, limiter):
    zero = torch.zeros_like(a)
    if limiter == "minmod":
        return torch.where(a * b <= 0, zero, torch.where(a.abs() <= b.abs(), a, b))
    m = torch.where((2 * b).abs() < (2 * a).abs(), 2 * b, 2 * a)
    c = 0.5 * (a + b)
    return torch.where(a * b <= 0, zero, torch.where(c.abs() < m.abs(), c, m))


def _parabola(q, d):
    """Edges (low, high) of the cells two in from the block's ends along d, as offsets from the cell."""
    def at(s):
        return _part(q, d, s, 2)

    def mc(s):
        dl, dr, dc = at(s) - at(s - 1), at(s + 1) - at(s), 0.5 * (at(s + 1) - at(s - 1))
        m = torch.minimum(dc.abs(), 2.0 * torch.minimum(dl.abs(), dr.abs()))
        return torch.where(dl * dr > 0, torch.copysign(m, dc), torch.zeros_like(m))

    c = at(0)
    sm, s0, sp = mc(-1), mc(0), mc(1)
    hi = c + 0.5 * (at(1) - c) - (sp - s0) / 6.0
    lo = at(-1) + 0.5 * (c - at(-1)) - (s0 - sm) / 6.0
    ext = (hi - c) * (c - lo) <= 0
    D, Q = hi - lo, 6.0 * (c - 0.5 * (lo + hi))
    over = D * Q > D * D
    under = ~over & (-(D * D) > D * Q)
    nlo = torch.where(ext, c, torch.where(over, 3.0 * c - 2.0 * hi, lo))
    nhi = torch.where(ext, c, torch.where(under, 3.0 * c - 2.0 * lo, hi))
    return nlo - c, nhi - c


def _floored(q):
    return [torch.where(q[0] < RHO_FLOOR, torch.full_like(q[0], RHO_FLOOR), q[0]), q[1], q[2], q[3],
            torch.where(q[4] < P_FLOOR, torch.full_like(q[4], P_FLOOR), q[4])]


def _hllc(L, R, d):
    """HLLC flux along axis d (Davis speeds, star states of Batten et al.)."""
    n = 1 + d

    def side(q):
        E = q[4] / (GAMMA - 1.0) + 0.5 * q[0] * (q[1] * q[1] + q[2] * q[2] + q[3] * q[3])
        U = [q[0], q[0] * q[1], q[0] * q[2], q[0] * q[3], E]
        F = [q[n] * x for x in U]
        F[n] = F[n] + q[4]
        F[4] = F[4] + q[n] * q[4]
        return U, F, torch.sqrt(GAMMA * q[4] / q[0])

    (UL, FL, cL), (UR, FR, cR) = side(L), side(R)
    SL, SR = torch.minimum(L[n] - cL, R[n] - cR), torch.maximum(L[n] + cL, R[n] + cR)
    mL, mR = L[0] * (SL - L[n]), R[0] * (SR - R[n])
    S = (R[4] - L[4] + L[n] * mL - R[n] * mR) / (mL - mR)

    def star(q, U, F, SK, m):
        r = m / (SK - S)
        X = [r, r * q[1], r * q[2], r * q[3], r * (U[4] / q[0] + (S - q[n]) * (S + q[4] / m))]
        X[n] = r * S
        return [f + SK * (x - u) for f, x, u in zip(F, X, U)]

    TL, TR = star(L, UL, FL, SL, mL), star(R, UR, FR, SR, mR)
    return [torch.where(SL >= 0, a, torch.where(S >= 0, b, torch.where(SR > 0, c, e)))
            for a, b, c, e in zip(FL, TL, TR, FR)]


def _euler_step(U, dt, dx, limiter, fluxes=None):
    """U: five tensors (..., z, y, x) with two ghost cells per side (three for parabolas); the interior
    after one step.  fluxes: a list that receives the x, y and z face fluxes."""
    g = 3 if limiter == "ppm" else 2
    q = _prim(U)
    c = [_part(a, 0, 0, g - 1) for a in q]
    lo, hi, dq = [], [], []
    for d in range(3):
        if limiter == "ppm":
            e = [_parabola(a, d) for a in q]
            lo.append([x for x, _ in e])
            hi.append([y for _, y in e])
            dq.append([y - x for x, y in e])
        else:
            s = [_slope(k - _part(a, d, -1, 1), _part(a, d, 1, 1) - k, limiter) for a, k in zip(q, c)]
            lo.append([-0.5 * x for x in s])
            hi.append([0.5 * x for x in s])
            dq.append(s)
    t = [0, 0, 0, 0, 0]
    for d in range(3):
        s, un = dq[d], c[1 + d]
        a = [un * s[0] + c[0] * s[1 + d], un * s[1], un * s[2], un * s[3], GAMMA * c[4] * s[1 + d] + un * s[4]]
        a[1 + d] = a[1 + d] + s[4] / c[0]
        t = [x + y for x, y in zip(t, a)]
    qh = [x - (0.5 * dt / dx) * y for x, y in zip(c, t)]
    div = [0, 0, 0, 0, 0]
    for d in range(3):
        L = _floored([_face_part(x + y, d, 0) for x, y in zip(qh, hi[d])])
        R = _floored([_face_part(x + y, d, 1) for x, y in zip(qh, lo[d])])
        F = _hllc(L, R, d)
        if fluxes is not None:
            fluxes.append(torch.stack(F))
        n = F[0].shape[-1 - d] - 1
        div = [x + (f.narrow(-1 - d, 1, n) - f.narrow(-1 - d, 0, n)) for x, f in zip(div, F)]
    return [_part(u, 0, 0, g) - (dt / dx) * y for u, y in zip(U, div)]


def _mhd_prim(U):
    q = _prim([U[0], U[1], U[2], U[3], U[4] - 0.5 * (U[5] * U[5] + U[6] * U[6] + U[7] * U[7])])
    return q + [U[5], U[6], U[7], U[8]]


def _mhd_cons(q):
    E = q[4] / (GAMMA - 1.0) + 0.5 * q[0] * (q[1] * q[1] + q[2] * q[2] + q[3] * q[3]) + \
        0.5 * (q[5] * q[5] + q[6] * q[6] + q[7] * q[7])
    return [q[0], q[0] * q[1], q[0] * q[2], q[0] * q[3], E, q[5], q[6], q[7], q[8]]


def _mhd_flux(q, d, ch):
    un, Bn = q[1 + d], q[5 + d]
    pt = q[4] + 0.5 * (q[5] * q[5] + q[6] * q[6] + q[7] * q[7])
    F = [q[0] * un] + [q[0] * un * q[1 + k] - Bn * q[5 + k] for k in range(3)]
    F[1 + d] = F[1 + d] + pt
    F.append((_mhd_cons(q)[4] + pt) * un - Bn * (q[1] * q[5] + q[2] * q[6] + q[3] * q[7]))
    F += [un * q[5 + k] - q[1 + k] * Bn for k in range(3)]
    F[5 + d] = q[8]
    return F + [ch * ch * Bn]


def _fast(q, d):
    a2, b2 = GAMMA * q[4] / q[0], (q[5] * q[5] + q[6] * q[6] + q[7] * q[7]) / q[0]
    r = (a2 + b2) ** 2 - 4.0 * a2 * q[5 + d] * q[5 + d] / q[0]
    return torch.sqrt(0.5 * (a2 + b2 + torch.sqrt(r.clamp_min(0.0))))


def _mhd_speed_max(U):
    m = []
    for z in range(0, U.shape[1], 32):
        q = _mhd_prim([u[z:z + 32].double() for u in U])
        m.append(sum(q[1 + d].abs() + _fast(q, d) for d in range(3)).max())
    return torch.stack(m).max().reshape(1)


def _hll(L, R, d, ch):
    B = 0.5 * (L[5 + d] + R[5 + d]) - (R[8] - L[8]) / (2.0 * ch)
    P = 0.5 * (L[8] + R[8]) - 0.5 * ch * (R[5 + d] - L[5 + d])
    L, R = list(L), list(R)
    L[5 + d], R[5 + d], L[8], R[8] = B, B, P, P
    cL, cR = _fast(L, d), _fast(R, d)
    SL, SR = torch.minimum(L[1 + d] - cL, R[1 + d] - cR), torch.maximum(L[1 + d] + cL, R[1 + d] + cR)
    F = []
    for fl, fr, ul, ur in zip(_mhd_flux(L, d, ch), _mhd_flux(R, d, ch), _mhd_cons(L), _mhd_cons(R)):
        mid = (SR * fl - SL * fr + SL * SR * (ur - ul)) / (SR - SL)
        F.append(torch.where(SL >= 0, fl, torch.where(SR <= 0, fr, mid)))
    F[5 + d], F[8] = P, ch * ch * B
    return F


def _mhd_step(U, dt, dx, limiter):
    ch = (CFL / 3.0) * dx / dt
    q = _mhd_prim(U)
    c = [_part(a, 0, 0, 1) for a in q]
    lo, hi, dF = [], [], [0] * 9
    for d in range(3):
        s = [_slope(k - _part(a, d, -1, 1), _part(a, d, 1, 1) - k, limiter) for a, k in zip(q, c)]
        lo.append([k - 0.5 * x for k, x in zip(c, s)])
        hi.append([k + 0.5 * x for k, x in zip(c, s)])
        dF = [t + (h - l) for t, h, l in zip(dF, _mhd_flux(hi[d], d, ch), _mhd_flux(lo[d], d, ch))]

    def half_step(w):
        return _mhd_prim([u - (0.5 * dt / dx) * f for u, f in zip(_mhd_cons(w), dF)])

    div = [0] * 9
    for d in range(3):
        F = _hll([_face_part(x, d, 0) for x in half_step(hi[d])], [_face_part(x, d, 1) for x in half_step(lo[d])], d, ch)
        n = F[0].shape[-1 - d] - 1
        div = [x + (f.narrow(-1 - d, 1, n) - f.narrow(-1 - d, 0, n)) for x, f in zip(div, F)]
    out = [_part(u, 0, 0, 2) - (dt / dx) * y for u, y in zip(U, div)]
    out[8] = out[8] * torch.exp(-ALPHA * ch * dt / dx)
    return out


def _periodic(U, g, step, nz=16):
    """step applied to z slabs of the periodic box U (fields, z, y, x), ghosted by g cells."""
    Z = U.shape[1]
    nz = max(1, min(Z, nz * 262144 // (U.shape[2] * U.shape[3])))
    out = torch.empty(U.shape, dtype=F64, device=U.device)
    for z in range(0, Z, nz):
        n = min(nz, Z - z)
        W = U[:, torch.arange(z - g, z + n + g, device=U.device) % Z].double()
        for d in (-1, -2):
            m = W.shape[d]
            W = torch.cat([W.narrow(d, m - g, g), W, W.narrow(d, 0, g)], dim=d)
        out[:, z:z + n] = torch.stack(step(list(W)))
    return out


def _box_step(U, dt, dx, limiter):
    return _periodic(U, 3 if limiter == "ppm" else 2, lambda W: _euler_step(W, dt, dx, limiter))


def _adjoint_inputs(case, seed):
    U = _white_gas(_shape(case), seed, 0.3, jitter=0.3)
    lam = _randn(U.shape, _gen(seed + 1))
    return U.to(_dtype(case)).contiguous(), lam.to(_dtype(case)).contiguous(), 1.0 / case["nx"]


def exact(case, seed):
    path, lim = case["path"], case["limiter"]
    if path == "step":
        U, dx = _box_gas(case, seed)
        out = _box_step(U, _cfl_dt(U, dx), dx, lim)
        return dict(U=list(out), dt=_cfl_dt(out, dx))
    if path == "run":
        U, dx = _box_gas(case, seed)
        U = U.double()
        hist = [_cfl_dt(U, dx)]
        for _ in range(case["steps"]):
            U = _box_step(U, hist[-1], dx, lim)
            hist.append(_cfl_dt(U, dx))
        return dict(U=list(U), dt=torch.cat(hist))
    if path == "patches":
        return _exact_patches(case, seed)
    if path == "octs":
        G, dx = _oct_gas(case, seed)
        dt = _oct_dt(G, dx)
        out = [torch.stack(_euler_step([g.double() for g in G[:, i:i + 32768]], dt, dx, lim))
               for i in range(0, G.shape[1], 32768)]
        return dict(U=list(torch.cat(out, dim=1)))
    if path == "octlevel":
        U, pos, dx = _octlevel_gas(case, seed)
        return dict(U=list(_to_octs(_box_step(U, _cfl_dt(U, dx), dx, lim))), order=None, nbr=None)
    if path == "adjoint":
        U, lam, dx = _adjoint_inputs(case, seed)
        dt = _cfl_dt(U, dx)
        V = U.double().requires_grad_(True)
        out = torch.stack(_euler_step(list(_wrap_pad(V, 2)), dt, dx, lim))
        return dict(lam=list(torch.autograd.grad(out, V, lam.double())[0]))
    if path == "mhd":
        U = _magnetised_gas(_shape(case), seed).to(_dtype(case))
        dx = 1.0 / case["nx"]
        dt = CFL * dx / _mhd_speed_max(U)
        out = _periodic(U, 2, lambda W: _mhd_step(W, dt, dx, lim), 8)
        return dict(U=list(out), dt=CFL * dx / _mhd_speed_max(out))
    return _exact_amr(case, seed)


def _exact_patches(case, seed):
    rows, U, window = _patch_gas(case, seed)
    speed = _speed(U)
    at = _offsets(rows, 0)
    flat = torch.zeros((5, int(at[-1])), dtype=F64, device=DEV)
    dt_next = torch.empty(len(rows), dtype=F64, device=DEV)
    groups = {}
    for p, r in enumerate(rows):
        groups.setdefault(r[:3], []).append(p)
    for n, members in groups.items():
        per = max(1, 4000000 // ((n[0] + 4) * (n[1] + 4) * (n[2] + 4)))
        for i in range(0, len(members), per):
            ps = members[i:i + per]
            W = torch.stack([window(U, rows[p]) for p in ps], dim=1).double()
            dx = torch.tensor([rows[p][4] for p in ps], dtype=F64, device=DEV)
            smax = torch.stack([window(speed, rows[p], 0) for p in ps]).amax(dim=(1, 2, 3))
            b = (-1, 1, 1, 1)
            V = torch.stack(_euler_step(list(W), (CFL * dx / smax).view(b), dx.view(b), case["limiter"]))
            dt_next[torch.tensor(ps, device=DEV)] = CFL * dx / _speed(V).amax(dim=(1, 2, 3))
            for k, p in enumerate(ps):
                _patch_view(flat, at[p], rows[p], 0).copy_(V[:, k])
    return dict(U=list(flat), dt=dt_next)


def _prolonged(C):
    """The fine level prolonged from the periodic coarse level with MinMod slopes."""
    out = C
    for d in (-1, -2, -3):
        s = 0.25 * _slope(C - torch.roll(C, 1, d), torch.roll(C, -1, d) - C, "minmod")
        for k in (-1, -2, -3):  # the slope in the axes refined so far, then both halves of axis d
            if k > d:
                s = s.repeat_interleave(2, k)
        out = torch.stack([out - s, out + s], dim=out.dim() + d + 1).flatten(out.dim() + d, out.dim() + d + 1)
    return out


def _level_fluxes(U, dt, dx, limiter):
    """The periodic step of a level and its face fluxes (x, y, z low faces with the last high one)."""
    F = []
    out = torch.stack(_euler_step(list(_wrap_pad(U, 2)), dt, dx, limiter, F))
    return out, F


def _registers(F, origins, dims, dt):
    """dt * F through the six boundary faces of each box."""
    rows = []
    for o, n in zip(origins, dims):
        parts = []
        for d in range(3):
            for side in (0, 1):
                f = F[d].select(-1 - d, o[d] + side * n[d])  # five (slow, fast) planes
                a, b = [k for k in (2, 1, 0) if k != d]
                parts.append(f[:, o[a]:o[a] + n[a], o[b]:o[b] + n[b]].reshape(5, -1))
        rows.append(torch.cat(parts, dim=1).reshape(-1))
    return dt * torch.stack(rows)


def _exact_amr(case, seed):
    coarse, fine, origins, dx = _amr_gas(case, seed)
    lim, e = case["limiter"], case["edge"]
    dtc, dtf = _amr_dt(coarse, fine, dx)
    coarse, fine = coarse.double(), fine.double()
    covered = torch.zeros(fine.shape[1:], dtype=torch.bool, device=DEV)
    for x, y, z in origins:
        covered[z:z + e, y:y + e, x:x + e] = True
    new, FC = _level_fluxes(coarse, dtc, dx, lim)
    FF = None
    for theta in (0.0, 0.5):
        level = torch.where(covered, fine, _prolonged((1.0 - theta) * coarse + theta * new))
        fine, F = _level_fluxes(level, dtf, 0.5 * dx, lim)
        FF = F if FF is None else [a + b for a, b in zip(FF, F)]
    half = [tuple(v // 2 for v in o) for o in origins]
    creg = _registers(FC, half, [(e // 2,) * 3] * len(half), dtc)
    freg = _registers(FF, origins, [(e,) * 3] * len(half), dtf)
    under = covered[::2, ::2, ::2]
    for d in range(3):  # coarse cells beside a covered one: the fine fluxes in place of the coarse
        ax = -1 - d
        n = coarse.shape[ax]
        f = FF[d].index_select(ax, torch.arange(0, 2 * n + 1, 2, device=DEV))
        for k in range(3):
            if k != d:
                m = f.shape[-1 - k]
                f = 0.5 * (f.index_select(-1 - k, torch.arange(0, m, 2, device=DEV)) +
                           f.index_select(-1 - k, torch.arange(1, m, 2, device=DEV)))
        diff = dtc * FC[d] - dtf * f
        up = torch.roll(under, -1, ax)    # the next cell is covered: its low face is our high face
        down = torch.roll(under, 1, ax)
        new = new + torch.where(up, diff.narrow(ax, 1, n), 0.0) / dx - torch.where(down, diff.narrow(ax, 0, n), 0.0) / dx
    Z, Y, X = _shape(case)
    mean = fine.reshape(5, Z, 2, Y, 2, X, 2).mean(dim=(2, 4, 6))
    new = torch.where(under, mean, new)
    # the last substep writes interiors only; its buffer's ghost cells keep their initial zeros
    C = torch.zeros((5, len(origins), e + 4, e + 4, e + 4), dtype=F64, device=DEV)
    for p, (x, y, z) in enumerate(origins):
        C[:, p, 2:-2, 2:-2, 2:-2] = fine[:, z:z + e, y:y + e, x:x + e]
    return dict(coarse=list(new), fine=list(C), coarse_fluxes=creg, fine_fluxes=freg)
