"""Performance cases: what a user of the solver has it do, at the sizes and options of real use.

Each case hands the library initial states, advances them by SSP-RK3 steps through the public
entry points and takes the whole result back: single grids of the paper's test cases (small,
where launches and latency count), a batch of many uneven grids, a large curvilinear grid, 3D
volumes with passive scalars, in FP32 and FP64. States that live on the GPU go through
`set_state_device` / `get_state_device`, host-resident ones through `roeam_step_host_f32`, and
3D ones through page-locked host arrays. FP32 results are returned as float32.

`exact` restates the scheme (Section 6.2 of the paper, finite volumes, SSP-RK3, the time-step
rule of include/roeam.h) in plain 64-bit torch on ghost-padded cells, without the library.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1711_09272_gb300 import (Batch, Batch3, roeam3_get_state, roeam3_set_state, roeam_step_host_f32)

PERIODIC, WALL, INFLOW, OUTFLOW = 0, 1, 2, 3
GAMMA = 1.4
CFL = 0.5
F64 = torch.float64
DEV = "cuda"


# ----------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call: one small FP32 grid loaded, advanced by one step and read back, as a
        # coupled solver does every time step; launches and latency are all of it
        {"name": "one_step_96x65_fp32", "flow": "smooth", "ni": 96, "nj": 65, "prec": 32, "recon": 0, "steps": 1},
        # the accuracy study: isentropic vortex, FP64, first order
        {"name": "vortex_64_fp64", "flow": "vortex", "ni": 64, "nj": 64, "prec": 64, "recon": 0, "steps": 20},
        # low-Mach convergence run in FP64 with its monitors (residual norm, conserved totals)
        {"name": "gresho_256_fp64", "flow": "gresho", "ni": 256, "nj": 256, "prec": 64, "recon": 1, "steps": 10},
        # the same flow in production precision
        {"name": "gresho_256_fp32", "flow": "gresho", "ni": 256, "nj": 256, "prec": 32, "recon": 1, "steps": 50},
        # odd-even decoupling duct: a thin curvilinear grid with walls, inflow and outflow
        {"name": "quirk_800x20_fp32", "flow": "quirk", "ni": 800, "nj": 20, "prec": 32, "recon": 0, "steps": 64,
         "eps1": 0},
        # shock diffraction over a solid corner, Cartesian with walls
        {"name": "corner_400_fp32", "flow": "corner", "ni": 400, "nj": 400, "prec": 32, "recon": 0, "steps": 40},
        # parameter study: 512 uneven periodic grids advanced together (the benchmark workload)
        {"name": "batch_512_fp32", "flow": "batch", "count": 512, "prec": 32, "recon": 0, "steps": 8},
        # the same batch kept in host memory, one step per call
        {"name": "batch_512_host_fp32", "flow": "batch", "count": 512, "prec": 32, "recon": 0, "steps": 1, "host": 1},
        # a smaller second-order study
        {"name": "batch_96_vanleer_fp32", "flow": "batch", "count": 96, "prec": 32, "recon": 2, "steps": 8},
        # the largest 2D grid: Mach-3 flow over a step, warped grid, solid block, van Leer
        {"name": "warped_4096_fp32", "flow": "warped", "ni": 4096, "nj": 4096, "prec": 32, "recon": 2, "steps": 4},
        # 3D Taylor-Green vortex with one passive scalar, production precision
        {"name": "tgv_256_fp32", "flow": "tgv", "ni": 256, "nj": 256, "nk": 256, "nscal": 1, "prec": 32, "steps": 20},
        # the 3D accuracy study
        {"name": "tgv_64_fp64", "flow": "tgv", "ni": 64, "nj": 64, "nk": 64, "nscal": 2, "prec": 64, "steps": 4},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    flow = rng.choice(["smooth", "vortex", "gresho", "quirk", "corner", "batch", "warped", "tgv"])
    if flow == "smooth":
        return {"flow": flow, "ni": size(16, 640), "nj": size(16, 640), "prec": 32, "recon": rng.randrange(3), "steps": 1}
    if flow == "vortex":
        return {"flow": flow, "ni": size(32, 256), "nj": size(32, 256), "prec": 64, "recon": rng.randrange(3),
                "steps": rng.randrange(4, 21)}
    if flow == "gresho":
        prec = rng.choice([32, 64])
        n = size(64, 640 if prec == 32 else 300)
        return {"flow": flow, "ni": n, "nj": n + rng.randrange(-9, 10), "prec": prec, "recon": rng.randrange(3),
                "steps": rng.randrange(20, 60) if prec == 32 else rng.randrange(4, 13)}
    if flow == "quirk":
        return {"flow": flow, "ni": size(200, 1600), "nj": size(10, 80), "prec": 32, "recon": 0,
                "steps": rng.randrange(20, 65), "eps1": rng.randrange(2)}
    if flow == "corner":
        return {"flow": flow, "ni": size(100, 900), "nj": size(100, 900), "prec": 32, "recon": 0,
                "steps": rng.randrange(10, 41)}
    if flow == "batch":
        c = {"flow": flow, "count": size(16, 512), "prec": 32, "recon": rng.choice([0, 0, 2]), "steps": rng.randrange(2, 9)}
        return dict(c, steps=1, host=1) if rng.random() < 0.25 else c
    if flow == "warped":
        return {"flow": flow, "ni": size(256, 4096), "nj": size(256, 4096), "prec": 32, "recon": 2,
                "steps": rng.randrange(1, 5)}
    prec = rng.choice([32, 64])
    hi = 224 if prec == 32 else 80
    return {"flow": flow, "ni": size(32, hi), "nj": size(32, hi), "nk": size(32, hi), "nscal": rng.randrange(4),
            "prec": prec, "steps": rng.randrange(8, 21) if prec == 32 else rng.randrange(1, 5)}


# ----------------------------------------------------------------------------- inputs
def params(**kw):
    p = dict(gamma=GAMMA, m_ref=0.5, u_ref=1.0, eps2=0.05, eps1=0, use_s1=1, recon=0, xi_form=0)
    p.update(kw)
    return SimpleNamespace(**p)


def grid(ni, nj, dx=1.0, dy=1.0, bc=(PERIODIC,) * 4, inflow=(1.0, 0.0, 0.0, 1.0), xv=None, yv=None, solid=None, **p):
    return SimpleNamespace(ni=ni, nj=nj, dx=dx, dy=dy, bc=bc, inflow=inflow, xv=xv, yv=yv, solid=solid,
                           params=params(**p))


def centres(s):
    """Cell centres (x, y), each [nj, ni], on the GPU."""
    if s.xv is None:
        x = (torch.arange(s.ni, device=DEV, dtype=F64) + 0.5) * s.dx
        y = (torch.arange(s.nj, device=DEV, dtype=F64) + 0.5) * s.dy
        return x[None, :].expand(s.nj, s.ni), y[:, None].expand(s.nj, s.ni)
    return tuple(0.25 * (v[:-1, :-1] + v[:-1, 1:] + v[1:, :-1] + v[1:, 1:])
                 for v in (torch.from_numpy(s.xv).to(DEV), torch.from_numpy(s.yv).to(DEV)))


def conserved(r, u, v, p):
    return torch.stack([r, r * u, r * v, p / (GAMMA - 1.0) + 0.5 * r * (u * u + v * v)])


def modes(x, y, rng, n=4):
    """A smooth field of unit size, periodic over the unit square in (x, y)."""
    f = torch.zeros_like(x)
    for _ in range(n):
        kx, ky, ph = rng.integers(1, 5), rng.integers(1, 5), rng.uniform(0, 2 * math.pi)
        f = f + rng.uniform(0.2, 0.5) * torch.sin(2 * math.pi * (kx * x + ky * y) + ph)
    return f


def batch_sizes(count):
    """(ni, nj) of each grid of a batch: 32..512 by 32..256, by the case alone."""
    rng = np.random.default_rng([count, 20171127])
    return [(int(rng.integers(32, 513)), int(rng.integers(32, 257))) for _ in range(count)]


def flow_2d(c, seed):
    """The grids of a 2D case and their states [4, nj, ni] (float64, on the GPU)."""
    rng = np.random.default_rng([seed, 20171127])
    flow, recon = c["flow"], c["recon"]
    if flow == "batch":
        grids, states = [], []
        for ni, nj in batch_sizes(c["count"]):
            mach, ang = 10.0 ** rng.uniform(-3.0, math.log10(20.0)), rng.uniform(0, 2 * math.pi)
            s = grid(ni, nj, 1.0 / ni, 1.0 / ni, m_ref=max(mach, 1e-3), u_ref=mach, recon=recon)
            x, y = centres(s)
            Ly = nj / ni
            bump = []
            for _ in range(2):
                cx, cy = rng.uniform(0, 1), rng.uniform(0, Ly)
                bx, by = torch.remainder(x - cx + 0.5, 1.0) - 0.5, torch.remainder(y - cy + 0.5 * Ly, Ly) - 0.5 * Ly
                bump.append(1.0 + 0.1 * torch.exp(-50.0 * (bx * bx + by * by)))
            one = torch.ones_like(bump[0])
            grids.append(s)
            states.append(conserved(bump[0], mach * math.cos(ang) * one, mach * math.sin(ang) * one, bump[1] / GAMMA))
        return grids, states
    ni, nj = c["ni"], c["nj"]
    if flow == "smooth":   # a periodic subsonic flow
        s = grid(ni, nj, 1.0 / ni, 1.0 / nj, m_ref=0.4, u_ref=0.5, recon=recon)
        x, y = centres(s)
        f = [modes(x, y, rng) for _ in range(4)]
        return [s], [conserved(1 + 0.1 * f[0], 0.4 + 0.2 * f[1], -0.2 + 0.2 * f[2], 1 + 0.1 * f[3])]
    if flow == "vortex":   # isentropic vortex on [0, 10]^2
        s = grid(ni, nj, 10.0 / ni, 10.0 / nj, m_ref=0.5, u_ref=0.5 * math.sqrt(GAMMA), recon=recon)
        x, y = centres(s)
        cx, cy, ang = rng.uniform(0, 10), rng.uniform(0, 10), rng.uniform(0, 2 * math.pi)
        dx, dy = torch.remainder(x - cx + 5.0, 10.0) - 5.0, torch.remainder(y - cy + 5.0, 10.0) - 5.0
        r2 = dx * dx + dy * dy
        amp = 5.0 / (2 * math.pi) * torch.exp(0.5 * (1 - r2))
        T = 1 - (GAMMA - 1) * 25.0 / (8 * GAMMA * math.pi ** 2) * torch.exp(1 - r2)
        r = T ** (1 / (GAMMA - 1))
        u0 = 0.5 * math.sqrt(GAMMA)
        return [s], [conserved(r, u0 * math.cos(ang) - amp * dy, u0 * math.sin(ang) + amp * dx, r ** GAMMA)]
    if flow == "gresho":   # Gresho vortex at M = 0.01 with a checkerboard of noise on p
        s = grid(ni, nj, 1.0 / ni, 1.0 / nj, m_ref=0.01, u_ref=1.0, recon=recon)
        x, y = centres(s)
        dx, dy = x - 0.5, y - 0.5
        q = torch.sqrt(dx * dx + dy * dy).clamp_min(1e-300)
        p0 = 1.0 / (GAMMA * 1e-4)
        w = torch.where(q < 0.2, 5 * q, torch.where(q < 0.4, 2 - 5 * q, 0 * q))
        mid = 4 - 4 * math.log(0.2) + 12.5 * q * q - 20 * q + 4 * torch.log(q)
        p = p0 + torch.where(q < 0.2, 12.5 * q * q, torch.where(q < 0.4, mid, torch.full_like(q, 4 * math.log(2.0) - 2)))
        noise = torch.from_numpy(rng.uniform(0.5, 1.5, (nj, ni))).to(DEV)
        sign = 1 - 2 * ((torch.arange(ni, device=DEV)[None, :] + torch.arange(nj, device=DEV)[:, None]) % 2)
        return [s], [conserved(torch.ones_like(q), -w * dy / q, w * dx / q, p + 1e-3 * sign * noise)]
    if flow == "quirk":    # Mach-6 shock in a duct whose centreline is perturbed
        xv, yv = np.meshgrid(np.arange(ni + 1.0), np.arange(nj + 1.0))
        yv[nj // 2] += 1e-3 * rng.uniform(0.5, 1.0, ni + 1) * np.where(np.arange(ni + 1) % 2 == 0, 1, -1)
        post = (1512 / 205, 175 / 36, 0.0, 251 / 6)
        s = grid(ni, nj, bc=(INFLOW, OUTFLOW, WALL, WALL), inflow=post, xv=xv, yv=yv, m_ref=6.0, u_ref=post[1],
                 eps1=c["eps1"], recon=recon)
        x, _ = centres(s)
        left = x < rng.uniform(10, 0.2 * ni)
        z = torch.zeros_like(x)
        return [s], [conserved(torch.where(left, post[0], z + 1.4), torch.where(left, post[1], z), z,
                               torch.where(left, post[3], z + 1.0))]
    if flow == "corner":   # Mach-5.09 shock diffracting over a solid block
        xs, yc = rng.uniform(0.05, 0.08), rng.uniform(0.4, 0.6)
        post = (7.04108, 4.07794, 0.0, 30.05942)
        s = grid(ni, nj, 1.0 / ni, 1.0 / nj, bc=(INFLOW, OUTFLOW, OUTFLOW, WALL), inflow=post, m_ref=1.0,
                 u_ref=post[1], recon=recon)
        x, y = centres(s)
        s.solid = ((x < xs) & (y < yc)).to(torch.uint8).cpu().numpy()
        z = torch.zeros_like(x)
        return [s], [conserved(torch.where(x < xs, post[0], z + 1.4), torch.where(x < xs, post[1], z), z,
                               torch.where(x < xs, post[3], z + 1.0))]
    # warped: Mach-3 flow over a forward-facing step on a warped grid, some way into the run (smooth
    # disturbances and a pressure and density jump in the stream)
    dx, dy = 3.0 / ni, 1.0 / nj
    X = torch.arange(ni + 1, device=DEV, dtype=F64)[None, :] * dx
    Y = torch.arange(nj + 1, device=DEV, dtype=F64)[:, None] * dy
    w = torch.sin(16 * math.pi * X / 3) * torch.sin(16 * math.pi * Y)
    solid = np.zeros((nj, ni), np.uint8)
    solid[:max(1, round(0.2 * nj)), round(0.2 * ni):] = 1
    s = grid(ni, nj, dx, dy, bc=(INFLOW, OUTFLOW, WALL, WALL), inflow=(1.4, 3.0, 0.0, 1.0),
             xv=(X + 0.1 * dx * w).cpu().numpy(), yv=(Y + 0.1 * dy * w).cpu().numpy(), solid=solid, m_ref=3.0, u_ref=3.0,
             recon=recon)
    x, y = centres(s)
    f = [modes(x / 3, y, rng) for _ in range(4)]
    jump = ((x - rng.uniform(0.8, 2.2)) ** 2 + (y - rng.uniform(0.4, 0.8)) ** 2 < 0.04).to(F64)
    return [s], [conserved(1.4 * (1 + 0.05 * f[0] + 0.6 * jump), 3 + 0.1 * f[1], 0.1 * f[2], 1 + 0.05 * f[3] + jump)]


def flow_3d(c, seed):
    """Taylor-Green vortex (M = 0.1) of a random phase, with smooth scalars: grid and state."""
    rng = np.random.default_rng([seed, 20171127])
    n = (c["ni"], c["nj"], c["nk"])
    d = [2 * math.pi / k for k in n]
    s = SimpleNamespace(ni=n[0], nj=n[1], nk=n[2], dx=d[0], dy=d[1], dz=d[2], bc=(PERIODIC,) * 6,
                        inflow=(1.0, 0.0, 0.0, 0.0, 1.0), nscal=c["nscal"], params=params(m_ref=0.1))
    x, y, z = (((torch.arange(n[a], device=DEV, dtype=F64) + 0.5) * d[a] + rng.uniform(0, 2 * math.pi))
               .reshape([-1 if 2 - b == a else 1 for b in range(3)]) for a in range(3))
    u, v = torch.sin(x) * torch.cos(y) * torch.cos(z), -torch.cos(x) * torch.sin(y) * torch.cos(z)
    w = 0.1 * torch.sin(x + y) * torch.sin(z)
    p = 1.0 / (GAMMA * 0.01) + (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2) / 16
    r = 1 + 0.05 * torch.sin(x + y + z)
    rows = [r, r * u, r * v, r * w, p / (GAMMA - 1) + 0.5 * r * (u * u + v * v + w * w)]
    rows += [r * 0.5 * (1 + torch.sin(x + k) * torch.sin(y) * torch.sin(z)) for k in range(c["nscal"])]
    return s, torch.stack(rows)


def prepare(case, seed):
    """The handle and the buffers that a program keeps, and the initial state."""
    st = SimpleNamespace(case=case)
    if case["flow"] == "tgv":
        s, U = flow_3d(case, seed)
        st.U = torch.empty(U.shape, dtype=F64, pin_memory=True).copy_(U)
        st.out = torch.empty(U.shape, dtype=F64, pin_memory=True)
        st.batch = Batch3([s], precision=case["prec"])
        return st
    grids, states = flow_2d(case, seed)
    st.batch = Batch(grids, precision=case["prec"])
    U = torch.cat([u.reshape(-1) for u in states])
    if case.get("host"):
        st.U = torch.empty(U.shape, dtype=torch.float32, pin_memory=True).copy_(U)
        st.out = torch.empty(U.shape, dtype=torch.float32, pin_memory=True)
    else:
        st.U, st.out = U, torch.empty_like(U)
    return st


def run(st):
    """Loads the state, advances it and takes the result back."""
    c, b = st.case, st.batch
    if c["flow"] == "tgv":
        roeam3_set_state(b.handle, 0, st.U)
        b.step(CFL, nsteps=c["steps"])
        roeam3_get_state(b.handle, 0, st.out)
        return st.out if c["prec"] == 64 else st.out.to(DEV, non_blocking=True).float()
    if c.get("host"):
        roeam_step_host_f32(b.handle, CFL, 0.0, c["steps"], st.U, st.out)
        return st.out
    stream = torch.cuda.current_stream().cuda_stream
    b.set_state_device(st.U, -1, stream)
    b.step(CFL, nsteps=c["steps"])
    b.get_state_device(st.out, -1, stream)
    if c["prec"] == 32:
        return st.out.float()
    if c["flow"] == "gresho":   # the run's monitors
        return {"state": st.out, "norm": b.residual_norm(0), "totals": b.totals(0)}
    return st.out


def cells_of(c):
    if c["flow"] == "tgv":
        return c["ni"] * c["nj"] * c["nk"]
    return c["ni"] * c["nj"] if "ni" in c else sum(a * b for a, b in batch_sizes(c["count"]))


def work(case):
    """Bytes: the initial state in and the result out, once each, in the types run() passes. Flops of
    the scheme per cell and stage, counted from its formulas: about 160 per face (Roe averages,
    Mach functions, dissipation, assembly; 9 more per scalar), 75 per cell (primitives, detector
    ratios, stage update), 56 per face for a limited reconstruction, 30 per curvilinear face."""
    c, n = case, cells_of(case)
    if c["flow"] == "tgv":
        nv = 5 + c["nscal"]
        face, faces, cell = 175 + 9 * c["nscal"], 3, 100
        size_in, size_out = 8, 8
    else:
        nv, faces, cell = 4, 2, 75
        face = 160 + (56 if c["recon"] else 0) + (30 if c["flow"] in ("quirk", "warped") else 0)
        size_in = 4 if c.get("host") else 8
        size_out = 4 if c["prec"] == 32 else 8
    return {"bytes": float(n * nv * (size_in + size_out)), "flops": float(n * c["steps"] * 3 * (faces * face + cell))}


# ----------------------------------------------------------------------------- 64-bit values
def f_mach(m):
    """Eq. 98."""
    return torch.clamp(m * torch.sqrt(4 + (1 - m * m) ** 2) / (1 + m * m), max=1.0).where(m < 1, torch.ones_like(m))


def side(r, un, ut, p, k=()):
    """One side of a face: ut and k are lists of further velocity components and of scalars."""
    q2 = un * un + sum(t * t for t in ut)
    c2 = GAMMA * p / r
    return SimpleNamespace(r=r, un=un, ut=ut, p=p, k=k, c2=c2, H=c2 / (GAMMA - 1) + 0.5 * q2, m=torch.sqrt(q2 / c2))


def roe_am(L, R, s1, par):
    """Eqs. 85-101 (102-109 with eps1, in 2D): the flux per unit face, [mass, normal momentum,
    tangential momenta, energy, scalars]."""
    a, b = torch.sqrt(L.r), torch.sqrt(R.r)

    def mean(x, y):
        return (a * x + b * y) / (a + b)

    rho, U, H = a * b, mean(L.un, R.un), mean(L.H, R.H)
    ts, ks = [mean(x, y) for x, y in zip(L.ut, R.ut)], [mean(x, y) for x, y in zip(L.k, R.k)]
    du, dt = R.un - L.un, [y - x for x, y in zip(L.ut, R.ut)]
    dq2 = du * du + sum(t * t for t in dt)
    c2 = mean(L.c2, R.c2) + 0.5 * (GAMMA - 1) * rho / (a + b) ** 2 * dq2
    c, dp = torch.sqrt(c2), R.p - L.p
    M, Mb = 0.5 * (L.m + R.m), U.abs() / c
    f, fb = f_mach(M), f_mach(Mb)
    sub = torch.sign(U + c) - torch.sign(U - c)
    Up = torch.clamp(U.abs() - fb * sub / 4 * torch.clamp(du, min=0), min=0)
    xi = torch.clamp((0.5 * (L.un + R.un)).abs() + (1 - fb ** 8) * du / 2, min=0)
    if par.eps1:
        dq = torch.sqrt(dq2)
        big = dq >= 1e-5 * par.u_ref
        nx = torch.where(big, du / dq.clamp_min(1e-300), torch.ones_like(dq))
        ny = torch.where(big, dt[0] / dq.clamp_min(1e-300), torch.zeros_like(dq))
        frr = (nx * (nx * U + ny * ts[0])).abs() + (ny * (nx * ts[0] - ny * U)).abs()
        xi = torch.maximum(xi, (1 - fb ** 8) * f ** 8 * torch.minimum(par.eps2 * c, frr))
    sm = torch.sign(U) * torch.minimum(Up, c)
    dpp = sm / c * dp + (1 - s1 + s1 * f) * torch.clamp(c - Up, min=0) * rho * du
    th = torch.clamp(torch.maximum(M * M, par.m_ref ** 2), max=1.0)
    ct = 0.5 * torch.sqrt(4 * c2 * th + (1 - th) ** 2 * U * U)
    Ut = 0.5 * (1 + th) * U
    term = torch.clamp(ct - Up, min=0) + (1 - th) * (Up - U * torch.sign(Ut) * torch.minimum(Ut.abs(), ct) / (2 * ct))
    rdUp = s1 * (1 - f ** 8) * term * dp / (th * c2)   # rho delta U_p
    dUu = 0.5 * sm / c * du                            # delta U_u
    gL, gR = L.r * (L.un + xi - dUu), R.r * (R.un - xi - dUu)
    out = [gL + gR - rdUp, gL * L.un + gR * R.un - rdUp * U + L.p + R.p - dpp]
    out += [gL * x + gR * y - rdUp * t for x, y, t in zip(L.ut, R.ut, ts)]
    out += [gL * L.H + gR * R.H - rdUp * H]
    out += [gL * x + gR * y - rdUp * k for x, y, k in zip(L.k, R.k, ks)]
    return [0.5 * x for x in out]


def ratio(r0, p0, r1, p1):
    """Eq. 97."""
    return torch.minimum(torch.minimum(p0, p1) / torch.maximum(p0, p1), torch.minimum(r0, r1) / torch.maximum(r0, r1))


def speed(un, q2, c2, mr):
    """|U| + max(c, c~ / theta)."""
    th = torch.clamp(torch.maximum(q2 / c2, mr * mr), max=1.0)
    ct = 0.5 * torch.sqrt(4 * c2 * th + (1 - th) ** 2 * un * un)
    return un.abs() + torch.where(th < 1, torch.maximum(torch.sqrt(c2), ct / th), torch.sqrt(c2))


class Padded:
    """All grids of a 2D case as one flat list of cells, each grid padded by two ghost layers."""

    def __init__(self, grids):
        G = len(grids)
        long = dict(device=DEV, dtype=torch.int64)
        parts = {k: [] for k in ("src", "gid", "wall_x", "wall_y", "inflow", "solid", "inner", "pitch")}
        base = cbase = 0
        for g, s in enumerate(grids):
            W, Hh = s.ni + 4, s.nj + 4
            i, kx = self.resolve(torch.arange(-2, s.ni + 2, **long), s.ni, s.bc[0], s.bc[1])
            j, ky = self.resolve(torch.arange(-2, s.nj + 2, **long), s.nj, s.bc[2], s.bc[3])
            full = (Hh, W)
            parts["src"].append((cbase + j[:, None] * s.ni + i[None, :]).reshape(-1))
            parts["gid"].append(torch.full((W * Hh,), g, **long))
            parts["pitch"].append(torch.full((W * Hh,), W, **long))
            fl = (kx == 2)[None, :] | (ky == 2)[:, None]
            parts["inflow"].append(fl.expand(full).reshape(-1))
            parts["wall_x"].append(((kx == 1)[None, :] & ~(kx == 2)[None, :]).expand(full).reshape(-1))
            parts["wall_y"].append(((ky == 1)[:, None] & ~(kx == 2)[None, :]).expand(full).reshape(-1))
            sol = torch.zeros((s.nj, s.ni), device=DEV, dtype=torch.bool) if s.solid is None else \
                torch.from_numpy(s.solid).to(DEV).bool()
            parts["solid"].append(sol[j][:, i].reshape(-1) & ~fl.expand(full).reshape(-1))
            at = base + torch.arange(W * Hh, **long).reshape(full)
            parts["inner"].append(at[2:-2, 2:-2].reshape(-1))
            base, cbase = base + W * Hh, cbase + s.ni * s.nj
        for k in ("src", "gid", "wall_x", "wall_y", "inflow", "solid", "inner"):
            setattr(self, k, torch.cat(parts[k]))
        pitch = torch.cat(parts["pitch"])
        at = torch.arange(base, **long)
        self.w, self.e = (at - 1).clamp_min(0), (at + 1).clamp_max(base - 1)
        self.s, self.n = (at - pitch).clamp_min(0), (at + pitch).clamp_max(base - 1)
        self.wall = self.wall_x | self.wall_y
        self.grids, self.G = grids, G
        gid = self.gid

        def per(f, at=gid):
            v = torch.tensor([float(f(s)) for s in grids], device=DEV, dtype=F64)
            return v[0] if G == 1 else v[at]

        p0 = grids[0].params
        self.par = SimpleNamespace(m_ref=per(lambda s: s.params.m_ref), u_ref=per(lambda s: s.params.u_ref),
                                   eps1=p0.eps1, eps2=p0.eps2)
        self.recon, self.curv = p0.recon, grids[0].xv is not None
        inner_gid = gid[self.inner]
        self.mr_inner = per(lambda s: s.params.m_ref, inner_gid)
        self.gid_inner = inner_gid
        one, zero = torch.ones((), device=DEV, dtype=F64), torch.zeros((), device=DEV, dtype=F64)
        if not self.curv:
            self.fx = (one, zero, per(lambda s: s.dy))    # unit normal and length of the west face
            self.fy = (zero, one, per(lambda s: s.dx))
            self.wn = (self.fx[:2], self.fy[:2])
            self.cx = (one, zero, per(lambda s: s.dy, inner_gid))
            self.cy = (zero, one, per(lambda s: s.dx, inner_gid))
            self.V = per(lambda s: s.dx * s.dy, inner_gid)
            return
        s = grids[0]                                      # (one curvilinear grid per case)
        xv, yv = torch.from_numpy(s.xv).to(DEV), torch.from_numpy(s.yv).to(DEV)
        I = torch.arange(-2, s.ni + 2, **long)
        J = torch.arange(-2, s.nj + 2, **long)

        def vec(sx, sy, i, j):
            l = torch.sqrt(sx * sx + sy * sy)
            i, j = i.clamp(0, l.shape[1] - 1), j.clamp(0, l.shape[0] - 1)
            return tuple(v[j][:, i].reshape(-1) for v in (sx / l, sy / l, l))

        self.fx = vec(yv[1:] - yv[:-1], xv[:-1] - xv[1:], I, J)
        self.fy = vec(yv[:, :-1] - yv[:, 1:], xv[:, 1:] - xv[:, :-1], I, J)
        # normals of the boundary faces that the W/E and S/N wall ghost cells are mirrored about
        gx, gy = torch.where(I < 0, 0, s.ni), torch.where(J < 0, 0, s.nj)
        self.wn = (vec(yv[1:] - yv[:-1], xv[:-1] - xv[1:], gx, J)[:2],
                   vec(yv[:, :-1] - yv[:, 1:], xv[:, 1:] - xv[:, :-1], I, gy)[:2])
        sx, sy = yv[1:] - yv[:-1], xv[:-1] - xv[1:]
        self.cx = self.unit(0.5 * (sx[:, 1:] + sx[:, :-1]), 0.5 * (sy[:, 1:] + sy[:, :-1]))
        sx, sy = yv[:, :-1] - yv[:, 1:], xv[:, 1:] - xv[:, :-1]
        self.cy = self.unit(0.5 * (sx[1:] + sx[:-1]), 0.5 * (sy[1:] + sy[:-1]))
        d1x, d1y = xv[1:, 1:] - xv[:-1, :-1], yv[1:, 1:] - yv[:-1, :-1]
        d2x, d2y = xv[1:, :-1] - xv[:-1, 1:], yv[1:, :-1] - yv[:-1, 1:]
        self.V = (0.5 * (d1x * d2y - d1y * d2x)).reshape(-1)

    @staticmethod
    def unit(sx, sy):
        l = torch.sqrt(sx * sx + sy * sy)
        return (sx / l).reshape(-1), (sy / l).reshape(-1), l.reshape(-1)

    @staticmethod
    def resolve(x, n, lo, hi):
        """Source index and kind (0 copy, 1 wall mirror, 2 inflow) of cell indices in -2 .. n + 1."""
        kind = torch.zeros_like(x)
        src = x.clone()
        for out, bc, edge in ((x < 0, lo, 0), (x >= n, hi, n - 1)):
            if bc == PERIODIC:
                v = x % n
            elif bc == OUTFLOW:
                v = torch.full_like(x, edge)
            elif bc == INFLOW:
                v = torch.zeros_like(x)
            else:
                v = torch.where(x < 0, -1 - x, 2 * n - 1 - x)
            src = torch.where(out, v, src)
            kind = torch.where(out, {WALL: 1, INFLOW: 2}.get(bc, 0), kind)
        return src.clamp(0, n - 1), kind

    @staticmethod
    def mirror(u, v, n):
        un = 2 * (u * n[0] + v * n[1])
        return u - un * n[0], v - un * n[1]

    def prims(self, U):
        r = U[0]
        u, v = U[1] / r, U[2] / r
        return r, u, v, (GAMMA - 1) * (U[3] - 0.5 * r * (u * u + v * v))

    def rate(self, U):
        """Largest rate per grid."""
        r, u, v, p = self.prims(U)
        c2, q2 = GAMMA * p / r, u * u + v * v
        lam = sum(speed(u * n[0] + v * n[1], q2, c2, self.mr_inner) * n[2] for n in (self.cx, self.cy)) / self.V
        solid = self.solid[self.inner]
        lam = torch.where(solid, torch.zeros_like(lam), lam)
        return torch.zeros(self.G, device=DEV, dtype=F64).scatter_reduce(0, self.gid_inner, lam, "amax")

    def limited(self, a, b):
        if self.recon == 1:
            m = torch.where(a.abs() < b.abs(), a, b)
        else:
            m = 2 * a * b.abs() / (a.abs() + b.abs()).clamp_min(1e-300)
        return torch.where(torch.sign(a) * torch.sign(b) > 0, m, torch.zeros_like(a))

    def face(self, q, back, ahead, n, s1):
        """Flux through the face between cell `back` of each cell and the cell itself, in global
        components times the face length."""
        A, B = [x[back] for x in q], q
        fA, fB = (self.solid | self.wall)[back], self.solid | self.wall
        sA = self.solid[back]
        L, R = list(A), list(B)
        if self.recon:
            M0, M3 = [x[back[back]] for x in q], [x[ahead] for x in q]
            if self.solid.any():
                m0, m3 = list(A), list(B)
                m0[1], m0[2] = self.mirror(A[1], A[2], (n[0][back], n[1][back]) if self.curv else n)
                m3[1], m3[2] = self.mirror(B[1], B[2], (n[0][ahead], n[1][ahead]) if self.curv else n)
                M0 = [torch.where(self.solid[back[back]], x, y) for x, y in zip(m0, M0)]
                M3 = [torch.where(self.solid[ahead], x, y) for x, y in zip(m3, M3)]
            L = [a + 0.5 * self.limited(a - m, b - a) for m, a, b in zip(M0, A, B)]
            R = [b - 0.5 * self.limited(b - a, m - b) for a, b, m in zip(A, B, M3)]
            ok = (L[0] > 0) & (L[3] > 0) & (R[0] > 0) & (R[3] > 0) & ~fA & ~fB
            L = [torch.where(ok, x, a) for x, a in zip(L, A)]
            R = [torch.where(ok, x, b) for x, b in zip(R, B)]
        if self.wall.any() or self.solid.any():
            mA, mB = list(B), list(A)
            mA[1], mA[2] = self.mirror(B[1], B[2], n)
            mB[1], mB[2] = self.mirror(A[1], A[2], n)
            L = [torch.where(fA, x, y) for x, y in zip(mA, L)]
            R = [torch.where(fB & ~fA, x, y) for x, y in zip(mB, R)]
        lr = [side(r, n[0] * u + n[1] * v, [n[0] * v - n[1] * u], p) for r, u, v, p in (L, R)]
        F = roe_am(*lr, s1, self.par)
        F = [F[0], n[0] * F[1] - n[1] * F[2], n[1] * F[1] + n[0] * F[2], F[3]]
        both = sA & self.solid
        return [torch.where(both, torch.zeros_like(x), x * n[2]) for x in F]

    def residual(self, U):
        """-(1 / V) sum of outward fluxes, of U [4, cells]."""
        r, u, v, p = (x[self.src] for x in self.prims(U))
        if self.inflow.any():
            g = self.grids[0].inflow
            r, u, v, p = (torch.where(self.inflow, w, x) for w, x in zip(g, (r, u, v, p)))
        if self.wall.any():
            mu, mv = self.mirror(u, v, self.wn[1])
            m = self.wall_y & ~self.inflow
            u, v = torch.where(m, mu, u), torch.where(m, mv, v)
            mu, mv = self.mirror(u, v, self.wn[0])
            u, v = torch.where(self.wall_x, mu, u), torch.where(self.wall_x, mv, v)
        q = (r, u, v, p)
        w, e, s, n = self.w, self.e, self.s, self.n
        Px, Py = ratio(r[w], p[w], r, p), ratio(r[s], p[s], r, p)
        if self.solid.any():
            Px = torch.where(self.solid | self.solid[w], torch.ones_like(Px), Px)
            Py = torch.where(self.solid | self.solid[s], torch.ones_like(Py), Py)
        Pyn, Pxe = Py[n], Px[e]
        ax = torch.stack([Px, Py[w], Pyn[w], Py, Pyn]).amin(0)
        ay = torch.stack([Py, Px[s], Pxe[s], Px, Pxe]).amin(0)
        Fx = self.face(q, w, e, self.fx, f_mach(ax) ** 8)
        Fy = self.face(q, s, n, self.fy, f_mach(ay) ** 8)
        k = self.inner
        R = torch.stack([(x[k] - x[e[k]] + y[k] - y[n[k]]) / self.V for x, y in zip(Fx, Fy)])
        return torch.where(self.solid[k], torch.zeros_like(R), R)

    def split(self, flat):
        """[cells of each grid as 4 planes, concatenated] -> [4, cells]."""
        out, at = [], 0
        for s in self.grids:
            m = 4 * s.ni * s.nj
            out.append(flat[at:at + m].reshape(4, -1))
            at += m
        return torch.cat(out, 1)

    def join(self, U):
        out, at = [], 0
        for s in self.grids:
            out.append(U[:, at:at + s.ni * s.nj].reshape(-1))
            at += s.ni * s.nj
        return torch.cat(out)


def ssp_rk3(U, dt, R):
    U1 = U + dt * R(U)
    U2 = 0.75 * U + 0.25 * (U1 + dt * R(U1))
    return U / 3 + 2.0 / 3 * (U2 + dt * R(U2))


def residual_3d(U, d, par):
    """Periodic 3D residual of U [5 + nscal, nk, nj, ni]."""
    r = U[0]
    vel = [U[1 + a] / r for a in range(3)]
    p = (GAMMA - 1) * (U[4] - 0.5 * r * sum(t * t for t in vel))
    ks = [x / r for x in U[5:]]
    dims = (2, 1, 0)   # array dimension of the axes x, y, z

    def back(x, a):
        return torch.roll(x, 1, dims[a])

    def ahead(x, a):
        return torch.roll(x, -1, dims[a])

    P = [ratio(back(r, a), back(p, a), r, p) for a in range(3)]
    both = [torch.minimum(P[a], ahead(P[a], a)) for a in range(3)]
    out = torch.zeros_like(U)
    for a in range(3):
        s = P[a]
        for b in range(3):
            if b != a:
                s = torch.minimum(s, torch.minimum(both[b], back(both[b], a)))
        ts = [vel[b] for b in range(3) if b != a]
        R = side(r, vel[a], ts, p, ks)
        L = side(back(r, a), back(vel[a], a), [back(t, a) for t in ts], back(p, a), [back(k, a) for k in ks])
        F = roe_am(L, R, f_mach(s) ** 8, par)
        rows = [0, 1 + a] + [1 + b for b in range(3) if b != a] + list(range(4, U.shape[0]))
        for k, f in zip(rows, F):
            out[k] += (f - ahead(f, a)) / d[a]
    return out


def exact(case, seed):
    """What run() returns for these inputs, in 64 bits."""
    c = case
    if c["flow"] == "tgv":
        s, U = flow_3d(c, seed)
        d, mr = (s.dx, s.dy, s.dz), torch.tensor(s.params.m_ref, device=DEV, dtype=F64)
        par = SimpleNamespace(m_ref=mr, eps1=0)
        for _ in range(c["steps"]):
            vel = [U[1 + a] / U[0] for a in range(3)]
            q2 = sum(t * t for t in vel)
            c2 = GAMMA * (GAMMA - 1) * (U[4] / U[0] - 0.5 * q2)
            dt = CFL / sum(speed(vel[a], q2, c2, mr) / d[a] for a in range(3)).max()
            U = ssp_rk3(U, dt, lambda X: residual_3d(X, d, par))
        return U
    grids, states = flow_2d(c, seed)
    P = Padded(grids)
    U = P.split(torch.cat([u.reshape(-1) for u in states]))
    for _ in range(c["steps"]):
        dt = (CFL / P.rate(U))[P.gid_inner]
        U = ssp_rk3(U, dt, P.residual)
    if c["prec"] == 64 and c["flow"] == "gresho":
        R = P.residual(U)
        return {"state": P.join(U), "norm": R.square().mean(1).sqrt(), "totals": (U * P.V).sum(1)}
    return P.join(U)
