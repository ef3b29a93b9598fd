"""Performance cases of the STG-LBM channel library.

A case is one call sequence of a user's program on lattices it already holds:
so many steps of a channel (``Channel.step``), of a probed channel
(``Channel.step_probed``), of a batch (``Batch.step``), or steps followed by a
statistics read-out (``Channel.stats``).  The listed cases are the workloads
of this repository's configurations, tests and benchmark, from the 64x32x32
parity channel to the refined 1536x256x384 one; ``draw`` gives others of the
same ranges (0.07 to 20 million cells, both lane-friendly and odd sizes, every
storage, collision, streaming scheme, boundary and option).

Fields of a case:
  nx, ny, nz     lattice (of a batch: the members' half-heights h are given
                 by ``heights`` and each is a 12h x 2h x 3h channel)
  storage        fp32 | fp16s (binary16, to nearest) | fp16sr (binary16, stochastic)
  streaming      pull | aa (in place)
  collision      regularized | bgk
  bc_x           stg (inlet/outlet) | periodic (driven by ``force``)
  sponge         length of the sponge zone before the outlet (0: none)
  modes          Fourier modes of the inlet
  probes         velocity probes sampled after every step (0: none)
  readout        True: the pass ends with the statistics read-out
  steps          time steps of one pass
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_2205_02774_gb300.channel import Channel
from paper_2205_02774_gb300.serving import Batch

TAU0, C_SMAG, T_FILTER, MACH, STATS_EVERY, CHECK_EVERY = 0.52, 0.01, 4.0, 0.0516, 10, 100
C_L, N_FV, RE_TAU = 3.0, 96, 180.0
SPONGE_K, SPONGE_P = 1000.0, 3.0

# D3Q19 in the order of the library's population arrays
VEL = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
       (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
       (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
OPP = [VEL.index((-a, -b, -c)) for a, b, c in VEL]
WGT = [1 / 3 if i == 0 else 1 / 18 if i < 7 else 1 / 36 for i in range(19)]


def _case(nx, ny, nz, steps, storage="fp32", streaming="pull", collision="regularized", bc_x="stg", sponge=0.0,
          modes=200, probes=0, readout=False, force=0.0, heights="", name=None):
    c = dict(nx=nx, ny=ny, nz=nz, steps=steps, storage=storage, streaming=streaming, collision=collision, bc_x=bc_x,
             sponge=sponge, modes=modes, probes=probes, readout=readout, force=force, heights=heights)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one step of the parity channel, as a program that couples
        # something of its own to every step makes it; latency only
        _case(64, 32, 32, 1, modes=100, name="single_step_64x32x32_fp32"),
        # the parity channel's own run: 200 steps, all launches and dependent small kernels
        _case(64, 32, 32, 200, modes=100, name="parity_64x32x32_fp32"),
        # a small job of the served stream (h = 20, the smallest it draws), binary16 storage
        _case(240, 40, 60, 100, storage="fp16sr", name="served_240x40x60_fp16sr"),
        # time series for the auto-correlation of a mid-size channel: 64 probes, every step
        _case(384, 64, 96, 100, probes=64, name="probed_384x64x96_fp32"),
        # the production channel in plain FP32
        _case(768, 128, 192, 20, name="production_768x128x192_fp32"),
        # the production channel with the paper's sponge zone (0.4 half-heights), binary16 to nearest
        _case(768, 128, 192, 20, storage="fp16s", sponge=25.6, name="sponge_768x128x192_fp16s"),
        # half the memory: the one-lattice in-place update
        _case(768, 128, 192, 20, storage="fp16sr", streaming="aa", name="inplace_768x128x192_fp16sr"),
        # the paper's literal collision
        _case(768, 128, 192, 20, storage="fp16sr", collision="bgk", name="bgk_768x128x192_fp16sr"),
        # a grid whose streamwise node count is odd (end points included), nothing divides anything
        _case(385, 65, 97, 20, name="odd_385x65x97_fp32"),
        # the body-force-driven doubly periodic channel, with its statistics read at the end
        _case(256, 128, 128, 20, collision="bgk", bc_x="periodic", force=1e-7, readout=True,
              name="forced_256x128x128_fp32"),
        # an ensemble of channels of the batched configuration's half-heights in one batch
        _case(0, 0, 0, 20, heights="16,24,32,48,64,16,24,32,48,64,16,24,32,48,24,32",
              name="ensemble_16_channels_fp32"),
        # the refined channel, the benchmark's workload: the largest
        _case(1536, 256, 384, 20, storage="fp16sr", name="refined_1536x256x384_fp16sr"),
    ]


def draw(rng: random.Random):
    if rng.random() < 0.1:
        hs = [rng.choice((16, 20, 24, 27, 32, 40, 48)) for _ in range(rng.randint(3, 12))]
        return _case(0, 0, 0, rng.choice((20, 40, 50)), storage=rng.choice(("fp32", "fp16sr")),
                     heights=",".join(map(str, hs)))
    cells = math.exp(rng.uniform(math.log(7e4), math.log(2e7)))
    h = (cells / 72.0) ** (1.0 / 3.0)
    # the configurations' 12h x 2h x 3h, up to a third longer or shorter each way
    nx, ny, nz = (max(m, round(k * h * math.exp(rng.uniform(-0.3, 0.3)))) for k, m in ((12, 16), (2, 8), (3, 8)))
    shape = rng.random()
    if shape < 0.3:
        nx |= 1
    elif shape < 0.5:
        nx += nx % 2
    else:
        nx += -nx % 4
    storage = rng.choice(("fp32", "fp16s", "fp16sr"))
    streaming = "aa" if nx % 2 == 0 and rng.random() < 0.25 else "pull"
    collision = "bgk" if rng.random() < 0.25 else "regularized"
    bc_x = "periodic" if rng.random() < 0.2 else "stg"
    sponge = float(round(0.2 * ny, 1)) if bc_x == "stg" and rng.random() < 0.2 else 0.0
    probes = rng.choice((8, 64, 500)) if rng.random() < 0.15 else 0
    readout = not probes and rng.random() < 0.25
    most = max(1, int(1.5e9 / (nx * ny * nz)))
    steps = min(most, rng.choice((1, 10, 20, 33, 50, 100, 200)))
    if streaming == "aa":
        steps += steps % 2
    return _case(nx, ny, nz, steps, storage, streaming, collision, bc_x, sponge, rng.choice((50, 100, 200)), probes,
                 readout, 1e-7 if bc_x == "periodic" else 0.0)


# ------------------------------------------------------------------ inputs

def _profile(re_tau):
    """A RANS channel profile at the centres of a tanh-stretched grid (wall units, half-height 1)."""
    i = np.arange(N_FV + 1)
    faces = 1.0 + np.tanh(2.0 * (2.0 * i / N_FV - 1.0)) / np.tanh(2.0)
    y = 0.5 * (faces[:-1] + faces[1:])
    yp = np.minimum(y, 2.0 - y) * re_tau
    U = np.log1p(0.41 * yp) / 0.41 + 7.8 * (1.0 - np.exp(-yp / 11.0) - yp / 11.0 * np.exp(-yp / 3.0))
    s = (yp / 15.0) ** 2
    k = 18.0 * s / (1.0 + s) ** 2 + 0.8 * (1.0 - np.exp(-yp / 30.0))
    eps = re_tau / (0.41 * (yp + 8.0))
    R = np.zeros((N_FV, 6))
    R[:, 0], R[:, 1], R[:, 2] = 1.1 * k, 0.4 * k, 0.5 * k
    R[:, 3] = -(1.0 - y) * (1.0 - np.exp(-yp / 26.0)) ** 2
    return SimpleNamespace(y_c=y, U=U, k=k, eps=eps, R=R, U_bulk=float(np.sum(U * np.diff(faces)) / 2.0),
                           nu_phys=1.0 / re_tau, h_phys=1.0)


def _members(case):
    """The lattices of a case: (nx, ny, nz, Re_tau) each."""
    if not case["heights"]:
        return [(case["nx"], case["ny"], case["nz"], RE_TAU)]
    hs = [int(h) for h in case["heights"].split(",")]
    return [(12 * h, 2 * h, 3 * h, (180.0, 395.0)[m % 2]) for m, h in enumerate(hs)]


def _initial_state(nx, ny, nz, storage, seed):
    """A channel flow in progress, in the storage format (f_i - w_i), on the GPU: the mean profile with
    smooth fluctuations of a few per cent of it, small density waves and cell-to-cell non-equilibrium."""
    dev = "cuda"
    gen = torch.Generator(device=dev).manual_seed(seed)
    r = random.Random(seed)
    x, y, z = (torch.arange(n, device=dev, dtype=torch.float32) for n in (nx, ny, nz))
    x, y, z = x[None, None, :], y[None, :, None], z[:, None, None]
    eta = (2.0 * y + 1.0) / ny - 1.0

    def smooth(amp):
        out = torch.zeros((nz, ny, nx), device=dev)
        for _ in range(2):
            kx, ky, kz = r.randint(1, 6), r.randint(0, 3), r.randint(1, 4)
            ph = 2.0 * math.pi * (kx * x / nx + kz * z / nz + r.random())
            out += amp * r.gauss(0, 1) * torch.cos(ph) * torch.cos(math.pi * ky * (y + 0.5) / ny)
        return out

    env = 1.0 - eta ** 6
    u = [0.03 * (1.0 - eta ** 4) + env * smooth(1e-3), env * smooth(1e-3), env * smooth(1e-3)]
    drho = smooth(2e-4)
    rho, uu = 1.0 + drho, u[0] ** 2 + u[1] ** 2 + u[2] ** 2
    out = torch.empty((19, nz, ny, nx), device=dev, dtype=torch.float32 if storage == "fp32" else torch.float16)
    for i, c in enumerate(VEL):
        cu = sum(s * v for s, v in zip(c, u) if s)
        geq = drho + rho * (3.0 * cu + 4.5 * cu * cu - 1.5 * uu)
        noise = torch.randn((nz, ny, nx), device=dev, generator=gen)
        out[i] = WGT[i] * (geq + 1e-3 * noise)
    return out


def _probe_cells(case, seed):
    r = np.random.default_rng(seed)
    return np.stack([r.integers(0, n, case["probes"]) for n in (case["nx"], case["ny"], case["nz"])], axis=1)


_stream = None


def prepare(case, seed):
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()  # the program's solver stream
    chs = []
    for m, (nx, ny, nz, re_tau) in enumerate(_members(case)):
        stg = case["bc_x"] == "stg"
        ch = Channel(nx, ny, nz, profile=_profile(re_tau) if stg else None, tau0=TAU0, c_smag=C_SMAG,
                     force=(case["force"], 0.0, 0.0), storage=case["storage"], collision=case["collision"],
                     bc_x=case["bc_x"], stats_every=STATS_EVERY, check_every=CHECK_EVERY, n_modes=case["modes"],
                     C_l=C_L, t_filter=T_FILTER, mach_target=MACH, seed=seed + m, stream=_stream,
                     sponge=(case["sponge"], SPONGE_K, SPONGE_P), streaming=case["streaming"])
        s = _initial_state(nx, ny, nz, case["storage"], seed + m).cpu()
        ch.set_state(s.numpy() if case["storage"] == "fp32" else s.view(torch.int16).numpy().view(np.uint16))
        chs.append(ch)
    batch = None
    if case["heights"]:
        batch = Batch(stream=_stream)
        for ch in chs:
            batch.add(ch)
    if case["probes"]:
        chs[0].set_probes(_probe_cells(case, seed))
    return SimpleNamespace(case=case, chs=chs, batch=batch)


class _Device:
    """A device array of the library as torch sees it."""

    def __init__(self, ptr, shape, typestr):
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": shape, "typestr": typestr, "version": 3}


def run(state):
    case, out = state.case, {}
    if state.batch:
        state.batch.step(case["steps"])
    elif case["probes"]:
        out["probe_u"] = state.chs[0].step_probed(case["steps"])
    else:
        state.chs[0].step(case["steps"])
    for m, ch in enumerate(state.chs):
        pops, inlet = ch.device_state()
        out["populations%d" % m] = torch.as_tensor(
            _Device(pops, ch.shape, "<f4" if ch.storage == "fp32" else "<f2"), device="cuda")
        if case["bc_x"] == "stg":
            out["inlet%d" % m] = torch.as_tensor(_Device(inlet, (3, ch.nz, ch.ny), "<f4"), device="cuda")
    if case["readout"]:
        # time- and span-averaged profiles <u_a>, <u_a u_b> as a program keeps them (sums of FP32 velocities)
        ch = state.chs[0]
        s = ch.stats()
        if s["n_samples"]:
            n = s["n_samples"] * ch.nz
            out["mean_u"] = (s["mean_sum"] / n).astype(np.float32)
            out["mean_uu"] = (s["rey_sum"] / n).astype(np.float32)
        out["mass"] = np.float32(s["mass"])
    return out


def work(case):
    e = 4 if case["storage"] == "fp32" else 2
    bts = fl = 0.0
    for nx, ny, nz, _ in _members(case):
        cells = nx * ny * nz
        bts += case["steps"] * cells * 38 * e  # 19 populations read, 19 written
        fl += case["steps"] * cells * 300
        if case["bc_x"] == "stg":  # tables read, plane and filter state written; a cosine term is about 12 operations
            bts += case["steps"] * (4.0 * case["modes"] * (2 * ny + nz) + 36.0 * ny * nz)
            fl += case["steps"] * 12.0 * case["modes"] * ny * nz
        bts += case["steps"] // STATS_EVERY * 144.0 * nx * ny  # running sums read and written
        if case["readout"]:
            bts += 72.0 * nx * ny + 19 * cells * e
    bts += 12.0 * case["steps"] * case["probes"]
    return {"bytes": bts, "flops": fl}


# ------------------------------------------------------------------ the same in 64 bits

def _uniform(seed, n):
    """SplitMix64 (Steele, Lea & Flood 2014), top 53 bits."""
    m, s, out = (1 << 64) - 1, seed & ((1 << 64) - 1), []
    for _ in range(n):
        s = (s + 0x9E3779B97F4A7C15) & m
        z = ((s ^ (s >> 30)) * 0xBF58476D1CE4E5B9) & m
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
        out.append(((z ^ (z >> 31)) >> 11) / float(1 << 53))
    return np.array(out)


class _Inlet:
    """The inlet velocity plane of step t in 64 bits, (3, nz, ny)."""

    def __init__(self, ny, nz, re_tau, n_modes, seed):
        p = _profile(re_tau)
        top, cx = 2.0 * p.h_phys, 2.0 * p.h_phys / ny
        su = MACH / math.sqrt(3.0) / p.U.max()
        y = (np.arange(ny) + 0.5) * cx
        yy = np.concatenate(([0.0], p.y_c, [top]))

        def at(v, lo=0.0, hi=0.0):
            return np.interp(y, yy, np.concatenate(([lo], v, [hi])))

        k, eps = at(p.k), at(p.eps, p.eps[0], p.eps[-1])
        R = [at(p.R[:, c]) * su * su for c in range(6)]
        dw = np.minimum(y, top - y)
        le = np.minimum(2.0 * dw, C_L * k ** 1.5 / eps) / cx
        leta = (p.nu_phys ** 3 / eps) ** 0.25 / cx
        lcut = 2.0
        kcut = 2.0 * math.pi / lcut
        kmin, kmax = math.pi / le.max(), 1.5 * kcut
        ratio = (kmax / kmin) ** (1.0 / (n_modes - 1)) if n_modes > 1 else 1.0
        kn = kmin * ratio ** np.arange(n_modes)
        dk = kn * (1.0 - 1.0 / ratio) if n_modes > 1 else np.ones(1)
        x = kn[:, None] * le[None, :] / (2.0 * math.pi)
        e = x ** 4 / (1.0 + 2.4 * x * x) ** (17.0 / 6.0)
        e *= np.exp(-(12.0 * kn[:, None] * leta[None, :] / (2.0 * math.pi)) ** 2)
        e *= np.exp(-(4.0 * np.maximum(kn - 0.9 * kcut, 0.0) / kcut) ** 3)[:, None]
        e *= dk[:, None]
        u = _uniform(seed, 4 * n_modes).reshape(n_modes, 4)
        Phi, Th, et = 2 * math.pi * u[:, 0], np.arccos(1.0 - 2.0 * u[:, 1]), 2 * math.pi * u[:, 2]
        st, ct, sp, cp, se, ce = (f(a) for a in (Th, Phi, et) for f in (np.sin, np.cos))
        t64 = dict(device="cuda", dtype=torch.float64)
        self.amp = torch.tensor(np.sqrt(6.0 * e / e.sum(0)), **t64)  # (N, ny)
        self.sig = torch.tensor(np.stack([cp * ct * ce - sp * se, sp * ct * ce + cp * se, -st * ce]), **t64)
        self.om = torch.tensor(-2.0 * math.pi * st * cp * p.U_bulk * su / le.max(), **t64)
        self.phi = torch.tensor(2.0 * math.pi * u[:, 3], **t64)
        self.A = torch.tensor((kn * st * sp)[:, None] * (np.arange(ny) + 0.5), **t64)
        self.B = torch.tensor((kn * ct)[:, None] * np.arange(nz), **t64)
        a11 = np.sqrt(np.maximum(R[0], 0.0))
        inv = np.divide(1.0, a11, out=np.zeros(ny), where=a11 > 0)
        a21, a31 = R[3] * inv, R[4] * inv
        a22 = np.sqrt(np.maximum(R[1] - a21 ** 2, 0.0))
        a32 = np.divide(R[5] - a21 * a31, a22, out=np.zeros(ny), where=a22 > 0)
        a33 = np.sqrt(np.maximum(R[2] - a31 ** 2 - a32 ** 2, 0.0))
        self.L = [torch.tensor(a, **t64) for a in (a11, a21, a22, a31, a32, a33)]
        self.U = torch.tensor(at(p.U) * su, **t64)
        self.uf, self.a = None, math.exp(-1.0 / T_FILTER)

    def plane(self, t):
        # cos(y part + z part) by the addition theorem: two products per component
        ph = self.B + (self.phi + self.om * t)[:, None]
        Ca, Sa = self.amp * torch.cos(self.A), self.amp * torch.sin(self.A)
        Cb, Sb = torch.cos(ph), torch.sin(ph)
        v = [(Cb * s[:, None]).T @ Ca - (Sb * s[:, None]).T @ Sa for s in self.sig]
        l11, l21, l22, l31, l32, l33 = self.L
        u = torch.stack([l11 * v[0], l21 * v[0] + l22 * v[1], l31 * v[0] + l32 * v[1] + l33 * v[2]])
        self.uf = u if self.uf is None else self.a * self.uf + (1.0 - self.a) * u
        out = self.uf.clone()
        out[0] += self.U
        return out


_PAIRS = [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]


class _Lattice:
    """The step in 64 bits on g_i = f_i - w_i, [19][nz][ny][nx], the pull scheme."""

    def __init__(self, case, nx, ny, nz):
        t64 = dict(device="cuda", dtype=torch.float64)
        self.case, self.n = case, (nx, ny, nz)
        c = torch.tensor(VEL, **t64)
        self.w = torch.tensor(WGT, **t64)
        cc = torch.stack([c[:, a] * c[:, b] for a, b in _PAIRS], 1)
        # moments (rho, j, sum c c g) of 19 values, and 19 values w (a0 + c.B + c.A.c) of ten coefficients
        self.M = torch.cat([torch.ones(19, 1, **t64), c, cc], 1).T.contiguous()
        self.N = self.w[:, None] * torch.cat([torch.ones(19, 1, **t64), c, cc[:, :3], 2.0 * cc[:, 3:]], 1)
        f = torch.zeros(nx, **t64)
        if case["sponge"] > 0:
            xi = (torch.arange(nx, **t64) - (nx - 1 - case["sponge"])) / case["sponge"]
            f = torch.where(xi >= 0, SPONGE_K * xi.clamp(min=0) ** SPONGE_P, 0.0)
        self.nuf = f + 1.0

    def eq(self, drho, u):
        """Coefficients of the shifted equilibrium."""
        rho = 1.0 + drho
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        return [drho - 1.5 * rho * uu] + [3.0 * rho * v for v in u] + [4.5 * rho * u[a] * u[b] for a, b in _PAIRS]

    def values(self, co):
        co = torch.stack(co)
        return (self.N @ co.reshape(10, -1)).reshape((19,) + co.shape[1:])

    def moments(self, g, F):
        m = (self.M @ g.reshape(19, -1)).reshape((10,) + g.shape[1:])
        rho = 1.0 + m[0]
        u = [(m[1] + 0.5 * F) / rho, m[2] / rho, m[3] / rho]
        pi = [m[4 + k] - rho * u[a] * u[b] - (m[0] / 3.0 if a == b else 0.0) for k, (a, b) in enumerate(_PAIRS)]
        return m[0], u, pi, [m[1], m[2], m[3]]

    def rebuild(self, g, drho, u, sign):
        """Regularized boundary node: unknown directions (c_x of that sign) take the opposite's non-equilibrium."""
        geq = self.values(self.eq(drho, u))
        neq = g - geq
        neq = torch.stack([neq[OPP[i]] if VEL[i][0] == sign else neq[i] for i in range(19)])
        pi = (self.M @ neq.reshape(19, -1)).reshape((10,) + g.shape[1:])
        tr = pi[0]
        P = [pi[4 + k] - (tr / 3.0 if a == b else 0.0) for k, (a, b) in enumerate(_PAIRS)]
        z = torch.zeros_like(tr)
        return geq + self.values([-1.5 * (P[0] + P[1] + P[2]), z, z, z] + [4.5 * p for p in P])

    def step(self, f, ubc, sums):
        nx, ny, nz = self.n
        case, F = self.case, self.case["force"]
        stg = case["bc_x"] == "stg"
        out = torch.empty_like(f)
        slab = max(1, min(nz, int(4e6 // (nx * ny))))
        for z0 in range(0, nz, slab):
            zz = torch.arange(z0, min(nz, z0 + slab), device="cuda")
            g = torch.empty((19, len(zz), ny, nx), device="cuda", dtype=torch.float64)
            for i, (cx, cy, cz) in enumerate(VEL):
                s = f[i].index_select(0, (zz - cz) % nz)
                g[i] = torch.roll(s, (cy, cx), (1, 2))
                if cy:  # half-way bounce-back
                    row = 0 if cy > 0 else ny - 1
                    g[i, :, row] = f[OPP[i]][zz[0]:zz[-1] + 1, row]
            if stg:
                x0 = g[:, :, :, 0]
                u = [v[zz] for v in ubc]
                par = sum(x0[i] for i in range(19) if VEL[i][0] == 0)
                lv = sum(x0[i] for i in range(19) if VEL[i][0] < 0)
                g[:, :, :, 0] = self.rebuild(x0, (par + 2.0 * lv + u[0]) / (1.0 - u[0]), u, 1)
                _, u, _, _ = self.moments(g[:, :, :, nx - 2].contiguous(), F)
                g[:, :, :, nx - 1] = self.rebuild(g[:, :, :, nx - 1].contiguous(), torch.zeros_like(u[0]), u, -1)
            drho, u, pi, j = self.moments(g, F)
            if sums is not None:
                for a in range(3):
                    sums[0][a] += u[a].sum(0)
                for k, (a, b) in enumerate(_PAIRS):
                    sums[1][k] += (u[a] * u[b]).sum(0)
            rho = 1.0 + drho
            qh = torch.sqrt(sum(p * p * (1.0 if a == b else 2.0) for p, (a, b) in zip(pi, _PAIRS)))
            tau = 0.5 * TAU0 + torch.sqrt((TAU0 * rho) ** 2 + 18.0 * math.sqrt(2.0) * C_SMAG * qh) / (2.0 * rho)
            tau = 0.5 + self.nuf * (tau - 0.5)
            om = 1.0 / tau
            co = self.eq(drho, u)
            if case["collision"] == "regularized":
                km = 1.0 - om
                co[0] = co[0] - 1.5 * km * (pi[0] + pi[1] + pi[2])
                for k in range(6):
                    co[4 + k] = co[4 + k] + 4.5 * km * pi[k]
                if F:  # first-order non-equilibrium part, -F/2
                    co[1] = co[1] - 1.5 * km * F
            else:
                co = [om * v for v in co]
            if F:
                kf = 1.0 - 0.5 * om
                co[0] = co[0] - 3.0 * kf * u[0] * F
                co[1] = co[1] + 3.0 * kf * F
                for k, (a, b) in enumerate(_PAIRS):
                    uF = (u[b] if a == 0 else 0.0) + (u[a] if b == 0 else 0.0)
                    co[4 + k] = co[4 + k] + 4.5 * kf * F * uF
            r = self.values(co)
            if case["collision"] == "bgk":
                r += (1.0 - om) * g
            out[:, zz[0]:zz[-1] + 1] = r
        return out


def exact(case, seed):
    cells = sum(nx * ny * nz for nx, ny, nz, _ in _members(case))
    if cells * case["steps"] > 3.2e9:
        return None
    out = {}
    for m, (nx, ny, nz, re_tau) in enumerate(_members(case)):
        f = _initial_state(nx, ny, nz, case["storage"], seed + m).double()
        lat = _Lattice(case, nx, ny, nz)
        stg = case["bc_x"] == "stg"
        inlet = _Inlet(ny, nz, re_tau, case["modes"], seed + m) if stg else None
        t64 = dict(device="cuda", dtype=torch.float64)
        sums = (torch.zeros((3, ny, nx), **t64), torch.zeros((6, ny, nx), **t64))
        samples, ubc, series = 0, None, []
        if case["probes"]:
            px, py, pz = torch.tensor(_probe_cells(case, seed), device="cuda").T
        for t in range(case["steps"]):
            ubc = inlet.plane(t) if stg else None
            sampling = (t + 1) % STATS_EVERY == 0
            samples += sampling
            f = lat.step(f, ubc, sums if sampling and case["readout"] else None)
            if case["probes"]:
                mo = lat.M @ f[:, pz, py, px]
                mo[1] -= 0.5 * case["force"]
                series.append((mo[1:4] / (1.0 + mo[0])).T)
        if series:
            out["probe_u"] = torch.stack(series).cpu().numpy()
        if case["readout"]:
            if samples:
                out["mean_u"] = (sums[0] / (samples * nz)).cpu().numpy()
                out["mean_uu"] = (sums[1] / (samples * nz)).cpu().numpy()
            out["mass"] = np.float64(f.sum().item() + nx * ny * nz)
        # in place, after an even number of steps population i is kept in the opposite slot
        out["populations%d" % m] = f[OPP] if case["streaming"] == "aa" else f
        if stg:
            out["inlet%d" % m] = ubc
    return out
