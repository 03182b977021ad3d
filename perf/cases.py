"""What a user of this framework has it do, as measurable cases.

Most cases advance one fluid-structure problem (or a batch of them) by some
coarse steps through `Simulation` and read the whole state back, as a program
does that writes a results file or samples a trajectory every few steps.  Two
more cover the learned sub-stepper's training step and the tensor-core GEMM.

Each listed case carries the options that select it; `draw` varies sizes,
spacings and options over the same ranges.  `exact` restates a coarse step of
the method in 64 bits in plain torch, pair by pair.

Fields held on the device in single precision (or summed from single-precision
pair terms: the time averages) come back as float32, as a results file stores
them; positions, which are held and advanced in 64 bits, come back as such.
"""
import math

import numpy as np
import torch

import fsi_cases
from paper_1911_13255_gb300 import Mpnn, Simulation, gemm_bf16


def listed():
    return [
        # the smallest call: an interactive session that takes one step at a time and looks at the result
        dict(name="box_2d_single_step", kind="box2d", nx=16, ny=12, steps=1),
        # the paper's flow-induced vibration (cylinder with an elastic flag, D/10), sampled every 20 steps
        dict(name="flag_channel_2d", kind="flag", cells_D=10, ratio=2, steps=20),
        # the paper's dam break through an elastic gate at 1 mm, every 20 steps
        dict(name="dam_gate_2d", kind="dam", dp_mm=1.0, ratio=2, steps=20),
        # the same at half the spacing: 56k fluid particles and a body of 6.4k
        dict(name="dam_gate_2d_fine", kind="dam", dp_mm=0.5, ratio=2, steps=20),
        # the pulsatile venous valve, whose stable setting is one time step for both phases
        dict(name="valve_2d_single_rate", kind="valve", wo=10.0, steps=20),
        # a parameter study: 32 channels of uneven size advanced as one batch, all states read
        dict(name="flag_batch_32", kind="batch", n=32, nf_hi=60000, steps=10),
        # a medium 3-D tank with a clamped plate and a free surface
        dict(name="tank_3d", kind="box3d", nx=48, ny=36, nz=36, steps=10),
        # the 3-D duct with a flexible plate at 1/8 of the benchmark's size
        dict(name="duct_3d_eighth", kind="duct", ny=50, cadence=1, steps=10),
        # the same with the paper's neighbour lists held over an advection step (Algorithm 1)
        dict(name="duct_3d_eighth_held", kind="duct", ny=50, cadence=2, steps=10),
        # the benchmark's duct: 3.0M fluid, 65k solid, 0.5M wall particles
        dict(name="duct_3d_full", kind="duct", ny=100, cadence=1, steps=10),
        # fitting the learned sub-stepper: one Adam step over 32 copies of the flag's graph
        dict(name="mpnn_train_step", kind="mpnn", replicas=32, flag_len=3.5),
        # the tensor-core GEMM by itself at a large shape
        dict(name="gemm_bf16_large", kind="gemm", M=16384, N=256, K=4096, bias=False),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["box2d", "flag", "flag", "dam", "dam", "valve", "batch", "box3d", "duct", "duct", "mpnn", "gemm"])
    steps = int(round(_log(rng, 1, 20)))
    if kind == "box2d":
        return dict(kind=kind, nx=int(_log(rng, 14, 60)), ny=int(_log(rng, 11, 50)), steps=rng.choice([1, 1, 2, 3]))
    if kind == "flag":
        return dict(kind=kind, cells_D=int(round(_log(rng, 10, 28))), ratio=rng.choice([1, 2, 2, 3]), steps=steps)
    if kind == "dam":
        return dict(kind=kind, dp_mm=round(_log(rng, 0.45, 2.0), 3), ratio=rng.choice([1, 2, 2]), steps=steps)
    if kind == "valve":
        return dict(kind=kind, wo=round(_log(rng, 1.0, 10.0), 2), steps=steps)
    if kind == "batch":
        return dict(kind=kind, n=rng.randint(3, 32), nf_hi=int(_log(rng, 12000, 60000)), steps=rng.randint(1, 10))
    if kind == "box3d":
        return dict(kind=kind, nx=int(_log(rng, 9, 70)), ny=int(_log(rng, 7, 50)), nz=int(_log(rng, 7, 50)),
                    steps=rng.randint(1, 10))
    if kind == "duct":
        return dict(kind=kind, ny=int(_log(rng, 40, 90)), cadence=rng.choice([1, 1, 2]), steps=rng.randint(1, 10))
    if kind == "mpnn":
        return dict(kind=kind, replicas=int(round(_log(rng, 1, 32))), flag_len=round(rng.uniform(2.0, 4.0), 2))
    return dict(kind=kind, M=128 * int(round(_log(rng, 1, 150))), N=16 * int(round(_log(rng, 1, 32))),
                K=64 * int(round(_log(rng, 1, 128))), bias=rng.random() < 0.5)


# --------------------------------------------------------------------------
# inputs (from the seed alone)
# --------------------------------------------------------------------------

def _problems(case, seed):
    """The raw arrays and constants of the problem instances of a case."""
    k = case["kind"]
    if k == "box2d":
        return [fsi_cases.tiny_box(seed=seed, nx=case["nx"], ny=case["ny"])]
    if k == "flag":
        # the reading set of the framework's long runs: 12 dp_F inflow buffer, reinitialisation every 3 steps
        c = fsi_cases.channel_flag(seed=seed, dpF=0.1 / case["cells_D"], ratio=case["ratio"])
        c.n_reinit, c.inflow_width = 3, 12 * c.f_dp
        return [c]
    if k == "dam":
        return [fsi_cases.dam_gate(seed=seed, dpF=case["dp_mm"] * 1e-3, ratio=case["ratio"])]
    if k == "valve":
        return [fsi_cases.venous_valve(seed=seed, wo=case["wo"])]
    if k == "batch":
        # one family of channels and flags; the seed moves their particles
        cs = fsi_cases.flag_batch(seed=0, n=case["n"], nf_hi=case["nf_hi"])
        rng = np.random.default_rng(seed)
        for c in cs:
            c.n_reinit, c.inflow_width = 3, 12 * c.f_dp
            c.f_r = fsi_cases.jitter(c.f_r, c.f_dp, 1e-3, rng)
            c.f_r[:, 0] %= c.Lx
            c.s_r0 = fsi_cases.jitter(c.s_r0, c.s_dp, 1e-3, rng)
        return cs
    if k == "box3d":
        # a tank of water at rest under its own weight, c0 and the plate's stiffness in proportion
        c = fsi_cases.tiny_box_3d(seed=seed, n=(case["nx"], case["ny"], case["nz"]), c0=40.0)
        c.s_E = 2e5
        c.f_p = c.f_p + c.f_rho0 * 9.81 * (case["ny"] * c.f_dp - c.f_r[:, 1])
        return [c]
    return [fsi_cases.duct_plate_3d(seed=seed, scale=100.0 / case["ny"])]


FIN, NOUT, WIDTH, LAYERS = 64, 16, 128, 3   # the network's padded input, output and hidden widths


def _network(case, seed):
    """Graph of the flag's body, weights, and one batch of normalised samples with its targets and mask."""
    rng = np.random.default_rng(seed)
    c = fsi_cases.channel_flag(seed=seed, flag_len=case["flag_len"])
    n, h, V = c.ns, 1.3 * c.s_dp, c.s_dp ** 2
    d = c.s_r0[:, None, :] - c.s_r0[None, :, :]
    r = np.sqrt((d * d).sum(2))
    rows, idx = np.nonzero((r < 2 * h) & ~np.eye(n, dtype=bool))
    ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))]).astype(np.int64)
    rq, a = r[rows, idx], 7.0 / (4.0 * math.pi * h * h)
    q = rq / h
    w = V * a * (1 - 0.5 * q) ** 4 * (1 + 2 * q)
    g = (h * V * -5.0 * a / h * q * (1 - 0.5 * q) ** 3 / rq)[:, None] * d[rows, idx]
    z, parts = WIDTH * 4, []
    for out, inp, scale in [(WIDTH, FIN, 1.0)] + [(WIDTH, z, 1.0)] * LAYERS + [(NOUT, WIDTH, 0.1)]:
        lim = math.sqrt(6.0 / inp) * scale
        parts += [rng.uniform(-lim, lim, out * inp), np.zeros(out)]
    theta = np.concatenate(parts).astype(np.float32)
    N = n * case["replicas"]
    x = np.zeros((N, FIN), np.float32)
    x[:, :14] = rng.normal(size=(N, 14))
    t = np.zeros((N, NOUT), np.float32)
    t[:, :4] = rng.normal(size=(N, 4))
    mask = np.tile((c.s_cons == 0).astype(np.uint8), case["replicas"])
    return (ptr, idx.astype(np.int64), w, g), rows, theta, x, t, mask


def _matrices(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.randn(case["M"], case["K"], generator=gen, device="cuda").bfloat16()
    B = torch.randn(case["N"], case["K"], generator=gen, device="cuda").bfloat16()
    bias = torch.randn(case["N"], generator=gen, device="cuda") if case["bias"] else None
    return A, B, bias


def prepare(case, seed):
    if case["kind"] == "gemm":
        A, B, bias = _matrices(case, seed)
        out = torch.empty(case["M"], case["N"], device="cuda")
        return dict(kind="gemm", A=A, B=B, bias=bias, out=out)
    stream = torch.cuda.Stream()
    if case["kind"] == "mpnn":
        graph, _, theta, x, t, mask = _network(case, seed)
        net = Mpnn(2, graph, replicas=case["replicas"], stream=stream)
        net.set_params(theta)
        return dict(kind="mpnn", net=net, stream=stream, x=torch.from_numpy(x).cuda(), t=torch.from_numpy(t).cuda(),
                    mask=mask)
    cs = _problems(case, seed)
    if case["kind"] == "box2d":
        # a session on the default stream, stepping by hand
        sim = Simulation.from_case(cs[0])
    elif case["kind"] == "batch":
        sim = Simulation.from_cases(cs, stream=stream)
    else:
        sim = Simulation.from_case(cs[0], stream=stream)
    if case["kind"] == "valve":
        sim.set_time_stepping("single_solid")
    if case.get("cadence", 1) != 1:
        sim.set_advection_cadence(case["cadence"])
    return dict(kind=case["kind"], sim=sim, stream=stream, steps=case["steps"], rho0=[c.f_rho0 for c in cs])


def _fields(sim, rho0):
    """The whole state of the selected instance."""
    f, s = sim.get_fluid(), sim.get_solid()
    return dict(f_r=f["r"], f_v=f["v"], f_drho=(f["rho"] - rho0).astype(np.float32), f_rate=f["drho"],
                f_acc=f["dvdt"], s_r=s["r"], s_v=s["v"], s_F=s["F"].astype(np.float32),
                s_vbar=s["vbar"].astype(np.float32), s_abar=s["abar"].astype(np.float32), s_force=s["fF"],
                s_n=s["nrm"])


def _join(states):
    return {k: np.concatenate([s[k] for s in states]) for k in states[0]}


def run(state):
    if state["kind"] == "gemm":
        return gemm_bf16(state["A"], state["B"], bias=state["bias"], out=state["out"])
    if state["kind"] == "mpnn":
        loss = state["net"].train_step(state["x"], state["t"], state["mask"], lr=1e-3)
        return dict(loss=np.float32(loss), theta=state["net"].get_params())
    sim = state["sim"]
    if state["kind"] == "box2d":
        for _ in range(state["steps"]):
            sim.step()
    else:
        sim.run(state["steps"])
    sim.sync()   # reports a run-away or timed-out step
    if state["kind"] != "batch":
        return _fields(sim, state["rho0"][0])
    return _join([_fields(sim.select(b), rho0) for b, rho0 in enumerate(state["rho0"])])


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def _counts(case):
    """(dim, fluid, solid, wall particles, solid sub-steps per coarse step), from the geometry."""
    k = case["kind"]
    if k == "box2d":
        return 2, case["nx"] * case["ny"] - 8, 32, 8 * (case["nx"] + case["ny"]), 2
    if k == "flag":
        n, r = case["cells_D"], case["ratio"]
        return 2, int(102.5 * n * n), int(1.485 * (n * r) ** 2), 200 * n, max(1, r)
    if k == "dam":
        p, r = case["dp_mm"], case["ratio"]
        return 2, int(14000 / p ** 2), int(405 * (r / p) ** 2), int(4222 / p), 12 * r
    if k == "valve":
        return 2, 12718, 288, 2560, 1
    if k == "batch":
        hi = case["nf_hi"]
        return 2, int(case["n"] * (hi - 2000) / math.log(hi / 2000)), 560 * case["n"], 2250 * case["n"], 8
    if k == "box3d":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        return 3, nx * ny * nz, 64 * int(round(0.6 * ny)), (nx + 8) * (ny + 6) * (nz + 8) - nx * (ny + 2) * nz, 3
    n = case["ny"]
    return 3, 3 * n ** 3, int(0.0646 * n ** 3), int(49.9 * n * n), 14


def work(case):
    if case["kind"] == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return dict(bytes=2 * (M * K + N * K) + 4 * M * N + (4 * N if case["bias"] else 0), flops=2 * M * N * K)
    if case["kind"] == "mpnn":
        N = int((316 + 80 * case["flag_len"]) * case["replicas"])
        P = WIDTH * FIN + LAYERS * WIDTH * 4 * WIDTH + NOUT * WIDTH
        # samples, targets and mask read, parameters and two moments read and written; forward and two backward products
        return dict(bytes=N * (4 * FIN + 4 * NOUT + 1) + 24 * P, flops=6 * N * P)
    D, nf, ns, nw, K = _counts(case)
    pairs_f, pairs_s = (20, 20) if D == 2 else (76, 66)
    # per coarse step: the fluid state read and written, wall positions and normals read, the solid state read and written
    fluid, solid = 8 * D + 4 * D + 8, 16 * D + 8 * D + 4 * (D * D + 2 * D)
    step = 2 * fluid * nf + 12 * D * nw + 2 * solid * ns
    # the state read back: fluid r, v, rho, rates; solid r, v, F, averages, force, normal
    out = nf * (8 * D + 4 * D + 8 + 4 + 4 * D) + ns * (24 * D + 8 * D * D + 12 * D)
    flops = nf * pairs_f * (55 + 30 + 4) + ns * K * (2 * pairs_s * 11 * (D - 1) + 80)
    return dict(bytes=case["steps"] * step + out, flops=case["steps"] * flops)


# --------------------------------------------------------------------------
# the same in 64 bits
# --------------------------------------------------------------------------

def _pairs(A, B, rc, lx, same):
    """All (i, j) with |A_i - B_j| < rc (minimal image in x of period lx when lx > 0), by a cell grid."""
    dev, D = A.device, A.shape[1]
    empty = torch.zeros(0, dtype=torch.int64, device=dev)
    if len(A) == 0 or len(B) == 0:
        return empty, empty
    lo = torch.minimum(A.min(0).values, B.min(0).values)
    hi = torch.maximum(A.max(0).values, B.max(0).values)
    if lx > 0:
        lo[0], hi[0] = 0.0, lx
    nc = torch.clamp(((hi - lo) / rc).floor(), min=1).long()
    edge = (hi - lo) / nc
    edge = torch.where(edge > 0, edge, torch.ones_like(edge))
    if lx > 0 and nc[0] < 3:
        raise ValueError("a periodic period needs at least three cells")

    def cells(X):
        return torch.minimum(torch.clamp(((X - lo) / edge).floor().long(), min=0), nc - 1)

    mul = torch.ones_like(nc)
    for k in range(1, D):
        mul[k] = mul[k - 1] * nc[k - 1]
    key, order = torch.sort((cells(B) * mul).sum(1))
    start = torch.searchsorted(key, torch.arange(int(nc.prod()) + 1, device=dev))
    offs = torch.cartesian_prod(*[torch.arange(-1, 2, device=dev)] * D)
    I, J = [], []
    for a0 in range(0, len(A), 1 << 20):
        Ac = A[a0:a0 + (1 << 20)]
        ca = cells(Ac)
        for o in offs:
            c = ca + o
            if lx > 0:
                c[:, 0] %= nc[0]
            ok = ((c >= 0) & (c < nc)).all(1)
            i = ok.nonzero()[:, 0]
            kc = (c[i] * mul).sum(1)
            cnt = start[kc + 1] - start[kc]
            ii = torch.repeat_interleave(i, cnt)
            first = torch.repeat_interleave(start[kc] - (torch.cumsum(cnt, 0) - cnt), cnt)
            jj = order[torch.arange(len(ii), device=dev) + first]
            d = Ac[ii] - B[jj]
            if lx > 0:
                d[:, 0] -= lx * torch.round(d[:, 0] / lx)
            keep = (d * d).sum(1) < rc * rc
            if same:
                keep &= ii + a0 != jj
            I.append(ii[keep] + a0)
            J.append(jj[keep])
    return torch.cat(I), torch.cat(J)


class _Exact:
    """One problem advanced in 64 bits: momentum, continuity, ghost coupling, reinitialisation and solid sub-steps
    pair by pair at the positions of the step (or at those of the last rebuild when they are held)."""

    CHUNK = 1 << 23

    def __init__(self, c, mode, cadence):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        T = lambda a: torch.as_tensor(np.asarray(a, np.float64), device=dev)  # noqa: E731
        self.c, self.mode, self.cadence, D = c, mode, cadence, c.dim
        self.g = T(c.gravity[:D])
        self.fr, self.fv = T(c.f_r).clone(), T(c.f_v).clone()
        self.B = c.f_rho0 * c.f_c0 ** 2 / 7
        self.rho = c.f_rho0 * (T(c.f_p) / self.B + 1) ** (1 / 7)
        self.rate, self.acc = torch.zeros_like(self.rho), torch.zeros_like(self.fv)
        self.wr, self.wn = T(c.w_r), T(c.w_n)
        self.free = T(c.s_cons) == 0
        self.sr0, self.sn0 = T(c.s_r0), T(c.s_n0)
        self.sr, self.sv, self.sn = self.sr0.clone(), T(c.s_v0) * self.free[:, None], self.sn0.clone()
        self.vbar, self.abar = self.sv.clone(), torch.zeros_like(self.sv)
        self.force = torch.zeros_like(self.sv)
        self.F = torch.eye(D, dtype=torch.float64, device=dev).repeat(c.ns, 1, 1)
        self.hF, self.hS = 1.3 * c.f_dp, 1.3 * c.s_dp
        self.mF, self.VW, self.VS = c.f_rho0 * c.f_dp ** D, c.w_dp ** D, c.s_dp ** D
        self.lx = c.Lx if c.periodic_x else 0.0
        self.mu = c.s_E / (2 * (1 + c.s_nu))
        self.lam = 2 * self.mu * c.s_nu / (1 - 2 * c.s_nu)
        self.cS = math.sqrt(c.s_E / (3 * (1 - 2 * c.s_nu)) / c.s_rho0)
        if c.ns:
            self.sa, self.sb = _pairs(self.sr0, self.sr0, 2 * self.hS, 0.0, True)
            d = self.sr0[self.sa] - self.sr0[self.sb]
            r = d.norm(dim=1)
            self.sg = self.VS * (self.dW(r, self.hS) / r)[:, None] * d
            self.B0 = torch.linalg.inv(self.rows(c.ns, self.sa, -d[:, :, None] * self.sg[:, None, :]))
        n = np.arange(-3, 4) * c.f_dp
        lat = np.stack(np.meshgrid(*[n] * D), -1).reshape(-1, D)
        self.sigma0 = float(self.W(T(np.linalg.norm(lat, axis=1)), self.hF).sum())
        self.t, self.k = 0.0, 0
        speed = lambda v: float(v.norm(dim=1).max()) if len(v) else 0.0  # noqa: E731
        self.vF, self.vS, self.aS = speed(self.fv), speed(self.sv), 0.0

    # Wendland C2
    def alpha(self, h):
        return 7 / (4 * math.pi * h * h) if self.c.dim == 2 else 21 / (16 * math.pi * h ** 3)

    def W(self, r, h):
        a = torch.clamp(1 - 0.5 * r / h, min=0)
        return self.alpha(h) * a ** 4 * (1 + 2 * r / h)

    def dW(self, r, h):
        a = torch.clamp(1 - 0.5 * r / h, min=0)
        return -5 * self.alpha(h) / h * (r / h) * a ** 3

    @staticmethod
    def rows(n, i, v):
        return torch.zeros((n,) + tuple(v.shape[1:]), dtype=v.dtype, device=v.device).index_add_(0, i, v)

    def eos(self, rho):
        return self.B * ((rho / self.c.f_rho0) ** 7 - 1)

    def steps_of_time(self):
        c = self.c
        ac = 0.6 * self.hF / (c.f_c0 + self.vF)
        ds = 1e300
        if c.ns:
            ds = 0.6 * min(self.hS / (self.cS + self.vS), math.sqrt(self.hS / self.aS) if self.aS > 0 else 1e300)
        if self.mode == "single_solid":
            return min(ac, ds), 1
        return ac, (int(math.floor(ac / ds)) + 1 if c.ns else 1)

    def inflow(self, r):
        c = self.c
        U, H = c.inflow_U, c.inflow_H
        y = torch.clamp(r[:, 1] - c.inflow_y0, 0, H)
        if c.inflow_profile == 2:
            w, b = 2 * math.pi / c.inflow_period, c.inflow_wo / math.sqrt(2)
            s = 2 * y / H - 1
            p, q = b * (1 + s), b * (1 - s)
            g = math.cosh(2 * b) + math.cos(2 * b)
            return U / (w * g) * ((p.sinh() * q.sin() + q.sinh() * p.sin()) * math.cos(w * self.t)
                                  + (g - p.cosh() * q.cos() - q.cosh() * p.cos()) * math.sin(w * self.t))
        u = 6 * U * y * (H - y) / H ** 2
        if c.inflow_profile == 3:
            z = torch.clamp(r[:, 2] - c.inflow_z0, 0, c.inflow_Hz)
            u = u * 6 * z * (c.inflow_Hz - z) / c.inflow_Hz ** 2
        return u

    def drift(self, dt):
        self.rho = self.rho + 0.5 * dt * self.rate
        self.fr = self.fr + 0.5 * dt * self.fv
        if self.lx:
            x = self.fr[:, 0]
            x = torch.where(x >= self.c.x_lo + self.lx, x - self.lx, torch.where(x < self.c.x_lo, x + self.lx, x))
            self.fr[:, 0] = x

    def over(self, ij, Rj):
        """Chunks (i, j, d, r) of a pair list between the fluid and another set, at the pair geometry."""
        for q in range(0, len(ij[0]), self.CHUNK):
            i, j = ij[0][q:q + self.CHUNK], ij[1][q:q + self.CHUNK]
            d = self.gf[i] - Rj[j]
            if self.lx:
                d[:, 0] -= self.lx * torch.round(d[:, 0] / self.lx)
            yield i, j, d, d.norm(dim=1)

    def boundary(self, solid):
        if solid:
            return self.FS, self.gs, self.vbar, self.abar, self.sn, self.VS
        z = torch.zeros_like(self.wr)
        return self.FW, self.wr, z, z, self.wn, self.VW

    def ghost(self, i, a, d, p, ab, n):
        gn = ((self.g - ab[a]) * n[a]).sum(1)
        pd = p[i] + self.rho[i] * torch.clamp(-gn, min=0) * torch.clamp((d * n[a]).sum(1), min=0)
        return pd, self.c.f_rho0 * (pd / self.B + 1) ** (1 / 7)

    def step(self):
        c, D, hF = self.c, self.c.dim, self.hF
        nf = len(self.fr)
        dt, K = self.steps_of_time()
        if c.inflow_on:
            inb = (self.fr[:, 0] >= c.x_lo) & (self.fr[:, 0] < c.x_lo + c.inflow_width)
            u = torch.zeros_like(self.fv)
            u[:, 0] = self.inflow(self.fr)
            self.fv = torch.where(inb[:, None], u, self.fv)
        self.drift(dt)
        if self.k % self.cadence == 0:
            self.gf, self.gs = self.fr.clone(), self.sr.clone()
            rc = 2 * hF
            self.FF = _pairs(self.gf, self.gf, rc, self.lx, True)
            self.FW = _pairs(self.gf, self.wr, rc, self.lx, False)
            self.FS = _pairs(self.gf, self.gs, rc, self.lx, False)
        if c.n_reinit and self.k % c.n_reinit == 0:
            s = self.W(torch.zeros(1, dtype=torch.float64, device=self.fr.device), hF).repeat(nf)
            for ij, R, f in ((self.FF, self.gf, 1.0), (self.FW, self.wr, self.VW / c.f_dp ** D),
                             (self.FS, self.gs, self.VS / c.f_dp ** D)):
                for i, j, d, r in self.over(ij, R):
                    s.index_add_(0, i, f * self.W(r, hF))
            self.rho = c.f_rho0 * s / self.sigma0
            if c.free_surface:
                self.rho = torch.clamp(self.rho, min=c.f_rho0)
            if c.ns:
                n = torch.einsum("nji,nj->ni", torch.linalg.inv(self.F), self.sn0)
                self.sn = n / n.norm(dim=1, keepdim=True)
        p, rho, v = self.eos(self.rho), self.rho, self.fv
        V = self.mF / rho
        a = torch.zeros_like(v)
        for i, j, d, r in self.over(self.FF, self.gf):
            w = self.dW(r, hF) / r
            UL, UR = -(v[i] * d).sum(1) / r, -(v[j] * d).sum(1) / r
            du = UL - UR
            beta = torch.clamp(3 * torch.clamp(du, min=0), max=c.f_c0)
            ps = 0.5 * (p[i] + p[j]) + 0.25 * (rho[i] + rho[j]) * beta * du
            a.index_add_(0, i, (V[j] * w)[:, None] * (-2 * ps[:, None] * d + 2 * c.f_eta * (v[i] - v[j])))
        self.force = torch.zeros_like(self.sv)
        for solid in (False, True):
            ij, R, vb, ab, n, Va = self.boundary(solid)
            for i, b, d, r in self.over(ij, R):
                pd, rd = self.ghost(i, b, d, p, ab, n)
                w = self.dW(r, hF)
                pb = (p[i] * rd + pd * rho[i]) / (rho[i] + rd)
                f = Va * ((-2 * pb * w / r)[:, None] * d
                          + (4 * c.f_eta * w / (r + 0.01 * hF))[:, None] * (v[i] - vb[b]))
                a.index_add_(0, i, f)
                if solid:
                    self.force.index_add_(0, b, -V[i][:, None] * f)
        self.acc = a / rho[:, None] + self.g
        self.fv = v = v + dt * self.acc
        self.vF = float(v.norm(dim=1).max())
        rate = torch.zeros_like(rho)
        for i, j, d, r in self.over(self.FF, self.gf):
            du = -((v[i] - v[j]) * d).sum(1) / r
            diff = 0.5 * du - (p[i] - p[j]) / ((rho[i] + rho[j]) * c.f_c0)
            rate.index_add_(0, i, -V[j] * self.dW(r, hF) * diff)
        for solid in (False, True):
            ij, R, vb, ab, n, Va = self.boundary(solid)
            for i, b, d, r in self.over(ij, R):
                pd, rd = self.ghost(i, b, d, p, ab, n)
                du = -((v[i] - vb[b]) * d).sum(1) / r
                diff = du + (pd - p[i]) / ((rho[i] + rd) * c.f_c0)
                rate.index_add_(0, i, -Va * self.dW(r, hF) * diff)
        self.rate = 2 * rho * rate
        self.drift(dt)
        if c.ns:
            self.solid(dt, K)
        self.t, self.k = self.t + dt, self.k + 1

    def F_rate(self):
        M = self.rows(self.c.ns, self.sa, (self.sv[self.sb] - self.sv[self.sa])[:, :, None] * self.sg[:, None, :])
        return M @ self.B0

    def solid(self, dt, K):
        c, h = self.c, dt / K
        eye = torch.eye(c.dim, dtype=torch.float64, device=self.sr.device)
        free = self.free[:, None]
        r0, v0 = self.sr.clone(), self.sv.clone()
        Fd, vmax, amax = self.F_rate(), 0.0, 0.0
        for _ in range(K):
            self.F = self.F + 0.5 * h * Fd
            self.sr = self.sr + 0.5 * h * self.sv * free
            Ci = torch.linalg.inv(self.F.mT @ self.F)
            lnJ = torch.log(torch.linalg.det(self.F))[:, None, None]
            P = self.F @ (self.mu * (eye - Ci) + self.lam * lnJ * Ci)
            Q = P @ self.B0
            f = self.rows(c.ns, self.sa, ((Q[self.sa] + Q[self.sb]) @ self.sg[:, :, None])[:, :, 0])
            acc = (f / c.s_rho0 + self.force / (c.s_rho0 * self.VS) + self.g) * free
            self.sv = self.sv + h * acc
            amax, vmax = max(amax, float(acc.norm(dim=1).max())), max(vmax, float(self.sv.norm(dim=1).max()))
            Fd = self.F_rate()
            self.F = self.F + 0.5 * h * Fd
            self.sr = self.sr + 0.5 * h * self.sv * free
        self.vbar, self.abar = (self.sr - r0) / dt, (self.sv - v0) / dt
        self.vS, self.aS = vmax, amax

    def fields(self):
        o = dict(f_r=self.fr, f_v=self.fv, f_drho=self.rho - self.c.f_rho0, f_rate=self.rate, f_acc=self.acc,
                 s_r=self.sr, s_v=self.sv, s_F=self.F, s_vbar=self.vbar, s_abar=self.abar, s_force=self.force,
                 s_n=self.sn)
        return {k: t.cpu().numpy() for k, t in o.items()}


def _exact_training_step(case, seed):
    (ptr, idx, w, g), rows, theta, x, t, mask = _network(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    T = lambda a: torch.as_tensor(np.asarray(a, np.float64), device=dev)  # noqa: E731
    n, R = len(ptr) - 1, case["replicas"]
    rep = lambda a: torch.cat([torch.as_tensor(a, device=dev) + r * n for r in range(R)])  # noqa: E731
    i, j, coef = rep(rows), rep(idx), [T(w).repeat(R)] + [T(g[:, k]).repeat(R) for k in range(2)]
    th = T(theta).requires_grad_()
    parts, o = [], 0
    for out, inp in [(WIDTH, FIN)] + [(WIDTH, 4 * WIDTH)] * LAYERS + [(NOUT, WIDTH)]:
        parts.append((th[o:o + out * inp].reshape(out, inp), th[o + out * inp:o + out * inp + out]))
        o += out * inp + out
    silu = torch.nn.functional.silu
    h = silu(T(x) @ parts[0][0].T + parts[0][1])
    for W, b in parts[1:-1]:
        d = h[j] - h[i]
        z = torch.cat([h] + [torch.zeros_like(h).index_add(0, i, k[:, None] * d) for k in coef], 1)
        h = h + silu(z @ W.T + b)
    out = h @ parts[-1][0].T + parts[-1][1]
    m = T(mask)
    loss = (((out[:, :4] - T(t)[:, :4]) * m[:, None]) ** 2).sum() / m.sum()
    gr, = torch.autograd.grad(loss, th)
    # the first Adam step: both bias-corrected moments are the gradient's own
    new = th - 1e-3 * gr / (gr.abs() + 1e-8)
    return dict(loss=float(loss.detach()), theta=new.detach().cpu().numpy())


def exact(case, seed):
    if case["kind"] == "gemm":
        A, B, bias = _matrices(case, seed)
        C = A.double() @ B.double().T
        return C if bias is None else C + bias.double()
    if case["kind"] == "mpnn":
        return _exact_training_step(case, seed)
    mode = "single_solid" if case["kind"] == "valve" else "multiple"
    done = []
    for c in _problems(case, seed):
        e = _Exact(c, mode, case.get("cadence", 1))
        for _ in range(case["steps"]):
            e.step()
        done.append(e.fields())
    return _join(done) if case["kind"] == "batch" else done[0]
