"""Performance cases of the lattice Boltzmann library: what its users run.

Four kinds of program, each through the public entry points of the Python binding:

* ``advance``: a program keeps a handle and alternates ``lb_ks_step`` with reading the
  density (and, for long-time statistics, the energies) of every run;
* ``solve``: a job per batch, ``lb_ks_batch_init`` from host memory, the steps, the
  density back to host memory, ``lb_ks_free``;
* ``front``: the paper's travelling front with fixed-value ends, the batch of one time
  step of the stability map (every spacing and relaxation time at once), as a ``solve``;
* ``collapse``: ``advance`` at tau = 1 with the density-only kernel.

Periodic lattices have lengths log-uniform in [nmin, nmax] (the same for every seed) and
start from 16 low Fourier modes with random amplitudes and phases, the very long ones
from 64 modes in the band the equation amplifies; relaxation times are uniform in
[tau_lo, tau_hi], spacings in [dx, (1 + spread) dx].
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1711_03540_gb300 as lb

PRECISION = {"f64": lb.F64, "f32": lb.F32, "f16s": lb.F16S}
KERNEL = {"auto": lb.KERNEL_AUTO, "stream": lb.KERNEL_STREAM, "collapse": lb.KERNEL_COLLAPSE}
STORED_BYTES = {"f64": 8, "f32": 4, "f16s": 2}

# The travelling front of the paper's Table 5.
FRONT_L, FRONT_B = 60.0, 3.0
FRONT_K = 0.5 * math.sqrt(11.0 / 19.0)
FRONT_A = 15.0 / 19.0 * math.sqrt(11.0 / 19.0)
FRONT_LEFT = FRONT_B - 30.0 / 19.0 * math.sqrt(11.0 / 19.0)
FRONT_RIGHT = 2.0 * FRONT_B - FRONT_LEFT


def _case(name, kind, scheme, precision, nruns, nmin, nmax, dx, dt, tau_lo, tau_hi, steps, kernel="auto",
          recentre=0, energy=False, out="host", modes=16, spread=0.0):
    c = {"kind": kind, "scheme": scheme, "precision": precision, "nruns": nruns, "nmin": nmin, "nmax": nmax,
         "dx": dx, "dt": dt, "tau_lo": tau_lo, "tau_hi": tau_hi, "steps": steps, "kernel": kernel,
         "recentre": recentre, "energy": energy, "out": out, "modes": modes,
         "spread": spread}
    if name:
        c["name"] = name
    return c


def listed():
    l32 = 32.0 * math.pi
    return [
        # One small lattice in the defaults, the paper's L = 32 pi box with D1Q5: the smallest
        # long-running job; a step is all latency.
        _case("one_512_d1q5_f64", "advance", 5, "f64", 1, 512, 512, l32 / 512, 5e-5, 1.0, 1.0, 1000),
        # One finely resolved lattice in the defaults (D1Q7, T = 150 takes 3e7 such steps).
        _case("one_4096_d1q7_f64", "advance", 7, "f64", 1, 4096, 4096, l32 / 4096, 5e-6, 3.0, 3.0, 1000),
        # A first try or a parity check: three tiny lattices of odd length, created, stepped, read, freed.
        _case("tiny_3_d1q7_f64", "solve", 7, "f64", 3, 61, 161, 0.1, 1e-4, 1.5, 3.0, 200),
        # The FP64 reference of a small parameter study with the original scheme.
        _case("batch_200_d1q5_f64", "advance", 5, "f64", 200, 200, 2000, 0.1, 1e-4, 1.5, 3.0, 400),
        # The FP64 reference run of the full ensemble of uneven lattices.
        _case("ensemble_4096_d1q7_f64", "advance", 7, "f64", 4096, 256, 8192, 0.1, 1e-4, 1.5, 3.0, 64, out="device"),
        # One time step of the stability and accuracy map: two spacings x 61 relaxation times.
        _case("front_122_d1q7_f64", "front", 7, "f64", 122, 301, 601, 0.1, 1e-4, 1.5, 2.4, 1000),
        # The benchmark ensemble as a job: host density in, 1000 FP32 steps with the guard, host density out.
        _case("ensemble_4096_d1q7_f32", "solve", 7, "f32", 4096, 256, 8192, 0.1, 1e-4, 1.5, 3.0, 1000, recentre=500),
        # A handful of lattices of the same kind: far too few to fill the chip one block each.
        _case("batch_24_d1q7_f32", "advance", 7, "f32", 24, 256, 8192, 0.1, 1e-4, 1.5, 3.0, 1000, recentre=500),
        # Long-time statistics in scaled FP16: 1000 steps, then the energies and a snapshot.
        _case("chaos_1024_d1q7_f16s", "advance", 7, "f16s", 1024, 220, 4000, 0.05, 1e-4, 3.0, 3.0, 1000,
              recentre=500, energy=True, spread=1.0),
        # One very long lattice, default kernel choice.
        _case("long_2p24_d1q7_f32", "advance", 7, "f32", 1, 1 << 24, 1 << 24, 0.1, 1e-4, 1.51, 1.51, 320,
              recentre=500, out="device", modes=64),
        # The same in scaled FP16 on the streaming kernel (a state read and written once per step).
        _case("long_2p24_d1q7_f16s_stream", "advance", 7, "f16s", 1, 1 << 24, 1 << 24, 0.1, 1e-4, 1.51, 1.51, 100,
              kernel="stream", out="device", modes=64),
        # The ensemble at tau = 1 on the density-only kernel.
        _case("collapse_4096_d1q7_f32", "collapse", 7, "f32", 4096, 256, 8192, 0.2, 5e-5, 1.0, 1.0, 1000,
              kernel="collapse", recentre=500, out="device", spread=0.05),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["advance", "advance", "advance", "solve", "front", "collapse"])
    scheme = rng.choice([5, 7, 7])
    if kind == "front":
        ntau = rng.randint(5, 61)
        return _case(None, "front", scheme, "f64", 2 * ntau, 301, 601, 0.1, rng.choice([2e-5, 5e-5, 1e-4]), 1.5,
                     rng.uniform(1.9, 2.4), _log_int(rng, 100, 1000))
    if kind == "collapse":
        precision, kernel = rng.choice(["f32", "f64"]), "collapse"
        dx, dt, tau_lo, tau_hi = 0.2, 5e-5, 1.0, 1.0
    else:
        precision, kernel = rng.choice(["f64", "f64", "f32", "f32", "f16s"]), "auto"
        dx, dt, tau_lo, tau_hi = rng.choice([(0.1, 1e-4, 1.5, 3.0), (0.0625, 1e-4, 3.0, 3.0), (0.1, 5e-5, 1.6, 2.6)])
    # at most what a few tens of milliseconds of the slowest path hold
    most = 4e8 if precision == "f64" else 4e9
    nruns = _log_int(rng, 1, 4096)
    nmin = _log_int(rng, 16, 2000)
    nmax = _log_int(rng, nmin, max(nmin, min(8192, 1.2e7 / nruns)))
    if nruns == 1 and precision != "f64" and kind == "advance" and rng.random() < 0.5:
        nmin = nmax = _log_int(rng, 1 << 16, 1 << 24)
    steps = int(min(_log_int(rng, 100, 1000), max(20.0, most / (nruns * 0.5 * (nmin + nmax)))))
    # a snapshot wanted by more GPU work stays on the device, the others go to the host
    return _case(None, kind, scheme, precision, nruns, nmin, nmax, dx, dt, tau_lo, tau_hi, steps, kernel,
                 0 if precision == "f64" else 500, rng.random() < 0.3 and kind != "solve",
                 "host" if kind == "solve" else rng.choice(["host", "device"]), spread=0.05)


# ---------------------------------------------------------------- inputs


def _lengths(case):
    if case["kind"] == "front":  # half the runs at dx, half at 2 dx: nodes on [0, 60], both ends included
        half = case["nruns"] // 2
        return np.array([case["nmax"]] * half + [case["nmin"]] * (case["nruns"] - half), dtype=np.int64)
    g = np.random.Generator(np.random.PCG64(20171109 + case["nruns"]))
    u = g.uniform(math.log(case["nmin"]), math.log(case["nmax"]), case["nruns"])
    return np.maximum(7, np.round(np.exp(u))).astype(np.int64)


def _inputs(case, seed):
    """(N, L, dt, tau) as numpy arrays and rho0 as a device tensor, all from the seed."""
    N = _lengths(case)
    R = case["nruns"]
    g = np.random.Generator(np.random.PCG64(seed))
    dt = np.full(R, float(case["dt"]))
    dev = torch.device("cuda")
    if case["kind"] == "front":
        half = R // 2
        taus = np.linspace(case["tau_lo"], case["tau_hi"], half)
        tau = np.concatenate([taus, taus[: R - half]]) + g.uniform(0.0, 0.01)
        L = np.full(R, FRONT_L)
        x0 = FRONT_L / 3.0 + g.uniform(-1.0, 1.0)
        parts = []
        for n in N:
            z = np.tanh(FRONT_K * (np.arange(n) * (FRONT_L / (n - 1)) - x0))
            parts.append(FRONT_B + FRONT_A * (-9.0 * z + 11.0 * z ** 3))
        return N, L, dt, tau, torch.from_numpy(np.concatenate(parts)).to(dev)
    L = N * (float(case["dx"]) * (1.0 + g.uniform(0.0, case["spread"], R)))
    tau = g.uniform(case["tau_lo"], case["tau_hi"], R) if case["tau_hi"] > case["tau_lo"] else np.full(R, case["tau_lo"])
    modes = case["modes"]
    amp = g.uniform(0.0, 1e-2, (modes, R))
    phase = g.uniform(0.0, 2 * math.pi, (modes, R))
    if modes > 16:  # wavenumbers up to 1.2
        m = np.stack([g.choice(np.arange(1, int(1.2 * l / (2 * math.pi)) + 1), modes, replace=False) for l in L], 1)
    else:
        m = np.repeat(np.arange(1, modes + 1)[:, None], R, 1)
    Nd = torch.from_numpy(N).to(dev)
    run = torch.repeat_interleave(torch.arange(R, device=dev), Nd)
    off = torch.cumsum(Nd, 0) - Nd
    x = torch.arange(run.numel(), device=dev) - off[run]
    n = Nd[run]
    rho0 = torch.zeros(run.numel(), dtype=torch.float64, device=dev)
    am, ph, mm = torch.from_numpy(amp).to(dev).float(), torch.from_numpy(phase).to(dev).float(), torch.from_numpy(m).to(dev)
    for k in range(modes):  # the phase m x / N reduced exactly, then single precision
        a, p, q = (v[k][run] if R > 1 else v[k, 0] for v in (am, ph, mm))
        turn = torch.remainder(q * x, n).double() / n
        rho0 += a * torch.cos((2 * math.pi * turn).float() + p)
    return N, L, dt, tau, rho0


class _State:
    """A program's handle and buffers."""

    handle = None

    def __del__(self):
        if self.handle:
            lb.lb_ks_free(self.handle)


def prepare(case, seed):
    N, L, dt, tau, rho0 = _inputs(case, seed)
    s = _State()
    s.case, s.N, s.L, s.dt, s.tau = case, N, L, dt, tau
    s.opts = lb.lb_ks_default_opts(precision=PRECISION[case["precision"]], kernel=KERNEL[case["kernel"]],
                                   recentre_every=case["recentre"])
    total = int(N.sum())
    s.energy = np.empty(len(N)) if case["energy"] else None
    if case["kind"] in ("solve", "front"):
        s.rho0 = rho0.cpu().pin_memory()
        s.rho = torch.empty(total, dtype=torch.float64, pin_memory=True)
        if case["kind"] == "front":
            s.left, s.right = np.full(len(N), FRONT_LEFT), np.full(len(N), FRONT_RIGHT)
    else:
        s.rho = torch.empty(total, dtype=torch.float64, device="cuda") if case["out"] == "device" else np.empty(total)
        torch.cuda.synchronize()
        s.handle = lb.lb_ks_batch_init(case["scheme"], N, L, dt, tau, rho0, s.opts)
    return s


def run(s):
    c = s.case
    if c["kind"] in ("solve", "front"):
        if c["kind"] == "front":
            h = lb.lb_ks_batch_init_reservoir(c["scheme"], s.N, s.L, s.dt, s.tau, s.rho0, s.left, s.right, s.opts)
        else:
            h = lb.lb_ks_batch_init(c["scheme"], s.N, s.L, s.dt, s.tau, s.rho0, s.opts)
        try:
            lb.lb_ks_step(h, c["steps"])
            lb.lb_ks_rho(h, s.rho)
        finally:
            lb.lb_ks_free(h)
        return {"rho": s.rho}
    lb.lb_ks_step(s.handle, c["steps"])
    got = {}
    if s.energy is not None:
        lb.lb_ks_mass_energy(s.handle, None, s.energy)
        got["energy"] = s.energy
    lb.lb_ks_rho(s.handle, s.rho)
    got["rho"] = s.rho
    return got


def work(case):
    sites = float(_lengths(case).sum())
    planes = 1 if case["kind"] == "collapse" else case["scheme"]
    # multiplies and adds of one site's step, a fused multiply-add as two
    flops = {("collapse", 5): 21, ("collapse", 7): 31}.get((case["kind"], case["scheme"]),
                                                          27 if case["scheme"] == 5 else 39)
    state = planes * STORED_BYTES[case["precision"]] * sites
    # a kept handle's populations read once and written once, or a job's density in; the density out
    first = 8 * sites if case["kind"] in ("solve", "front") else 2 * state
    per_step = 2 * state * case["steps"] if case["kernel"] == "stream" else first
    return {"bytes": per_step + 8 * sites, "flops": flops * sites * case["steps"]}


# ---------------------------------------------------------------- the method in plain FP64


def _weights(Q):
    w = {0: [1, 0, 0, 0, 0], 1: [0, 2 / 3, -2 / 3, -1 / 12, 1 / 12], 2: [-5 / 4, 2 / 3, 2 / 3, -1 / 24, -1 / 24],
         4: [1 / 4, -1 / 6, -1 / 6, 1 / 24, 1 / 24]}
    w = {k: v + [0] * (Q - 5) for k, v in w.items()}
    w[6] = [-1 / 36, 1 / 48, 1 / 48, -1 / 120, -1 / 120, 1 / 720, 1 / 720][:Q]
    return w


def _equilibrium(Q, dx, dt, tau):
    """A_i, B_i of f^eq_i = A_i rho + B_i rho^2, arrays [Q, runs] (Sec. 2, Table 2)."""
    t2 = 2 * tau ** 2 - tau
    t3 = 6 * tau ** 3 - 6 * tau ** 2 + tau
    t4 = (tau - 1) * (24 * tau ** 3 - 12 * tau ** 2 + 2 * tau + 1) + 1
    J = dt / (2 * dx)
    K = -2 * dt * tau / (dx ** 2 * t2)
    M = -24 * dt * tau / (dx ** 4 * t4)
    E = 0 * M
    if Q == 7:
        E = 120 * tau * dt / (t4 * dx ** 4)
        M = M - 24 * dt ** 2 * tau / (dx ** 4 * t4) * (t2 / (2 * tau) - t3 / t2)
    w = _weights(Q)
    A = np.stack([w[0][i] + K * w[2][i] + M * w[4][i] + E * w[6][i] for i in range(Q)])
    B = np.stack([J * w[1][i] for i in range(Q)])
    return A, B


def exact(case, seed):
    N, L, dt, tau, rho0 = _inputs(case, seed)
    dev, Q = rho0.device, case["scheme"]
    front = case["kind"] == "front"
    C = (Q - 1) // 2
    ghost = C if front else 0
    A, B = _equilibrium(Q, L / (N - 1 if front else N), dt, tau)
    Nd = torch.from_numpy(N).to(dev)
    W = Nd + 2 * ghost  # sites of a run with its ghost nodes
    run_of = torch.repeat_interleave(torch.arange(len(N), device=dev), W)
    off = (torch.cumsum(W, 0) - W)[run_of]
    x = torch.arange(run_of.numel(), device=dev) - off - ghost
    n = Nd[run_of]
    if front:
        first = torch.cumsum(Nd, 0) - Nd
        rho = rho0[first[run_of] + x.clamp(min=0).minimum(n - 1)]
        rho = torch.where(x <= 0, FRONT_LEFT, torch.where(x >= n - 1, FRONT_RIGHT, rho))
        fixed = (x <= 0) | (x >= n - 1)
    else:
        rho = rho0
    At, Bt = (torch.from_numpy(v).to(dev) for v in (A, B))
    w = torch.from_numpy(1.0 / tau).to(dev)[run_of]
    speeds = [0, 1, -1, 2, -2, 3, -3][:Q]
    src = []
    for c in speeds:
        y = x - c
        y = y.clamp(min=-ghost).minimum(n - 1 + ghost) if front else torch.remainder(y, n)
        src.append((off + ghost + y).to(torch.int32))
    f = [At[i][run_of] * rho + Bt[i][run_of] * rho * rho for i in range(Q)]
    held = [v[fixed] for v in f] if front else None
    if len(N) == 1:  # one lattice: the constants are numbers
        w = float(1.0 / tau[0])
        Aw, Bw = [float(v) * w for v in A[:, 0]], [float(v) * w for v in B[:, 0]]
    else:
        Aw, Bw = [At[i][run_of] * w for i in range(Q)], [Bt[i][run_of] * w for i in range(Q)]
    for _ in range(case["steps"]):
        rho = f[0].clone()
        for v in f[1:]:
            rho += v
        rho2 = rho * rho
        f = [torch.index_select(v + (Aw[i] * rho + Bw[i] * rho2 - w * v), 0, src[i]) for i, v in enumerate(f)]
        if front:
            for v, b in zip(f, held):
                v[fixed] = b
    rho = sum(f[1:], f[0])
    if front:
        rho = rho[(x >= 0) & (x < n)]
    got = {"rho": rho}
    if case["energy"]:
        got["energy"] = torch.zeros(len(N), dtype=torch.float64, device=dev).index_add_(0, run_of, rho * rho).cpu().numpy()
    if case["out"] == "host":
        got["rho"] = rho.cpu() if case["kind"] in ("solve", "front") else rho.cpu().numpy()
    return got
