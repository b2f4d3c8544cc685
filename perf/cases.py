"""The work that a user of this framework has it do, as measurable cases.

Each case is one pass through the public entry points: a device advanced and
read back, a closed loop of short calls, a batch of uneven devices, a gradient
pass, a whole fit evaluation, the torch.autograd front end, and the sweep on
caller-owned memory.  ``prepare`` makes what the user's program holds before
the call, ``run`` is the call, ``work`` the bytes and operations that it cannot
do without, and ``exact`` the gradient outputs in plain numpy.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_2511_09413_gb300 import kmc as K
from paper_2511_09413_gb300 import workloads as W

# Hop base probabilities at Ea = 0.40 eV, 300 K, 1e12 Hz: P0 = 3.8e-4 at
# dt = 1e-9 s (moves are rare) and 0.17 at dt = 5e-7 s (moves in every step).
DT_RARE, DT_DENSE = 1e-9, 5e-7


def listed():
    return [
        # A program that reacts to what it reads: sets the next ten voltages,
        # advances ten steps and reads the traces.  The smallest calls.
        dict(name="control_loop_64x100", kind="loop", rails=64, sites=100, zones=10, open=False,
             barriers=False, fill=0.125, dt=DT_RARE, rule=0, protocol="pulse", steps=10),
        # The plain small device (64 rails x 100 sites), a thousand steps per
        # call: one warp's latency per step.
        dict(name="relaxation_64x100", kind="steps", rails=64, sites=100, zones=10, open=False,
             barriers=False, fill=0.125, dt=DT_RARE, rule=0, protocol="pulse", steps=1000),
        # A device of the published timing table's size (16,000 rails x 200
        # sites), blocking, rare moves.
        dict(name="relaxation_16000x200", kind="steps", rails=16000, sites=200, zones=10, open=False,
             barriers=False, fill=0.25, dt=DT_RARE, rule=0, protocol="pulse", steps=1000),
        # The benchmark device: open electrodes, a barrier per site, triangular
        # sweep.  The largest.
        dict(name="hysteresis_65536x1024", kind="steps", rails=65536, sites=1024, zones=10, open=True,
             barriers=True, fill=0.25, dt=DT_RARE, rule=0, protocol="triangle", steps=5000),
        # Sixteen replicas of the adjoint device (4,096 x 512), moves in every
        # step.
        dict(name="replicas_65536x512", kind="steps", rails=65536, sites=512, zones=10, open=False,
             barriers=False, fill=0.2, dt=DT_DENSE, rule=0, protocol="pulse", steps=1600),
        # The longest rails with the most zones, half full, open electrodes.
        dict(name="long_rails_2500x2048", kind="steps", rails=2500, sites=2048, zones=32, open=True,
             barriers=False, fill=0.5, dt=DT_DENSE, rule=0, protocol="triangle", steps=1500),
        # The even/odd-bond update rule.
        dict(name="brick_wall_8192x1000", kind="steps", rails=8192, sites=1000, zones=10, open=False,
             barriers=False, fill=0.3, dt=DT_DENSE, rule=1, protocol="pulse", steps=1500),
        # The sweep on caller-owned device memory, odd sizes, open electrodes.
        dict(name="caller_owned_3001x777", kind="noalloc", rails=3001, sites=777, zones=7, open=True,
             barriers=False, fill=0.25, dt=DT_RARE, rule=0, protocol="triangle", steps=2000),
        # Spike-timing devices of uneven sizes advanced together.
        dict(name="spike_batch_32", kind="batch", devices=32, sizes=7, steps=1000),
        # Backward pass of four replicas of the adjoint device, weights on the
        # current and on every zone count.
        dict(name="gradient_16384x512", kind="grad", rails=16384, sites=512, zones=10, open=False,
             fill=0.2, dt=DT_DENSE, steps=600, weights="both"),
        # One loss and gradient of the material fit on a shortened protocol
        # (batch creation, forward, curves, backward).
        dict(name="fit_eval_12", kind="fit", devices=12, sizes=11, pulses=1),
        # The torch.autograd front end on a small device: creation, forward and
        # backward.
        dict(name="autograd_256x100", kind="autograd", rails=256, sites=100, zones=10, open=False,
             fill=0.2, dt=DT_DENSE, steps=500),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps"] * 8 + ["loop"] + ["noalloc"] * 2 + ["batch"] * 2 + ["grad"] * 3 +
                      ["autograd"] * 2)
    if kind == "batch":
        return dict(kind=kind, devices=rng.randint(4, 32), sizes=rng.randint(1, 999),
                    steps=_log(rng, 100, 900))
    rails = _log(rng, 16, 65536)
    sites = _log(rng, 16, 2048)
    c = dict(kind=kind, rails=rails, sites=sites,
             zones=rng.choice([10, 10, 10, rng.randint(1, 16), min(32, sites)]),
             open=rng.random() < 0.4, fill=round(rng.uniform(0.05, 0.5), 3),
             dt=rng.choice([DT_RARE, DT_DENSE]))
    if kind == "loop":
        c["steps"] = rng.randint(1, 50)
        c["rails"] = min(rails, 4096)
    elif kind in ("grad", "autograd"):
        c["steps"] = _log(rng, 50, 2000)
        c["rails"] = min(rails, 32768 if kind == "grad" else 2048)
        most = 6e9 if kind == "grad" else 2e9
    else:
        c["steps"] = _log(rng, 50, 4000)
        most = 6e10
    if kind != "loop":
        c["steps"] = max(8, min(c["steps"], int(most / (c["rails"] * c["sites"]))))
    if kind == "grad":
        c["weights"] = rng.choice(["both", "current", "zones"])
    if kind in ("steps", "loop", "noalloc"):
        c["rule"] = 1 if rng.random() < 0.15 else 0
        c["protocol"] = rng.choice(["pulse", "triangle"])
        c["barriers"] = kind == "steps" and c["rails"] * c["sites"] <= 8e6 and rng.random() < 0.3
    return c


# ------------------------------------------------------------------- inputs

def _device(c, seed):
    open_ = bool(c["open"])
    # exchange of about 0.86 per step at the benchmark's rate (1e9 Hz, 1e-9 s)
    # and of the same order where the step is longer
    k_e = (1e9 if c["dt"] == DT_RARE else 1e6) if open_ else 0.0
    return W.Device(R=c["rails"], L=c["sites"], Z=c["zones"], electrodes=1 if open_ else 0, dt=c["dt"],
                    k_e=k_e, rho_e=c["fill"] if open_ else 0.0, seed=int(seed) & 0x7fffffff,
                    instance=int(seed) % 1000, rule=c.get("rule", 0))


def _protocol(c, seed, n):
    """n voltages of a periodic protocol, starting at a phase of the seed's."""
    if c["protocol"] == "triangle":
        period = W.triangle_protocol(2.0, 100000, 1)
    else:
        period = W.potentiation_protocol(1, 0)
    phase = int(np.random.default_rng(seed).integers(len(period)))
    return np.resize(np.roll(period, -phase), n)


def _weights(c, seed):
    rng = np.random.default_rng(seed)
    n, Z = c["steps"], c["zones"]
    wJ = rng.normal(size=n) if c["weights"] != "zones" else None
    wZ = rng.normal(size=(n, Z)) / c["sites"] if c["weights"] != "current" else None
    return wJ, wZ


def _pulse(c, seed):
    """A write pulse and its relaxation, the pulse's share of the seed's."""
    on = int(c["steps"] * np.random.default_rng(seed).uniform(0.2, 0.6))
    return W.relaxation_protocol(on, 1.0, c["steps"])


class _Stepper:
    """A device and the voltages of many passes ahead."""

    def __init__(self, c, seed):
        self.c, self.n = c, c["steps"]
        self.dev = _device(c, seed)
        passes = max(64, min(50000, int(2e6 / self.n)))
        self.V = _protocol(c, seed, passes * self.n)
        self.Ea = (W.normal_barriers(c["rails"], c["sites"], 0.40, 0.02, seed)
                   if c["barriers"] else None)
        self.open()

    def open(self):
        self.sim = K.Sim(self.dev, self.V, 1, fill=self.c["fill"], Ea_site=self.Ea)

    def step(self):
        if self.sim.t + self.n > len(self.V):
            self.sim.close()
            self.open()
        t = self.sim.t
        if self.c["kind"] == "loop":
            K.kmc_set_voltage(self.sim.h, t, self.V[t:t + self.n])
        self.sim.step_n(self.n)
        J, Zc = self.sim.traces(t, self.n)
        return J, Zc, self.sim.occupancy()


class _CallerOwned:
    """Occupancy, voltages and traces in the caller's own device memory."""

    def __init__(self, c, seed):
        self.c, self.n, self.t = c, c["steps"], 0
        self.dev = _device(c, seed)
        R, L = c["rails"], c["sites"]
        self.stride = (L + 15) // 16 * 16
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        self.occ = torch.zeros((R, self.stride), dtype=torch.uint8, device="cuda")
        self.occ[:, :L] = torch.rand((R, L), device="cuda", generator=g) < c["fill"]
        self.N0 = self.occ.sum(dim=1, dtype=torch.int32)
        self.V = torch.from_numpy(_protocol(c, seed, self.n)).cuda()
        self.J = torch.zeros(self.n, dtype=torch.int64, device="cuda")
        self.Zc = torch.zeros((self.n, c["zones"]), dtype=torch.int64, device="cuda")
        self.params = K.params_from_device(self.dev, 2)

    def step(self):
        K.kmc_sweep_noalloc(self.params, self.occ.data_ptr(), self.stride, self.N0.data_ptr(),
                            self.V.data_ptr(), self.t, self.n, self.J.data_ptr(), self.Zc.data_ptr(),
                            torch.cuda.current_stream().cuda_stream)
        self.t += self.n
        return self.J, self.Zc, self.occ


class _Batch:
    """Spike-timing devices of uneven sizes, their pulses inside the window."""

    def __init__(self, c, seed):
        self.n = c["steps"]
        passes = max(16, int(100000 / self.n))
        devs, Vs, fills, _ = W.stdp_batch(c["devices"], seed=c["sizes"])
        # the window from a phase of the seed's on, repeated
        phase = 2000 * int(np.random.default_rng(seed).integers(20, 60))
        self.Vs = [np.resize(np.roll(V, -phase), passes * self.n) for V in Vs]
        self.devs = [dataclasses.replace(d, seed=int(seed) & 0x7fffffff) for d in devs]
        self.fills = fills
        self.open()

    def open(self):
        self.b = K.Batch(self.devs, self.Vs, [1] * len(self.devs), fills=self.fills)

    def step(self):
        if self.b.t + self.n > len(self.Vs[0]):
            self.b.close()
            self.open()
        t = self.b.t
        self.b.step_n(self.n)
        J, Zc, Jr, occ = [], [], [], []
        for i in range(len(self.devs)):
            j, z = self.b.traces(i, t, self.n)
            J.append(j)
            Zc.append(z)
            Jr.append(self.b.rail_current(i))
            occ.append(self.b.occupancy(i).reshape(-1))
        return np.stack(J), np.stack(Zc), np.concatenate(Jr), np.concatenate(occ)


class _Gradient:
    """A device after its forward pass, and the weights of its observable."""

    def __init__(self, c, seed):
        self.sim = K.Sim(_device(c, seed), _pulse(c, seed), 1, fill=c["fill"])
        self.sim.step_n(c["steps"])
        self.wJ, self.wZ = _weights(c, seed)

    def step(self):
        g, se = self.sim.grad(self.wJ, self.wZ)
        return {"grad": g, "stderr": se}


class _Fit:
    """The devices, protocol and target curves of a material fit."""

    def __init__(self, c, seed):
        from paper_2511_09413_gb300.fit import MaterialFit
        devs, V, fills, samples = W.fit_batch(c["devices"], seed=c["sizes"], n_pulses=c["pulses"],
                                              forget_steps=0)
        devs = [dataclasses.replace(d, seed=int(seed) & 0x7fffffff) for d in devs]
        rng = np.random.default_rng(seed)
        tau = rng.uniform(500.0, 2000.0, size=(len(devs), 1))
        target = 0.1 + 0.05 * (1.0 - np.exp(-(samples[None, :] + 1.0) / tau))
        self.fit = MaterialFit(devs, V, fills, samples, target)

    def step(self):
        s = self.fit.loss_and_grad(0.40, 1.0)
        return {"loss": s.loss, "grad": s.grad, "stderr": s.stderr}


class _Autograd:
    """Parameters that require gradients and the weights of a loss."""

    def __init__(self, c, seed):
        self.c, self.dev, self.V = c, _device(c, seed), _pulse(c, seed)
        wJ, wZ = _weights(dict(c, weights="both"), seed)
        self.wJ, self.wZ = torch.from_numpy(wJ), torch.from_numpy(wZ)

    def step(self):
        from paper_2511_09413_gb300.autograd import simulate
        d = self.dev
        theta = torch.tensor([d.Ea, d.nu, d.kappa, self.c["fill"]], dtype=torch.float64,
                             requires_grad=True)
        J, Zc = simulate(theta, d, self.V, self.c["steps"])
        loss = (self.wJ * J).sum() + (self.wZ * Zc).sum()
        loss.backward()
        return {"J": J.detach(), "Zc": Zc.detach(), "grad": theta.grad}


_KINDS = {"steps": _Stepper, "loop": _Stepper, "noalloc": _CallerOwned, "batch": _Batch,
          "grad": _Gradient, "fit": _Fit, "autograd": _Autograd}


def prepare(case, seed):
    K.load()
    return _KINDS[case["kind"]](case, int(seed))


def run(state):
    return state.step()


# --------------------------------------------------------------------- work

# Integer operations of one Philox4x32-10 block (ten rounds of two widening
# multiplies and four exclusive ors) and of one trial pair besides its draw
# (exclusion, two comparisons, conflict, move).
_PHILOX_OPS, _TRIAL_OPS = 60, 12


def _sweep_work(rails, sites, zones, fill, steps, rule=0, open_=False, barriers=False):
    # ions with a free neighbour (half of the bonds under the even/odd rule)
    per_step = rails * (sites * fill * ((1 - fill * fill) if rule == 0 else (1 - fill)) +
                        (2 if open_ else 0))
    occ = rails * sites
    return {"bytes": 2 * occ + 8 * steps * (2 + zones) + (8 * occ if barriers else 0),
            "flops": per_step * steps * (_PHILOX_OPS + _TRIAL_OPS)}


def work(case):
    c = case
    if c["kind"] in ("steps", "loop", "noalloc"):
        return _sweep_work(c["rails"], c["sites"], c["zones"], c["fill"], c["steps"], c["rule"],
                           c["open"], c["barriers"])
    if c["kind"] in ("grad", "autograd"):
        w = _sweep_work(c["rails"], c["sites"], c["zones"], c["fill"], c["steps"], 0, c["open"])
        passes = 2 if c["kind"] == "autograd" else 1
        # the score of a rail's zones per step: two weights, four products
        score = 20.0 * c["rails"] * c["zones"] * c["steps"]
        return {"bytes": passes * w["bytes"], "flops": passes * w["flops"] + score}
    if c["kind"] == "batch":
        # the means of the devices' log-uniform sizes
        one = _sweep_work(16128 / math.log(64), 1920 / math.log(16), 10, 0.225, c["steps"])
        return {k: v * c["devices"] for k, v in one.items()}
    steps = 2000 * c["pulses"]
    one = _sweep_work(6144 / math.log(4), 768 / math.log(4), 10, 0.2, steps)
    score = 20.0 * (6144 / math.log(4)) * 10 * steps
    return {"bytes": 2 * one["bytes"] * c["devices"],
            "flops": (2 * one["flops"] + score) * c["devices"]}


# -------------------------------------------------------------------- exact

_KB = 8.6173e-5      # eV/K


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on uint64 arrays that hold 32-bit words."""
    M0, M1, mask = np.uint64(0xD2511F53), np.uint64(0xCD9E8D57), np.uint64(0xFFFFFFFF)
    s = np.uint64(32)
    for i in range(10):
        a, b = M0 * c0, M1 * c2
        r0 = np.uint64((k0 + 0x9E3779B9 * i) & 0xFFFFFFFF)
        r1 = np.uint64((k1 + 0xBB67AE85 * i) & 0xFFFFFFFF)
        c0, c1, c2, c3 = (b >> s) ^ c1 ^ r0, b & mask, (a >> s) ^ c3 ^ r1, a & mask
    return c0, c1, c2, c3


def _uniforms(dev, t, site, rail):
    word = np.zeros_like(site)
    x = _philox(site, rail, word + np.uint64(t), word + np.uint64(dev.instance),
                dev.seed & 0xFFFFFFFF, dev.seed >> 32)
    s, d = np.uint64(32), np.uint64(11)
    return ((((x[1] << s) | x[0]) >> d).astype(np.float64) * 2.0 ** -53,
            (((x[3] << s) | x[2]) >> d).astype(np.float64) * 2.0 ** -53)


def _replay(dev, V, n, fill, step):
    """Every step of the synchronous rule on all rails in 64 bits; calls
    step(t, zone counts [R, Z], per-rail current, score increments)."""
    R, L, Z = dev.R, dev.L, dev.Z
    open_ = dev.electrodes == 1
    site = np.broadcast_to(np.arange(L, dtype=np.uint64), (R, L)).copy()
    rail = np.broadcast_to(np.arange(R, dtype=np.uint64)[:, None], (R, L)).copy()
    occ = _uniforms(dev, 0xFFFFFFFF, site, rail)[0] < fill
    zone = ((np.arange(L) + 1) * Z + L - 1) // L - 1
    bnd = (np.arange(Z) * L) // Z
    w = np.bincount(zone, minlength=Z).astype(np.float64)
    N0 = occ.sum(axis=1)
    kT = _KB * dev.T
    x = 2.0 * dev.nu * math.exp(-dev.Ea / kT) * dev.dt
    P0 = -math.expm1(-x)
    E = -math.expm1(-2.0 * dev.k_e * dev.dt)
    bgd = N0[:, None] * w / L
    for t in range(n):
        Nz = np.add.reduceat(occ.astype(np.int64), bnd, axis=1)
        C = Nz - bgd
        Q = np.cumsum(C, axis=1) - 0.5 * C
        dq = Q - (Q @ w / L)[:, None]
        B = np.exp(-((V[t] - dev.kappa * dev.alpha * dq) / L) / kT)
        inv = 1.0 / (1.0 + B)
        c = dev.alpha * dq / (L * kT)
        Bk, ik, ck = B[:, zone], inv[:, zone], c[:, zone]
        uR, uL = _uniforms(dev, t, site, rail)
        base_R = np.full((R, L), P0)
        base_L = np.full((R, L), P0)
        right = np.zeros((R, L), dtype=bool)
        left = np.zeros((R, L), dtype=bool)
        right[:, :-1] = occ[:, :-1] & ~occ[:, 1:]
        left[:, 1:] = occ[:, 1:] & ~occ[:, :-1]
        inner_R, inner_L = right.copy(), left.copy()
        if open_:
            e = occ[:, 0]
            left[:, 0] = e                                  # extraction
            right[~e, 0] = True                             # injection
            base_L[:, 0] = E * (1.0 - dev.rho_e)
            base_R[~e, 0] = E * dev.rho_e
            e = occ[:, -1]
            right[:, -1] = e
            left[~e, -1] = True
            base_R[:, -1] = E * (1.0 - dev.rho_e)
            base_L[~e, -1] = E * dev.rho_e
        pL, pR = base_L * ik, base_R * ik * Bk
        aR, aL = right & (uR <= pR), left & (uL <= pL)
        wR = np.where(right, np.where(pR < 1.0, (aR - pR) / np.where(pR < 1.0, 1.0 - pR, 1.0), 1.0), 0.0)
        wL = np.where(left, np.where(pL < 1.0, (aL - pL) / np.where(pL < 1.0, 1.0 - pL, 1.0), 1.0), 0.0)
        inner = (wR * inner_R + wL * inner_L).sum(axis=1)
        kappa = (wR * ik * ck - wL * (1.0 - ik) * ck).sum(axis=1)
        eta = (left * (aL - pL) - right * (aR - pR)).sum(axis=1)
        mR, mL = occ & aR & ~aL, occ & aL & ~aR
        inj0, injL = ~occ[:, 0] & aR[:, 0] & open_, ~occ[:, -1] & aL[:, -1] & open_
        into_R = np.concatenate([inj0[:, None], mR[:, :-1]], axis=1)
        into_L = np.concatenate([mL[:, 1:], injL[:, None]], axis=1)
        clash = into_R & into_L
        into_R &= ~clash
        into_L &= ~clash
        mR[:, :-1] &= ~clash[:, 1:]
        mL[:, 1:] &= ~clash[:, :-1]
        inj0, injL = into_R[:, 0], into_L[:, -1]
        J = (mL.sum(axis=1) - mR.sum(axis=1) - inj0.astype(np.int64) + injL.astype(np.int64))
        step(t, Nz, J, inner, kappa, eta)
        occ = (occ & ~mR & ~mL) | into_R | into_L
    return N0, x, P0, kT


def _gradient(dev, V, n, fill, wJ, wZ):
    """Gradient and standard error of the likelihood-ratio estimator with
    leave-one-out baselines and the current's innovation as control variate."""
    steps = []
    N0, x, P0, kT = _replay(dev, V, n, fill, lambda *a: steps.append(a[1:]))
    R = dev.R
    W_, K_ = np.zeros(R), np.zeros(R)
    GW, GK, G1 = np.zeros(R), np.zeros(R), np.zeros(R)
    for t, (Nz, J, inner, kappa, eta) in enumerate(steps):
        f = np.zeros(R)
        if wZ is not None:
            f = (Nz - (Nz.sum(axis=0) - Nz) / (R - 1)) @ wZ[t]
        if wJ is not None:
            f = f - wJ[t] * eta
        GW += f * W_
        GK += f * K_
        G1 += f
        W_ += inner
        K_ += kappa
        if wJ is not None:
            f = wJ[t] * (J - (J.sum() - J) / (R - 1))
            GW += f * W_
            GK += f * K_
            G1 += f
    rho = (N0 - dev.L * fill) / (fill * (1.0 - fill))
    G = np.stack([-(x / kT) * math.exp(-x) / P0 * GW, (x / dev.nu) * math.exp(-x) / P0 * GW, GK,
                  rho * G1], axis=1)
    return G.sum(axis=0), np.sqrt(R / (R - 1.0) * ((G - G.mean(axis=0)) ** 2).sum(axis=0)), steps


def exact(case, seed):
    c = case
    if c["kind"] not in ("grad", "autograd") or c["rails"] * c["sites"] * c["steps"] > 2e7:
        return None
    seed = int(seed)
    dev, V = _device(c, seed), _pulse(c, seed)
    wJ, wZ = _weights(c if c["kind"] == "grad" else dict(c, weights="both"), seed)
    g, se, steps = _gradient(dev, V, c["steps"], c["fill"], wJ, wZ)
    if c["kind"] == "grad":
        return {"grad": g, "stderr": se}
    J = np.array([s[1].sum() for s in steps], dtype=np.float64)
    Zc = np.array([s[0].sum(axis=0) for s in steps], dtype=np.float64)
    return {"J": J, "Zc": Zc, "grad": g}
