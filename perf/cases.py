"""The work that programs built on this library have it do, as cases that can
be timed and compared: the operators on device buffers (accelerations, Kepler
drift, training of the guess network), the energy diagnostic, and whole step
calls on the disks and the ensemble.

A step case is one segment of an integration as a host program drives it: the
state in from pinned host memory, a few steps, the state and the encounter
records out.
"""
import math

import numpy as np
import torch

import paper_1007_3458_gb300 as qym
from paper_1007_3458_gb300 import guess
from paper_1007_3458_gb300 import workloads as W

FP64, MIXED = qym.QYM_KICK_FP64, qym.QYM_KICK_MIXED


def listed():
    return [
        # The smallest acceleration call: the 260-body disk, all launches and latency.
        dict(name="accel_mixed_260", kind="accel", prec="mixed", bodies=260),
        # The FP64 kick at the paper's 10240 bodies (its Tables 2 and 3).
        dict(name="accel_fp64_10240", kind="accel", prec="fp64", bodies=10240),
        # The default kick on the 16384-body disk.
        dict(name="accel_mixed_16384", kind="accel", prec="mixed", bodies=16384),
        # E_Kep with the step's default solver on a disk's worth of bodies.
        dict(name="kepler_laguerre_16384", kind="kepler", n=16384, solver="laguerre", guess="standard"),
        # E_Kep started from the trained network, Newton in FP64.
        dict(name="kepler_mlp_262144", kind="kepler", n=262144, solver="newton", guess="mlp"),
        # E_Kep of the 1,048,576 test particles, FP32 steps first.
        dict(name="kepler_newton32_1m", kind="kepler", n=1048576, solver="newton32", guess="standard"),
        # Training of the guess network: eight minibatches of the default fit.
        dict(name="train_131072", kind="train", rows=131072, batch=16384),
        # The energy diagnostic that every run's error is quoted from.
        dict(name="energy_16384", kind="energy", system="disk", bodies=16384),
        # The 260-body disk with the paper's FP64 kick: a step is latency.
        dict(name="step_260_fp64", kind="step", system="disk", prec="fp64", bodies=260, steps=16),
        # The 16384-body disk with the default kick.
        dict(name="step_16384_mixed", kind="step", system="disk", prec="mixed", bodies=16384, steps=8),
        # The batch of 512 systems of 64 to 4096 bodies.
        dict(name="step_ensemble_512", kind="step", system="ensemble", prec="mixed", systems=512, steps=2),
        # The dense-encounter disk: embryos in 262080 planetesimals.
        dict(name="step_262144_mixed", kind="step", system="embryos", prec="mixed", bodies=262144, steps=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["accel", "accel", "kepler", "kepler", "train", "energy", "step", "step", "step"])
    if kind == "accel":
        prec = rng.choice(["mixed", "fp64"])
        return dict(kind=kind, prec=prec, bodies=_log(rng, 65, 32767 if prec == "mixed" else 16384))
    if kind == "kepler":
        g = rng.choice(["standard", "standard", "mlp"])
        return dict(kind=kind, n=_log(rng, 1000, 1 << 20), guess=g,
                    solver=rng.choice(["laguerre", "newton", "newton32"]))
    if kind == "train":
        return dict(kind=kind, rows=_log(rng, 4096, 262144), batch=_log(rng, 1024, 16384))
    system = rng.choice(["disk", "ensemble"] if kind == "energy" else ["disk", "disk", "ensemble", "embryos"])
    if kind == "energy":
        if system == "disk":
            return dict(kind=kind, system=system, bodies=_log(rng, 200, 24000))
        return dict(kind=kind, system=system, systems=_log(rng, 4, 128))
    if system == "ensemble":
        return dict(kind=kind, system=system, prec="mixed", systems=_log(rng, 4, 256),
                    steps=rng.randint(1, 4))
    if system == "embryos":
        return dict(kind=kind, system=system, prec="mixed", bodies=_log(rng, 20000, 150000),
                    steps=rng.randint(1, 3))
    prec = rng.choice(["mixed", "mixed", "fp64"])
    return dict(kind=kind, system=system, prec=prec, steps=rng.randint(1, 16),
                bodies=_log(rng, 200, 16384 if prec == "mixed" else 2048))


def _workload(case, seed):
    seed = int(seed) % (1 << 32)
    if case.get("system", "disk") == "ensemble":
        # the ensemble's sizes (the same for every seed), each system drawn from the seed
        sizes = np.random.default_rng(3).integers(64, 4097, case["systems"])
        parts = [W.ensemble(1, int(k), int(k), seed=[seed, i]) for i, k in enumerate(sizes)]
        offsets = np.concatenate([[0], np.cumsum([len(p.m) for p in parts])]).astype(np.int64)
        return W.Workload("ensemble", *(np.concatenate([getattr(p, k) for p in parts]) for k in "mqv"),
                          offsets, parts[0].tau, case["steps"] if "steps" in case else 0,
                          eps_H=parts[0].eps_H)
    n = case["bodies"]
    if case.get("system") == "embryos":
        return W.embryo_disk(64, n - 64, seed=seed)
    # planetesimal masses of the 260-body and the 16384-body disk
    return W.outer_disk(n - 4, 1e-9 if n < 4096 else 1e-10, seed=seed)


def _soa(a):
    return torch.from_numpy(np.ascontiguousarray(a.T)).cuda()


def _pinned(a):
    return torch.from_numpy(np.ascontiguousarray(a)).pin_memory()


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "accel":
        w = _workload(case, seed)
        prec = MIXED if case["prec"] == "mixed" else FP64
        rows = len(w.m)
        s.update(rows=rows, prec=prec, m=torch.from_numpy(w.m).cuda(), q=_soa(w.q),
                 a=torch.empty((3, rows), dtype=torch.float64, device="cuda"),
                 work=torch.empty(qym.qym_accel_workspace_bytes(rows, prec), dtype=torch.uint8,
                                  device="cuda"))
    elif kind == "kepler":
        n = case["n"]
        q, v, dt = W.test_particles(n, seed=int(seed) % (1 << 32))
        s.update(n=n, dt=dt, q0=_soa(q), v0=_soa(v),
                 solver=dict(laguerre=qym.QYM_SOLVER_LAGUERRE, newton=qym.QYM_SOLVER_NEWTON,
                             newton32=qym.QYM_SOLVER_NEWTON32)[case["solver"]],
                 guess=qym.QYM_GUESS_MLP if case["guess"] == "mlp" else qym.QYM_GUESS_STANDARD,
                 status=torch.zeros(1, dtype=torch.int32, device="cuda"), mlp=None)
        s["q1"], s["v1"] = torch.empty_like(s["q0"]), torch.empty_like(s["v0"])
        if case["guess"] == "mlp":
            # a network fitted to other particles' solves, as a program would keep it
            tq, tv, tdt = W.test_particles(65536, seed=5)
            wts, _ = guess.fit(guess.log_particle_rows(tq, tv, tdt, 1), batch=4096, epochs=20)
            s["mlp"] = torch.from_numpy(wts).cuda()
    elif kind == "train":
        rows = W.mlp_rows_synthetic(case["rows"], int(seed) % (1 << 32))
        w = torch.from_numpy(W.mlp_init(0, rows[:, :4], rows[:, 4])).cuda()
        batches = -(-case["rows"] // case["batch"])
        s.update(rows=torch.from_numpy(rows).cuda(), w=w, m=torch.zeros_like(w), v=torch.zeros_like(w),
                 t=0, batches=batches,
                 losses=torch.empty(batches, dtype=torch.float32, device="cuda"),
                 work=torch.empty(qym.qym_mlp_workspace_bytes(), dtype=torch.uint8, device="cuda"))
    else:
        w = _workload(case, seed)
        prec = FP64 if case.get("prec") == "fp64" else MIXED
        s.update(tau=w.tau, sim=qym.Simulation(w.m, w.q, w.v, w.offsets, eps_H=w.eps_H, kick_prec=prec))
        if kind == "step":
            host = [_pinned(w.q), _pinned(w.v), _pinned(np.empty_like(w.q)), _pinned(np.empty_like(w.v))]
            # room for the encounter records of a call; unused rows hold -1
            s.update(host=host, arrays=[t.numpy() for t in host],
                     records=np.full((max(1024, len(w.m) // 2) * case["steps"], 3), -1), used=0)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "accel":
        qym.qym_accel_dev(s["rows"], s["m"], s["q"], s["a"], 1.0, s["prec"], s["work"])
        return s["a"]
    if kind == "kepler":
        qym.qym_kepler_drift_dev(s["n"], s["q0"], s["v0"], s["q1"], s["v1"], 1.0, s["dt"], s["solver"],
                                 s["guess"], s["mlp"], status=s["status"])
        return s["q1"], s["v1"], s["status"]
    if kind == "train":
        qym.qym_mlp_train_dev(s["w"], s["m"], s["v"], s["t"], s["rows"], case["rows"], case["batch"], 1,
                              2e-3, 2e-5, s["losses"], s["work"])
        s["t"] += s["batches"]
        return s["w"], s["m"], s["v"], s["losses"]
    if kind == "energy":
        return s["sim"].energy()
    q0, v0, q, v = s["arrays"]
    sim = s["sim"]
    sim.set_state(q0, v0)
    sim.step(s["tau"], case["steps"])
    qym.qym_get_state(sim.ctx, q, v)
    found = sim.encounters()
    s["records"][:len(found)] = found
    s["records"][len(found):s["used"]] = -1
    s["used"] = len(found)
    return q, v, s["records"]


def _nbodies(case):
    """(rows, sum over systems of N (N - 1)); an ensemble's by its mean size."""
    if case.get("system", "disk") == "ensemble":
        n = 0.5 * (64 + 4096)
        n2 = (4096.0 ** 3 - 64.0 ** 3) / (3.0 * (4096 - 64))  # mean of N^2
        return case["systems"] * n, case["systems"] * n2
    n = case["bodies"]
    return n, float(n) * (n - 1)


def work(case):
    kind = case["kind"]
    if kind == "kepler":
        # state in and out; two evaluations of Kepler's equation, f and g functions
        return {"bytes": 96.0 * case["n"], "flops": 250.0 * case["n"]}
    if kind == "train":
        # forward and both backward products of 4-64-64-1; rows read once, the
        # weights and moments read and written once
        return {"bytes": 20.0 * case["rows"] + 24.0 * qym.QYM_MLP_NW,
                "flops": 6.0 * case["rows"] * (4 * 64 + 64 * 64 + 64)}
    rows, pairs = _nbodies(case)
    if kind == "accel":
        return {"bytes": 56.0 * rows, "flops": 20.0 * pairs}
    if kind == "energy":
        return {"bytes": 56.0 * rows, "flops": 0.5 * 11.0 * pairs}
    # two kicks a step (20 flops a pair) and the drift; the state in and out
    return {"bytes": 96.0 * rows, "flops": case["steps"] * (40.0 * pairs + 250.0 * rows)}


def _exact_accel(w, G=1.0):
    m = torch.from_numpy(w.m).cuda()
    q = torch.from_numpy(np.ascontiguousarray(w.q)).cuda()
    qb, gm = q[1:], G * m[1:]
    a = torch.zeros_like(q)
    for i in range(0, len(qb), 1024):
        d = qb[None, :, :] - qb[i:i + 1024, None, :]
        r2 = (d * d).sum(-1)
        f = torch.where(r2 > 0, gm / (r2 * r2.sqrt()), torch.zeros_like(r2))
        a[1 + i:1 + i + 1024] = (f[:, :, None] * d).sum(1)
    return a.T.contiguous()


def _exact_drift(q, v, dt):
    """Elliptic drift about mu = 1 by the difference of eccentric anomalies."""
    q, v = _soa(q), _soa(v)
    r0 = (q * q).sum(0).sqrt()
    alpha = 2.0 / r0 - (v * v).sum(0)
    a = 1.0 / alpha
    n = alpha * alpha.sqrt()
    ec, es = 1.0 - r0 * alpha, (q * v).sum(0) * alpha.sqrt()
    M = n * dt
    E = M.clone()
    for _ in range(40):  # Laguerre-Conway: M = E - ec sin E + es (1 - cos E)
        sn, cs = torch.sin(E), torch.cos(E)
        F = E - ec * sn + 2.0 * es * torch.sin(0.5 * E) ** 2 - M
        F1 = 1.0 - ec * cs + es * sn
        F2 = ec * sn + es * cs
        E = E - 5.0 * F / (F1 + torch.sqrt((16.0 * F1 * F1 - 20.0 * F * F2).abs()))
    sh2 = 2.0 * torch.sin(0.5 * E) ** 2  # 1 - cos E
    f = 1.0 - a / r0 * sh2
    g = (a * r0 * torch.sin(E) + a * (q * v).sum(0) * a.sqrt() * sh2) * alpha.sqrt()
    q1 = f * q + g * v
    r1 = (q1 * q1).sum(0).sqrt()
    fd = -torch.sin(E) * a.sqrt() / (r0 * r1)
    gd = 1.0 - a / r1 * sh2
    return q1, fd * q + gd * v


def _exact_train(case, seed):
    """The same Adam steps in 64 bits; the matrices rounded to bf16 where they are used."""
    rows32 = W.mlp_rows_synthetic(case["rows"], int(seed) % (1 << 32))
    w = torch.from_numpy(W.mlp_init(0, rows32[:, :4], rows32[:, 4])).cuda().double()
    rows = torch.from_numpy(rows32).cuda().double()
    m, v = torch.zeros_like(w), torch.zeros_like(w)
    mean, std, om, osd = w[4545:4549].clone(), w[4549:4553].clone(), w[4553].clone(), w[4554].clone()
    n, batch = case["rows"], case["batch"]
    S = -(-n // batch)
    losses = []
    for s in range(S):
        r = rows[s * batch:(s + 1) * batch]
        wb = w.clone()
        for lo, hi in ((0, 256), (320, 4416), (4480, 4544)):
            wb[lo:hi] = w[lo:hi].bfloat16().double()
        wb.requires_grad_(True)
        h = ((r[:, :4] - mean) / std) @ wb[:256].reshape(64, 4).T + wb[256:320]
        h = torch.nn.functional.gelu(h, approximate="tanh") @ wb[320:4416].reshape(64, 64).T + wb[4416:4480]
        y = torch.nn.functional.gelu(h, approximate="tanh") @ wb[4480:4544] + wb[4544]
        loss = ((y - (r[:, 4] - om) / osd) ** 2).mean()
        loss.backward()
        g = wb.grad
        g[4545:] = 0.0
        losses.append(loss.detach())
        lr = 2e-5 + 0.5 * (2e-3 - 2e-5) * (1.0 + math.cos(math.pi * s / S))
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        w = w - lr * (m / (1 - 0.9 ** (s + 1))) / ((v / (1 - 0.999 ** (s + 1))).sqrt() + 1e-8)
    return w, m, v, torch.stack(losses)


def _exact_energy(w):
    E = []
    for s in range(w.nsys):
        lo, hi = int(w.offsets[s]), int(w.offsets[s + 1])
        m, q, v = (torch.from_numpy(np.ascontiguousarray(x[lo:hi])).cuda() for x in (w.m, w.q, w.v))
        m0, mb, qb = m[0], m[1:], q[1:]
        # heliocentric to barycentric velocities
        vb = v[1:] - (mb[:, None] * v[1:]).sum(0) / m.sum()
        S = (mb[:, None] * vb).sum(0)
        e = (S * S).sum() / (2.0 * m0) + (0.5 * mb * (vb * vb).sum(1)).sum()
        e = e - (m0 * mb / (qb * qb).sum(1).sqrt()).sum()
        for i in range(0, len(qb), 1024):
            d = qb[i:i + 1024, None, :] - qb[None, :, :]
            r2 = (d * d).sum(-1)
            p = torch.where(r2 > 0, mb[None, :] / r2.sqrt(), torch.zeros_like(r2))
            e = e - 0.5 * (mb[i:i + 1024] * p.sum(1)).sum()
        E.append(e)
    return torch.stack(E)


def exact(case, seed):
    kind = case["kind"]
    if kind == "accel":
        return _exact_accel(_workload(case, seed))
    if kind == "kepler":
        q, v, dt = W.test_particles(case["n"], seed=int(seed) % (1 << 32))
        return (*_exact_drift(q, v, dt), None)
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "energy":
        return _exact_energy(_workload(case, seed))
    return None  # the hybrid step with its encounters has no short 64-bit form
