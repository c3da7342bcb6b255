"""What a program that integrates GLD systems with this package does, as cases to be timed and compared.

A case is one of three kinds:
  run    one system: GLD.step(steps), then its velocities and unwrapped displacements are read (and the
         VACF where it is on) -- what every simulation and analysis loop does;
  batch  many uneven independent systems stepped together by a Batch;
  serve  a standing Server that gets a handful of requests, runs them and hands the results back.

Sizes, densities, time steps, memory lengths and kernels are those of the package's workloads
(paper_1808_00270_gb300.inputs) and of its tests.  Results are FP32 on the device and come back in FP64
arrays; they are returned as the FP32 numbers they are.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_1808_00270_gb300 import ARR_DISP, ARR_HIST, ARR_VEL, GLD, Batch, Server, inputs

GIVEN_HISTORY = 2_000_000  # particles x memory slots up to which prepare() hands a history over


def _run(name=None, *, n, m_max, steps, density=0.1, r_c=2.0, dt=0.005, tau_s=0.5, tau_p=0.3, tail=False, hist="f32",
         kahan=False, terms="pair", memory="ring", pair_noise=0, vacf_len=0, vacf_stride=1, first=0):
    c = dict(kind="run", n=n, m_max=m_max, steps=steps, density=density, r_c=r_c, dt=dt, tau_s=tau_s, tau_p=tau_p,
             tail=tail, hist=hist, kahan=kahan, terms=terms, memory=memory, pair_noise=pair_noise, vacf_len=vacf_len,
             vacf_stride=vacf_stride, first=first)
    return dict(c, name=name) if name else c


def _batch(name=None, *, systems, n_lo, n_hi, steps, mix=4):
    c = dict(kind="batch", systems=systems, n_lo=n_lo, n_hi=n_hi, steps=steps, mix=mix)
    return dict(c, name=name) if name else c


def _serve(name=None, *, requests, n_lo, n_hi, steps_lo, steps_hi, mix=5):
    c = dict(kind="serve", requests=requests, n_lo=n_lo, n_hi=n_hi, steps_lo=steps_lo, steps_hi=steps_hi, mix=mix)
    return dict(c, name=name) if name else c


def listed():
    suspension = dict(r_c=2.5, tail=True, m_max=400)
    return [
        # the oracle-sized system of inputs.SMALL: launches and latencies are all there is
        _run("small_n64_m32", n=64, density=0.125, m_max=32, dt=0.01, tau_s=0.2, tau_p=0.1, steps=64),
        # one step at a time: a program that couples something else to every step
        _run("single_step_n4096_m200", n=4096, m_max=200, steps=1),
        # inputs.MEDIUM with its VACF: the everyday parameter study
        _run("medium_n4096_m200", n=4096, m_max=200, steps=256, vacf_len=200, vacf_stride=20),
        # a resumed run written out every 50 steps: ragged in size, memory and steps, off every block boundary
        _run("ragged_n10007_m257", n=10007, m_max=257, steps=50, first=77),
        # inputs.LARGE_QUARTER
        _run("suspension_n65536_m400", n=65536, steps=128, vacf_len=400, vacf_stride=40, **suspension),
        # inputs.LARGE, the benchmark's system and VACF
        _run("suspension_n262144_m400", n=262144, steps=256, vacf_len=400, vacf_stride=40, **suspension),
        # half the history bytes, sums compensated
        _run("bf16_kahan_n100003_m400", n=100003, steps=64, hist="bf16", kahan=True, **suspension),
        # the paper's general kernel: pair and self-difference terms with perpendicular factors
        _run("general_n20000_m400", n=20000, steps=64, terms="general", **suspension),
        # the auxiliary-variable form of the memory
        _run("modes_n65536_m400", n=65536, steps=128, memory="modes", **suspension),
        # the pair-correlated random force (fluctuation-dissipation balance of the pair friction)
        _run("pair_noise_n32768_m200", n=32768, m_max=200, density=0.05, steps=64, pair_noise=8),
        # replicas: inputs.batch_systems, an eighth of its systems
        _batch("batch_64_systems", systems=64, n_lo=256, n_hi=16384, steps=256),
        # the serving trace's mix, its smaller requests
        _serve("serve_16_requests", requests=16, n_lo=512, n_hi=16384, steps_lo=128, steps_hi=448),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    u = rng.random()
    if u < 0.12:
        return _batch(systems=log_int(4, 64), n_lo=256, n_hi=log_int(1024, 16384), steps=64 * rng.randint(1, 4),
                      mix=rng.randint(1, 10 ** 6))
    if u < 0.2:
        lo = rng.randint(64, 256)
        return _serve(requests=log_int(2, 16), n_lo=512, n_hi=log_int(1024, 16384), steps_lo=lo,
                      steps_hi=lo + rng.randint(1, 192), mix=rng.randint(1, 10 ** 6))
    n = log_int(64, 200000)
    m = log_int(64, 800)
    steps = rng.choice([1, 7, 33, 50, 64, 100, 128, 256])
    suspension = rng.random() < 0.5
    kw = dict(n=n, m_max=m, steps=steps, density=round(math.exp(rng.uniform(math.log(0.02), math.log(0.2))), 4),
              r_c=2.5 if suspension else 2.0, tail=suspension)
    if n / kw["density"] < 1000.0:  # a box of at least four cutoffs
        kw["density"] = round(n / 1000.0, 4)
    if rng.random() < 0.4:
        kw["vacf_len"] = rng.choice([50, 100, 200, 400])
        kw["vacf_stride"] = kw["vacf_len"] // 10
    option = rng.random()
    if option < 0.15:
        kw["hist"] = "bf16"
        kw["kahan"] = rng.random() < 0.5
    elif option < 0.25:
        kw["kahan"] = True
    elif option < 0.35:
        kw["terms"] = "general"
    elif option < 0.45:
        kw["terms"] = "self"
    elif option < 0.55:
        kw["memory"] = "modes"
    elif option < 0.62 and not suspension and kw["density"] <= 0.06 and m >= 128:  # a positive semi-definite balance
        kw["pair_noise"] = rng.choice([4, 8])
    if n * m <= GIVEN_HISTORY and rng.random() < 0.5:
        kw["first"] = rng.randint(1, 5000)
    return _run(**kw)


# ---- inputs ------------------------------------------------------------------------------------
def _workload(c, seed):
    return inputs.Workload("case", n=c["n"], box=inputs.box_for_density(c["n"], c["density"]), m_max=c["m_max"],
                           dt=c["dt"], r_c=c["r_c"], tau_s=c["tau_s"], tau_p=c["tau_p"], steps=c["steps"],
                           tail=c["tail"], seed=seed)


def _f32(x):
    return np.asarray(x, dtype=np.float32)


def _initial(c, seed):
    """Workload, positions and velocities (numbers that FP32 holds), and the history where it is handed over."""
    w = _workload(c, seed)
    pos, vel = inputs.initial_state(w)
    pos, vel = _f32(pos).astype(np.float64), _f32(vel).astype(np.float64)
    pos[pos >= w.box] = 0.0
    hist = None
    if c["n"] * c["m_max"] <= GIVEN_HISTORY:  # displacements of one step: dt v, remembered for a few steps
        hist = _f32(inputs.random_history(w.n, w.m_max, scale=w.dt, seed=seed + 1)).astype(np.float64)
    return w, pos, vel, hist


def _terms(c, w):
    """set_kernels arguments and perpendicular factors of the case's terms."""
    ks = inputs.self_kernel_samples(w)
    if c["terms"] == "self":
        return dict(Ks=ks), None
    g, f, dr = inputs.pair_kernel_tables(w)
    if c["pair_noise"]:
        f = 0.2 * f  # the balance needs a positive semi-definite friction matrix
    if c["terms"] == "general":
        return dict(Ks=ks, g=g, f=f, dr=dr, gs=0.5 * g, fs=0.3 * f), dict(fp=0.4 * f, fs=0.1 * f)
    return dict(Ks=ks, g=g, f=f, dr=dr), None


def _system(w, pos, vel, **kw):
    return GLD(n=w.n, box=w.box, dt=w.dt, m_max=w.m_max, r_c=w.r_c, A_cons=w.A_cons, pos=pos, vel=vel, mass=w.mass,
               kT=w.kT, seed=w.seed, **kw)


def _prepare_run(c, seed):
    w, pos, vel, hist = _initial(c, seed)
    kw = dict(hist_dtype=c["hist"], kahan=c["kahan"])
    if c["vacf_len"]:
        kw.update(vacf_len=c["vacf_len"], vacf_stride=c["vacf_stride"], vacf_burnin=1)
    sim = _system(w, pos, vel, **kw)
    terms, perp = _terms(c, w)
    sim.set_kernels(**terms)
    if perp:
        sim.set_perpendicular(**perp)
    if hist is not None:
        if c["first"]:
            sim.set_step(c["first"])
        sim.set(ARR_HIST, hist)
    if c["memory"] == "modes":
        sim.set_memory_modes(*inputs.memory_modes(w))
    if c["pair_noise"]:
        sim.set_pair_noise(c["pair_noise"], lam=2.0)
    if hist is None:  # the history fills as it does in use: by stepping
        sim.step(-(-w.m_max // 64) * 64)
    sim.sync()
    return dict(kind="run", sim=sim, steps=c["steps"], vacf=bool(c["vacf_len"]))


def _members(c, seed):
    """The systems of the case's mix, their initial states and noise from the seed."""
    return [dataclasses.replace(w, seed=seed * 1000 + k) for k, w in enumerate(
        inputs.batch_systems(c["systems"], seed=c["mix"], n_range=(c["n_lo"], c["n_hi"])))]


def _prepare_batch(c, seed):
    b, systems = Batch(), []
    for w in _members(c, seed):
        pos, vel = inputs.initial_state(w)
        g = _system(w, pos, vel)
        gk, f, dr = inputs.pair_kernel_tables(w)
        g.set_kernels(inputs.self_kernel_samples(w), g=gk, f=f, dr=dr)
        b.add(g)
        systems.append(g)
    b.step(448)  # every history full
    b.sync()
    return dict(kind="batch", batch=b, systems=systems, steps=c["steps"])


def _trace(c, seed):
    trace = inputs.serve_trace(c["requests"], rate=1e6, seed=c["mix"], n_range=(c["n_lo"], c["n_hi"]),
                               step_range=(c["steps_lo"], c["steps_hi"]))
    return [dataclasses.replace(r, w=dataclasses.replace(r.w, seed=seed * 1000 + k)) for k, r in enumerate(trace)]


def _prepare_serve(c, seed):
    reqs = []
    for r in _trace(c, seed):
        w = r.w
        pos, vel = inputs.initial_state(w)
        gk, f, dr = inputs.pair_kernel_tables(w)
        reqs.append(dict(n=w.n, box=w.box, dt=w.dt, m_max=w.m_max, r_c=w.r_c, pos=pos, vel=vel,
                         Ks=inputs.self_kernel_samples(w), g=gk, f=f, dr=dr, steps=r.steps, mass=w.mass, kT=w.kT,
                         A_cons=w.A_cons, seed=w.seed, vacf_len=100, vacf_stride=10, vacf_burnin=1, keep_state=True))
    return dict(kind="serve", server=Server(hbm_budget=60_000_000_000), requests=reqs)


def prepare(case, seed):
    return {"run": _prepare_run, "batch": _prepare_batch, "serve": _prepare_serve}[case["kind"]](case, seed)


def run(state):
    if state["kind"] == "run":
        sim = state["sim"]
        sim.step(state["steps"])
        out = dict(vel=_f32(sim.get(ARR_VEL)), disp=_f32(sim.get(ARR_DISP)))
        if state["vacf"]:
            out["vacf"] = _f32(sim.vacf()[0])
        return out
    if state["kind"] == "batch":
        state["batch"].step(state["steps"])
        return dict(vel=np.concatenate([_f32(g.get(ARR_VEL)) for g in state["systems"]]),
                    disp=np.concatenate([_f32(g.get(ARR_DISP)) for g in state["systems"]]))
    srv, reqs = state["server"], state["requests"]
    ids = [srv.submit(arrival=0.0, **q) for q in reqs]
    srv.drain()
    got = [srv.result(i) for i in ids]
    moved = []
    for r, q in zip(got, reqs):  # displacement over the run, nearest image
        d = r["pos"] - q["pos"]
        moved.append(_f32(d - q["box"] * np.round(d / q["box"])))
    return dict(vel=np.concatenate([_f32(r["vel"]) for r in got]), moved=np.concatenate(moved),
                vacf=np.stack([_f32(r["vacf"]) for r in got]))


# ---- work --------------------------------------------------------------------------------------
def _work(n, m, steps, density, r_c, nacc, elem, ring=True):
    """Bytes: state in and out, the history once, the new displacements.  Flops: the memory sums, the noise's moving
    average, and about 60 per neighbour within the cutoff for both forces."""
    h = m - 1
    pairs = density * 4.18879 * r_c ** 3
    byts = n * (16.0 * 3 * 2 + 3 * elem * (h + min(steps, h)))
    mem = 2.0 * 3 * n * nacc * (h if ring else 32)
    return byts, steps * (mem + 2.0 * 3 * n * (2 * h + 1) + 60.0 * n * pairs)


def work(case):
    if case["kind"] == "run":
        nacc = {"self": 1, "pair": 2, "general": 3}[case["terms"]]
        b, f = _work(case["n"], case["m_max"], case["steps"], case["density"], case["r_c"], nacc,
                     2 if case["hist"] == "bf16" else 4, case["memory"] == "ring")
        if case["pair_noise"]:  # one filter and one neighbour sweep per degree
            f += case["steps"] * case["pair_noise"] * case["n"] * (
                6.0 * (2 * case["m_max"] - 1) + 40.0 * case["density"] * 4.18879 * case["r_c"] ** 3)
        return {"bytes": b, "flops": f}
    if case["kind"] == "batch":
        ws = [(w, case["steps"]) for w in _members(case, 0)]
    else:
        ws = [(r.w, r.steps) for r in _trace(case, 0)]
    both = [_work(w.n, w.m_max, s, w.density, w.r_c, 2, 4) for w, s in ws]
    return {"bytes": sum(b for b, _ in both), "flops": sum(f for _, f in both)}


# ---- the same in 64 bits -----------------------------------------------------------------------
def _gauss(seed, particles, times):
    """Unit Gaussians W[time, particle, 3]: Philox4x32-10 (Salmon et al., SC'11) keyed by the seed, counter
    (particle, low and high words of time + 2^62, 0), and Box-Muller on the top 23 bits of each word."""
    t = (times.astype(np.int64) + (1 << 62)).astype(np.uint64)
    shape = (len(times), len(particles))
    c = [np.broadcast_to(particles.astype(np.uint64)[None, :], shape).copy(),
         np.broadcast_to((t & np.uint64(0xFFFFFFFF))[:, None], shape).copy(),
         np.broadcast_to((t >> np.uint64(32))[:, None], shape).copy(), np.zeros(shape, np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    low, sh = np.uint64(0xFFFFFFFF), np.uint64(32)
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> sh) ^ c[1] ^ np.uint64(k0), p1 & low, (p0 >> sh) ^ c[3] ^ np.uint64(k1), p0 & low]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    u = [((x >> np.uint64(9)).astype(np.float64) + 0.5) / 8388608.0 for x in c]
    r0, r1 = np.sqrt(-2.0 * np.log(u[0])), np.sqrt(-2.0 * np.log(u[2]))
    return np.stack([r0 * np.cos(2 * np.pi * u[1]), r0 * np.sin(2 * np.pi * u[1]), r1 * np.cos(2 * np.pi * u[3])], -1)


def _random_force(seed, n, kd, kT, dt, first, steps):
    """F^R[step, particle, 3] = sum_s A_s W_{n+s}, A_s the inverse transform of the square root of the noise target's."""
    m = len(kd)
    c = kT / dt * kd * np.where(np.arange(m) == 0, 2.0, 1.0)
    L = 2 * m - 1
    spec = np.fft.fft(np.concatenate([c, c[:0:-1]])).real
    a = np.fft.fftshift(np.fft.ifft(np.sqrt(np.maximum(spec, 0.0))).real)  # A_s at s + m - 1
    w = _gauss(seed, np.arange(n), np.arange(first - (m - 1), first + steps + m - 1))
    out = np.empty((steps, n, 3))
    for t in range(steps):
        out[t] = np.tensordot(a, w[t:t + L], axes=(0, 0))
    return out


def exact(case, seed):
    """One pass of a small `run` case as the discrete equations give it in 64 bits, particles pair by pair."""
    c = case
    if (c["kind"] != "run" or c["n"] * c["m_max"] > GIVEN_HISTORY or c["hist"] != "f32" or c["pair_noise"]
            or c["n"] ** 2 * c["steps"] > 2e9 or c["n"] > 6000 or c["vacf_len"]):
        return None
    w, pos, vel, hist = _initial(c, seed)
    terms, perp = _terms(c, w)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    f64 = dict(dtype=torch.float64, device=dev)
    dt, M, box, m = w.dt, w.mass, w.box, w.m_max

    def weights(x):  # continuous samples to the delta comb's weights
        return np.asarray(x, dtype=np.float64).reshape(-1) * dt * np.where(np.arange(m) == 0, 0.5, 1.0)

    kd = weights(terms["Ks"])
    noise = torch.tensor(_random_force(w.seed, w.n, kd, w.kT, dt, c["first"], c["steps"]), **f64)
    rows = [kd] + [weights(terms[k]) for k in ("g", "gs") if k in terms]
    coef = torch.tensor(np.stack(rows)[:, 1:], **f64)  # m = 1 ..
    zero = [float(r[0]) for r in rows]

    def table(x):
        return None if x is None else torch.tensor(np.asarray(x, dtype=np.float64).reshape(-1), **f64)

    fpar = [table(terms.get("f")), table(terms.get("fs"))]
    fper = [table(perp["fp"] if perp else None), table(perp["fs"] if perp else None)]
    x, v = torch.tensor(pos, **f64), torch.tensor(vel, **f64)
    h = torch.tensor(hist, **f64)
    disp = torch.zeros_like(x)

    def pairs(x):
        d = x[:, None, :] - x[None, :, :]
        d -= box * torch.round(d / box)
        r2 = (d * d).sum(-1)
        r2.fill_diagonal_(math.inf)
        i, j = torch.nonzero(r2 < w.r_c ** 2, as_tuple=True)
        r = r2[i, j].sqrt()
        return i, j, d[i, j] / r[:, None], r

    def radial(t, r):
        s = r / terms["dr"]
        k = s.floor().long().clamp(max=len(t) - 2)
        return t[k] + (s - k) * (t[k + 1] - t[k])

    def conservative(p):
        i, _, e, r = p
        return torch.zeros_like(x).index_add_(0, i, (2 * w.A_cons / w.r_c * (1 - r / w.r_c))[:, None] * e)

    b = 1.0 / (1.0 + dt * zero[0] / (2 * M))
    a = b * (1.0 - dt * zero[0] / (2 * M))
    p = pairs(x)
    fc = conservative(p)
    for t in range(c["steps"]):
        S = torch.tensordot(coef, h, dims=([1], [0]))  # [terms, n, 3]
        fd = -S[0] / dt
        i, j, e, r = p
        for q, (par, per) in enumerate(zip(fpar, fper)):  # pair term on the neighbour, self-difference on itself
            if par is None:
                continue
            of = j if q == 0 else i
            y = zero[1 + q] * v[of] + S[1 + q][of] / dt
            ey = (e * y).sum(-1, keepdim=True) * e
            force = radial(par, r)[:, None] * ey
            if per is not None:
                force = force + radial(per, r)[:, None] * (y - ey)
            fd = fd.index_add(0, i, -force)
        step = b * dt * v + b * dt * dt / (2 * M) * (fc + fd + noise[t])
        x = torch.remainder(x + step, box)
        disp = disp + step
        h = torch.cat([step[None], h[:-1]])
        p = pairs(x)
        new = conservative(p)
        v = a * v + dt / (2 * M) * (a * fc + new) + b * dt / M * (fd + noise[t])
        fc = new
    return dict(vel=v.cpu().numpy(), disp=disp.cpu().numpy())
