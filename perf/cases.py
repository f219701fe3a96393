"""Timed workloads of the lattice library, through its public Python binding.

Four kinds of work, as programs use the library:

- ``evolve``: one simulation job on one lattice: load the initial state from
  (page-locked) host arrays, take ``steps`` leapfrog steps, read energies, scale
  factor, means and variances every ``every`` steps (0: only at the end), and
  take the complete staggered state (the checkpoint form) back to the host.
- ``batch``: a group of lattices of uneven dimension and size advanced together,
  then every member's state back on the host.  The members go on from pass to
  pass, as in the serving loop's step chunks.
- ``outputs``: the read-outs of a resident state: energies, means, variances and
  every field's power spectrum.
- ``moments``: means and variances of field arrays the caller already holds in
  device memory (the allocation-free call).

Checkpoints and read-outs of FP32 runs are kept in FP32, the precision such a run
has; those of FP64 runs in FP64.  Inputs follow the repository's recipe (Gaussian
random fields with |d_k|^2 = 1/(2 omega_k), random phases, modes above N/4
removed), drawn on the device, at the tests' larger amplitude 1e-2: at 1e-4 the
variance and the gradient energy of an FP32 run are the rounding of phi ~ 1.
Sides above 256 keep the spacing of the 256^3 run (the box grows with the
lattice), so FP32's rounding times 1/dx^2 stays that of the ordinary runs.
"""
import math

import numpy as np
import torch

from paper_0712_0813_gb300 import capi
from paper_0712_0813_gb300.icgen import courant_dt

Q = (0.8, 5.0, 40.0)      # couplings of the four-field model; two fields take 1.2
AMP = 1e-2
PHI0_OVER_MPL = 0.342
L2_BYTES = 96e6           # a state up to about this size need not leave the chip between steps


# ---- the cases ---------------------------------------------------------------

def _evolve(name, dims, N, nf, precision, expansion, steps, every=0):
    c = {"kind": "evolve", "dims": dims, "N": N, "nf": nf, "precision": precision,
         "expansion": expansion, "steps": steps, "every": every}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the plain FP64 run (32^3, box 20, dt 0.05, 1000 steps, no expansion): small
        # lattices, parameter scans, where a step is a few microseconds
        _evolve("plain_32cube_f64", 3, 32, 2, "f64", False, 1000),
        # the smallest 3D lattice of the serving mix, FP32, expanding
        _evolve("small_64cube_f32", 3, 64, 2, "f32", True, 1000),
        # the expanding 256^3 run, FP32, with its statistics read every 50 steps
        _evolve("cube256_f32", 3, 256, 2, "f32", True, 400, 50),
        # the same run in FP64 (the reference precision)
        _evolve("cube256_f64", 3, 256, 2, "f64", True, 200, 100),
        # four fields on 512^3, FP32: the largest job
        _evolve("cube512_4field_f32", 3, 512, 4, "f32", True, 250),
        # an odd side in 3D (no aligned rows), FP32
        _evolve("odd_383cube_f32", 3, 383, 2, "f32", True, 300, 100),
        # a large odd 2D lattice, FP32, without expansion
        _evolve("odd_6001sq_f32", 2, 6001, 2, "f32", False, 400, 200),
        # a 2D lattice in FP64, expanding
        _evolve("sq1024_f64", 2, 1024, 2, "f64", True, 500, 100),
        # the 1D lattice of the mixed batch, alone
        _evolve("line_65536_f32", 1, 65536, 2, "f32", True, 1000),
        # the 96-lattice mixed batch: 32 each of 1D 65536, 2D 1024^2, 3D 64..192
        {"name": "batch_mix_96_f32", "kind": "batch", "per_kind": 32, "side_min": 64, "side_max": 192,
         "precision": "f32", "steps": 200},
        # all outputs of a resident 256^3 FP32 state
        {"name": "outputs_256cube_f32", "kind": "outputs", "dims": 3, "N": 256, "nf": 2, "precision": "f32"},
        # moments of four 128^3 FP32 arrays that another allocator owns
        {"name": "moments_128cube_x4_f32", "kind": "moments", "n": 128 ** 3, "nf": 4, "precision": "f32"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["evolve"] * 7 + ["batch", "outputs", "moments"])
    precision = rng.choice(["f32", "f32", "f64"])
    nf = rng.choice([1, 2, 2, 2, 3, 4])
    if kind == "moments":
        return {"kind": kind, "n": _log_int(rng, 1000, 1 << 26), "nf": nf, "precision": precision}
    if kind == "batch":
        return {"kind": kind, "per_kind": rng.randint(2, 24), "side_min": 32, "side_max": rng.choice([96, 128, 160]),
                "precision": precision, "steps": rng.randint(20, 80) if precision == "f32" else rng.randint(5, 20)}
    dims = rng.choice([1, 2, 2, 3, 3, 3, 3])
    N = _log_int(rng, *{1: (1000, 1 << 22), 2: (48, 6144), 3: (16, 448)}[dims])
    r = rng.random()
    if r < 0.35:
        N |= 1                                  # odd sides
    elif r < 0.7:
        N = max(16, N // 32 * 32)               # the usual multiples of 32
    if kind == "outputs":
        N = min(N, {1: 1 << 20, 2: 4096, 3: 320}[dims])
        return {"kind": kind, "dims": dims, "N": N, "nf": nf, "precision": precision}
    site_steps = 2.5e9 if precision == "f32" else 5e8
    steps = int(max(20, min(1000, site_steps * rng.uniform(0.5, 1.0) / (N ** dims * nf))))
    return _evolve(None, dims, N, nf, precision, rng.random() < 0.6, steps, rng.choice([0, 50, 100]))


# ---- inputs ------------------------------------------------------------------

def _couplings(nf):
    return (1.2,) if nf == 2 else Q[:nf - 1]


def _box(N):
    return 20.0 * max(1.0, N / 256.0)


def _dt(dims, N, L, q):
    return courant_dt(dims, N, L, 1.0, q)


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _random_field(dims, N, L, m2, mean, gen, dev):
    """(f, u) on the device: one field's Gaussian random field and its velocity."""
    axis = torch.fft.fftfreq(N, d=1.0 / N, dtype=torch.float64, device=dev) ** 2
    n2 = (torch.fft.rfftfreq(N, d=1.0 / N, dtype=torch.float64, device=dev) ** 2).reshape((1,) * (dims - 1) + (-1,))
    for d in range(dims - 1):
        n2 = n2 + axis.reshape((1,) * d + (-1,) + (1,) * (dims - 1 - d))
    keep = (n2 > 0) & (n2 <= (N / 4.0) ** 2)
    omega = torch.sqrt(n2 * (2.0 * math.pi / L) ** 2 + m2)
    theta = torch.rand(n2.shape, dtype=torch.float64, device=dev, generator=gen) * (2.0 * math.pi)
    c = torch.polar(torch.where(keep, torch.sqrt(0.5 / omega), torch.zeros_like(omega)), theta)
    scale = AMP * math.sqrt(float(N) ** dims)
    f = torch.fft.irfftn(c, s=(N,) * dims).mul_(scale).add_(mean)
    u = torch.fft.irfftn(c.mul_(omega), s=(N,) * dims).mul_(scale)
    return f, u


def _fields(dims, N, L, nf, q, seed, dev):
    gen = torch.Generator(device=dev).manual_seed(int(seed) * 7919 + 17)
    masses = [3.0] + list(q)
    for i in range(nf):
        yield _random_field(dims, N, L, masses[i], 1.0 if i == 0 else 0.0, gen, dev)


def _host(shape):
    return torch.empty(shape, dtype=torch.float64, pin_memory=torch.cuda.is_available())


def _host_fields(dims, N, L, nf, q, seed):
    f0, u0 = _host((nf, N ** dims)), _host((nf, N ** dims))
    for i, (f, u) in enumerate(_fields(dims, N, L, nf, q, seed, _device())):
        f0[i].copy_(f.reshape(-1))
        u0[i].copy_(u.reshape(-1))
    return f0.numpy(), u0.numpy()


def _batch_specs(case, seed):
    """(dims, N, q, phi0, expansion) of the members; the 3D sides are multiples of 32."""
    rng = np.random.default_rng([int(seed), 96])
    sides = list(range(case["side_min"], case["side_max"] + 1, 32))
    fixed = np.random.default_rng(5)            # the mix's shapes belong to the case, not to the inputs
    specs = []
    for k in range(3 * case["per_kind"]):
        dims = 1 + k // case["per_kind"]
        N = 65536 if dims == 1 else 1024 if dims == 2 else int(fixed.choice(sides))
        q = (float(math.exp(rng.uniform(math.log(0.5), math.log(20.0)))),)
        L = _box(N)
        specs.append({"dims": dims, "N": N, "L": L, "q": q, "expansion": k % 2 == 0,
                      "dt": courant_dt(dims, N, L, 1.0, q, amp=4.0)})
    return specs


def prepare(case, seed):
    f32 = case["precision"] == "f32"
    if case["kind"] == "moments":
        gen = torch.Generator(device="cuda").manual_seed(int(seed) + 3)
        f = torch.randn((case["nf"], case["n"]), device="cuda", generator=gen,
                        dtype=torch.float32 if f32 else torch.float64).mul_(1e-3)
        f[0].add_(1.0)
        return {"case": case, "f": f, "mean": torch.zeros(case["nf"], dtype=torch.float64, device="cuda"),
                "var": torch.zeros(case["nf"], dtype=torch.float64, device="cuda")}
    if case["kind"] == "batch":
        specs = _batch_specs(case, seed)
        sims, total = [], 0
        for k, s in enumerate(specs):
            sim = capi.Simulation(dims=s["dims"], N=s["N"], L=s["L"], dt=s["dt"], nfields=2, q=s["q"],
                                  expansion=s["expansion"], precision=case["precision"])
            f0, u0 = _host_fields(s["dims"], s["N"], s["L"], 2, s["q"], int(seed) * 1000 + k)
            sim.set_fields(f0, u0)
            sims.append(sim)
            total += f0.size
        state = {"case": case, "sims": sims, "batch": capi.Batch(sims), "image": _host((2, total))}
        if f32:
            state["keep"] = torch.zeros((2, total), dtype=torch.float32)
            state["keep"].fill_(1.0)            # touch the pages once
        return state
    dims, N, nf = case["dims"], case["N"], case["nf"]
    q, L = _couplings(nf), _box(N)
    f0, u0 = _host_fields(dims, N, L, nf, q, seed)
    sim = capi.Simulation(dims=dims, N=N, L=L, dt=_dt(dims, N, L, q), nfields=nf, q=q,
                          expansion=case.get("expansion", True), precision=case["precision"])
    state = {"case": case, "sim": sim, "f0": f0, "u0": u0}
    if case["kind"] == "outputs":
        sim.set_fields(f0, u0)
        return state
    state["image"] = _host((2, f0.size))
    if f32:
        state["keep"] = torch.zeros((2, f0.size), dtype=torch.float32)
        state["keep"].fill_(1.0)                # touch the pages once
    return state


# ---- one pass ----------------------------------------------------------------

def _checkpoint(state):
    """The run's state, f then v, as the run keeps it: in FP32 for an FP32 run."""
    return state["keep"].copy_(state["image"]) if "keep" in state else state["image"]


def _series(rows, dtype):
    """Per-quantity arrays of a run's read-outs."""
    return {name: np.array([r[name] for r in rows], dtype=dtype) for name in rows[0]}


def _bins(case):
    return int(math.ceil(math.sqrt(case["dims"]) * (case["N"] // 2))) + 2 if case["dims"] > 1 \
        else min(case["N"] // 2 + 2, 2048)


def _read(sim):
    e = sim.energy()
    mean, var = sim.means_variances()
    return {"K": e["K"], "G": e["G"], "V": e["V"], "E": e["E"], "a": e["a"], "ap": e["ap"], "mean": mean, "var": var}


def run(state):
    case = state["case"]
    dtype = np.float32 if case["precision"] == "f32" else np.float64
    if case["kind"] == "moments":
        f = state["f"]
        capi.ce_moments_noalloc(f.data_ptr(), capi.CE_F32 if dtype == np.float32 else capi.CE_F64, case["n"],
                                case["nf"], torch.cuda.current_stream().cuda_stream, state["mean"].data_ptr(),
                                state["var"].data_ptr())
        return {"mean": state["mean"], "var": state["var"]}
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
        at, a = 0, []
        f, v = state["image"].numpy()
        for sim in state["sims"]:
            n = 2 * sim.sites
            _, _, sc = capi.ce_get_fields(sim.handle, 2, sim.sites, capi.CE_VEL_STAGGERED,
                                          out=(f[at:at + n], v[at:at + n]))
            a.append((sc.a, sc.ap_half))
            at += n
        return {"state": _checkpoint(state), "a": np.array(a, dtype=dtype)}
    sim = state["sim"]
    if case["kind"] == "outputs":
        out = _series([_read(sim)], dtype)
        for i in range(case["nf"]):
            k, p, n = sim.spectrum(i, _bins(case))
            out["k%d" % i], out["count%d" % i] = k, n
            # the fluctuation bins; phi's zero mode (S <phi>)^2 stands apart
            out["power%d" % i], out["zero%d" % i] = p[1:].astype(dtype), p[:1].astype(dtype)
        if case["nf"] > 1:
            del out["zero1"]                    # rounding noise: chi has no zero mode
        for i in range(2, case["nf"]):
            del out["zero%d" % i]
        return out
    sim.set_fields(state["f0"], state["u0"])
    left, rows = case["steps"], []
    while left > 0:
        n = min(left, case["every"] or left)
        sim.step(n)
        left -= n
        rows.append(_read(sim))
    _, _, sc = capi.ce_get_fields(sim.handle, case["nf"], sim.sites, capi.CE_VEL_STAGGERED,
                                  out=tuple(state["image"].numpy()))
    return {"state": _checkpoint(state), "read": _series(rows, dtype),
            "a": np.array([sc.a, sc.ap_half], dtype=dtype)}


# ---- what a pass cannot do without ----------------------------------------------

def _evolve_work(dims, S, nf, es, steps):
    """A step reads f and v and writes both, unless the state fits on the chip;
    about 12 + 6 dims operations a field and site."""
    state = 2.0 * nf * S * es
    return (2.0 * state * steps if state > L2_BYTES else 2.0 * state), (12.0 + 6.0 * dims) * nf * S * steps


def work(case):
    es = 4 if case["precision"] == "f32" else 8
    if case["kind"] == "moments":
        return {"bytes": float(es * case["n"] * case["nf"]), "flops": 4.0 * case["n"] * case["nf"]}
    if case["kind"] == "batch":
        b = fl = 0.0
        specs = _batch_specs(case, 0)
        total = sum(2.0 * 2 * s["N"] ** s["dims"] * es for s in specs)
        for s in specs:
            fl += _evolve_work(s["dims"], s["N"] ** s["dims"], 2, es, case["steps"])[1]
        b = 2.0 * total * case["steps"] if total > L2_BYTES else 2.0 * total
        return {"bytes": b + total / es * 8, "flops": fl}
    S, nf, dims = case["N"] ** case["dims"], case["nf"], case["dims"]
    if case["kind"] == "outputs":
        # the state once, and a transform of every field
        return {"bytes": 2.0 * nf * S * es, "flops": nf * S * (12.0 + 6.0 * dims + 2.5 * math.log2(S))}
    b, fl = _evolve_work(dims, S, nf, es, case["steps"])
    return {"bytes": b + 2.0 * 2 * nf * S * 8, "flops": fl}


# ---- the same in 64 bits, plain torch ---------------------------------------------

class _Plain:
    """The leapfrog of one lattice in FP64, operation by operation."""

    def __init__(self, dims, N, L, dt, nf, q, expansion, seed):
        self.dims, self.N, self.dt, self.nf, self.q, self.expansion = dims, N, dt, nf, q, expansion
        self.idx2 = (N / L) ** 2
        self.kappa2 = 8.0 * math.pi / 3.0 * PHI0_OVER_MPL ** 2
        fu = list(_fields(dims, N, L, nf, q, seed, _device()))
        self.f, self.v = [x[0] for x in fu], [x[1] for x in fu]
        self.a, self.ap, self.app = 1.0, 0.0, 0.0
        G, V = self.sums()
        if expansion:
            K = sum(float((u * u).mean()) for u in self.v) * 0.5
            self.ap = math.sqrt(self.kappa2 * (K + sum(G) + V))
            self.app = -self.ap ** 2 + self.kappa2 * (2.0 * sum(G) + 3.0 * V)
            for f, v in zip(self.f, self.v):
                v.add_(f, alpha=self.ap)
        self.kick(0.5 * dt)
        self.ap += 0.5 * dt * self.app

    def sums(self):
        G = []
        for f in self.f:
            g = torch.zeros((), dtype=torch.float64, device=f.device)
            for d in range(self.dims):
                g += (torch.roll(f, -1, d) - f).square_().mean()
            G.append(0.5 * self.idx2 * float(g))
        phi2 = self.f[0] * self.f[0]
        w = phi2 * 0.25
        for q, chi in zip(self.q, self.f[1:]):
            w += 0.5 * q * chi * chi
        return G, float((phi2 * w).mean())

    def force(self, i):
        f, phi = self.f[i], self.f[0]
        acc = f * (-2.0 * self.dims)
        for d in range(self.dims):
            acc += torch.roll(f, 1, d)
            acc += torch.roll(f, -1, d)
        acc *= self.idx2
        if i == 0:
            w = phi * phi
            for q, chi in zip(self.q, self.f[1:]):
                w += q * chi * chi
            acc -= w * phi
        else:
            acc -= self.q[i - 1] * phi * phi * f
        if self.expansion:
            acc.add_(f, alpha=self.app / self.a)
        return acc

    def kick(self, h):
        forces = [self.force(i) for i in range(self.nf)]
        for v, F in zip(self.v, forces):
            v.add_(F, alpha=h)

    def step(self):
        dt = self.dt
        for f, v in zip(self.f, self.v):
            f.add_(v, alpha=dt)
        if self.expansion:
            G, V = self.sums()
            self.a += dt * self.ap
            Q_ = self.kappa2 * (2.0 * sum(G) + 3.0 * V) / self.a
            C = 2.0 * self.ap + dt * Q_
            u = 2.0 * C / (1.0 + math.sqrt(1.0 + dt * C / self.a))
            self.app = (u - 2.0 * self.ap) / dt
            self.ap = u - self.ap
        self.kick(dt)

    def read(self):
        G, V = self.sums()
        ap = self.ap - 0.5 * self.dt * self.app
        K, mean, var = [], [], []
        for i, f in enumerate(self.f):
            u = self.v[i] - 0.5 * self.dt * self.force(i) - ap / self.a * f
            K.append(0.5 * float((u * u).mean()))
            m = float(f.mean())
            mean.append(m)
            var.append(float((f - m).square_().mean()))
        return {"K": K, "G": G, "V": V, "E": sum(K) + sum(G) + V, "a": self.a, "ap": ap, "mean": mean, "var": var}

    def spectrum(self, i, nbins):
        F = torch.fft.rfftn(self.f[i])
        N, dims = self.N, self.dims
        axis = torch.fft.fftfreq(N, d=1.0 / N, dtype=torch.float64, device=F.device) ** 2
        x = torch.fft.rfftfreq(N, d=1.0 / N, dtype=torch.float64, device=F.device) ** 2
        n2 = x.reshape((1,) * (dims - 1) + (-1,))
        for d in range(dims - 1):
            n2 = n2 + axis.reshape((1,) * d + (-1,) + (1,) * (dims - 1 - d))
        weight = torch.full_like(x, 2.0)
        weight[0] = 1.0
        if N % 2 == 0:
            weight[-1] = 1.0
        weight = weight.expand(n2.shape)
        b = torch.floor(torch.sqrt(n2) + 0.5).long().reshape(-1)
        keep = b < nbins
        p2 = (weight * (F.real ** 2 + F.imag ** 2)).reshape(-1)
        n = torch.bincount(b[keep], weight.reshape(-1)[keep], minlength=nbins)
        p = torch.bincount(b[keep], p2[keep], minlength=nbins)
        return torch.where(n > 0, p / n, torch.zeros_like(p)), n

    def state(self):
        return torch.stack([torch.cat([x.reshape(-1) for x in xs]) for xs in (self.f, self.v)])


def exact(case, seed):
    if case["kind"] == "moments":
        f = prepare(case, seed)["f"].double()
        return {"mean": f.mean(1), "var": f.var(1, unbiased=False)}
    if case["kind"] == "batch":
        states, a = [], []
        for k, s in enumerate(_batch_specs(case, seed)):
            p = _Plain(s["dims"], s["N"], s["L"], s["dt"], 2, s["q"], s["expansion"], int(seed) * 1000 + k)
            for _ in range(case["steps"]):
                p.step()
            states.append(p.state())
            a.append((p.a, p.ap))
        return {"state": torch.cat(states, dim=1), "a": np.array(a)}
    dims, N, nf = case["dims"], case["N"], case["nf"]
    q, L = _couplings(nf), _box(N)
    p = _Plain(dims, N, L, _dt(dims, N, L, q), nf, q, case.get("expansion", True), seed)
    if case["kind"] == "outputs":
        out = _series([p.read()], np.float64)
        for i in range(nf):
            power, n = p.spectrum(i, _bins(case))
            out["k%d" % i], out["count%d" % i] = 2.0 * math.pi / L * torch.arange(_bins(case), dtype=torch.float64), n
            out["power%d" % i] = power[1:]
            if i == 0:
                out["zero0"] = power[:1]
        return out
    rows, left = [], case["steps"]
    while left > 0:
        n = min(left, case["every"] or left)
        for _ in range(n):
            p.step()
        left -= n
        rows.append(p.read())
    return {"state": p.state(), "read": _series(rows, np.float64), "a": np.array([p.a, p.ap])}
