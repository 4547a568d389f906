"""Performance cases of the library: what its users have it do, over the sizes they do it at.

A case is a dict of plain values.  listed() names the fixed ones, draw() gives more of the same ranges; prepare() makes a
case's inputs and handles from a seed, run() makes one pass through the public entry points, work() says what a pass
cannot do without, and exact() computes a pass's outputs in 64 bits with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2211_15630_gb300 as A

DEV = "cuda"


# ------------------------------------------------------------------ cases --
def _box(n, rho, aspect=1.0):
    """Sides of a box of n particles at density rho, at least four interaction radii each."""
    ly = max(math.sqrt(n / rho / aspect), 4.0)
    return max(ly * aspect, 4.0), ly


def _case(kind, n=0, **kw):
    """A particle case with the defaults of the library's own workloads (R = 1, periodic, one species, uniform start)."""
    c = {"kind": kind, "n": n, "model": "vm", "rho": 2.0, "aspect": 1.0, "eta": 0.45, "v": 0.5, "dt": 0.01,
         "order": 1, "walls": False, "kn": 0, "species": 1, "start": "uniform", "steps": 20, "bins": 128}
    c.update(kw)
    return c


def listed():
    return [
        # the library's default system (1000 particles, 32 x 32): p(t) of a short run, where launches and latency are all
        dict(_case("trace", 1000, rho=1000 / 1024, eta=0.4, steps=200), name="trace_n1000"),
        # the small workload (8192 particles, L = 64): moments, Binder cumulant and histograms measured on the fly
        dict(_case("measure", 8192, eta=0.4, steps=40), name="measure_n8192"),
        # an odd-sized mixture of three species with non-reciprocal couplings (Langevin), a few thousand to 1e5 particles
        dict(_case("step", 50021, model="langevin", v=1.0, eta=0.3, species=3, steps=50), name="species_langevin_n50021"),
        # the surrogate's data: 524,288 particles in 512 x 512, a 128 x 128 frame every 10 steps
        dict(_case("frames", 524288, eta=0.4, steps=10, bins=128), name="frames_n524288"),
        # the Brownian workload: overdamped Langevin alignment, 2^20 particles between four reflecting walls
        dict(_case("step", 1 << 20, model="langevin", rho=2.0004, v=1.0, eta=math.sqrt(0.2), walls=True, steps=50),
             name="brownian_walls_n2^20"),
        # a flocking state (half of the particles in dense aligned flocks), a ragged number of particles in an oblong box
        dict(_case("step", 1000003, eta=0.3, aspect=1.3, start="flocks", steps=16), name="flocks_n1000003"),
        # nematic Vicsek particles at high density
        dict(_case("step", 300000, model="nvm", rho=4.0, eta=0.2, steps=16), name="nvm_rho4_n300000"),
        # metric-free Vicsek, the six nearest neighbours
        dict(_case("step", 1 << 20, kn=6, rho=2.0004, steps=10), name="metric_free_k6_n2^20"),
        # a phase-diagram sweep: replicas of 2^10 to 2^16 particles at mixed densities and noises, measured, one frame each
        dict(_case("ensemble", 0, replicas=64, nmax_log2=16.0, steps=40, bins=32), name="ensemble_64"),
        # the large workload end to end: a checkpoint restored from host memory, 16 steps, the state read back
        dict(_case("restore", 1 << 24, rho=2.0004, steps=16), name="restore_n2^24"),
        # one training step of the surrogate at its training batch
        {"kind": "train", "batch": 32, "h": 128, "w": 128, "conserve": 3, "apps": 1, "name": "train_b32_128x128"},
        # a rollout of one state 100 particle steps ahead
        {"kind": "predict", "batch": 1, "h": 128, "w": 128, "conserve": 3, "apps": 10, "name": "predict_b1_128x128"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["trace", "measure", "step", "step", "step", "metric_free", "frames", "restore", "ensemble", "train",
                       "predict"])
    if kind in ("train", "predict"):
        return {"kind": kind, "batch": _log(rng, 1, 32), "h": 16 * rng.randint(3, 8), "w": 16 * rng.randint(3, 8),
                "conserve": rng.choice([0, 3]), "apps": 1 if kind == "train" else rng.randint(1, 10)}
    c = dict(rho=rng.choice([0.5, 1.0, 2.0, 4.0]), eta=round(rng.uniform(0.1, 0.7), 3), aspect=round(rng.uniform(0.7, 1.4), 3))
    if kind == "trace":
        return _case(kind, _log(rng, 500, 20000), steps=rng.randint(50, 200), **c)
    if kind == "measure":
        return _case(kind, _log(rng, 4000, 150000), steps=rng.randint(20, 40), **c)
    if kind == "frames":
        return _case(kind, _log(rng, 100000, 1 << 22), steps=10, bins=rng.choice([64, 128, 181, 256, 512]), **c)
    if kind == "restore":
        return _case(kind, _log(rng, 1 << 19, 1 << 23), steps=rng.randint(5, 16), **c)
    if kind == "metric_free":
        return _case("step", _log(rng, 20000, 1 << 20), kn=rng.randint(3, 12), steps=rng.randint(3, 10), **c)
    if kind == "ensemble":
        return _case(kind, 0, replicas=_log(rng, 16, 64), nmax_log2=round(rng.uniform(12.0, 16.0), 2), steps=rng.randint(20, 40),
                     bins=32)
    model = rng.choice(["vm", "nvm", "langevin"])
    c.update(model=model, walls=rng.choice([False, True]) and model != "nvm", start=rng.choice(["uniform", "flocks"]))
    if model == "langevin":
        c.update(v=1.0, order=rng.choice([1, 1, 2]))
    steps = rng.randint(5, 30 if model == "langevin" else 16)
    return _case("step", _log(rng, 20000, 1 << 21), steps=steps, species=rng.choice([1, 1, 3]), **c)


# ----------------------------------------------------------------- inputs --
MODELS = {"vm": 0, "langevin": 1, "nvm": 2}


def _systems(case, seed):
    """The systems of a case as dicts (one, or the replicas of an ensemble)."""
    if case["kind"] != "ensemble":
        n = case["n"]
        lx, ly = _box(n, case["rho"], case["aspect"])
        s = dict(n=n, lx=lx, ly=ly, v=case["v"], eta=case["eta"], seed=1000 + seed)
        if case["species"] > 1:
            k = case["species"]
            cnt = [n // k] * (k - 1)
            # unequal speeds, noises and chiralities; couplings that are not reciprocal
            s.update(counts=cnt + [n - sum(cnt)], vs=[case["v"] * (1.0 - 0.2 * a) for a in range(k)],
                     etas=[case["eta"] * (1.0 + 0.3 * a) for a in range(k)], omegas=[0.1 * a for a in range(k)],
                     gammas=[[1.0 if a == b else 0.5 * (1 + a - b) for b in range(k)] for a in range(k)])
        return [s]
    g = np.random.default_rng(seed)
    out = []
    for r in range(case["replicas"]):
        n = int(round(2.0 ** g.uniform(10.0, case["nmax_log2"])))
        lx, ly = _box(n, float(g.choice([0.5, 1.0, 2.0, 4.0])))
        out.append(dict(n=n, lx=lx, ly=ly, v=case["v"], eta=float(g.uniform(0.1, 0.7)), seed=1000 + 977 * seed + r))
    return out


def _params(case, s):
    p = A.aap_params_default(n=s["n"], lx=s["lx"], ly=s["ly"], r=1.0, v=s["v"], eta=s["eta"], dt=case["dt"], gamma=1.0,
                             order=case["order"], model=MODELS[case["model"]], bx=int(case["walls"]), by=int(case["walls"]),
                             kn=case["kn"], seed=s["seed"])
    if "counts" in s:
        A.set_species(p, s["counts"], s["vs"], s["etas"], s["omegas"], s["gammas"])
    return p


def _start(case, s, seed):
    """Positions and orientations (FP64, on the GPU): uniform and isotropic, or half of them in aligned flocks."""
    g = torch.Generator(device=DEV)
    g.manual_seed(7919 * seed + 17)
    n, lx, ly = s["n"], s["lx"], s["ly"]
    u = torch.rand((3, n), generator=g, device=DEV, dtype=torch.float64)
    x, y, th = u[0] * lx, u[1] * ly, (2.0 * u[2] - 1.0) * math.pi
    if case["start"] == "flocks":
        nf = max(1, n // 400)                                   # flocks of about 200 particles, some three radii wide
        m = n // 2
        f = torch.randint(0, nf, (m,), generator=g, device=DEV)
        c = torch.rand((3, nf), generator=g, device=DEV, dtype=torch.float64)
        d = torch.randn((3, m), generator=g, device=DEV, dtype=torch.float64)
        x[:m] = torch.remainder(c[0][f] * lx + 1.5 * d[0], lx)
        y[:m] = torch.remainder(c[1][f] * ly + 1.5 * d[1], ly)
        th[:m] = (2.0 * c[2][f] - 1.0) * math.pi + 0.3 * d[2]
        perm = torch.randperm(n, generator=g, device=DEV)
        x, y, th = x[perm], y[perm], th[perm]
    th = (torch.remainder(th + math.pi, 2.0 * math.pi) - math.pi).float().clamp(-3.1415925, 3.1415925)
    return x.clamp(0.0, lx * (1.0 - 1e-12)), y.clamp(0.0, ly * (1.0 - 1e-12)), th


def _pinned(n):
    return (torch.empty(n, dtype=torch.float64, pin_memory=True).numpy(),
            torch.empty(n, dtype=torch.float64, pin_memory=True).numpy(),
            torch.empty(n, dtype=torch.float32, pin_memory=True).numpy())


class _Held:
    """A library handle, destroyed with the state that holds it."""

    def __init__(self, h, destroy):
        self.h, self.destroy = h, destroy

    def __del__(self):
        self.destroy(self.h)


def _fields(case, seed):
    """Coarse-grained fields like those of a Vicsek state at density 2 (batch, 3, h, w), the noises, the fields 10 steps on."""
    g = torch.Generator(device=DEV)
    g.manual_seed(104729 * seed + 3)
    b, h, w = case["batch"], case["h"], case["w"]
    z = torch.randn((b, 6, h, w), generator=g, device=DEV)
    k = torch.ones((1, 1, 5, 5), device=DEV) / 5.0
    z = torch.nn.functional.conv2d(torch.nn.functional.pad(z.reshape(-1, 1, h, w), (2, 2, 2, 2), mode="circular"), k)
    z = z.reshape(b, 6, h, w)
    f = torch.empty((b, 3, h, w), device=DEV)
    f[:, 0] = 2.0 * torch.exp(0.4 * z[:, 0])
    f[:, 1:] = f[:, :1] * (0.3 + 0.5 * torch.tanh(z[:, 1:3]))
    t = f + 0.15 * z[:, 3:]
    eta = 0.3 + 0.2 * torch.rand((b,), generator=g, device=DEV)
    return f.contiguous(), t.contiguous(), eta


LAYERS = ((16, 32, 4, 32), (32, 32, 32, 32), (32, 32, 32, 32), (32, 8, 32, 3))   # cin, cout padded; cin, cout used


def _weights(seed):
    """He-uniform weights of a network some way into its training, in the library's layout ([co][tap][ci], then biases)."""
    g = np.random.default_rng(seed + 31)
    out = []
    for cin, cout, ci, co in LAYERS:
        w = np.zeros((cout, 9, cin), np.float32)
        w[:co, :, :ci] = g.uniform(-1.0, 1.0, (co, 9, ci)) * math.sqrt(6.0 / (9.0 * ci)) * (0.1 if co == 3 else 1.0)
        bias = np.zeros(cout, np.float32)
        bias[:co] = 0.05 * g.normal(size=co) * (0.1 if co == 3 else 1.0)
        out += [w.reshape(-1), bias]
    return np.concatenate(out)


def prepare(case, seed):
    A.load()
    st = {"case": case}
    stream = torch.cuda.current_stream().cuda_stream
    kind = case["kind"]
    if kind in ("train", "predict"):
        f, t, eta = _fields(case, seed)
        p = A.aap_sur_params_default(nbx=case["w"], nby=case["h"], max_batch=case["batch"], conserve=case["conserve"])
        h = A.aap_sur_create(p, stream)
        st.update(held=_Held(h, A.aap_sur_destroy), f=f, t=t, eta=eta, out=torch.empty_like(f))
        A.aap_sur_set_params(h, _weights(seed))
        return st
    ss = _systems(case, seed)
    nb = case["bins"]
    if kind == "ensemble":
        h = A.aap_ens_create([_params(case, s) for s in ss], stream)
        st.update(held=_Held(h, A.aap_ens_destroy), fields=torch.empty((len(ss), 3, nb, nb), device=DEV))
        return st
    s = ss[0]
    h = A.aap_create(_params(case, s), stream)
    st.update(held=_Held(h, A.aap_destroy), n=s["n"])
    if kind == "frames":
        st["fields"] = torch.empty((3, nb, nb), device=DEV)
    else:
        st["out"] = _pinned(s["n"])
    x, y, th = _start(case, s, seed)
    if kind == "restore":
        st["start"] = _pinned(s["n"])
        for a, b in zip(st["start"], (x, y, th)):
            a[:] = b.cpu().numpy()
    else:
        A.aap_set_state(h, x.cpu().numpy(), y.cpu().numpy(), th.cpu().numpy(), 0)
    return st


# ------------------------------------------------------------------- pass --
def run(st):
    case, h = st["case"], st["held"].h
    kind = case["kind"]
    if kind == "train":
        loss = A.aap_sur_train_step(h, st["f"].data_ptr(), st["t"].data_ptr(), st["eta"].data_ptr(), case["batch"])
        return {"loss": loss, "grads": A.aap_sur_get_grads(h), "params": A.aap_sur_get_params(h)}
    if kind == "predict":
        A.aap_sur_predict(h, st["f"].data_ptr(), st["eta"].data_ptr(), case["batch"], case["apps"], st["out"].data_ptr())
        return {"fields": st["out"]}
    steps, nb = case["steps"], case["bins"]
    if kind == "ensemble":
        A.aap_ens_measure(h, steps)
        for r in range(case["replicas"]):
            A.aap_ens_coarse_grain(h, r, nb, nb, st["fields"][r].data_ptr())
        return {"phi_mean": A.aap_ens_phi_mean(h), "fields": st["fields"]}
    if kind == "frames":
        A.aap_step(h, steps)
        A.aap_coarse_grain(h, nb, nb, st["fields"].data_ptr())
        return {"fields": st["fields"]}
    out = {}
    if kind == "restore":
        A.aap_set_state(h, *st["start"], step=0)
    if kind == "trace":
        out["p"] = A.aap_phi_trace(h, steps)
    elif kind == "measure":
        A.aap_clear_results(h)
        A.aap_measure(h, steps)
        r = A.aap_get_results(h)
        th_hist, nb_hist = A.aap_get_histograms(h, 100, 100)
        out.update(p=np.array(r.p[:]), q=np.array(r.q[:]), nbar=np.array(r.nbar[:]), binder=r.binder, theta_hist=th_hist,
                   nbr_hist=nb_hist)
    else:
        A.aap_step(h, steps)
    out["x"], out["y"], out["theta"] = A.aap_get_state(h, st["n"], out=st["out"])
    return out


def work(case):
    """Bytes and operations of a pass.  The records (16 bytes a particle) are read and written once in a pass, and once in every
    step of it when both copies are larger than what the chip holds (about 128 MB); the operations of a step are a distance
    test and a sum for every neighbour (8) and some 60 for the noise, the angle and the streaming."""
    kind = case["kind"]
    if kind in ("train", "predict"):
        pix = case["batch"] * case["h"] * case["w"]
        macs = 9 * sum(ci * co for _, _, ci, co in LAYERS)
        weights = 4 * sum(co * 9 * ci + co for ci, co, _, _ in LAYERS)
        if kind == "predict":
            return {"bytes": 24 * pix + weights, "flops": 2 * macs * pix * case["apps"]}
        # forward, data gradients (not of the first layer) and weight gradients; weights, two moments, gradients
        data = 9 * sum(ci * co for _, _, ci, co in LAYERS[1:])
        return {"bytes": 24 * pix + 7 * weights, "flops": 2 * (2 * macs + data) * pix}
    if kind == "ensemble":
        tot, nbr = sum(s["n"] for s in _systems(case, 0)), math.pi * 2.0
    else:
        tot, nbr = case["n"], float(case["kn"] or math.pi * case["rho"])
    byts = 32.0 * tot * (case["steps"] if 32 * tot > 1 << 27 else 1)
    if kind in ("frames", "ensemble"):
        byts += 16.0 * tot + 12.0 * case["bins"] ** 2 * case.get("replicas", 1)
    else:
        byts += (40.0 if kind == "restore" else 20.0) * tot
    return {"bytes": byts, "flops": tot * case["steps"] * (8.0 * (nbr + 1.0) + 60.0)}


# ----------------------------------------------- the same passes in 64 bits --
M32 = 0xFFFFFFFF


def _philox(ids, step, seed):
    """Philox4x32-10 words 0 and 1, counter (id, step, 0), key = seed (Salmon et al., SC'11), in int64 arithmetic."""
    c0, c1 = ids.clone(), torch.full_like(ids, step & M32)
    c2, c3 = torch.full_like(ids, (step >> 32) & M32), torch.zeros_like(ids)
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57                # products mod 2^64
        c0, c1, c2, c3 = ((p1 >> 32) & M32) ^ c1 ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c3 ^ k1, p0 & M32
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1


def _uniform(w):
    return ((w >> 9).double() + 0.5) * 2.0 ** -23


def _wrap(t):
    return torch.remainder(t + math.pi, 2.0 * math.pi) - math.pi


class _Exact:
    """Systems stepped together in FP64: image particles around every box, cells, neighbours by cell rows."""

    def __init__(self, case, ss, states):
        self.case, self.ss = case, ss
        self.x, self.y, self.th = (torch.cat([s[k].double() for s in states]) for k in range(3))
        n = [s["n"] for s in ss]
        self.n = sum(n)
        rep = torch.tensor(n, device=DEV)
        self.sys = torch.repeat_interleave(torch.arange(len(ss), device=DEV), rep)
        self.ids = torch.cat([torch.arange(k, device=DEV) for k in n])
        per = lambda f: torch.tensor([float(f(s)) for s in ss], device=DEV, dtype=torch.float64)
        self.L = (per(lambda s: s["lx"]), per(lambda s: s["ly"]))
        side = lambda s: math.sqrt(s["lx"] * s["ly"] * case["kn"] / (s["n"] * math.pi)) if case["kn"] else 1.0
        cells = [[max(1, math.floor(s[k] / side(s))) for s in ss] for k in ("lx", "ly")]
        self.ring = 3 if case["kn"] else 1
        self.nc = [torch.tensor(c, device=DEV) for c in cells]
        self.pad = [c + 2 * self.ring for c in self.nc]
        size = self.pad[0] * self.pad[1]
        self.off = torch.cumsum(size, 0) - size
        self.ncell = int(size.sum())
        seeds = [s["seed"] for s in ss]
        self.seed = seeds[0] if len(ss) == 1 else torch.tensor(seeds, device=DEV)[self.sys]
        s0 = ss[0]
        if "counts" in s0:
            self.sp = torch.repeat_interleave(torch.arange(len(s0["counts"]), device=DEV), torch.tensor(s0["counts"], device=DEV))
            pick = lambda v: torch.tensor(v, device=DEV, dtype=torch.float64)[self.sp]
            self.v, self.eta, self.omega = pick(s0["vs"]), pick(s0["etas"]), pick(s0["omegas"])
            self.gamma = torch.tensor(s0["gammas"], device=DEV, dtype=torch.float64)
        else:
            self.sp, self.omega, self.gamma = None, 0.0, None
            self.v, self.eta = per(lambda s: s["v"])[self.sys], per(lambda s: s["eta"])[self.sys]
        self.step = 0

    def images(self):
        """Every particle with its images around the box: coordinates, angle, system, index of the original."""
        refl = self.case["walls"]
        x, y, th, sy, src = self.x, self.y, self.th, self.sys, torch.arange(self.n, device=DEV)
        for axis in (0, 1):
            q = x if axis == 0 else y
            L = self.L[axis][sy]
            w = self.ring * (L / self.nc[axis][sy])
            parts = [(x, y, th, sy, src)]
            for low in (True, False):
                near = torch.nonzero((q < w) if low == refl else (q >= L - w)).reshape(-1)
                Ls = L[near]
                qq = q[near]
                img = (-qq if low else 2.0 * Ls - qq) if refl else (qq - Ls if low else qq + Ls)
                t = th[near]
                if refl:
                    t = (math.pi - t) if axis == 0 else -t
                parts.append((img if axis == 0 else x[near], y[near] if axis == 0 else img, t, sy[near], src[near]))
            x, y, th, sy, src = (torch.cat(v) for v in zip(*parts))
        return x, y, th, sy, src

    def sort(self):
        x, y, th, sy, src = self.images()
        cell = [torch.clamp(torch.floor(q / (self.L[a][sy] / self.nc[a][sy])).long() + self.ring, torch.zeros_like(sy),
                            self.pad[a][sy] - 1) for a, q in enumerate((x, y))]
        c = self.off[sy] + cell[1] * self.pad[0][sy] + cell[0]
        c, o = torch.sort(c)
        start = torch.zeros(self.ncell + 1, device=DEV, dtype=torch.long)
        start[1:] = torch.cumsum(torch.bincount(c, minlength=self.ncell), 0)
        own = torch.nonzero(o < self.n).reshape(-1)             # originals, in cell order
        return x[o], y[o], th[o], src[o], start, own, o[own], c[own], self.pad[0][sy[o[own]]]

    def metric(self):
        """Per particle: sums over its neighbours (complex exponentials, or weighted sines) and their number."""
        X, Y, T, src, start, own, who, c, row = self.sort()
        cT, sT = torch.cos(self.case["order"] * T), torch.sin(self.case["order"] * T)
        a, b, n = (torch.zeros(self.n, device=DEV, dtype=torch.float64) for _ in range(3))
        xi, yi, ci, si = X[own], Y[own], cT[own], sT[own]
        a1, b1, n1 = torch.zeros_like(xi), torch.zeros_like(xi), torch.zeros_like(xi)
        model = self.case["model"]
        for d in (-1, 0, 1):
            first = start[c + d * row - 1]
            length = start[c + d * row + 2] - first
            k = 0
            live = torch.nonzero(length > 0).reshape(-1)
            while live.numel():
                j = first[live] + k
                hit = ((X[j] - xi[live]) ** 2 + (Y[j] - yi[live]) ** 2 <= 1.0) & (j != own[live])
                i, j = live[hit], j[hit]
                if model == "langevin":
                    t = ci[i] * sT[j] - si[i] * cT[j]
                    if self.sp is not None:
                        t = t * self.gamma[self.sp[who[i]], self.sp[src[j]]]
                    a1[i] += t
                else:
                    f = 1.0 if model == "vm" else torch.where(ci[i] * cT[j] + si[i] * sT[j] < 0.0, -1.0, 1.0).double()
                    a1[i] += f * cT[j]
                    b1[i] += f * sT[j]
                n1[i] += 1.0
                k += 1
                live = live[length[live] > k]
        a[who], b[who], n[who] = a1, b1, n1
        return a, b, n

    def nearest(self):
        """The same over the kn nearest (Vicsek); every window of 7 x 7 cells is checked to reach far enough."""
        k = self.case["kn"]
        X, Y, T, src, start, own, who, c, row = self.sort()
        a, b, n = (torch.zeros(self.n, device=DEV, dtype=torch.float64) for _ in range(3))
        reach = self.ring * float(torch.minimum(self.L[0] / self.nc[0], self.L[1] / self.nc[1])[0])
        for lo in range(0, own.numel(), 1 << 17):
            sl = slice(lo, lo + (1 << 17))
            q, cc, rr = own[sl], c[sl], row[sl]
            cand = []
            for d in range(-self.ring, self.ring + 1):
                first = start[cc + d * rr - self.ring]
                length = start[cc + d * rr + self.ring + 1] - first
                m = torch.arange(int(length.max()), device=DEV)
                cand.append(torch.where(m[None] < length[:, None], first[:, None] + m[None], -1))
            j = torch.cat(cand, 1)
            d2 = (X[j] - X[q][:, None]) ** 2 + (Y[j] - Y[q][:, None]) ** 2
            d2[(j < 0) | (j == q[:, None])] = math.inf
            dk, at = torch.topk(d2, k, 1, largest=False)
            j = torch.gather(j, 1, at)
            far = torch.nonzero(dk[:, -1] > reach * reach).reshape(-1)
            if far.numel():                                     # sparse spots: against everything
                for f in range(0, far.numel(), 64):
                    qf = q[far[f:f + 64]]
                    d2 = (X[None] - X[qf][:, None]) ** 2 + (Y[None] - Y[qf][:, None]) ** 2
                    d2[torch.arange(qf.numel(), device=DEV), qf] = math.inf
                    j[far[f:f + 64]] = torch.topk(d2, k, 1, largest=False)[1]
            a[who[sl]] = torch.cos(T[j]).sum(1)
            b[who[sl]] = torch.sin(T[j]).sum(1)
            n[who[sl]] = float(k)
        return a, b, n

    def advance(self):
        """One time step; returns |Omega_i| of the state before it."""
        cs = self.case
        a, b, n = self.nearest() if cs["kn"] else self.metric()
        w0, w1 = _philox(self.ids, self.step, self.seed)
        u0 = _uniform(w0)
        if cs["model"] == "langevin":
            dt = cs["dt"]
            gz = torch.sqrt(-2.0 * torch.log(u0)) * torch.cos(2.0 * math.pi * _uniform(w1))
            th = self.th + dt * a / (1.0 + n) + self.omega * dt + self.eta * math.sqrt(dt) * gz
            go, d = self.th, self.v * dt
        else:
            ang = torch.atan2(b + torch.sin(self.th), a + torch.cos(self.th))
            th = ang + self.omega + self.eta * math.pi * (2.0 * u0 - 1.0)
            go, d = th, self.v
        q = [self.x + d * torch.cos(go), self.y + d * torch.sin(go)]
        for k in (0, 1):
            L = self.L[k][self.sys]
            if cs["walls"]:
                low, high = q[k] < 0.0, q[k] > L
                q[k] = torch.where(low, -q[k], torch.where(high, 2.0 * L - q[k], q[k]))
                th = torch.where(low | high, (math.pi - th) if k == 0 else -th, th)
            else:
                q[k] = torch.remainder(q[k], L)
        self.x, self.y = q
        self.th = _wrap(th)
        self.step += 1
        return n

    def per_system(self, v):
        return torch.zeros(len(self.ss), device=DEV, dtype=torch.float64).index_add_(0, self.sys, v)

    def polar(self, o=1):
        count = torch.tensor([s["n"] for s in self.ss], device=DEV)
        return torch.hypot(self.per_system(torch.cos(o * self.th)), self.per_system(torch.sin(o * self.th))) / count

    def fields(self, nb):
        """Density and polarisation per unit area of nb x nb bins, for every system."""
        R = len(self.ss)
        ix = torch.clamp((self.x * nb / self.L[0][self.sys]).long(), 0, nb - 1)
        iy = torch.clamp((self.y * nb / self.L[1][self.sys]).long(), 0, nb - 1)
        out = torch.zeros((3, R * nb * nb), device=DEV, dtype=torch.float64)
        at = (self.sys * nb + iy) * nb + ix
        for k, v in enumerate((torch.ones_like(self.x), torch.cos(self.th), torch.sin(self.th))):
            out[k].index_add_(0, at, v)
        return out.reshape(3, R, nb, nb).transpose(0, 1) * (nb * nb / (self.L[0] * self.L[1]))[:, None, None, None]


def _initial(s):
    """The library's initial state of a replica: uniform and isotropic from Philox with tag 1."""
    ids = torch.arange(s["n"], device=DEV)
    c0, c1, c2, c3 = ids.clone(), torch.zeros_like(ids), torch.zeros_like(ids), torch.ones_like(ids)
    k0, k1 = s["seed"] & M32, s["seed"] >> 32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & M32) ^ c1 ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c3 ^ k1, p0 & M32
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return s["lx"] * _uniform(c0), s["ly"] * _uniform(c1), (math.pi * (2.0 * _uniform(c2) - 1.0)).float()


def _exact_particles(case, seed):
    ss = _systems(case, seed)
    kind, steps, nb = case["kind"], case["steps"], case["bins"]
    # the Vicsek models are chaotic: from FP32 rounding, single trajectories part within some 20 steps and the averages over
    # a small system within some 50, so that a longer pass has no 64-bit value to be compared with
    chaotic = case["model"] != "langevin"
    if chaotic and steps > 50:
        return None
    lost = chaotic and steps > 16
    e = _Exact(case, ss, [_initial(s) if kind == "ensemble" else _start(case, s, seed) for s in ss])
    p, q, nbar = [], [], []
    th_hist, nb_hist = (torch.zeros(100, device=DEV, dtype=torch.float64) for _ in range(2))
    watched = kind in ("trace", "measure", "ensemble")
    for _ in range(steps):
        if watched:
            p.append(e.polar())
            q.append(e.polar(2))
            if kind == "measure":
                th_hist += torch.bincount(torch.clamp(((e.th + math.pi) * (100 / (2.0 * math.pi))).long(), 0, 99), minlength=100)
        n = e.advance()
        if kind == "measure":
            nbar.append(n.mean()[None])
            nb_hist += torch.bincount(torch.clamp(n.long(), max=99), minlength=100)
    if kind == "ensemble":
        return {"phi_mean": torch.stack(p).mean(0), "fields": None if lost else e.fields(nb)}
    if kind == "frames":
        return {"fields": None if lost else e.fields(nb)[0]}
    out = {}
    if kind == "trace":
        out["p"] = torch.cat(p + [e.polar()])
    if kind == "measure":
        mom = lambda v: torch.stack([(torch.cat(v) ** k).mean() for k in (1, 2, 3, 4)])
        pm = mom(p)
        out.update(p=pm, q=mom(q), nbar=mom(nbar), binder=float(1.0 - pm[3] / (3.0 * pm[1] ** 2)),
                   theta_hist=th_hist / th_hist.sum(), nbr_hist=nb_hist / nb_hist.sum())
    out.update(x=None, y=None, theta=None) if lost else out.update(x=e.x, y=e.y, theta=e.th)
    return out


def _exact_network(case, seed):
    f, t, eta = _fields(case, seed)
    f, t, eta = f.double(), t.double(), eta.double()
    flat = torch.tensor(_weights(seed), device=DEV, dtype=torch.float64, requires_grad=case["kind"] == "train")
    ws, at = [], 0
    for cin, cout, _, _ in LAYERS:
        w = flat[at:at + cout * 9 * cin].reshape(cout, 3, 3, cin).permute(0, 3, 1, 2)
        at += cout * 9 * cin
        ws.append((w, flat[at:at + cout]))
        at += cout
    scale = torch.tensor([0.5, 0.5, 0.5], device=DEV, dtype=torch.float64).reshape(1, 3, 1, 1)
    one = torch.tensor([1.0, 0.0, 0.0], device=DEV, dtype=torch.float64).reshape(1, 3, 1, 1)
    keep = torch.tensor([case["conserve"] & 1, case["conserve"] & 2, case["conserve"] & 2], device=DEV).bool().double()
    ch = ((eta - 0.4) / 0.1)[:, None, None, None].expand(-1, 1, case["h"], case["w"])

    def net(u):
        a = torch.cat([u, ch, torch.zeros((u.shape[0], 12) + u.shape[2:], device=DEV, dtype=torch.float64)], 1)
        for k, (w, b) in enumerate(ws):
            a = torch.nn.functional.pad(a, (1, 1, 1, 1), mode="circular")
            # a convolution as nine products, sample by sample in size
            a = sum(torch.einsum("bchw,oc->bohw", a[:, :, dy:dy + case["h"], dx:dx + case["w"]], w[:, :, dy, dx])
                    for dy in range(3) for dx in range(3)) + b[None, :, None, None]
            a = torch.relu(a) if k < 3 else a[:, :3]
        return u + a - keep.reshape(1, 3, 1, 1) * a.mean((2, 3), keepdim=True)

    u = f * scale - one
    if case["kind"] == "predict":
        for _ in range(case["apps"]):
            u = net(u)
        return {"fields": (u + one) / scale}
    loss = ((net(u) - (t * scale - one)) ** 2).mean()
    loss.backward()
    g = flat.grad
    # Adam's first step: the moments' bias corrections leave lr g / (|g| + eps)
    return {"loss": float(loss), "grads": g, "params": flat.detach() - 1e-3 * g / (g.abs() + 1e-8)}


def exact(case, seed):
    return _exact_network(case, seed) if case["kind"] in ("train", "predict") else _exact_particles(case, seed)
