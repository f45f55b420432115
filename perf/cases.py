"""Performance cases of the hologram library: what its users have it do, each a
pass through the public entry points (``Plan.solve``, ``Plan.batch``,
``Plan.host_batch``, ``Plan.submit`` / ``wait``).

A case names a kind of call and its sizes:
  solve   one whole hologram (``cswgs_solve_ex``): start state, iterations,
          final pass;
  step    iterations from a caller's state without the final pass (a program
          that tracks moving spots re-weights them between frames);
  final   the final pass alone from a caller's state: the phase map, the spot
          intensities, e and u;
  batch   a captured batch of holograms, run again and again;
  host    the host-buffer form of a batch: spots in host memory, phase maps
          into pinned host memory;
  serve   requests submitted to the serving loop and waited for.
`mix` > 0 gives every hologram of a batch or stream its own size (the sizes
come from that number, the spots from the seed).

What comes back.  A phase map is returned as the field behind the SLM,
A e^{i Phi}, so that a pixel at the 0 / 2 pi seam is not a whole turn away
from itself.  Where the field at the SLM all but vanishes the phase of a pixel
is arbitrary to any rounding before it, so over a million pixels no two correct
solvers agree on each one once spot states were computed: large solves return
the spot states they end in (w, theta, I_n, e, u), from which the map follows,
and the maps themselves are returned by the final passes from a given state and
by the small whole solves.  Batches and the serving loop give e and u for each
hologram beside the maps that they write.
"""
import math
import types

import numpy as np
import torch

from paper_2003_05293_gb300 import Plan

_CHOICES = (512, 768, 1024, 1152)


def _case(name, call, P, N, c, I, **kw):
    d = dict(name=name, call=call, P=P, N=N, c=c, I=I, precision="fp32", count=1, mix=0, gamma=10.0,
             pattern="cloud", aperture="square", waist=0.0, subset="fresh", weighted=False)
    d.update(kw)
    return d


def listed():
    return [
        # the smallest whole hologram: launches and host work
        _case("solve_tiny", "solve", 64, 10, 0.25, 10, gamma=5.0),
        # one compressed iteration between two frames, spots of unequal target amplitude
        _case("step_medium", "step", 512, 100, 0.125, 1, weighted=True),
        # a real-time loop's hologram on a full SLM: one at a time, latency counts
        _case("solve_large", "solve", 1152, 100, 0.125, 30),
        # few spots (optical traps), sparse subset
        _case("solve_few_spots", "solve", 1152, 10, 0.0625, 30),
        # the paper's optics: round aperture, Gaussian beam, windowed subsets, a
        # 6 x 6 grid of traps
        _case("solve_paper_optics", "solve", 1152, 36, 0.125, 30, pattern="grid", aperture="round", waist=652.0,
              subset="windows"),
        # the map, intensities and metrics of a state found before, many spots
        _case("final_dense", "final", 1152, 300, 1.0, 0),
        # the double-precision solver, whole
        _case("solve_fp64", "solve", 512, 100, 0.125, 10, precision="fp64"),
        # throughput: many holograms at once, as a quality study or a
        # stimulation experiment queues them
        _case("batch_large", "batch", 1152, 100, 0.125, 30, count=64),
        # holograms of uneven size in one batch
        _case("batch_mixed", "batch", 1152, 300, 0.125, 30, count=64, mix=1),
        # the half-precision option
        _case("batch_fp16", "batch", 1152, 100, 0.125, 30, count=64, precision="fp32_fp16sincos"),
        # end to end with host buffers: regular trap grids, maps to pinned memory
        _case("host_grid", "host", 1152, 100, 0.125, 30, count=16, pattern="grid"),
        # a burst of requests of very different size through the serving loop
        _case("serve_burst", "serve", 1152, 1000, 0.125, 20, count=32, mix=2, gamma=20.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _even(x):
    return 2 * max(1, int(round(x / 2.0)))


def draw(rng):
    call = rng.choice(["solve", "solve", "solve", "step", "final", "batch", "batch", "host", "serve"])
    precision = "fp32"
    P, N = _even(_log(rng, 48, 1152)), int(round(_log(rng, 5, 400)))
    c = 2.0 ** -rng.randint(1, 5) if rng.random() < 0.7 else round(rng.uniform(0.03, 1.0), 3)
    I = rng.choice([3, 5, 10, 20, 30])
    kw = dict(gamma=rng.choice([5.0, 10.0, 20.0]), weighted=rng.random() < 0.3)
    if call in ("batch", "host", "serve"):
        P = _even(_log(rng, 200, 1152))
        count = int(round(_log(rng, 4, 64 if call == "batch" else 24)))
        N = min(N, 300)
        kw.update(count=count, mix=rng.randint(3, 10**6) if call == "serve" or rng.random() < 0.5 else 0)
        if call == "batch" and rng.random() < 0.25:
            precision = "fp32_fp16sincos"
    elif call == "step":
        I = rng.randint(1, 3)
    elif call == "final":
        I, c = 0, 1.0
    elif call == "solve" and rng.random() < 0.2:
        precision, P, N, I = "fp64", _even(_log(rng, 48, 512)), min(N, 100), min(I, 10)
    if precision != "fp64" and rng.random() < 0.3:
        kw.update(aperture="round", waist=round(rng.uniform(0.4, 0.7) * P, 1), subset=rng.choice(["fresh", "windows"]))
    d = _case("", call, P, N, c, I, precision=precision, **kw)
    del d["name"]
    return d


# ------------------------------------------------------------------ inputs --

def _rotation(rng):
    a, b, g = rng.uniform(0.0, 2.0 * np.pi, 3)

    def rz(t):
        return np.array([[np.cos(t), -np.sin(t), 0.0], [np.sin(t), np.cos(t), 0.0], [0.0, 0.0, 1.0]])

    rx = np.array([[1.0, 0.0, 0.0], [0.0, np.cos(b), -np.sin(b)], [0.0, np.sin(b), np.cos(b)]])
    return rz(a) @ rx @ rz(g)


def _spots(rng, pattern, P, N, gamma):
    """(N, 3): tilts in cycles across the aperture, defocus in waves: a random 3D
    cloud, or a square grid of traps (the first N of it) turned in space."""
    if pattern == "grid":
        n = math.isqrt(N - 1) + 1
        g = (np.arange(n) - (n - 1) / 2.0) * (P / (4.0 * n))
        pts = np.array([[x, y, 0.0] for x in g for y in g])[:N] @ _rotation(rng).T
        return np.ascontiguousarray(pts * np.array([1.0, 1.0, 0.2]))
    xyz = rng.uniform(-0.25 * P, 0.25 * P, (N, 3))
    xyz[:, 2] = rng.uniform(-gamma, gamma, N)
    return xyz


def _sizes(case):
    """(P, N) of every hologram of the case."""
    if not case["mix"]:
        return [(case["P"], case["N"])] * case["count"]
    rng = np.random.Generator(np.random.PCG64(case["mix"]))
    out = []
    for _ in range(case["count"]):
        P = int(rng.choice([p for p in _CHOICES if p <= case["P"]] or [case["P"]]))
        if case["call"] == "serve":   # the values of a mixed stream: few, some, many spots
            N = min(case["N"], int(rng.choice([10, 100, 1000])))
        else:
            N = int(rng.integers(min(10, case["N"]), case["N"] + 1))
        out.append((P, N))
    return out


def _problems(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    extra = {}
    if case["aperture"] != "square" or case["waist"] or case["subset"] != "fresh":
        extra = dict(aperture=case["aperture"], waist=case["waist"], subset_mode=case["subset"])
    out = []
    for P, N in _sizes(case):
        out.append(types.SimpleNamespace(
            P=P, N=N, c=case["c"], iterations=case["I"], extra=extra, seed=int(rng.integers(0, 2**63 - 1)),
            xyz=_spots(rng, case["pattern"], P, N, case["gamma"]),
            amp=rng.uniform(0.5, 1.5, N) if case["weighted"] else None))
    return out, rng


_plans = {}


def _plan(case):
    """The plan that a program keeps for all its calls of a precision; a serving
    loop (sized by its first request) has one of its own."""
    key = case["precision"]
    if case["call"] == "serve":
        key = repr(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _plans:
        _plans[key] = Plan(precision=case["precision"], max_batch=64, mem_cap_bytes=8 << 30)
    return _plans[key]


def _amplitude(P, aperture, waist, device="cuda"):
    """A of the light at the SLM, 0 outside the aperture."""
    x = torch.arange(P, device=device, dtype=torch.float64) - P // 2
    rho2 = x[:, None] ** 2 + x[None, :] ** 2
    A = torch.exp(-rho2 / waist**2) if waist else torch.ones_like(rho2)
    return A * (rho2 <= (P // 2) ** 2) if aperture == "round" else A


def _keeps_map(case):
    """The calls whose maps are compared (the module's docstring says why)."""
    return case["call"] == "final" or (case["call"] == "solve" and (case["P"] <= 96 or case["precision"] == "fp64"))


def prepare(case, seed):
    plan = _plan(case)
    pbs, rng = _problems(case, seed)
    s = types.SimpleNamespace(case=case, plan=plan, pbs=pbs, batch=None, outs=None)
    call = case["call"]
    if call in ("solve", "step", "final"):
        pb = pbs[0]
        s.out = torch.empty(pb.P, pb.P, device="cuda") if call != "step" else None
        if _keeps_map(case):
            s.A = _amplitude(pb.P, case["aperture"], case["waist"]).float()
        s.kw = dict(P=pb.P, c=pb.c, iterations=pb.iterations, seed=pb.seed, amp=pb.amp, out=s.out, state=True,
                    **pb.extra)
        if call != "solve":   # a state of earlier iterations
            s.kw.update(init_w=np.exp(rng.normal(0.0, 0.3, pb.N)), init_theta=rng.uniform(-np.pi, np.pi, pb.N))
        if call == "step":
            s.kw.update(full_iterations=0, first_iteration=7, final_pass=False)
    elif call == "host":
        s.outs = [torch.empty(pb.P * pb.P, pin_memory=True).numpy() for pb in pbs]
        s.batch = plan.host_batch(pbs, s.outs)
    else:
        s.outs = [torch.empty(pb.P, pb.P, device="cuda") for pb in pbs]
        if call == "batch":
            s.batch = plan.batch(pbs, s.outs)
    return s


def run(s):
    call = s.case["call"]
    if call in ("solve", "step", "final"):
        r = s.plan.solve(s.pbs[0].xyz, **s.kw)
        out = {"w": r["w"].astype(np.float32), "theta": r["theta"].astype(np.float32)} if call != "final" else {}
        if s.case["precision"] == "fp64":
            out = {"w": r["w"], "theta": r["theta"]}
        if call != "step":
            out.update(I=r["I"].astype(np.float32), e=r["e"], u=r["u"])
            if _keeps_map(s.case):
                out["field"] = torch.polar(s.A, s.out)
        return out
    if call == "batch":
        s.batch.run()
        rs = s.batch.results()
    elif call == "host":   # new spots every pass, as a caller that solves batch after batch gives them
        s.batch.update(s.pbs, s.outs)
        s.batch.run()
        rs = s.batch.results()
    else:
        tickets = [s.plan.submit(pb, o) for pb, o in zip(s.pbs, s.outs)]
        rs = [s.plan.wait(t) for t in tickets]
    return {k: np.array([r[k] for r in rs], dtype=np.float32) for k in ("e", "u")}


def _schedule(case):
    """(compressed iterations, full iterations, final pass)"""
    full = 0 if case["call"] == "step" else min(2, case["I"])
    return case["I"] - full, full, case["call"] != "step"


def work(case):
    sub, full, fin = _schedule(case)
    flops = bytes_ = 0.0
    for P, N in _sizes(case):
        D = P * P * (math.pi / 4.0 if case["aperture"] == "round" else 1.0)
        # one complex multiply-add per pixel of the pass and spot, back and forward
        flops += 16.0 * N * D * (sub * case["c"] + full + (1 if fin else 0))
        bytes_ += N * (24 + 8 * case["weighted"] + (16 if case["call"] in ("step", "final") else 0))
        bytes_ += N * (0 if case["call"] == "final" else 16) + (8 * N + 16 if fin else 0)
        if fin:
            bytes_ += 4.0 * P * P * (1 if not _keeps_map(case) else 3)
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------ the method, in 64 bits --

_M64 = (1 << 64) - 1


def _splitmix64(seed, k):
    z = (seed + (k + 1) * 0x9E3779B97F4A7C15) & _M64
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
    return z ^ (z >> 31)


def _mul32(h, m):
    """h * m mod 2^32 for h < 2^32 (64-bit signed arithmetic)."""
    return ((h & 0xFFFF) * m + ((((h >> 16) * m) & 0xFFFF) << 16)) & 0xFFFFFFFF


def _fmix32(h):
    h = h ^ (h >> 16)
    h = _mul32(h, 0x85EBCA6B)
    h = h ^ (h >> 13)
    h = _mul32(h, 0xC2B2AE35)
    return h ^ (h >> 16)


def _permutation(D, seed, j, k):
    """The keyed bijection of [0, D) at the positions k."""
    a = math.isqrt(D - 1) + 1 if D > 1 else 1
    b = -(-D // a)
    keys = [_splitmix64(seed, 2**32 + 4 * j + r) >> 32 for r in range(4)]

    def rect(k):
        L, R = k // b, k % b
        for r in range(4):
            p = a if r % 2 == 0 else b
            L, R = R, (L + ((_fmix32(R ^ keys[r]) * p) >> 32)) % p
        return L * b + R

    y = rect(k)
    while True:
        out = y >= D
        if not bool(out.any()):
            return y
        y[out] = rect(y[out])


class _Hologram:
    """One hologram by the paper's equations, with the separable factors of its
    lens-and-prism phases, in double precision."""

    def __init__(self, case, pb, dev):
        P = self.P = pb.P
        self.N, self.seed, self.windows, self.dev = pb.N, pb.seed, case["subset"] == "windows", dev
        self.A = _amplitude(P, case["aperture"], case["waist"], dev)
        x = torch.arange(P, device=dev, dtype=torch.float64) - P // 2
        inside = torch.ones(P, P, dtype=torch.bool, device=dev)
        if case["aperture"] == "round":
            inside = x[:, None] ** 2 + x[None, :] ** 2 <= (P // 2) ** 2
        self.pupil = inside.reshape(-1).nonzero().reshape(-1)
        self.D = int(self.pupil.numel())
        self.Mp = int(math.floor(pb.c * self.D))
        s = torch.from_numpy(np.ascontiguousarray(pb.xyz)).to(dev)

        def factor(tilt):
            t = tilt[:, None] / P * x + s[:, 2:3] / (P / 2.0) ** 2 * x * x
            return torch.polar(torch.ones_like(t), 2 * math.pi * (t - t.round()))

        self.C, self.R = factor(s[:, 0]), factor(s[:, 1])
        self.amp = torch.ones(pb.N, device=dev, dtype=torch.float64) if pb.amp is None else torch.from_numpy(pb.amp).to(dev)

    def back(self, w, th):
        return (self.R * torch.polar(w * self.amp, th)[:, None]).T @ self.C

    def forward(self, S, weight):
        n = S.abs()
        u = torch.where(n > 0, S / n, torch.ones_like(S)) * weight
        return ((u @ self.C.conj().T) * self.R.conj().T).sum(0)

    def subset(self, j):
        k = torch.arange(self.Mp, device=self.dev)
        if self.windows:
            k, j = (k + (j - 1) * self.Mp) % self.D, 0
        m = torch.zeros(self.P * self.P, device=self.dev, dtype=torch.float64)
        m[self.pupil[_permutation(self.D, self.seed, j, k)]] = 1.0
        return m.reshape(self.P, self.P)

    def solve(self, sub, full, fin, first_j=1, w=None, th=None):
        if w is None:
            w = torch.ones(self.N, device=self.dev, dtype=torch.float64)
            th = torch.tensor([2 * math.pi * (_splitmix64(self.seed, n) >> 11) * 2.0**-53 for n in range(self.N)],
                              device=self.dev, dtype=torch.float64)
        for i in range(sub + full):
            weight = self.A if i >= sub else self.A * self.subset(first_j + i)
            V = self.forward(self.back(w, th), weight)
            mag = V.abs()
            w, th = w * mag.mean() / mag, V.angle()
        out = {"w": w.cpu().numpy(), "theta": torch.remainder(th + math.pi, 2 * math.pi).sub(math.pi).cpu().numpy()}
        if fin:
            S = self.back(w, th)
            I = (self.forward(S, self.A) / self.A.sum()).abs() ** 2
            hi, lo = float(I.max()), float(I.min())
            out.update(I=I.cpu().numpy(), e=np.float64(I.sum().item()), u=np.float64(1 - (hi - lo) / (hi + lo)))
            out["field"] = torch.polar(self.A, S.angle())
        return out


def exact(case, seed):
    sub, full, fin = _schedule(case)
    pairs = sum(N * P * P for P, N in _sizes(case)) * (case["I"] + 1)
    if pairs > 4e11:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    pbs, rng = _problems(case, seed)
    if case["call"] in ("solve", "step", "final"):
        w = th = None
        if case["call"] != "solve":
            w = torch.from_numpy(np.exp(rng.normal(0.0, 0.3, pbs[0].N))).to(dev)
            th = torch.from_numpy(rng.uniform(-np.pi, np.pi, pbs[0].N)).to(dev)
        r = _Hologram(case, pbs[0], dev).solve(sub, full, fin, 7 if case["call"] == "step" else 1, w, th)
        if not _keeps_map(case):
            r.pop("field", None)
        if case["call"] == "final":
            del r["w"], r["theta"]
        return r
    got = [_Hologram(case, pb, dev).solve(sub, full, fin) for pb in pbs]
    return {k: np.array([g[k] for g in got]) for k in ("e", "u")}
