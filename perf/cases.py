"""The work that programs have this library do, as cases that can be timed and compared.

A case is one call of a public entry point on a batch of trajectories (Engine.evolve + observables,
qtraj_evolve_static, UnevenBatch, Server), from the smallest latency-bound call to several full waves of
the device, over the grid sizes N = 16 .. 16384, both precisions, both forms and both potentials.

Every step of a medium does the same work, so a case runs a segment of a medium (some tens of steps, like
the short media of the tests and of the autotuner) instead of the whole 10^4 steps.  That also keeps the
FP32 results comparable with 64-bit ones: rounding noise grows with N x steps.

Waiting-time jumps in FP32: a threshold that falls within the rounding of the norm moves a jump by a step,
after which two equally right programs return different records.  The large FP32 ensembles therefore take
seeds whose first jump lies beyond the segment ("quiet"; the waiting-time test runs in every step all the
same); trajectories with jumps are covered by the FP64 cases, whose jumps do not move, and by the smallest
FP32 one.

An FP32 context computes in single precision and reports through FP64 record fields; run() hands its
floating results on as single precision.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2107_06147_gb300 import batching, qtraj, serving

HBARC = 0.1973269804          # GeV fm
MASS, ALPHA, NC = 4.65, 0.3, 3.0
CF = (NC * NC - 1.0) / (2.0 * NC)
DR = 5.0 / 512                # grid spacing of the serving and uneven workloads (GeV^-1)
INT_FIELDS = ("l", "color", "n_jumps", "n_steps_exec", "flags", "first_jump_step", "last_jump_step", "jump_digest")


def listed():
    e = {"entry": "engine", "potential": 0, "deriv": 0, "dt": 0.001, "rmin": 0, "states": False, "gamma0": False,
         "fit": False}
    return [
        # a notebook or a unit test: 8 trajectories of the 512-point reference configuration in FP64, default
        # options (rMin on), final states fetched; the latency of a trajectory on an otherwise empty device
        dict(e, name="tiny_f64_n512", prec="f64", N=512, dr=20.0 / 512, batch=8, steps=300, rmin=1, states=True,
             quiet=False),
        # the same call in FP32
        dict(e, name="tiny_f32_n512", prec="f32", N=512, dr=20.0 / 512, batch=8, steps=96, rmin=1, states=True,
             quiet=False),
        # a latency-bound loop that may not allocate: the static entry on a small grid, 63 trajectories
        dict(e, name="static_f32_n256", entry="static", prec="f32", N=256, dr=5.0 / 256, batch=63, steps=96, quiet=True),
        # the small grid of the serving and uneven mixes, several waves (ragged)
        dict(e, name="ensemble_f32_n1024", prec="f32", N=1024, dr=DR, batch=9999, steps=16, quiet=True),
        # continuous batching: 20 requests of 64 .. 512 trajectories (log-spaced) on three grid sizes, submitted together
        dict(e, name="serve_f32", entry="serve", prec="f32", N=4096, dr=DR, batch=20, steps=16, quiet=True),
        # the headline workload: uniform N = 4096 batch of S and P wave states, kappa_hat in {4, 5, 6},
        # gamma_hat in {-3.5, 0}
        dict(e, name="uniform_f32_n4096", prec="f32", N=4096, dr=DR, batch=9216, steps=16, quiet=True),
        # the precision study's grid: N = 8192, L = 80, dt = 0.0005, 1S Gaussian, gamma_hat = 0
        dict(e, name="precision_f32_n8192", prec="f32", N=8192, dr=DR, batch=4096, steps=12, dt=0.0005, quiet=True,
             gamma0=True),
        # the largest grid
        dict(e, name="large_f32_n16384", prec="f32", N=16384, dr=DR, batch=1001, steps=8, quiet=True),
        # uneven batch: N in {1024 .. 8192}, every trajectory its own medium and lifetime, concurrent launches
        dict(e, name="uneven_f32", entry="uneven", prec="f32", N=8192, dr=DR, batch=3001, steps=16, quiet=True),
        # the isotropic KSU potential (deterministic), singlets
        dict(e, name="ksu_f32_n4096", prec="f32", N=4096, dr=DR, batch=1216, steps=16, potential=1, quiet=False),
        # the FP64 reference ensemble with jumps, singlets and octets, a kappa_hat(T) lattice fit among the media
        dict(e, name="ensemble_f64_n4096", prec="f64", N=4096, dr=DR, batch=600, steps=24, quiet=False, fit=True),
        # FP64 beyond the fused form's grid limit: the plain per-step form at N = 16384
        dict(e, name="plain_f64_n16384", entry="plain", prec="f64", N=16384, dr=DR, batch=40, steps=8, quiet=False),
    ]


def _cost(c):
    """Rough time of a pass (s) at ~2e7 (FP32) / 6e5 (FP64) trajectory-steps/s of N = 4096."""
    n = {"serve": 180.0, "uneven": 0.45}.get(c["entry"], 1.0) * c["batch"] * c["steps"]
    return n * c["N"] * math.log2(c["N"]) / (4096 * 12) / (6e5 if c["prec"] == "f64" else 1.2e7 if c["potential"] else 2e7)


def draw(rng):
    kind = rng.choice(["engine", "engine", "engine", "f64", "static", "uneven", "serve", "ksu", "plain"])
    c = {"entry": "engine", "potential": 0, "deriv": rng.choice([0, 0, 1]), "dt": rng.choice([0.001, 0.001, 0.0005]),
         "rmin": 0, "states": False, "gamma0": rng.random() < 0.3, "fit": False, "prec": "f32", "dr": DR, "quiet": True}
    if kind == "f64" or kind == "plain":
        c.update(prec="f64", quiet=False, entry="engine" if kind == "f64" else "plain", fit=rng.random() < 0.5,
                 N=2 ** (rng.randint(4, 13) if kind == "f64" else rng.randint(9, 14)))
    elif kind == "uneven":
        c.update(entry="uneven", N=8192)
    elif kind == "serve":
        c.update(entry="serve", N=4096)
    elif kind == "ksu":
        c.update(potential=1, quiet=False, N=2 ** rng.randint(8, 12))
    else:
        c.update(entry=kind, N=2 ** rng.randint(4, 14))
    if c["N"] <= 256:
        c["dr"] = 5.0 / 256
    # FP32: short segments (the rounding noise of the state grows with N and the steps)
    most = 300 if c["prec"] == "f64" else 96 if c["N"] <= 512 else 16 if c["N"] <= 4096 else 8
    lo, hi = (3, 24) if c["entry"] == "serve" else (1, 3000)
    while True:
        c["steps"] = int(round(math.exp(rng.uniform(math.log(4), math.log(max(5, most))))))
        c["batch"] = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        if _cost(c) <= 0.02:
            return c


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _philox(seeds, k):
    """Philox4x32-10, counter (k, 0, 0, 0), key = 64-bit seed: the (r, u_l, u_c) draws of waiting period k."""
    m32 = np.uint64(0xFFFFFFFF)
    c0 = np.broadcast_to(np.asarray(k, np.uint64), seeds.shape).copy()
    c1, c2, c3 = (np.zeros_like(c0) for _ in range(3))
    k0, k1 = seeds & m32, seeds >> np.uint64(32)
    for i in range(10):
        if i:
            k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m32, (k1 + np.uint64(0xBB67AE85)) & m32
        p0, p1 = np.uint64(0xD2511F53) * c0, np.uint64(0xCD9E8D57) * c2
        c0, c1, c2, c3 = (p1 >> np.uint64(32)) ^ c1 ^ k0, p1 & m32, (p0 >> np.uint64(32)) ^ c3 ^ k1, p0 & m32
    w = (c1 << np.uint64(32)) | c0
    return (((w >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53, (c2.astype(np.float64) + 0.5) * 2.0 ** -32,
            (c3.astype(np.float64) + 0.5) * 2.0 ** -32)


def _seeds(g, n, quiet):
    if not quiet:
        return g.integers(0, 2 ** 63, n, dtype=np.uint64)
    got = np.zeros(0, np.uint64)
    while len(got) < n:
        s = g.integers(0, 2 ** 63, 80 * n + 1000, dtype=np.uint64)
        got = np.concatenate([got, s[_philox(s, 0)[0] < 1.0 / 64]])
    return got[:n]


def _tf(T0, steps, dt):
    """Tf that ends a Bjorken medium from T0 at 0.6 fm/c after `steps` steps."""
    return T0 * (0.6 / (0.6 + (steps - 0.5) * HBARC * dt)) ** (1.0 / 3.0)


def _inputs(case, seed):
    """Per-trajectory grid size, initial state and medium (indices into lists) and Philox seed, all from the seed."""
    g = np.random.Generator(np.random.PCG64(seed))
    w = float(g.uniform(0.7, 0.9))
    inits = [("gauss", w, 1, 0, 0), ("coulomb", 0.0, 1, 0, 0), ("coulomb", 0.0, 2, 0, 0), ("gauss", w, 2, 1, 0)]
    if case["N"] >= 8192 and case["entry"] == "engine" and case["gamma0"]:
        inits = inits[:1]
    if not case["quiet"]:
        inits = inits + [("gauss", w, 3, 2, 1)]
    if case["potential"]:
        inits = [inits[0], inits[3]]
    kind, B, steps, dt = case["entry"], case["batch"], case["steps"], case["dt"]
    gam = (lambda: 0.0) if case["gamma0"] else (lambda: float(g.uniform(-3.5, 0.0)))
    n_req = None
    if kind == "serve":
        n_req = g.permutation(np.round(64.0 * 8.0 ** (np.arange(B) / max(1, B - 1))).astype(int))
        media = []
        for _ in range(B):
            T0 = float(g.uniform(0.35, 0.5))
            media.append((T0, _tf(T0, int(g.integers(max(2, steps // 2), steps + 1)), dt), float(g.uniform(3, 7)), gam()))
        mi = np.repeat(np.arange(B), n_req)
        si = np.repeat(g.integers(0, len(inits), B), n_req)
        Ns = np.repeat(np.array([1024, 2048, 4096])[np.arange(B) % 3], n_req)
    elif kind == "uneven":
        media = []
        for _ in range(B):
            T0 = float(g.uniform(0.35, 0.5))
            media.append((T0, _tf(T0, int(g.integers(max(2, steps // 4), steps + 1)), dt), float(g.uniform(3, 7)), gam()))
        mi, si = np.arange(B), g.integers(0, len(inits), B)
        Ns = g.permutation(np.array([1024, 2048, 4096, 8192])[np.arange(B) % 4])
    else:
        T0 = float(g.uniform(0.40, 0.45))
        dk, dg = float(g.uniform(-0.2, 0.2)), gam()
        media = [(T0, _tf(T0, steps, dt), k + dk, x * dg) for k in (4.0, 5.0, 6.0) for x in ((1.0,) if case["gamma0"] else (1.0, 0.0))]
        if case["fit"]:
            media[0] = media[0][:2] + (-1.0,) + media[0][3:]
        mi, si = (np.arange(B) // len(inits)) % len(media), np.arange(B) % len(inits)
        Ns = np.full(B, case["N"])
    seeds = _seeds(g, len(mi), case["quiet"])
    return {"inits": inits, "media": media, "si": si.astype(np.int32), "mi": mi.astype(np.int32), "Ns": Ns, "seeds": seeds,
            "n_req": n_req}


# ------------------------------------------------------------------------------------------------
# the calls
# ------------------------------------------------------------------------------------------------
class _Request(serving.Request):
    """A request whose trajectories have seeds of the caller's choice."""

    def descriptors(self):
        d = super().descriptors()
        d["seed"] = self.seeds
        return d


def _request(seeds, **fields):
    r = _Request(seed0=0, **fields)
    r.seeds = seeds
    return r


def _config(case, N):
    return qtraj.Config(N=N, L=N * case["dr"], dt=case["dt"], deriv_type=case["deriv"], use_rmin=case["rmin"],
                        precision=qtraj.FP32 if case["prec"] == "f32" else qtraj.FP64,
                        form=qtraj.PLAIN if case["entry"] == "plain" else qtraj.FUSED,
                        save_states=int(case["states"]), potential=case["potential"])


def prepare(case, seed):
    x = _inputs(case, seed)
    specs = [qtraj.init_spec(*s) for s in x["inits"]]
    media = [qtraj.medium(T0, 0.6, Tf, k, gm) for T0, Tf, k, gm in x["media"]]
    s = {"case": case, "specs": specs, "media": media, "x": x}
    if case["entry"] == "uneven":
        s["batch"] = batching.UnevenBatch(x["Ns"], [specs[i] for i in x["si"]], [media[i] for i in x["mi"]], dt=case["dt"],
                                          dr=case["dr"], use_rmin=0)
    elif case["entry"] == "serve":
        s["server"] = serving.Server(Ns=(1024, 2048, 4096), slots_per_n=2, dr=case["dr"], dt=case["dt"], specs=specs,
                                     cfg=qtraj.Config(dt=case["dt"], deriv_type=case["deriv"], precision=qtraj.FP32))
        first = np.concatenate([[0], np.cumsum(x["n_req"])[:-1]])
        s["requests"] = [dict(rid=i, N=int(x["Ns"][f]), init=int(x["si"][f]), T0=x["media"][i][0], Tf=x["media"][i][1],
                              kappa_hat=x["media"][i][2], gamma_hat=x["media"][i][3], ntraj=int(x["n_req"][i]),
                              seeds=x["seeds"][f:f + x["n_req"][i]]) for i, f in enumerate(first)]
    else:
        s["engine"] = qtraj.Engine(_config(case, case["N"]))
        if case["entry"] == "static":
            ip, up = ctypes.POINTER(ctypes.c_int), ctypes.POINTER(ctypes.c_uint64)
            s["args"] = ((qtraj.InitSpec * len(specs))(*specs), len(specs), x["si"].ctypes.data_as(ip),
                         (qtraj.Medium * len(media))(*media), len(media), x["mi"].ctypes.data_as(ip),
                         x["seeds"].ctypes.data_as(up))
            s["out"] = torch.zeros(case["batch"] * qtraj.OBS_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
        else:
            s["engine"].init(specs, case["batch"], x["si"])
    return s


def _records(case, obs):
    t = np.float32 if case["prec"] == "f32" else np.float64
    out = {f: obs[f].astype(t) for f in ("surv", "norm2")}
    out["overlap"] = np.stack([obs["ov_re"], obs["ov_im"]], -1).astype(t)
    out["r0"] = obs["r0"].copy()
    out.update((f, obs[f].copy()) for f in INT_FIELDS)
    return out


def run(state):
    case = state["case"]
    if case["entry"] == "uneven":
        return _records(case, state["batch"].run(state["x"]["seeds"]))
    if case["entry"] == "serve":
        srv = state["server"]
        reqs = [_request(**r) for r in state["requests"]]
        for r in reqs:
            srv.submit(r)
        left = len(reqs)
        while left:
            left -= len(srv.poll())
        srv.completed.clear()
        return _records(case, np.concatenate([r.obs for r in reqs]))
    e = state["engine"]
    if case["entry"] == "static":
        st = e.lib.qtraj_evolve_static(e.ctx, case["batch"], *state["args"], ctypes.c_void_p(state["out"].data_ptr()),
                                       ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if st:
            raise RuntimeError(e.lib.qtraj_last_error(e.ctx).decode())
        return _records(case, state["out"].cpu().numpy().view(qtraj.OBS_DTYPE))
    e.evolve(state["media"], state["x"]["seeds"], state["x"]["mi"])
    out = _records(case, e.observables())
    if case["states"]:
        out["states"] = e.states().astype(np.complex64 if case["prec"] == "f32" else np.complex128)
    return out


def work(case):
    """Two sine transforms of N complex points (5 N log2 N flops each), the kinetic factor (6 N), the two potential
    half-steps (12 N each) and the norm (4 N) of every trajectory-step; the descriptors (24 bytes) and initial states
    read and the records (192 bytes) and requested states written."""
    def one(N, steps):
        return steps * (10.0 * N * math.log2(N) + (34.0 + 60.0 * case["potential"]) * N)
    B = case["batch"]
    if case["entry"] == "serve":      # log-spaced 64 .. 512 trajectories a request; 3/4 of the steps on average
        n = B * (512 - 64) / math.log(8.0)
        return {"bytes": n * 216.0 + 3 * 7168 * 8.0, "flops": n / 3 * sum(one(N, 0.75 * case["steps"]) for N in (1024, 2048, 4096))}
    if case["entry"] == "uneven":
        return {"bytes": B * 216.0 + 3 * 15360 * 8.0,
                "flops": B / 4 * sum(one(N, 0.625 * case["steps"]) for N in (1024, 2048, 4096, 8192))}
    return {"bytes": B * 216.0 + 24.0 * case["N"] + (16.0 * B * case["N"] if case["states"] else 0.0),
            "flops": B * one(case["N"], case["steps"])}


# ------------------------------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ------------------------------------------------------------------------------------------------
def _state0(spec, r, dr):
    kind, w, n, l, _ = spec
    if kind == "gauss":
        a = (l + 1) * torch.log(r[1:]) - r[1:] ** 2 / (2 * w * w)
        u = torch.exp(a - a.max())
    else:
        u = _coulomb(n, l, r[1:])
    u = torch.cat([torch.zeros_like(r[:1]), u])
    return u / torch.sqrt((u * u).sum() * dr)


def _coulomb(n, l, r):
    x = 2.0 * r / (n * 2.0 / (MASS * CF * ALPHA))
    k, a = n - l - 1, 2 * l + 1
    p0, p1 = torch.ones_like(x), 1.0 + a - x
    for i in range(1, k):
        p0, p1 = p1, ((2 * i + 1 + a - x) * p1 - (i + a) * p0) / (i + 1)
    return r ** (l + 1) * torch.exp(-x / 2) * (p1 if k > 0 else p0)


def _dst(f):
    """S_k = sum_j f_j sin(pi j k / N) over the last axis, through the length-2N FFT of the odd extension."""
    N = f.shape[-1]
    return 0.5j * torch.fft.fft(torch.cat([f, torch.zeros_like(f[..., :1]), -f[..., 1:].flip(-1)], -1))[..., :N]


def _exact_group(case, N, inits, si, media, mi, seeds, dev):
    """The records and final states of trajectories on one grid."""
    dr, dt, B = case["dr"], case["dt"], len(si)
    c128, f64 = torch.complex128, torch.float64
    j = torch.arange(N, dtype=f64, device=dev)
    r = j * dr
    inv = torch.where(j > 0, 1.0 / torch.where(j > 0, r, torch.ones_like(r)), torch.zeros_like(r))
    u0 = torch.stack([_state0(s, r, dr) for s in inits])
    psi = u0[torch.as_tensor(si.astype(np.int64), device=dev)].to(c128)
    p = math.pi * j / (N * dr)
    Tk = p * p / MASS if case["deriv"] == 0 else 2.0 * (1.0 - torch.cos(p * dr)) / (MASS * dr * dr)
    KT = torch.polar(torch.full_like(Tk, 2.0 / N), -Tk * dt)
    l, c = (np.array([inits[i][q] for i in si]) for q in (3, 4))
    med = np.array([media[i] for i in mi])
    n_steps = np.ceil((0.6 * (med[:, 0] / med[:, 1]) ** 3 - 0.6) / (HBARC * dt)).astype(int)
    rr, ul, uc = _philox(seeds, np.zeros(B, np.uint64))
    nj = np.zeros(B, int)

    def t(v):
        return torch.as_tensor(np.asarray(v, np.float64), device=dev)[:, None]

    for n in range(n_steps.max()):
        on = np.nonzero(n < n_steps)[0]
        ix = torch.as_tensor(on, device=dev)
        T3 = med[on, 0] ** 3 * 0.6 / (0.6 + n * dt * HBARC)
        x = T3 ** (1.0 / 3.0) / 0.155
        fit = 1.0 / (0.00397 * x ** 1.5 - 0.08341 * x + 0.98031 * x ** 0.5 - 0.51889)
        kap = np.where(med[on, 2] < 0, fit, med[on, 2])
        f = np.where(c[on] == 0, 0.5, (NC * NC - 2.0) / (4.0 * (NC * NC - 1.0)))
        coul = np.where(c[on] == 0, -CF * ALPHA, ALPHA / (2.0 * NC))
        V = t(coul) * inv + t(l[on] * (l[on] + 1.0) / MASS) * inv * inv + t(f * med[on, 3] * T3) * r * r
        K = torch.polar(torch.exp(-t(f * kap * T3 * dt / 2) * r * r), -V * (dt / 2))
        K[:, 0] = 0.0
        y = psi[ix]
        y = K * _dst(KT * _dst(K * y))
        n2 = (torch.view_as_real(y) ** 2).sum((-1, -2)).cpu().numpy() * dr
        hit = n2 <= rr[on]
        for q in np.nonzero(hit)[0]:
            b = on[q]
            z = y[q] * r
            y[q] = z / torch.sqrt((z.abs() ** 2).sum() * dr)
            l_new = l[b] - 1 if ul[b] < l[b] / (2.0 * l[b] + 1.0) else l[b] + 1
            c[b] = 0 if c[b] == 1 and uc[b] < 2.0 / (NC * NC - 2.0) else 1
            l[b] = l_new
            nj[b] += 1
            v = _philox(seeds[b:b + 1], np.array([nj[b]], np.uint64))
            rr[b], ul[b], uc[b] = v[0][0], v[1][0], v[2][0]
        psi[ix] = y
    n2 = (torch.view_as_real(psi) ** 2).sum((-1, -2)) * dr
    surv, ov = np.zeros((B, 6)), np.zeros((B, 6), complex)
    for s, (bn, bl) in enumerate(((1, 0), (2, 0), (2, 1), (3, 0), (3, 1), (3, 2))):
        phi = _state0(("coulomb", 0.0, bn, bl, 0), r, dr)
        o = (psi @ phi.to(c128) * dr).cpu().numpy()
        o0 = (u0 @ phi * dr).cpu().numpy()
        m = (c == 0) & (l == bl)
        ov[m, s] = o[m]
        zero = np.array([q[4] != 0 or q[3] != bl or (q[0] == "coulomb" and q[2] != bn) for q in inits])
        d = np.where(zero, 1.0, o0 ** 2)[si]
        surv[m, s] = (np.abs(o) ** 2 / n2.cpu().numpy() / d)[m]
    return {"surv": surv, "overlap": np.stack([ov.real, ov.imag], -1), "norm2": n2.cpu().numpy(),
            "r0": _philox(seeds, np.zeros(B, np.uint64))[0]}, psi.cpu().numpy()


def exact(case, seed):
    """The floating fields of the records (and the states) as plain 64-bit arithmetic gives them; the KSU potential's
    vacuum basis is an eigensolver's result and its phi a special function: no value."""
    if case["potential"]:
        return None
    x = _inputs(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    out, states = None, None
    for N in sorted(set(int(v) for v in x["Ns"])):
        ids = np.nonzero(x["Ns"] == N)[0]
        step = max(1, (1 << 23) // N)          # trajectories at a time
        for a in range(0, len(ids), step):
            part = ids[a:a + step]
            rec, psi = _exact_group(case, N, x["inits"], x["si"][part], x["media"], x["mi"][part], x["seeds"][part], dev)
            if out is None:
                out = {f: np.zeros((len(x["si"]),) + v.shape[1:]) for f, v in rec.items()}
                states = np.zeros((len(x["si"]), N), complex) if case["states"] else None
            for f, v in rec.items():
                out[f][part] = v
            if case["states"]:
                states[part] = psi
    out.update((f, None) for f in INT_FIELDS)
    if case["states"]:
        out["states"] = states
    return out
