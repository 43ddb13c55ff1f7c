"""Performance cases: the work a program has this library do, over the range it takes.

A case is one pass of one of five kinds of work, each through the public entry points:

* ``d1q3``     a one-dimensional run sampled every step, read out through the API;
* ``d2q9``     a two-dimensional run of one or many replicas with its sampling, left as a
               checkpoint in pinned host memory or in the caller's own device workspace;
* ``lb3``      a three-dimensional run with time correlators at chosen wave vectors;
* ``spectra``  the standalone correlator sampler on device fields;
* ``train``    optimiser steps of the noise-scale network.

``listed`` has the fixed cases, ``draw`` more of the same ranges, ``prepare`` what a program
holds before the call, ``run`` one pass and its outputs, ``work`` the bytes and operations
a pass cannot do without, and ``exact`` the same outputs in 64 bits from plain torch.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1010_1233_gb300 import Sim, learned, workloads as W
from paper_1010_1233_gb300 import _lib as L
from paper_1010_1233_gb300.sim import spectra_accumulate, spectra_sizes

Q = {"D1Q3": 3, "D2Q9": 9, "D3Q15": 15, "D3Q19": 19}
HYDRO = "0,9,10"                        # density and velocity


def listed():
    return [
        # one-dimensional spectra in FP64, sampled every step: the d1q3_L64 workload
        dict(name="d1q3_64_fp64", kind="d1q3", nx=64, precision="fp64", fields="0,1", steps=2000, every=1),
        # a short run on the smallest sweep lattice: launches and latency
        dict(name="d2q9_64_short", kind="d2q9", recipe="one", nx=64, ny=64, replicas=1, precision="fp32",
             fields=HYDRO, steps=20, every=10, noise_mode=0, net=False, tune=False, out="checkpoint"),
        # all nine moment spectra of one 256^2 lattice: the d2q9_256 workload
        dict(name="d2q9_256_fp32", kind="d2q9", recipe="one", nx=256, ny=256, replicas=1, precision="fp32",
             fields="0,1,2,3,4,5,6,7,8", steps=2000, every=10, noise_mode=0, net=False, tune=False, out="checkpoint"),
        # the same in FP64, the precision of the theory comparisons
        dict(name="d2q9_256_fp64", kind="d2q9", recipe="one", nx=256, ny=256, replicas=1, precision="fp64",
             fields="0,1,2,3,4,5,6,7,8", steps=200, every=10, noise_mode=0, net=False, tune=False, out="checkpoint"),
        # the Galilean-invariance sweep, 64 uneven replicas in one context, with its launch tuning
        dict(name="d2q9_sweep64", kind="d2q9", recipe="sweep", nx=512, ny=512, replicas=64, precision="fp32",
             fields=HYDRO, steps=500, every=10, noise_mode=0, net=False, tune=True, out="checkpoint"),
        # the headline benchmark: 16384^2 with the noise-scale network, sampled every 20 steps
        dict(name="d2q9_16384_net", kind="d2q9", recipe="one", nx=16384, ny=16384, replicas=1, precision="fp32",
             fields=HYDRO, steps=40, every=20, noise_mode=0, net=True, tune=True, out="workspace"),
        # warm-up steps of an odd-sized box with the correlated noise of a moving fluid
        dict(name="d2q9_1510x1001_corr", kind="d2q9", recipe="one", nx=1510, ny=1001, replicas=1, precision="fp32",
             fields="", steps=100, every=0, noise_mode=1, net=False, tune=False, out="workspace"),
        # the D3Q15 benchmark box with time correlators
        dict(name="d3q15_512_fp32", kind="lb3", lattice="D3Q15", nx=512, ny=512, nz=512, precision="fp32",
             fields="0,4,9", steps=40, every=20, n_k=16, n_lags=8),
        # a ragged D3Q19 box
        dict(name="d3q19_190x126x70_fp32", kind="lb3", lattice="D3Q19", nx=190, ny=126, nz=70, precision="fp32",
             fields="0,4,9", steps=200, every=20, n_k=16, n_lags=8),
        # a small FP64 box, as the checks against the linear theory run it
        dict(name="d3q15_64x48x40_fp64", kind="lb3", lattice="D3Q15", nx=64, ny=48, nz=40, precision="fp64",
             fields="0,4,9", steps=60, every=10, n_k=8, n_lags=4),
        # the sampler on fields that another program holds on the device
        dict(name="spectra_3x1024x2048_fp32", kind="spectra", precision="fp32", n_fields=3, ny=1024, nx=2048),
        # optimiser steps of the noise-scale network on the sixteen training runs
        dict(name="train_16x4096", kind="train", runs=16, inputs=4096, n_k=4093, iters=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pow2(rng, lo, hi):
    return 1 << rng.randint(int(math.log2(lo)), int(math.log2(hi)))


def draw(rng):
    kind = rng.choice(("d1q3", "batch", "batch", "large", "ragged", "lb3", "lb3", "spectra", "spectra", "train"))
    if kind == "d1q3":
        nx, prec = _pow2(rng, 16, 1024), rng.choice(("fp64", "fp64", "fp32"))
        steps = min(_log(rng, 300, 6000), 400_000 // nx)
        return dict(kind="d1q3", nx=nx, precision=prec, fields=rng.choice(("0,1", "0,1,2", "0,1,2,9")), steps=steps,
                    every=rng.choice((1, 1, 2, 10)))
    if kind == "batch":                  # sampled replicas of 16^2 .. 1024^2
        prec = rng.choice(("fp32", "fp32", "fp64"))
        nx, ny = _pow2(rng, 16, 1024), _pow2(rng, 16, 1024)
        reps = _log(rng, 1, max(1, min(48, 3_000_000 // (nx * ny))))
        fields = rng.choice((HYDRO, "0,1,2,3,4,5,6,7,8", "0", "0,1,2,5", "0,1,2,3,4,5,6,7,8,9,10"))
        every = rng.choice((1, 5, 10, 20))
        v = nx * ny * reps
        budget = (6e8 if prec == "fp32" else 2e7) / (4 if every < 5 else 1)
        steps = max(8, min(_log(rng, 50, 1500), int(budget / v)))
        return dict(kind="d2q9", recipe="one" if reps == 1 else "same", nx=nx, ny=ny, replicas=reps, precision=prec,
                    fields=fields, steps=steps, every=every, noise_mode=0, net=prec == "fp32" and rng.random() < 0.3,
                    tune=False, out="checkpoint")
    if kind == "large":                  # one large sampled lattice
        nx = _pow2(rng, 1024, 16384)
        ny = _pow2(rng, 256, min(16384, (1 << 24) // nx))
        return dict(kind="d2q9", recipe="one", nx=nx, ny=ny, replicas=1, precision="fp32", fields=HYDRO,
                    steps=rng.randint(20, 60), every=rng.choice((10, 20)), noise_mode=0, net=rng.random() < 0.6,
                    tune=False, out="checkpoint")
    if kind == "ragged":                 # odd sizes without sampling, every noise form
        prec = rng.choice(("fp32", "fp32", "fp64"))
        nx, ny = 2 * _log(rng, 8, 2500), _log(rng, 1, 5000)
        budget = 2e9 if prec == "fp32" else 2e7
        steps = max(4, min(300, int(budget / (nx * ny))))
        return dict(kind="d2q9", recipe="one", nx=nx, ny=ny, replicas=1, precision=prec, fields="", steps=steps,
                    every=0, noise_mode=rng.choice((0, 1, 2)), net=prec == "fp32" and rng.random() < 0.4, tune=False,
                    out="workspace")
    if kind == "lb3":
        prec = rng.choice(("fp32", "fp32", "fp64"))
        nx, ny, nz = 2 * _log(rng, 4, 150), _log(rng, 6, 300), _log(rng, 4, 300)
        budget = 1.5e9 if prec == "fp32" else 1.5e7
        steps = max(4, min(200, int(budget / (nx * ny * nz))))
        return dict(kind="lb3", lattice=rng.choice(("D3Q15", "D3Q19")), nx=nx, ny=ny, nz=nz, precision=prec,
                    fields=rng.choice(("0,4,9", "0", "0,1,2,3")), steps=steps, every=rng.choice((1, 5, 20)),
                    n_k=rng.choice((4, 8, 16)), n_lags=rng.randint(1, 8))
    if kind == "spectra":
        prec = rng.choice(("fp32", "fp32", "fp64"))
        nx = _pow2(rng, 16, 16384 if prec == "fp32" else 8192)
        ny = _pow2(rng, 8, 16384 if prec == "fp32" else 4096)
        cap = 2e8 if prec == "fp32" else 2e7
        while nx * ny > cap / 3:
            ny //= 2
        f = rng.randint(1, max(1, min(9, int(cap / (nx * ny)))))
        return dict(kind="spectra", precision=prec, n_fields=f, ny=ny, nx=nx)
    return dict(kind="train", runs=_log(rng, 1, 24), inputs=_log(rng, 100, 8000), n_k=_log(rng, 200, 4000),
                iters=rng.randint(1, 20))


# ---------------------------------------------------------------------------
# Parameters of a case's replicas.

def _fields(case):
    return tuple(int(f) for f in case["fields"].split(",")) if case["fields"] else ()


def _replicas(case, seed):
    """Parameter dicts of the case's replicas; the seed sets the noise and the thermal start."""
    key = 1_000_003 * int(seed) + 17
    if case["kind"] == "d1q3":
        return [W.replica("D1Q3", case["nx"], 1, W.taus_d1q3(0.8), kT=1e-4, seed=key, init_mode=1,
                          fields=_fields(case))]
    if case["kind"] == "lb3":
        taus = W.taus_d3q15 if case["lattice"] == "D3Q15" else W.taus_d3q19
        return [W.replica3(case["nx"], case["ny"], case["nz"], taus(0.8, 0.8, 1.0), kT=1e-4, u0=(0.05, 0.02, 0.0),
                           seed=key, init_mode=1, fields=_fields(case), lattice=case["lattice"])]
    out = []
    for r in range(case["replicas"]):
        if case["recipe"] == "sweep":    # workloads.sweep64
            n = (64, 128, 256, 512)[r % 4]
            ts = 0.55 + 0.45 * ((29 * r) % 64) / 63.0
            out.append(W.replica("D2Q9", n, n, W.taus_d2q9(ts, ts, 1.0), kT=1e-4, u0=(0.02 * (r // 4), 0.0),
                                 seed=key + r, stream=r, init_mode=1, fields=_fields(case)))
        else:
            big = case["nx"] * case["ny"] > 1 << 24      # the benchmark starts uniform
            out.append(W.replica("D2Q9", case["nx"], case["ny"], W.taus_d2q9(0.6, 0.7, 1.0), kT=1e-4,
                                 u0=(0.1 - 0.003 * r, 0.05), seed=key + r, stream=r, init_mode=0 if big else 1,
                                 fields=_fields(case), noise_mode=case["noise_mode"]))
    return out


def _wave_vectors(case):
    """(kz, ky, kx) of the time correlators: the lowest axis and diagonal modes of the box."""
    out = []
    for m in range(case["n_k"]):
        k = m // 4 + 1
        kz, ky, kx = ((0, 0, k), (0, k, 0), (k, 0, 0), (k, k, k))[m % 4]
        out.append((kz % case["nz"], ky % case["ny"], kx % case["nx"]))
    return [k if any(k) else (0, 0, 1) for k in out]


def _pair_list(n):
    return [(a, b) for a in range(n) for b in range(a, n)]


def _align(x):
    return (x + 255) // 256 * 256


# ---------------------------------------------------------------------------
# prepare and run.

def prepare(case, seed):
    kind = case["kind"]
    if kind == "spectra":
        dt = torch.float32 if case["precision"] == "fp32" else torch.float64
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        shape = (case["n_fields"], case["ny"], case["nx"])
        fields = 0.01 * torch.randn(shape, generator=g, device="cuda", dtype=dt)
        nb, ns = spectra_sizes(*shape, case["precision"])
        return dict(case=case, fields=fields, sums=torch.zeros(ns, dtype=torch.float64, device="cuda"),
                    mean0=torch.zeros(shape[0], dtype=torch.float64, device="cuda"),
                    scratch=torch.empty(nb, dtype=torch.uint8, device="cuda"))
    if kind == "train":
        x, sp, g, w = _train_inputs(case, seed)
        return dict(case=case, trainer=learned.Trainer(x, learned.gram(sp, g), case["n_k"], w, lr=3e-3))
    sim = Sim(_replicas(case, seed), precision=case["precision"])
    state = dict(case=case, sim=sim)
    if kind == "lb3":
        sim.set_time_correlator(_wave_vectors(case), case["n_lags"])
    if kind == "d2q9":
        if case["net"]:
            sim.set_mlp(W.mlp_weights(int(seed), out_scale=0.1))
        if case["tune"]:
            sim.autotune(3)
        if case["out"] == "checkpoint":
            n = ctypes.c_size_t()
            L.check(L.lib().flb_save(sim._ctx, None, ctypes.byref(n)))
            state["blob"] = torch.empty(n.value, dtype=torch.uint8, pin_memory=True)
            state["parts"] = _checkpoint_parts(sim, case, n.value)
    return state


def _checkpoint_parts(sim, case, total):
    """Views of a checkpoint: 64 bytes of header, then per replica its populations and its
    pair sums (blocks of c columns, c the width that gives the checkpoint its size)."""
    rs = 4 if case["precision"] == "fp32" else 8
    pops = [9 * p["nx"] * p["ny"] * rs for p in sim.params]

    def sums(p, c):
        f = len(p["fields"])
        if not f:
            return 0
        pts = p["ny"] * (-(-(p["nx"] // 2 + 1) // c) * c)
        return f * _align(8 * pts) + f * (f - 1) // 2 * _align(16 * pts) + 8 * f

    for c in (16, 8, 4, 2, 1):
        if 64 + sum(pops) + sum(sums(p, c) for p in sim.params) == total:
            break
    else:
        raise RuntimeError("checkpoint of %d bytes" % total)
    parts, off = [], 64
    for p, n in zip(sim.params, pops):
        parts.append((off, n, sums(p, c)))
        off += n + sums(p, c)
    return parts


def _checkpoint(state):
    """flb_save into the program's pinned buffer: [populations, pair sums] of all replicas."""
    sim, blob = state["sim"], state["blob"]
    n = ctypes.c_size_t(blob.numel())
    L.check(L.lib().flb_save(sim._ctx, ctypes.c_void_p(blob.data_ptr()), ctypes.byref(n)))
    dt = torch.float32 if state["case"]["precision"] == "fp32" else torch.float64
    pops = [blob[o:o + n].view(dt) for o, n, _ in state["parts"]]
    sums = [blob[o + n:o + n + s].view(torch.float64) for o, n, s in state["parts"] if s]
    if len(pops) == 1:
        return pops + sums
    return [torch.cat(pops)] + ([torch.cat(sums)] if sums else [])


def _workspace(state):
    """The populations of a single replica in the caller's workspace, which begins with two
    256-byte aligned population buffers (the one of the step's parity holds the state)."""
    sim, p = state["sim"], state["sim"].params[0]
    rs = 4 if state["case"]["precision"] == "fp32" else 8
    dt = torch.float32 if rs == 4 else torch.float64
    n = Q[p["lattice"]] * p["nx"] * p["ny"] * p.get("nz", 1) * rs
    base = (sim.step & 1) * _align(n)
    return sim.workspace[base:base + n].view(dt)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "spectra":
        sums, mean0 = spectra_accumulate(state["fields"], state["sums"], state["mean0"], state["scratch"])
        return [sums, mean0]
    if kind == "train":
        t = state["trainer"].step(case["iters"])
        return [t.w, t.m, t.v, t.grad, t.loss, t.msq]
    sim = state["sim"].run(case["steps"], case["every"])
    if kind == "d1q3":
        f = _fields(case)
        return [sim.populations()] + [sim.correlator(0, f[a], f[b]) for a, b in _pair_list(len(f))]
    if kind == "lb3":
        f = _fields(case)
        return [_workspace(state)] + [sim.time_correlator(0, a, b) for a in f for b in f]
    if case["out"] == "checkpoint":
        return _checkpoint(state)
    if not case["fields"]:
        return [_workspace(state)]
    return [_workspace(state), _workspace_sums(state)]


def _workspace_sums(state):
    """The pair sums of a single large FP32 replica as one FP64 view of the workspace: after
    the two population buffers come the fields, the row spectra of two samples in tiles of
    16 columns, and the sums."""
    if "sums" not in state:
        sim, p = state["sim"], state["sim"].params[0]
        n = ctypes.c_size_t()
        L.check(L.lib().flb_save(sim._ctx, None, ctypes.byref(n)))
        size = n.value - 64 - 9 * p["nx"] * p["ny"] * 4          # a checkpoint holds exactly these sums
        v, f = p["nx"] * p["ny"], len(p["fields"])
        elems = f * p["ny"] * (-(-(p["nx"] // 2 + 1) // 16) * 16)
        off = 2 * _align(36 * v) + _align(4 * f * v) + 2 * _align(8 * elems)
        state["sums"] = sim.workspace[off:off + size].view(torch.float64)
    return state["sums"]


def work(case):
    """Bytes and operations of one pass.  A step reads and writes every population once; a
    sample reads its fields and reads and writes its FP64 sums; the operations are the
    moment transforms, relaxation and noise of a site (about 20 per population and 40 per
    normal), 5 n log2 n per transform and 8 per pair and wave vector."""
    kind = case["kind"]
    if kind == "train":
        n = case["runs"] * case["inputs"]
        per = 2 * (3 * 32 + 32 * 32 + 6 * 32)
        return {"bytes": case["iters"] * (12 * n + 1382 * 4 * 7), "flops": case["iters"] * 3 * per * n}
    if kind == "spectra":
        rs = 4 if case["precision"] == "fp32" else 8
        v, f = case["nx"] * case["ny"], case["n_fields"]
        pts = case["ny"] * (case["nx"] // 2 + 1)
        return {"bytes": f * v * rs + 2 * 8 * f * f * pts, "flops": f * 2.5 * v * math.log2(v) + 4 * f * f * pts}
    rs = 4 if case["precision"] == "fp32" else 8
    reps = _replicas(case, 0)
    q = Q[reps[0]["lattice"]]
    nc = q - (2 if q == 3 else 3 if q == 9 else 4)
    b = fl = 0.0
    samples = -(-case["steps"] // case["every"]) if case["every"] and case["fields"] else 0
    for p in reps:
        v, f = p["nx"] * p["ny"] * p.get("nz", 1), len(p["fields"])
        b += case["steps"] * 2.0 * q * v * rs
        fl += case["steps"] * v * (20.0 * q + 40.0 * nc + (2 * 1312 if case.get("net") else 0))
        if kind == "lb3":
            b += samples * f * v * rs
            fl += samples * 4.0 * f * v * max(1, case["n_k"] // 2)
        else:
            pts = p["ny"] * (p["nx"] // 2 + 1)
            b += samples * (f * v * rs + 16.0 * f * f * pts)
            fl += samples * (f * 2.5 * v * max(1.0, math.log2(v)) + 4.0 * f * f * pts)
    return {"bytes": b, "flops": fl}


# ---------------------------------------------------------------------------
# The same outputs in 64 bits with plain torch: the scheme of the paper written directly
# (dense moment transforms, the equilibrium of Eq. 2, the noise of Eq. 8), the counter-based
# generator with integers, transforms by torch.fft.

def exact(case, seed):
    kind = case["kind"]
    if kind == "spectra":
        if case["n_fields"] * case["nx"] * case["ny"] > 5e7:
            return None
        return _exact_spectra(prepare(case, seed)["fields"].double())
    if kind == "train":
        return _exact_train(case, seed)
    reps = _replicas(case, seed)
    sites = sum(p["nx"] * p["ny"] * p.get("nz", 1) for p in reps)
    if sites * case["steps"] > 3.5e9 or case["steps"] * len({(p["nx"], p["ny"]) for p in reps}) > 8000:
        return None
    net = None
    if case.get("net"):
        net = {k: torch.as_tensor(np.asarray(v, np.float32)).bfloat16().double().cuda()
               for k, v in W.mlp_weights(int(seed), out_scale=0.1).items()}
    order = {}
    for i, p in enumerate(reps):
        order.setdefault((p["nx"], p["ny"]), []).append(i)
    pops, samples = [None] * len(reps), None
    for idx in order.values():
        f, samples = _exact_run([reps[i] for i in idx], case, net)
        for b, i in enumerate(idx):
            g = f[:, b].reshape(f.shape[0], -1)
            if kind != "d1q3" and case["precision"] == "fp32":       # the stored deviation f - w rho0
                w = torch.as_tensor(_lattice(reps[i]["lattice"])[1], device="cuda")
                g = g - (w * reps[i]["rho0"])[:, None]
            pops[i] = g.reshape(-1)
    if kind == "d2q9":
        return [torch.cat(pops)] + ([None] if case["fields"] else [])
    p, f = reps[0], _fields(case)
    v = p["nx"] * p["ny"] * p.get("nz", 1)
    if kind == "d1q3":
        var = [3 * p["kT"] * p["rho0"] if x < 9 else p["kT"] / p["rho0"] for x in f]
        out = [pops[0].reshape(3, 1, p["nx"])]
        xk = torch.fft.fft(torch.stack(samples)[:, :, 0, 0], dim=-1)        # (n, F, nx)
        for a, b in _pair_list(len(f)):
            c = (xk[:, a] * xk[:, b].conj()).mean(0)
            c[0] = c[0] - xk[:, a, 0].real.mean() * xk[:, b, 0].real.mean()
            out.append((c / (v * math.sqrt(var[a] * var[b]))).reshape(1, -1))
        return out
    out = [pops[0]]
    var = 3 * p["kT"] * p["rho0"]
    x = torch.stack(samples) if samples else None                           # (n, F, K)
    for a in range(len(f)):
        for b in range(len(f)):
            rows = []
            for tau in range(case["n_lags"]):
                n = (x.shape[0] if x is not None else 0) - tau
                if n <= 0:                # no pair of samples at this lag yet
                    rows.append(torch.full((case["n_k"],), complex(math.nan, math.nan), dtype=torch.complex128,
                                           device="cuda"))
                else:
                    rows.append((x[tau:, a] * x[:n, b].conj()).sum(0) / n / (v * var))
            out.append(torch.stack(rows))
    return out


def _exact_spectra(x):
    f, ny, nx = x.shape
    k = torch.fft.rfft2(x)
    out = []
    for a, b in _pair_list(f):
        c = k[a] * k[b].conj()
        out.append(c.real.reshape(-1) if a == b else torch.view_as_real(c.contiguous()).reshape(-1))
    return [torch.cat(out), k[:, 0, 0].real.contiguous()]


def _train_inputs(case, seed):
    r, b = case["runs"], case["inputs"]
    x = W.mlp_inputs(r * b, int(seed)).astype(np.float32).reshape(r, b, 3)
    sp, g = W.correlator_tables(r, case["n_k"], int(seed) + 1)
    return x, sp, g, W.mlp_weights(int(seed) + 2, out_scale=0.1)


def _exact_train(case, seed):
    x, sp, g, w0 = _train_inputs(case, seed)
    r, k = case["runs"], case["n_k"]
    x = torch.as_tensor(x, device="cuda").double()
    target = torch.tensor([1, 0, 0, 1, 0, 1], dtype=torch.float64, device="cuda")[:, None]
    d = torch.as_tensor(sp, device="cuda") - target
    g = torch.as_tensor(g, device="cuda")
    w = torch.as_tensor(learned.pack(w0), device="cuda").double()
    m, v = torch.zeros_like(w), torch.zeros_like(w)
    b1, b2, lr, eps = (float(np.float32(t)) for t in (0.9, 0.999, 3e-3, 1e-8))
    grad = loss = msq = None
    d0 = d.abs().square().sum((1, 2))
    gd = torch.einsum("rpk,rcpk->rc", d.conj(), g).real
    h = torch.einsum("rcpk,repk->rce", g.conj(), g).real
    for t in range(1, case["iters"] + 1):
        w.requires_grad_(True)
        w1, w2, w3 = w[:96].view(32, 3), w[96:1120].view(32, 32), w[1120:1312].view(6, 32)
        a = torch.relu(x @ w1.T + w[1312:1344])
        a = torch.relu(a @ w2.T + w[1344:1376])
        s = 1 + a @ w3.T + w[1376:]
        msq = s.square().mean(1)
        e = msq - 1
        loss = ((d0 + 2 * (gd * e).sum(1) + torch.einsum("rc,rce,re->r", e, h, e)).sum()) / (r * 6 * k)
        grad, = torch.autograd.grad(loss, w)
        with torch.no_grad():
            m = b1 * m + (1 - b1) * grad
            v = b2 * v + (1 - b2) * grad * grad
            w = w.detach() - lr * (m / (1 - b1 ** t)) / (torch.sqrt(v / (1 - b2 ** t)) + eps)
    return [w, m, v, grad, loss.detach().reshape(1), msq.detach()]


def _mulhilo(a, b):
    """High and low words of the 64-bit product of 32-bit values held in int64."""
    lo = a * (b & 0xFFFF)
    p = a * (b >> 16) + (lo >> 16)
    return p >> 16, ((p & 0xFFFF) << 16) | (lo & 0xFFFF)


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 words of the counters (int64 tensors of 32-bit values) under keys k0, k1."""
    for _ in range(10):
        h0, l0 = _mulhilo(c0, 0xD2511F53)
        h1, l1 = _mulhilo(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1, c2, c3


def _box_muller(wa, wb):
    r = torch.sqrt(-2.0 * torch.log((wa.double() + 0.5) * 2.0 ** -32))
    th = 2.0 * math.pi * (wb.double() + 0.5) * 2.0 ** -32
    return r * torch.cos(th), r * torch.sin(th)


def _lattice(name):
    """Velocities (q, 3), weights (q), moment rows (q, q), number of conserved moments."""
    if name == "D1Q3":
        v = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0)], float)
        w = np.array([2 / 3, 1 / 6, 1 / 6])
        x = v[:, 0]
        return v, w, np.stack([x * 0 + 1, np.sqrt(3) * x, (3 * x * x - 1) / np.sqrt(2)]), 2
    if name == "D2Q9":
        v = np.array([(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0),
                      (1, -1, 0)], float)
        w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
        x, y = v[:, 0], v[:, 1]
        s = x * x + y * y
        rows = [x * 0 + 1, np.sqrt(3) * x, np.sqrt(3) * y, 1.5 * (x * x - y * y), 3 * x * y, 1.5 * s - 1,
                np.sqrt(1.5) * x * (3 * s - 4), np.sqrt(1.5) * y * (3 * s - 4), 2.25 * s * s - 3.75 * s + 0.5]
        return v, w, np.stack(rows), 3
    axes = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
    if name == "D3Q15":
        half = [(1, 1, 1), (1, 1, -1), (1, -1, 1), (-1, 1, 1)]
        w = np.array([2 / 9] + [1 / 9] * 6 + [1 / 72] * 8)
    else:
        half = [(1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]
        w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
    v = np.array(axes + [tuple(sg * c for c in e) for e in half for sg in (1, -1)], float)
    x, y, z = v.T
    s = x * x + y * y + z * z
    poly = [x * 0 + 1, x, y, z, x * x - y * y, x * x + y * y - 2 * z * z, x * y, y * z, z * x, s, x * s, y * s, z * s]
    if name == "D3Q15":
        poly += [x * y * z, s * s]
    else:
        poly += [x * (y * y - z * z), y * (z * z - x * x), z * (x * x - y * y), s * s, (x * x - y * y) * s,
                 (x * x + y * y - 2 * z * z) * s]
    rows = []
    for p in poly:                        # Gram-Schmidt in the norm weighted by w
        p = p.astype(float)
        for _ in range(2):
            for m in rows:
                p = p - (w * p * m).sum() * m
        rows.append(p / np.sqrt((w * p * p).sum()))
    return v, w, np.stack(rows), 4


def _exact_run(reps, case, net):
    """Populations (q, B, sites...) after the case's steps, and the samples taken: the sampled
    fields (d1q3) or their transforms at the chosen wave vectors (lb3)."""
    name, dev = reps[0]["lattice"], "cuda"
    v, w, m, nc = _lattice(name)
    q, d3 = len(w), name.startswith("D3")
    nx, ny, nz = reps[0]["nx"], reps[0]["ny"], reps[0].get("nz", 1)
    vol = nx * ny * nz
    t = lambda x: torch.as_tensor(np.asarray(x, float), device=dev)
    B = len(reps)
    V, Wt, M = t(v), t(w), t(m)
    N = (M * Wt).T.contiguous()                                   # f = N M
    col = lambda x: t(x).reshape(-1, 1)                           # one value per replica, over its sites
    rho0, kT = col([p["rho0"] for p in reps]), col([p["kT"] for p in reps])
    u0 = t([list(p["u0"]) + [0.0] * (3 - len(p["u0"])) for p in reps])
    if name == "D1Q3":
        u0[:, 1:] = 0
    tau = t([p["tau"][:q] for p in reps])                         # (B, q)
    key = [p["seed"] & 0xFFFFFFFFFFFFFFFF for p in reps]
    ki = lambda f: torch.tensor([f(k) for k in key], dtype=torch.int64, device=dev)
    k0, k1 = ki(lambda k: k & 0xFFFFFFFF), ki(lambda k: k >> 32)
    st = torch.tensor([p.get("stream", 0) for p in reps], dtype=torch.int64, device=dev)

    def equilibrium(rho, u):                                      # (B, n), (3, B, n) -> (q, B, n)
        cu = torch.einsum("ia,abn->ibn", V, u)
        return Wt[:, None, None] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u * u).sum(0))

    def words(counter, calls, steps):                             # (B, n), [calls], [steps] -> 4 x (S, C, B, n)
        c0 = counter[None, None]
        c1 = torch.as_tensor(steps, dtype=torch.int64, device=dev)[:, None, None, None]
        c2 = torch.as_tensor(calls, dtype=torch.int64, device=dev)[None, :, None, None]
        c3 = st[None, None, :, None]
        full = (len(steps), len(calls)) + tuple(counter.shape)
        return _philox(*(x.expand(full) for x in (c0, c1, c2, c3)), k0[None, None, :, None], k1[None, None, :, None])

    sites = torch.arange(vol, dtype=torch.int64, device=dev)[None].expand(B, vol)
    rho = rho0.expand(B, vol)
    u = u0.T[:, :, None].expand(3, B, vol)
    f = equilibrium(rho, u)
    if reps[0]["init_mode"] == 1:
        ncall = (q + 3) // 4
        a = words(sites, [c | 256 for c in range(ncall)], [0])
        n0, n1 = _box_muller(a[0][0], a[1][0])
        n2, n3 = _box_muller(a[2][0], a[3][0])
        z = torch.stack([n0, n1, n2, n3], 1).reshape(4 * ncall, B, vol)[:q]
        dm = torch.sqrt(3 * kT * rho0) * z
        dm[:nc] -= dm[:nc].mean(2, keepdim=True)
        f = f + torch.einsum("ia,abn->ibn", N, dm)
    itau = (1 / tau)[:, nc:].T[:, :, None]                        # (q - nc, B, 1)
    amp = torch.sqrt(3 * kT * rho0) * torch.sqrt(2 * tau - 1)[:, nc:].T[:, :, None] * itau
    root = None
    mode = reps[0].get("noise_mode", 0)
    if mode == 1:                                                 # correlated noise of the moving equilibrium
        root = []
        for i, p in enumerate(reps):
            feq = equilibrium(rho0[i:i + 1], u0[i][:, None, None])[:, 0, 0]
            cov = 3 * p["kT"] * (M * feq) @ M.T
            ti = 1 / tau[i]
            xi = (tau[i][:, None] + tau[i][None] - 1) * ti[:, None] * ti[None] * cov
            ev, vec = torch.linalg.eigh(xi[nc:, nc:])
            root.append((vec * ev.clamp(min=0).sqrt()) @ vec.T)
        root = torch.stack(root)
    # moments of the reference state, subtracted from the sampled fields
    ref = torch.einsum("ai,ib->ab", M, equilibrium(rho0, u0.T[:, :, None])[:, :, 0])[:, :, None]
    fid = _fields(case)
    phase = None
    if case["kind"] == "lb3":
        z, y, x = torch.meshgrid(*(torch.arange(n, device=dev) for n in (nz, ny, nx)), indexing="ij")
        phase = []
        for kz, ky, kx in _wave_vectors(case):
            a = (kz * z % nz).double() / nz + (ky * y % ny).double() / ny + (kx * x % nx).double() / nx
            phase.append(torch.polar(torch.ones_like(a), -2 * math.pi * a).reshape(-1))
        phase = torch.stack(phase)
    normals, chunk = {}, max(1, min(64, int(4e6 // (B * vol))))
    samples = []
    for step in range(case["steps"]):
        if step % chunk == 0:                                     # the normals of the next steps at once
            ss = list(range(step, min(step + chunk, case["steps"])))
            if name == "D2Q9":                                    # sites 2q, 2q + 1 share counter q
                a = words(sites[:, ::2] >> 1, [0, 1, 2], ss)
                twelve = torch.stack([a[k % 4][:, k // 4] for k in range(12)], 1)          # (S, 12, B, n/2)
                six = torch.stack([twelve[:, :6], twelve[:, 6:]], -1).reshape(len(ss), 6, B, vol)
                n0, n1 = _box_muller(six[:, 0::2], six[:, 1::2])
                z = torch.stack([n0, n1], 2).reshape(len(ss), 6, B, vol)
            else:
                a = words(sites, list(range((q - nc + 3) // 4)), ss)
                n0, n1 = _box_muller(a[0], a[1])
                n2, n3 = _box_muller(a[2], a[3])
                z = torch.stack([n0, n1, n2, n3], 2).reshape(len(ss), -1, B, vol)[:, :q - nc]
            normals = dict(zip(ss, z))
        g = f.reshape(q, B, nz, ny, nx)
        f = torch.stack([torch.roll(g[i], tuple(int(c) for c in v[i][::-1]), (1, 2, 3)) for i in range(q)])
        f = f.reshape(q, B, vol)
        rho = f.sum(0)
        u = torch.einsum("ia,ibn->abn", V, f) / rho
        mom = torch.einsum("ai,ibn->abn", M, f)
        if fid and case["every"] and step % case["every"] == 0 and case["kind"] != "d2q9":
            fl = [mom[k, 0] - ref[k, 0] if d3 or k < 9 else u[k - 9, 0] - u0[0, k - 9] for k in fid]
            fl = torch.stack(fl)                                  # (F, sites)
            samples.append(fl.to(torch.complex128) @ phase.T if phase is not None
                           else fl.reshape(len(fid), 1, 1, nx))
        z = normals[step]
        scale = 1.0
        if net is not None:                                       # bfloat16 operands, as documented
            bf = lambda x: x.bfloat16().double()
            a = bf(torch.stack([u[0], u[1], rho - rho0]))
            a = bf(torch.relu(torch.einsum("hi,ibn->hbn", net["W1"], a) + net["b1"][:, None, None]))
            a = bf(torch.relu(torch.einsum("hi,ibn->hbn", net["W2"], a) + net["b2"][:, None, None]))
            scale = 1 + torch.einsum("hi,ibn->hbn", net["W3"], a) + net["b3"][:, None, None]
        if root is not None:
            xi = scale * torch.einsum("bij,jbn->ibn", root, z)
        else:
            xi = scale * amp * z
            if mode == 2:
                xi = xi * torch.sqrt(rho / rho0)
        eq = torch.einsum("ai,ibn->abn", M[nc:], equilibrium(rho, u))
        f = f + torch.einsum("ia,abn->ibn", N[:, nc:], (eq - mom[nc:]) * itau + xi)
    return f, samples
