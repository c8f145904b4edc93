"""What this framework is measured on: simulations of diffusing walkers as a
user runs them, through the Python face of the C ABI.

A case is one program's call with its sizes:
  run         a kept substrate and sequence; rms_run and rms_read_signal
  simulate    the whole call from host arrays: substrate, sequence, run, read
  checkpoint  a run stopped half way, its walkers read to the host, resumed
  serve       a stream of requests given to a server, all results awaited
  setup       a new substrate and a new sequence, their b-values and a first
              look at the signal
  readout     rms_readout_noalloc over walker data that the caller holds

Every input (geometry, tissue tables, Philox key) is made from the seed; the
generators follow the recipes of rms_inputs (axons, Voronoi cells, cylinder),
on the GPU.
"""
import ctypes
import math
import types

import numpy as np
import torch

import paper_2012_06478_gb300 as rms
from paper_2012_06478_gb300 import _lib

FP64, FP32 = rms.RMS_FP64, rms.RMS_FP32


def listed():
    run = dict(kind="run", bits=32, shapes=1, dirs=30, nb=11, rec=20, relax="none", interaction="ec", absorb=False,
               morton=False, open_x=False, bath="live")
    return [
        # the smallest call: a quick look at one geometry (a smoke-sized run; launches and latency count)
        dict(run, name="cylinder-smallest", geometry="cylinder", nx=32, ny=32, nz=32, voxel=0.2, dt=1e-3,
             walkers=512, steps=400, dirs=3, nb=2, rec=8),
        # the plain-form check case end to end: host arrays in, signal and moments out
        dict(run, name="cylinder-fp64-simulate", kind="simulate", bits=64, geometry="cylinder", nx=32, ny=32, nz=32,
             voxel=0.2, dt=1e-3, walkers=10_000, steps=5000, dirs=3, nb=2, rec=100),
        # a medium request: the log-middle of the serving load's walkers and steps, one axon bundle
        dict(run, name="axons-64-medium", geometry="axons", nx=64, ny=64, nz=64, voxel=0.1, dt=2e-4,
             walkers=100_000, steps=7000, nb=5, rec=70),
        # the benchmark's substrate and walker count in the production form, a tenth of its steps
        dict(run, name="axons-fp32", geometry="axons", nx=200, ny=200, nz=400, voxel=0.1, dt=2e-4,
             walkers=1_000_000, steps=10_000, rec=10),
        # the same substrate in the plain form (reference-quality runs)
        dict(run, name="axons-fp64", bits=64, geometry="axons", nx=200, ny=200, nz=400, voxel=0.1, dt=2e-4,
             walkers=330_000, steps=3000, rec=10),
        # PGSE and five OGSE waveforms at once over T2 tissue with unequal D; labels the size of the L2
        dict(run, name="axons-ogse-t2", geometry="axons", nx=400, ny=400, nz=400, voxel=0.1, dt=4e-4,
             walkers=4_000_000, steps=1000, shapes=6, nb=5, rec=10, relax="t2", morton=True),
        # the largest: 512^3 cells, 1e7 walkers, T1 and T2, labels larger than the L2
        dict(run, name="voronoi-512", geometry="voronoi", nx=512, ny=512, nz=512, voxel=0.1, dt=1e-4,
             walkers=10_000_000, steps=1500, dirs=64, nb=8, rec=15, relax="t1t2", morton=True),
        # a plain-form stimulated-echo run that is stopped, stored and resumed, ragged sizes
        dict(run, name="checkpoint-fp64", kind="checkpoint", bits=64, geometry="voronoi", nx=101, ny=101, nz=101,
             voxel=0.1, dt=2e-4, walkers=50_001, steps=3001, nb=4, rec=7, relax="t1t2"),
        # magnetization transfer: absorbing membranes, walkers inside axons only, an open edge, ragged sizes
        dict(run, name="axons-absorbing", geometry="axons", nx=97, ny=131, nz=89, voxel=0.1, dt=2e-4,
             walkers=300_007, steps=3000, nb=5, rec=10, relax="t2", absorb=True, open_x=True, bath="dead"),
        # continuous batching: mixed geometries, walkers, steps and directions
        dict(kind="serve", name="serve-mixed", bits=32, requests=16, walkers_lo=10_000, walkers_hi=300_000,
             steps_lo=1000, steps_hi=8000, nmax=128),
        # a new substrate and a new long sequence with several waveforms (what a first run pays)
        dict(run, name="setup-axons", kind="setup", geometry="axons", nx=200, ny=200, nz=400, voxel=0.1, dt=2e-4,
             walkers=2048, steps=100_000, shapes=6, nb=5, rec=100, relax="t2", bath="dead"),
        # the signal of walker data that the caller holds, plain form
        dict(kind="readout", name="readout-1e6", walkers=1_000_000, shapes=1, dirs=30, nb=11),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run"] * 8 + ["simulate", "checkpoint", "serve", "setup", "readout", "readout"])
    if kind == "readout":
        return dict(kind=kind, walkers=_log(rng, 1000, 3_000_000), shapes=rng.choice([1, 1, 2, 6]),
                    dirs=rng.randint(3, 64), nb=rng.randint(1, 11))
    if kind == "serve":
        return dict(kind=kind, bits=rng.choice([32, 32, 64]), requests=rng.randint(4, 24), walkers_lo=3000,
                    walkers_hi=_log(rng, 10_000, 100_000), steps_lo=500, steps_hi=_log(rng, 1000, 5000),
                    nmax=rng.choice([48, 64, 128]))
    geometry = rng.choice(["cylinder", "axons", "axons", "voronoi"])
    # cubes, slabs and columns, odd edges among them
    n = _log(rng, 24, 300)
    nx, ny, nz = (max(16, int(n * rng.uniform(0.7, 1.3))) for _ in range(3))
    if geometry == "cylinder":
        nx = ny = min(nx, 100)
    elif geometry == "voronoi":
        nx = ny = nz = n
    bits = rng.choice([32, 32, 64])
    steps = _log(rng, 300, 6000)
    total = _log(rng, 1e6, 6e9 if bits == 32 else 6e8)
    walkers = min(4_000_000, max(500, total // steps))
    interaction = rng.choice(["ec"] * 6 + ["rs", "erl"])
    case = dict(kind=kind, bits=bits, geometry=geometry, nx=nx, ny=ny, nz=nz,
                voxel=0.2 if geometry == "cylinder" else 0.1, dt=1e-3 if geometry == "cylinder" else 2e-4,
                walkers=walkers, steps=steps, shapes=rng.choice([1, 1, 1, 2, 3, 6]), dirs=rng.randint(3, 64),
                nb=rng.randint(1, 11), rec=rng.randint(1, 30), relax=rng.choice(["none", "none", "t2", "t1t2"]),
                interaction=interaction, absorb=rng.random() < 0.15, morton=rng.random() < 0.15,
                open_x=rng.random() < 0.2, bath="dead" if geometry == "axons" and rng.random() < 0.2 else "live")
    if kind == "setup":
        case.update(walkers=2048, steps=_log(rng, 2000, 100_000))
    return case


# ---------------------------------------------------------------- geometry

def _cylinder(nx, nz, rng):
    c = np.arange(nx) + 0.5 - nx / 2.0
    r = nx * rng.uniform(0.28, 0.36)
    inside = (c[None, :] ** 2 + c[:, None] ** 2) <= r * r
    return torch.from_numpy(np.broadcast_to(inside.astype(np.int16), (nz, nx, nx)).copy()).cuda(), 2


def _axons(nx, ny, nz, voxel, rng):
    """Beaded, undulating axons (labels 1..n) in a bath (label 0), at the
    200-axon workload's areal density; one harmonic of undulation each."""
    n = max(2, int(round(200 * nx * ny / 40000.0)))
    Lx, Ly, Lz = nx * voxel, ny * voxel, nz * voxel
    r0 = np.sort(np.maximum(rng.gamma(6.25, 0.08, size=n), 0.15))[::-1]
    r0 = np.minimum(r0, 0.2 * min(Lx, Ly))
    cx, cy = np.zeros(n), np.zeros(n)
    for a in range(n):  # random sequential addition on the periodic cross-section
        shrink = 1.0
        while True:
            x, y = rng.uniform(0, Lx, 64), rng.uniform(0, Ly, 64)
            dx = np.abs(x[:, None] - cx[None, :a])
            dy = np.abs(y[:, None] - cy[None, :a])
            dx, dy = np.minimum(dx, Lx - dx), np.minimum(dy, Ly - dy)
            ok = np.all(dx * dx + dy * dy >= ((r0[:a] + shrink * r0[a]) ** 2)[None, :], axis=1)
            if ok.any():
                k = int(np.argmax(ok))
                cx[a], cy[a], r0[a] = x[k], y[k], shrink * r0[a]
                break
            shrink *= 0.98
    z = (np.arange(nz) + 0.5) * voxel
    lam = Lz / rng.integers(1, 3, size=n)
    w0 = 0.02 * lam * rng.uniform(0.5, 1.5, size=n)
    plane, ph = rng.uniform(0, 2 * np.pi, size=(2, n))
    wz = w0[:, None] * np.cos(2 * np.pi * z[None, :] / lam[:, None] + ph[:, None])
    rz = np.empty((n, nz))
    for a in range(n):
        nb = rng.poisson(Lz / 4.0)
        dz = np.abs(z[:, None] - rng.uniform(0, Lz, size=nb)[None, :])
        dz = np.minimum(dz, Lz - dz)
        rz[a] = r0[a] * (1.0 + (rng.uniform(0.2, 0.6, size=nb)[None, :] * np.exp(-2.0 * dz ** 2)).sum(axis=1))
    reach = rz.max(axis=1) + w0 + voxel
    px = torch.from_numpy((cx[:, None] + wz * np.cos(plane)[:, None]).astype(np.float32)).cuda()
    py = torch.from_numpy((cy[:, None] + wz * np.sin(plane)[:, None]).astype(np.float32)).cuda()
    rr = torch.from_numpy(rz.astype(np.float32)).cuda()
    best = torch.full((nz, ny, nx), 1.0, device="cuda")
    lab = torch.zeros((nz, ny, nx), dtype=torch.int16, device="cuda")
    for a in range(n):
        ix0, ix1 = math.floor((cx[a] - reach[a]) / voxel), math.ceil((cx[a] + reach[a]) / voxel)
        iy0, iy1 = math.floor((cy[a] - reach[a]) / voxel), math.ceil((cy[a] + reach[a]) / voxel)
        ix = torch.arange(ix0, min(ix1 + 1, ix0 + nx), device="cuda")
        iy = torch.arange(iy0, min(iy1 + 1, iy0 + ny), device="cuda")
        dx = (ix + 0.5)[None, None, :] * voxel - px[a][:, None, None]
        dy = (iy + 0.5)[None, :, None] * voxel - py[a][:, None, None]
        dx = dx - Lx * torch.round(dx / Lx)
        dy = dy - Ly * torch.round(dy / Ly)
        ratio = torch.sqrt(dx * dx + dy * dy) / rr[a][:, None, None]
        gx, gy = (ix % nx)[None, :], (iy % ny)[:, None]
        sub = best[:, gy, gx]
        take = ratio < sub
        best[:, gy, gx] = torch.where(take, ratio, sub)
        lab[:, gy, gx] = torch.where(take, torch.tensor(a + 1, dtype=torch.int16, device="cuda"), lab[:, gy, gx])
    return lab, n + 1


def _voronoi(n, rng):
    """Periodic Voronoi cells at the 512^3 workload's density."""
    cells = max(8, int(1000 * (n / 512.0) ** 3))
    p = torch.from_numpy(rng.uniform(0, n, size=(3, cells)).astype(np.float32)).cuda()
    g = torch.arange(n, device="cuda") + 0.5
    d = (g[None, :, None] - p[:, None, :]).abs()
    d = torch.minimum(d, n - d).square()  # [axis][coordinate][cell]
    lab = torch.empty((n, n, n), dtype=torch.int16, device="cuda")
    xy = d[1][:, None, :] + d[0][None, :, :]
    for z in range(n):
        lab[z] = (xy + d[2][z]).argmin(dim=2).to(torch.int16)
    return lab, cells


def _tissue(case, L, rng):
    """Per-label D, T2, T1 and per-pair kappa (and rho), by each geometry's recipe."""
    geometry = case["geometry"]
    D, T1, T2 = np.full(L, 2.0), np.full(L, math.inf), np.full(L, math.inf)
    if geometry == "cylinder":
        K = np.full((L, L), rng.uniform(0.0, 0.02))
    elif geometry == "axons":
        k = np.concatenate([[math.inf], np.exp(rng.uniform(math.log(0.005), math.log(0.05), size=L - 1))])
        with np.errstate(divide="ignore"):
            K = 1.0 / (1.0 / k[:, None] + 1.0 / k[None, :])
    else:
        D = rng.uniform(0.5, 2.5, size=L)
        K = np.triu(rng.uniform(0.0, 0.05, size=(L, L)), 1)
        K = K + K.T
    np.fill_diagonal(K, 0.0)
    if case["relax"] != "none":
        if geometry != "voronoi":
            D[0] = 1.5
        T2 = rng.uniform(40, 100, size=L)
    if case["relax"] == "t1t2":
        T1 = rng.uniform(600, 1000, size=L)
    dead = np.zeros(L, np.uint8)
    dead[0] = case["bath"] == "dead"
    rho = np.full((L, L), 0.02) if case["absorb"] else None
    return D, T2, T1, K, dead, rho


# ---------------------------------------------------------------- sequence

def _boxcar(t0, t1, n):
    k = np.arange(n, dtype=np.float64)
    return np.clip(np.minimum(t1, k + 1) - np.maximum(t0, k), 0.0, 1.0)


def _waveforms(shapes, dt, n):
    """Shape 0: PGSE; the others cosine OGSE of 1, 2, ... periods per lobe in
    the ratio of 20, 40, 60 ... Hz over the whole sequence."""
    d, D = (0.25 * n, 0.75 * n) if shapes == 1 else (0.03 * n, 0.07 * n)
    G = [_boxcar(0.0, d, n) - _boxcar(D, D + d, n)]
    t = np.arange(n + 1) * dt
    for f in range(1, shapes):
        w = 2.0 * f / (n * dt)  # the first fills the sequence with its two lobes
        lobe = []
        for start, sign in ((0.0, 1.0), (1.0 / w, -1.0)):
            tt = np.clip(t, start, start + 1.0 / w)
            lobe.append(sign * np.diff(np.sin(2 * np.pi * w * (tt - start)) / (2 * np.pi * w)) / dt)
        G.append(lobe[0] + lobe[1])
    return np.stack(G)


def _directions(n):
    k = np.arange(n) + 0.5
    z = 1.0 - 2.0 * k / n
    r = np.sqrt(1.0 - z * z)
    phi = np.pi * (3.0 - np.sqrt(5.0)) * k
    return np.stack([r * np.cos(phi), r * np.sin(phi), z], axis=1)


def _program(case, seed):
    """The arrays that a program has in hand before it calls the library."""
    rng = np.random.default_rng([int(seed), 7])
    if case["geometry"] == "cylinder":
        lab, L = _cylinder(case["nx"], case["nz"], rng)
    elif case["geometry"] == "axons":
        lab, L = _axons(case["nx"], case["ny"], case["nz"], case["voxel"], rng)
    else:
        lab, L = _voronoi(case["nx"], rng)
    D, T2, T1, K, dead, rho = _tissue(case, L, rng)
    n = case["steps"]
    mode = None
    if case["relax"] == "t1t2":  # T1 while the magnetisation is stored between the pulses
        mode = np.zeros(n, np.uint8)
        mode[n // 4: 3 * n // 4] = 1
    rec = np.unique(np.linspace(n / case["rec"], n, case["rec"]).astype(np.int64)).clip(1, n)
    return types.SimpleNamespace(
        labels=lab, voxel_um=case["voxel"], periodic=(0 if case["open_x"] else 1, 1, 1), D=D, T2=T2, T1=T1, kappa=K,
        dead=dead, rho=rho, conc=None, lam=-1.0, perm_model=0, dt=case["dt"], n_steps=n,
        G=_waveforms(case["shapes"], case["dt"], n), mode=mode, dirs=_directions(case["dirs"]),
        b=np.linspace(0.0, case["nb"] - 1.0, case["nb"]) if case["nb"] > 1 else np.array([1.0]),
        rec_steps=np.unique(rec), n_walkers=case["walkers"], seed=int(rng.integers(1, 2 ** 62)),
        interaction={"ec": rms.RMS_EC, "rs": rms.RMS_RS, "erl": rms.RMS_ERL}[case["interaction"]],
        precision=FP32 if case["bits"] == 32 else FP64, flags=rms.RMS_MORTON if case["morton"] else 0)


def _substrate(p):
    return rms.rms_create_substrate(p.labels, p.voxel_um, p.D, T2=p.T2, T1=p.T1, kappa=p.kappa, dead=p.dead,
                                    periodic=p.periodic, rho=p.rho)


def _sequence(sub, p):
    return rms.rms_set_sequence(sub, p.dt, p.G, p.dirs, p.b, p.rec_steps, mode=p.mode)


def _requests(case):
    """The sizes of a stream's requests: the load is the case's, its inputs the seed's."""
    rng = np.random.default_rng([case["requests"], case["walkers_hi"], case["steps_hi"], 11])
    out = []
    for r in range(case["requests"]):
        geometry = ["cylinder", "axons", "voronoi"][r % 3]
        n = [32, min(64, case["nmax"]), case["nmax"]][int(rng.integers(0, 3))]
        walkers, steps = (int(round(math.exp(rng.uniform(math.log(case[k + "_lo"]), math.log(case[k + "_hi"])))))
                          for k in ("walkers", "steps"))
        out.append(dict(kind="run", bits=case["bits"], geometry=geometry, nx=n, ny=n, nz=n, voxel=0.1, dt=2e-4,
                        walkers=walkers, steps=steps, shapes=1, dirs=int(rng.integers(6, 65)), nb=5, rec=10,
                        relax=["t2", "none", "t1t2"][r % 3], interaction="ec", absorb=False, morton=False,
                        open_x=False, bath="live"))
    return out


def _held_walkers(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    W, S = case["walkers"], case["shapes"]
    # phases of walkers in tissue: up to a few radians at the largest b; relaxation over an echo time
    phase = 0.4 * torch.randn((W, S, 3), generator=g, device="cuda", dtype=torch.float64)
    A = 0.5 * torch.rand(W, generator=g, device="cuda", dtype=torch.float64)
    bs = 1.0 + 0.25 * torch.rand(S, generator=g, device="cuda", dtype=torch.float64)
    dirs = torch.from_numpy(_directions(case["dirs"])).cuda()
    b = torch.linspace(0.0, case["nb"] - 1.0, case["nb"], dtype=torch.float64, device="cuda") + (case["nb"] == 1)
    return phase, A, bs, dirs, b


# ---------------------------------------------------------------- the cases

def prepare(case, seed):
    s = types.SimpleNamespace(kind=case["kind"])
    if s.kind == "readout":
        s.phase, s.A, s.bs, s.dirs, s.b = _held_walkers(case, seed)
        n = case["shapes"] * case["dirs"] * case["nb"]
        s.re, s.im = torch.zeros((2, n), dtype=torch.float64, device="cuda").unbind(0)
        s.asum = torch.zeros(1, dtype=torch.float64, device="cuda")
    elif s.kind == "serve":
        s.server = rms.Server(policy=rms.RMS_SERVE_FILL)
        s.requests = []
        for r, q in enumerate(_requests(case)):
            p = _program(q, int(seed) * 100 + r)
            sub = _substrate(p)
            s.requests.append((_sequence(sub, p), p))
            p.labels = None  # the substrate holds its own copy
    else:
        s.p = _program(case, seed)
        if s.kind == "simulate":
            s.p.labels = s.p.labels.cpu().numpy().view(np.uint16)
        elif s.kind != "setup":
            s.sub = _substrate(s.p)
            s.seq = _sequence(s.sub, s.p)
            s.p.labels = None
    return s


def run(s):
    if s.kind == "readout":
        rc = _lib.lib.rms_readout_noalloc(
            s.phase.data_ptr(), s.A.data_ptr(), s.phase.shape[0], s.phase.shape[1], s.bs.data_ptr(), s.dirs.shape[0],
            s.dirs.data_ptr(), s.b.numel(), s.b.data_ptr(), s.re.data_ptr(), s.im.data_ptr(), s.asum.data_ptr(),
            ctypes.c_void_p(rms.current_stream()))
        _lib.check(rc)
        return {"S_re": s.re, "S_im": s.im, "alpha_sum": s.asum}
    if s.kind == "serve":
        tickets = [s.server.submit(seq, p.n_walkers, p.seed, p.precision) for seq, p in s.requests]
        return [x for t in tickets for x in s.server.wait(t)[:2]]
    p = s.p
    if s.kind == "simulate":
        r = rms.simulate(p, p.precision, morton=bool(p.flags))
        return {"S": r["S"], "moments": r["moments"], "alpha_sum": r["alpha_sum"], "b_s": r["b_s"]}
    if s.kind == "setup":
        sub = _substrate(p)
        seq = _sequence(sub, p)
        bs = rms.rms_sequence_bvalues(seq)
        first = rms.rms_run(seq, p.n_walkers, p.seed, p.precision, p.flags, interaction=p.interaction,
                            step_end=min(200, p.n_steps))
        S, _, asum = rms.rms_read_signal(first)
        first.close()
        seq.close()
        sub.close()
        return {"S": S, "alpha_sum": asum, "b_s": bs}
    if s.kind == "checkpoint":
        half = max(1, p.n_steps // 2)
        a = rms.rms_run(s.seq, p.n_walkers, p.seed, p.precision, p.flags, interaction=p.interaction, step_end=half)
        stored = rms.rms_read_walkers(a)
        stored.update(step=half, moments=rms.rms_read_signal(a)[1])
        a.close()
        r = rms.rms_run(s.seq, p.n_walkers, p.seed, p.precision, p.flags, interaction=p.interaction, resume=stored)
        S, moments, asum = rms.rms_read_signal(r)
        w = rms.rms_read_walkers(r)
        r.close()
        return {"S": S, "moments": moments, "alpha_sum": asum, "i": w["i"], "o": w["o"], "c": w["c"], "A": w["A"],
                "phase": w["phase"], "stored_i": stored["i"], "stored_phase": stored["phase"]}
    r = rms.rms_run(s.seq, p.n_walkers, p.seed, p.precision, p.flags, interaction=p.interaction)
    S, moments, asum = rms.rms_read_signal(r)
    r.close()
    return {"S": S, "moments": moments, "alpha_sum": asum}


def work(case):
    """The label volume, the waveforms and the walker data read once, results
    written once; the method's operations per walker-step (a Philox call, the
    direction, three face times, 1.5 ds/l_p face events, the phase of each
    shape) and per read-out term (a dot product, a sine and a cosine, two sums)."""
    if case["kind"] == "readout":
        terms = case["walkers"] * case["shapes"] * case["dirs"] * case["nb"]
        return {"bytes": 8.0 * case["walkers"] * (3 * case["shapes"] + 1), "flops": 40.0 * terms}
    if case["kind"] == "serve":
        w = [work(q) for q in _requests(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    voxels = case["nx"] * case["ny"] * case["nz"]
    S, n, W = case["shapes"], case["steps"], case["walkers"]
    taken = min(200, n) if case["kind"] == "setup" else n
    byts = 2.0 * voxels + 8.0 * S * n + 16.0 * S * case["dirs"] * case["nb"] + 176.0 * case["rec"]
    flops = W * taken * (105.0 + 12.0 * S * (0.5 if S == 1 else 1.0)) + 40.0 * W * S * case["dirs"] * case["nb"]
    if case["kind"] == "setup":
        flops += 10.0 * S * n
    if case["kind"] == "checkpoint":
        byts += 3.0 * W * (84.0 + 24.0 * S)
    return {"bytes": byts, "flops": flops}


# ---------------------------------------------------------------- 64-bit reference

M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, key):
    k0, k1 = key & M32, key >> 32
    z = torch.zeros_like(c0)
    c = [c0, z + c1, z + c2, z + c3]
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # 64-bit products; the wrapped sign bit is the top bit
        c = [((p1 >> 32) & M32) ^ c[1] ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c[3] ^ k1, p0 & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def _threshold(P):
    return np.where(P >= 1.0, M32, np.minimum(np.floor(np.maximum(P, 0.0) * 4294967296.0), M32)).astype(np.int64)


class _Walk:
    """The method in plain torch, 64 bits, every walker of a case at once."""

    def __init__(self, p):
        dev = "cuda"
        self.p, self.L = p, len(p.D)
        self.lab = torch.as_tensor(np.ascontiguousarray(p.labels) if isinstance(p.labels, np.ndarray) else p.labels)
        self.lab = self.lab.cuda().view(torch.int16).reshape(-1).to(torch.int32)
        nz, ny, nx = p.labels.shape
        self.N = torch.tensor([nx, ny, nz], device=dev)
        self.stride = torch.tensor([1, nx, nx * ny], device=dev)
        self.per = torch.tensor([bool(x) for x in p.periodic], device=dev)
        ds = np.sqrt(6.0 * p.D * p.dt)
        alive = p.dead == 0
        live = alive[:, None] & alive[None, :] & ~np.eye(self.L, dtype=bool)
        num = p.kappa * (ds / p.D)[:, None] * (2.0 / 3.0)
        den = 1.0 + 0.5 * p.kappa * ((ds / p.D)[:, None] + (ds / p.D)[None, :]) * (2.0 / 3.0)
        self.T = torch.from_numpy(_threshold(np.where(live, num / den, 0.0)).reshape(-1)).cuda()
        self.Tmt = None
        if p.rho is not None:
            P = np.where(~np.eye(self.L, dtype=bool) & alive[:, None], p.rho * (ds / p.D)[:, None] * (2.0 / 3.0), 0.0)
            self.Tmt = torch.from_numpy(_threshold(P).reshape(-1)).cuda()
        self.s = torch.from_numpy(ds / p.voxel_um).cuda()
        self.rate = torch.from_numpy(np.stack([p.dt / p.T2, p.dt / p.T1, 0.0 * p.T2])).cuda()
        W = p.n_walkers
        self.w = torch.arange(W, device=dev, dtype=torch.int64)
        x, y = (_philox(self.w, 0, 0, (1 << 16) | k, p.seed) for k in (0, 1))
        start = torch.nonzero(torch.from_numpy(p.dead == 0).cuda()[self.lab.long()]).reshape(-1)
        vox = start[(x[0] * start.numel() + ((x[1] * start.numel()) >> 32)) >> 32]
        self.wc = torch.stack([vox % nx, (vox // nx) % ny, vox // (nx * ny)])
        self.i0, self.di = self.wc.clone(), torch.zeros_like(self.wc)
        self.o = (torch.stack([x[2], x[3], y[0]]).double() + 0.5) * 2.0 ** -32
        self.o0 = self.o.clone()
        self.c = self.lab[vox].long()
        self.A = torch.zeros(W, device=dev, dtype=torch.float64)
        self.phase = torch.zeros((W, p.G.shape[0], 3), device=dev, dtype=torch.float64)

    def displacement(self):
        return self.p.voxel_um * (self.di + (self.o - self.o0))

    def attempt(self, k, att, mode):
        """The step's state after draw `att`, and who was refused (RS, ERL)."""
        p, inf = self.p, math.inf
        o, wc, di, c, A = self.o, self.wc, self.di, self.c, self.A
        x = _philox(self.w, 0, k, (2 << 16) | att, p.seed)
        z = 1.0 - 2.0 * ((x[0].double() + 0.5) * 2.0 ** -32)
        r = torch.sqrt((1.0 - z) * (1.0 + z))
        phi = (x[1].double() + 0.5) * (2.0 ** -31 * math.pi)
        n = torch.stack([r * torch.cos(phi), r * torch.sin(phi), z])
        sc, rate = self.s[c], self.rate[mode][c]
        d = n * sc
        times = lambda: torch.where(d > 0, 1.0 - o, o) / d.abs()  # noqa: E731
        T = torch.where(d != 0, times(), inf)
        tau = torch.zeros_like(A)
        refused = torch.zeros_like(c, dtype=torch.bool)
        axis = torch.arange(3, device="cuda")[:, None]
        for ev in range(3):
            tmin, best = T.min(0)
            act = (tmin < 1.0) & ~refused
            span = torch.where(act, tmin - tau, 0.0)
            A = A + span * rate
            hit = (axis == best) & act
            up = d.gather(0, best[None])[0] > 0
            o = torch.where(hit, up.double(), (o + span * d).clamp(0.0, 1.0))
            T, tau = torch.where(hit, inf, T), torch.where(act, tmin, tau)
            Nb = self.N[best]
            q = wc.gather(0, best[None])[0] + torch.where(up, 1, -1)
            wall = ((q < 0) | (q >= Nb)) & ~self.per[best]
            q = q % Nb
            c2 = self.lab[(torch.where(hit, q, wc) * self.stride[:, None]).sum(0)].long()
            other = act & ~wall & (c2 != c)
            pair = c * self.L + c2
            if self.Tmt is not None:
                m = _philox(self.w, 0, k, (4 << 16) | att, p.seed)[ev]
                A = torch.where(other & (m < self.Tmt[pair]), inf, A)
            word = x[2 + ev] if ev < 2 else _philox(self.w, 0, k, (3 << 16) | att, p.seed)[0]
            cross = act & ~wall & ((c2 == c) | (word < self.T[pair]))
            back = act & ~cross
            moved = hit & cross
            wc = torch.where(moved, q, wc)
            di = di + torch.where(moved, torch.where(up, 1, -1), 0)
            o = torch.where(moved, 1.0 - up.double(), o)
            c = torch.where(cross, c2, c)
            rate = self.rate[mode][c]
            sn = self.s[c]
            re = cross & (sn != sc)
            d = torch.where(re, n * sn, d)
            T = torch.where(re & torch.isfinite(T), tau + times(), T)
            sc = torch.where(re, sn, sc)
            if p.interaction == rms.RMS_EC:
                flip = torch.where(hit & back, -1.0, 1.0)
                n, d = n * flip, d * flip
            else:
                refused = refused | back
        rem = 1.0 - tau
        return ((o + rem * d).clamp(0.0, 1.0), wc, di, c, A + rem * rate), A, refused

    def step(self, k):
        mode = int(self.p.mode[k - 1]) if self.p.mode is not None else 0
        if self.p.interaction == rms.RMS_EC:
            (self.o, self.wc, self.di, self.c, self.A), _, _ = self.attempt(k, 0, mode)
            return
        left = torch.ones_like(self.c, dtype=torch.bool)
        after = (self.o, self.wc, self.di, self.c, self.A + self.rate[mode][self.c])
        for att in range(1 if self.p.interaction == rms.RMS_RS else 64):
            new, A, refused = self.attempt(k, att, mode)
            take = left & ~refused
            after = tuple(torch.where(take, a, b) for a, b in zip(new, after))
            if self.Tmt is not None:  # a saturation met on a refused draw stays
                sat = left & torch.isinf(A)
                self.A = torch.where(sat, math.inf, self.A)
                after = after[:4] + (torch.where(sat, math.inf, after[4]),)
            left = left & refused
            if not bool(left.any()):
                break
        self.o, self.wc, self.di, self.c, self.A = after

    def moments(self):
        al, x = torch.exp(-self.A), self.displacement()
        m = [al.sum()]
        m += [(al * x[a] * x[b]).sum() for a in range(3) for b in range(a, 3)]
        m += [(al * x[a] * x[b] * x[c] * x[d]).sum()
              for a in range(3) for b in range(a, 3) for c in range(b, 3) for d in range(c, 3)]
        return torch.stack(m)

    def go(self, k0, k1):
        G = torch.from_numpy(self.p.dt * self.p.G).cuda()
        on = np.any(self.p.G != 0.0, axis=0)
        rec = set(int(r) for r in self.p.rec_steps)
        got = []
        for k in range(k0 + 1, k1 + 1):
            self.step(k)
            if on[k - 1]:
                self.phase += G[:, k - 1][None, :, None] * self.displacement().T[:, None, :]
            if k in rec:
                got.append(self.moments())
        return got


def _b_unit(p):
    """b of the unit waveform: dt sum F^2, F the running integral before each step."""
    F = np.concatenate([np.zeros((len(p.G), 1)), np.cumsum(p.dt * p.G, axis=1)[:, :-1]], axis=1)
    return p.dt * np.array([math.fsum(f * f) for f in F])


def _signal(phase, A, bs, dirs, b):
    al = torch.exp(-A)
    q = torch.sqrt(b[None, :] / bs[:, None])
    S = torch.empty((phase.shape[1], dirs.shape[0], b.numel()), dtype=torch.complex128, device="cuda")
    for s in range(phase.shape[1]):
        gp = phase[:, s] @ dirs.T
        for i in range(b.numel()):
            phi = q[s, i] * gp
            S[s, :, i] = torch.complex((al[:, None] * torch.cos(phi)).sum(0), -(al[:, None] * torch.sin(phi)).sum(0))
    return S / al.sum(), al.sum()


def exact(case, seed):
    if case["kind"] == "readout":
        phase, A, bs, dirs, b = _held_walkers(case, seed)
        S, asum = _signal(phase, A, bs, dirs, b)
        return {"S_re": S.real.reshape(-1), "S_im": S.imag.reshape(-1), "alpha_sum": asum.reshape(1)}
    if case["kind"] == "serve":
        return None  # thousands of steps for every request: minutes
    p = _program(case, seed)
    n = min(200, p.n_steps) if case["kind"] == "setup" else p.n_steps
    if n * max(1.0, p.n_walkers / 1e6) * (3.0 if case["interaction"] == "erl" else 1.0) > 3100:
        return None  # about 5 ms a step: over 20 s
    walk = _Walk(p)
    bs = _b_unit(p)
    half = max(1, n // 2) if case["kind"] == "checkpoint" else 0
    got = walk.go(0, half)
    stored_i, stored_phase = walk.i0 + walk.di, walk.phase.clone()
    got += walk.go(half, n)
    S, asum = _signal(walk.phase, walk.A, torch.from_numpy(bs).cuda(), torch.from_numpy(p.dirs).cuda(),
                      torch.from_numpy(p.b).cuda())
    out = {"S": S.cpu().numpy(), "alpha_sum": float(asum)}
    if case["kind"] in ("setup", "simulate"):
        out["b_s"] = bs
    if case["kind"] != "setup":
        out["moments"] = torch.stack(got).cpu().numpy()
    if case["kind"] == "checkpoint":
        out.update(i=None, o=walk.o.T.cpu().numpy(), c=None, A=walk.A.cpu().numpy(), phase=walk.phase.cpu().numpy(),
                   stored_i=None, stored_phase=stored_phase.cpu().numpy())
    return out
