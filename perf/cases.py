"""Performance cases: the work that a program using this package has it do.

Every case goes through the public entry points: out-of-core plans fed from
and read back into pinned host memory (set_field, step, get_field), the
stand-alone codecs, the in-core stencil runs and the differentiable wave
run.  The sizes are those of the benchmark's workloads and of the tests, or
generic; ``draw`` spreads them over the same ranges.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2109_05410_gb300 as ooc
from paper_2109_05410_gb300.autograd import WaveConfig

DX = 10.0  # grid spacing of the wave cases (m)
SOURCE_STEPS = 4096  # length of a wave plan's source series


def listed():
    return [
        # The headline: a 1024^3 heat field streamed through a 1 GiB device
        # budget as FR4 units at 16 bits per value, four steps per transfer.
        dict(name="heat_plan_1024", kind="plan", stencil="heat7", precision="fp32", nz=1024, ny=1024, nx=1024,
             rw="fr4", rw_rate=16, ro="fr4", ro_rate=16, k=4, steps=32, budget_mib=1024),
        # The paper's propagator with both its read-write levels and kappa
        # stored compressed (code 4), ten steps per transfer, source on.
        dict(name="wave_plan_512", kind="plan", stencil="wave25", precision="fp32", nz=512, ny=512, nx=512,
             rw="fr4", rw_rate=16, ro="fr4", ro_rate=16, k=10, steps=40, budget_mib=768),
        # The paper's precision: FP64 fields at 32 of every 64 bits.
        dict(name="heat_plan_fp64_512", kind="plan", stencil="heat7", precision="fp64", nz=512, ny=512, nx=512,
             rw="fr4", rw_rate=32, ro="fr4", ro_rate=32, k=4, steps=16, budget_mib=256),
        # One slab window of the headline, as the stand-alone codec sees it:
        # writing a unit ...
        dict(name="encode_window", kind="codec", op="encode", precision="fp32", nz=56, ny=1024, nx=1024, rate=16,
             corr=32.0),
        # ... and reading it back.
        dict(name="decode_window", kind="codec", op="decode", precision="fp32", nz=56, ny=1024, nx=1024, rate=16,
             corr=32.0),
        # A small field whose sides are no multiples of 4, there and back:
        # the smallest codec calls.
        dict(name="codec_ragged_small", kind="codec", op="roundtrip", precision="fp32", nz=37, ny=45, nx=133, rate=16,
             corr=3.0),
        # A stored snapshot with an error bound instead of a rate (the
        # variable-size mode), there and back.
        dict(name="codec_accuracy_512", kind="var", mode="accuracy", param=1e-4, nz=512, ny=512, nx=512, corr=32.0),
        # A double-precision window at 24 of every 64 bits, there and back.
        dict(name="codec_fp64_window", kind="codec", op="roundtrip", precision="fp64", nz=56, ny=1024, nx=1024,
             rate=24, corr=32.0),
        # In-core heat: a grid that fits the device, pairs of steps per launch.
        dict(name="heat_incore_512", kind="heat", entry="fused", nz=512, ny=512, nx=512, steps=10, corr=32.0),
        # A small in-core grid: launches count.
        dict(name="heat_small_128", kind="heat", entry="single", nz=128, ny=128, nx=128, steps=8, corr=16.0),
        # The in-core double-precision wave run that accuracy studies compare
        # single precision against.
        dict(name="wave_fp64_384", kind="wave64", nz=384, ny=384, nx=384, steps=10, corr=8.0),
        # A gradient of receiver traces with respect to the velocity model:
        # checkpointed forward run and adjoint.
        dict(name="adjoint_256", kind="adjoint", nz=256, ny=256, nx=256, steps=100, every=10, rate=16),
    ]


def _log_int(rng, lo, hi, multiple=1):
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(multiple, v // multiple * multiple)


def draw(rng):
    kind = rng.choice(["plan", "plan", "codec", "codec", "codec", "var", "heat", "heat", "wave64", "adjoint"])
    if kind == "plan":
        stencil = rng.choice(["heat7", "wave25"])
        precision = rng.choice(["fp32", "fp32", "fp64"])
        n = [_log_int(rng, 64, 512, 4) for _ in range(3)]
        if precision == "fp64":
            rates, k = [24, 32], rng.choice([4, 5] if stencil == "heat7" else [4, 10])
        else:
            rates, k = [8, 12, 16, 24], rng.choice([2, 4, 5] if stencil == "heat7" else [4, 10])
        rate = rng.choice(rates)
        # a budget for a quarter of the planes of every ring, and staging
        fields, esize = (2, 8) if stencil == "heat7" else (3, 8)
        halo = (1 if stencil == "heat7" else 4) * (k + 4)
        planes = n[0] // 4 + 2 * halo + 12
        mib = (4 * fields * esize * n[1] * n[2] * planes >> 20) + 2
        return dict(kind=kind, stencil=stencil, precision=precision, nz=n[0], ny=n[1], nx=n[2], rw="fr4", rw_rate=rate,
                    ro="fr4", ro_rate=rate, k=k, steps=k * rng.randint(2, 4) + rng.choice([0, 0, 1]), budget_mib=mib)
    if kind == "codec":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        m = 4 if precision == "fp64" or rng.random() < 0.6 else 1
        return dict(kind=kind, op=rng.choice(["encode", "decode", "roundtrip"]), precision=precision,
                    nz=_log_int(rng, 8, 128, m), ny=_log_int(rng, 16, 768, m), nx=_log_int(rng, 16, 768, m),
                    rate=rng.choice([24, 32] if precision == "fp64" else [8, 12, 16, 24]),
                    corr=rng.choice([4.0, 8.0, 16.0, 32.0]))
    if kind == "var":
        mode = rng.choice(["accuracy", "precision"])
        return dict(kind=kind, mode=mode, param=rng.choice([1e-2, 1e-3, 1e-4, 1e-5]) if mode == "accuracy"
                    else float(rng.choice([14, 16, 20])), nz=_log_int(rng, 8, 384), ny=_log_int(rng, 16, 384),
                    nx=_log_int(rng, 16, 384), corr=rng.choice([8.0, 16.0, 32.0]))
    if kind == "heat":
        return dict(kind=kind, entry=rng.choice(["single", "fused", "fp64"]), nz=_log_int(rng, 16, 512, 4),
                    ny=_log_int(rng, 16, 512, 4), nx=_log_int(rng, 16, 512, 4), steps=rng.randint(1, 12),
                    corr=rng.choice([8.0, 16.0, 32.0]))
    if kind == "wave64":
        return dict(kind=kind, nz=_log_int(rng, 16, 384, 4), ny=_log_int(rng, 16, 384, 4),
                    nx=_log_int(rng, 16, 384, 4), steps=rng.randint(1, 10), corr=8.0)
    return dict(kind=kind, nz=_log_int(rng, 32, 256, 4), ny=_log_int(rng, 32, 256, 4), nx=_log_int(rng, 32, 256, 4),
                steps=rng.randint(20, 60), every=rng.choice([5, 10]), rate=rng.choice([0, 16, 24]))


# ---- inputs --------------------------------------------------------------------

def _smooth(shape, corr, seed, dtype, terms=16):
    """A random field of unit variance and correlation length ``corr`` cells:
    a sum of separable cosine products, evaluated on the GPU in FP64."""
    nz, ny, nx = shape
    g = np.random.default_rng(seed)
    k, ph = g.normal(0.0, 1.0 / corr, size=(3, terms)), g.uniform(0.0, 2.0 * math.pi, size=(3, terms))

    def axis(n, a):
        i = torch.arange(n, dtype=torch.float64, device="cuda")
        return torch.cos(torch.outer(i, torch.from_numpy(k[a]).cuda()) + torch.from_numpy(ph[a]).cuda())

    x, y, z = axis(nx, 0), axis(ny, 1), axis(nz, 2) * math.sqrt(8.0 / terms)
    plane = (y[:, None, :] * x[None, :, :]).reshape(-1, terms).T.contiguous()
    out = torch.empty(shape, dtype=dtype, device="cuda")
    for z0 in range(0, nz, 32):
        out[z0:z0 + 32] = (z[z0:z0 + 32] @ plane).reshape(-1, ny, nx).to(dtype)
    return out


def _velocity(shape, seed):
    """Eight layers from 1500 to 4500 m/s, perturbed by 5 % (m/s, FP64)."""
    nz = shape[0]
    layer = torch.clamp(torch.arange(nz, device="cuda") * 8 // nz, max=7)
    v = (1500.0 + 3000.0 * layer.double() / 7.0)[:, None, None]
    return v * (1.0 + 0.05 * _smooth(shape, 8.0, seed, torch.float64).clamp(-1.0, 1.0))


def _ricker(n, dt, freq=15.0):
    a = (math.pi * freq * (np.arange(n) * dt - 1.0 / freq)) ** 2
    return (1.0 - 2.0 * a) * np.exp(-a)


def _shape(case):
    return case["nz"], case["ny"], case["nx"]


def _wave_inputs(case, seed, nw):
    """(kappa, p, p_prev, source point (x, y, z), source series), FP64: a
    wavefield under way in a layered model."""
    shape = _shape(case)
    v = _velocity(shape, seed)
    dt = 0.4 * DX / (4500.0 * 1.05)
    kappa = (v * (dt / DX)) ** 2
    p = 1e-3 * _smooth(shape, 8.0, seed + 1, torch.float64)
    src = (case["nx"] // 2, case["ny"] // 2, case["nz"] // 2)
    w = (_ricker(nw, dt) * float(kappa[src[2], src[1], src[0]]) * 1e-1).astype(np.float32)
    return kappa, p, 0.95 * p, src, w


def _adjoint_inputs(case, seed):
    shape = _shape(case)
    nz, ny, nx = shape
    v = _velocity(shape, seed).float()
    dt = 0.4 * DX / (4500.0 * 1.05)
    c = dt / DX
    src = (nx // 2, ny // 2, nz // 2)
    w = (_ricker(case["steps"], dt) * float((float(v[src[2], src[1], src[0]]) * c) ** 2)).astype(np.float32)
    rec = torch.tensor([(nz // 4 * ny + y) * nx + x for y in range(0, ny, 8) for x in range(0, nx, 8)],
                       dtype=torch.int64, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(seed)
    res = torch.randn((case["steps"], rec.numel()), generator=g, device="cuda")
    return v, WaveConfig(dt=dt, dx=DX, nsteps=case["steps"], rec=rec, src=src, w=w, every=case["every"],
                         rate=case["rate"]), res


def _pinned(t):
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h.numpy(), h  # the tensor owns the pinned block


def prepare(case, seed):
    kind, shape = case["kind"], _shape(case)
    s = dict(case=case)
    if kind == "plan":
        dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
        s["plan"] = plan = ooc.Plan(
            nx=case["nx"], ny=case["ny"], nz=case["nz"], stencil=case["stencil"], k=case["k"], rw_format=case["rw"],
            rw_rate=case["rw_rate"], ro_format=case["ro"], ro_rate=case["ro_rate"], precision=case["precision"],
            device_budget_bytes=case["budget_mib"] << 20)
        if case["stencil"] == "heat7":
            fields = [_smooth(shape, 32.0, seed, dtype)]
        else:
            kappa, p, pm, src, w = _wave_inputs(case, seed, SOURCE_STEPS)
            fields = [p.to(dtype), pm.to(dtype)]
            plan.set_field(2, _pinned(kappa.to(dtype))[0])
            plan.set_source(*src, w)
        s["in"] = [_pinned(f) for f in fields]
        s["out"] = [_pinned(torch.zeros_like(f)) for f in fields]
    elif kind == "codec":
        dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
        s["field"] = _smooth(shape, case["corr"], seed, dtype)
        enc = ooc.ooc_compress64 if dtype == torch.float64 else ooc.ooc_compress
        nbytes = ooc.ooc_compressed_bytes(case["nx"], case["ny"], case["nz"], case["rate"])
        s["stream"] = torch.zeros(nbytes, dtype=torch.uint8, device="cuda")
        s["decoded"] = torch.zeros_like(s["field"])
        if case["op"] == "decode":
            enc(s["field"], case["rate"], d_out=s["stream"])
    elif kind == "var":
        s["field"] = _smooth(shape, case["corr"], seed, torch.float32)
        s["mode"] = ooc.OOC_FR4_ACCURACY if case["mode"] == "accuracy" else ooc.OOC_FR4_PRECISION
        blocks = ((case["nx"] + 3) // 4) * ((case["ny"] + 3) // 4) * ((case["nz"] + 3) // 4)
        # room for a stream as large as the raw blocks
        s["stream"] = torch.zeros(256 * blocks, dtype=torch.uint8, device="cuda")
        s["index"] = torch.zeros(blocks + 1, dtype=torch.int64, device="cuda")
        s["decoded"] = torch.zeros_like(s["field"])
    elif kind == "heat":
        s["u"] = _smooth(shape, case["corr"], seed, torch.float64 if case["entry"] == "fp64" else torch.float32)
        s["tmp"] = torch.zeros_like(s["u"])
    elif kind == "wave64":
        s["kappa"], s["p"], s["pm"], s["src"], w = _wave_inputs(case, seed, case["steps"])
        s["w"] = w.astype(np.float64)
    else:
        v, s["cfg"], s["res"] = _adjoint_inputs(case, seed)
        s["v"] = v.requires_grad_(True)
    return s


# ---- one pass --------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "plan":
        plan = state["plan"]
        for f, (a, _) in enumerate(state["in"]):
            plan.set_field(f, a)
        plan.step(case["steps"])
        return [plan.get_field(f, a) for f, (a, _) in enumerate(state["out"])]
    if kind == "codec":
        f64 = case["precision"] == "fp64"
        enc, dec = (ooc.ooc_compress64, ooc.ooc_decompress64) if f64 else (ooc.ooc_compress, ooc.ooc_decompress)
        out = {}
        if case["op"] != "decode":
            out["stream"] = enc(state["field"], case["rate"], d_out=state["stream"])
        if case["op"] != "encode":
            out["decoded"] = dec(state["stream"], _shape(case), case["rate"], d_out=state["decoded"])
        return out
    if kind == "var":
        stream, index = ooc.ooc_compress_var(state["field"], state["mode"], case["param"], d_out=state["stream"],
                                             d_index=state["index"])
        decoded = ooc.ooc_decompress_var(stream, index, _shape(case), state["mode"], case["param"],
                                         d_out=state["decoded"])
        # the buffer that the stream is a part of (its length is the index's last entry)
        return {"stream": state["stream"], "index": index, "decoded": decoded}
    if kind == "heat":
        step = {"single": ooc.ooc_heat7_steps, "fused": ooc.ooc_heat7_steps_fused, "fp64": ooc.ooc_heat7_steps_f64}
        return step[case["entry"]](state["u"], state["tmp"], case["steps"])
    if kind == "wave64":
        return ooc.ooc_wave25_steps_f64(state["p"], state["pm"], state["kappa"], case["steps"], src=state["src"],
                                        w=state["w"])
    traces = ooc.wave_forward(state["v"], state["cfg"])
    (grad,) = torch.autograd.grad(traces, state["v"], state["res"])
    return {"traces": traces.detach(), "grad": grad}


# ---- what a pass cannot do without -------------------------------------------------

def work(case):
    n = case["nz"] * case["ny"] * case["nx"]
    kind = case["kind"]
    if kind == "plan":
        esize = 8 if case["precision"] == "fp64" else 4
        fields, flops = (1, 9) if case["stencil"] == "heat7" else (2, 35)
        return {"bytes": 2 * fields * esize * n, "flops": flops * n * case["steps"]}
    if kind == "codec":
        esize = 8 if case["precision"] == "fp64" else 4
        blocks = ((case["nx"] + 3) // 4) * ((case["ny"] + 3) // 4) * ((case["nz"] + 3) // 4)
        one = esize * n + 8 * case["rate"] * blocks
        return {"bytes": one * (2 if case["op"] == "roundtrip" else 1), "flops": 0}
    if kind == "var":
        return {"bytes": 2 * 4 * n, "flops": 0}  # the stream's size depends on the values
    if kind == "heat":
        return {"bytes": 2 * (8 if case["entry"] == "fp64" else 4) * n, "flops": 9 * n * case["steps"]}
    if kind == "wave64":
        return {"bytes": 5 * 8 * n, "flops": 35 * n * case["steps"]}
    # forward, replay and adjoint steps, and the gradient's Laplacian
    return {"bytes": 2 * 4 * n + 8 * case["steps"] * ((case["ny"] + 7) // 8) * ((case["nx"] + 7) // 8),
            "flops": 4 * 35 * n * case["steps"]}


# ---- the same in 64 bits -------------------------------------------------------------

C8 = (-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0)


def _add_neighbours(out, u, m, c):
    """out += c * (the six values m cells away), zero outside the grid."""
    for axis in range(3):
        n = u.shape[axis]
        if m < n:
            out.narrow(axis, m, n - m).add_(u.narrow(axis, 0, n - m), alpha=c)
            out.narrow(axis, 0, n - m).add_(u.narrow(axis, m, n - m), alpha=c)


def _laplacian8(p):
    out = p * (3.0 * C8[0])
    for m in range(1, 5):
        _add_neighbours(out, p, m, C8[m])
    return out


def _heat(u, steps, r=1.0 / 6.0):
    for _ in range(steps):
        v = u * (1.0 - 6.0 * r)
        _add_neighbours(v, u, 1, r)
        u = v
    return u


def _wave(p, pm, kappa, steps, src, w):
    for n in range(steps):
        q = kappa * _laplacian8(p) + 2.0 * p - pm
        q[src[2], src[1], src[0]] += float(w[n])
        p, pm = q, p
    return p, pm


def exact(case, seed):
    kind, shape = case["kind"], _shape(case)
    if kind == "plan":
        f64 = case["precision"] == "fp64"
        dtype = torch.float64 if f64 else torch.float32
        if case["stencil"] == "heat7":
            return [_heat(_smooth(shape, 32.0, seed, dtype).double(), case["steps"])]
        kappa, p, pm, src, w = _wave_inputs(case, seed, SOURCE_STEPS)
        return list(_wave(p.to(dtype).double(), pm.to(dtype).double(), kappa.to(dtype).double(), case["steps"], src,
                          w))
    if kind == "codec":
        if case["op"] == "encode":
            return None
        out = {"stream": None} if case["op"] == "roundtrip" else {}
        out["decoded"] = _smooth(shape, case["corr"], seed, torch.float64 if case["precision"] == "fp64"
                                 else torch.float32).double()
        return out
    if kind == "var":
        return {"stream": None, "index": None, "decoded": _smooth(shape, case["corr"], seed, torch.float32).double()}
    if kind == "heat":
        u = _smooth(shape, case["corr"], seed, torch.float64 if case["entry"] == "fp64" else torch.float32)
        return _heat(u.double(), case["steps"])
    if kind == "wave64":
        kappa, p, pm, src, w = _wave_inputs(case, seed, case["steps"])
        return _wave(p, pm, kappa, case["steps"], src, w)
    v, cfg, res = _adjoint_inputs(case, seed)
    v, res, c = v.double(), res.double(), cfg.dt / cfg.dx
    kappa = (v * c) ** 2
    p, pm = torch.zeros_like(v), torch.zeros_like(v)
    laps, traces = [], []
    for n in range(cfg.nsteps):
        lap = _laplacian8(p)
        laps.append(lap)
        q = kappa * lap + 2.0 * p - pm
        q[cfg.src[2], cfg.src[1], cfg.src[0]] += float(cfg.w[n])
        p, pm = q, p
        traces.append(p.flatten()[cfg.rec])
    mu1, mu2, grad = torch.zeros_like(v), torch.zeros_like(v), torch.zeros_like(v)
    for m in range(cfg.nsteps, 0, -1):
        mu = _laplacian8(kappa * mu1) + 2.0 * mu1 - mu2
        mu.view(-1)[cfg.rec] += res[m - 1]
        grad += mu * laps[m - 1]
        mu1, mu2 = mu, mu1
    return {"traces": torch.stack(traces), "grad": grad * 2.0 * v * c * c}
