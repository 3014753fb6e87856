"""The work that a user of this library has it do, as cases that can be timed.

Each case goes through the public binding (paper_2609_03922_gb300.spdba): solver
plans (set a field, advance some steps, read the field back), batched transforms,
the block activity scan with its classification, and the learned predictor.  The
sizes are those of the repository's own configurations, tests and benchmark.

listed() holds one case of each use, draw(rng) gives others of the same ranges.
exact(case, seed) writes the same computation out in 64 bits with torch alone.
"""
import math

import torch

from paper_2609_03922_gb300 import spdba

CH_DT, CH_KAPPA = 0.01, 1.0
RCD_DX, RCD_DT, RCD_D, RCD_CROSS = 0.5, 0.01, 0.5, 0.05
RCD_ALPHA, RCD_BETA, RCD_R, RCD_A = 1.0, 0.3, 1.0, 1.0
NLS_BETA2, NLS_GAMMA, NLS_H = -21.7, 1.3, 0.1
ENSEMBLE_SIDES = (128, 192, 256, 384, 512)


def listed():
    return [
        # one small 2-D run in double precision (the plain adaptive configuration): latency and launches
        {"name": "ch2d_128_f64", "kind": "ch", "dims": "128x128", "block": 16, "precision": 1, "half": 0,
         "steps": 40, "mode": 1, "measure": 0, "threshold": 1e-6, "tuned": False},
        # a small 3-D run with the half spectrum stored (the parity size of the benchmark)
        {"name": "ch3d_64_half", "kind": "ch", "dims": "64x64x64", "block": 8, "precision": 0, "half": 1,
         "steps": 40, "mode": 1, "measure": 0, "threshold": 1e-6, "tuned": False},
        # the headline configuration: 3-D 256^3, half spectrum stored, tuned as the benchmark does it
        {"name": "ch3d_256_half", "kind": "ch", "dims": "256x256x256", "block": 8, "precision": 0, "half": 1,
         "steps": 20, "mode": 1, "measure": 0, "threshold": 1e-6, "tuned": True},
        # unequal sides with a factor of three, default options (full spectrum), block energy as the measure
        {"name": "ch3d_ragged_full", "kind": "ch", "dims": "192x128x256", "block": 8, "precision": 0, "half": 0,
         "steps": 20, "mode": 1, "measure": 1, "threshold": 1e-6, "tuned": False},
        # the large grid of the predictor configuration, every mode updated (Regular)
        {"name": "ch3d_384_regular", "kind": "ch", "dims": "384x384x384", "block": 8, "precision": 0, "half": 1,
         "steps": 10, "mode": 0, "measure": 0, "threshold": 1e-6, "tuned": False},
        # the uneven ensemble: 64 2-D runs of five sizes in one plan
        {"name": "ch2d_ensemble64", "kind": "ensemble", "runs": 64, "largest": 512, "block": 16, "steps": 40,
         "threshold": 1e-6},
        # signal propagation: 64 signals of 2^12 .. 2^18 samples in one plan
        {"name": "nls_mixed64", "kind": "nls", "signals": 64, "emin": 12, "emax": 18, "precision": 0, "steps": 40,
         "mode": 1},
        # reaction-cross-diffusion with few components on a middling grid
        {"name": "rcd_64_m8", "kind": "rcd", "dims": "64x64x64", "block": 4, "components": 8, "precision": 0,
         "steps": 20, "mode": 1, "threshold": 1e-4},
        # the large reaction-cross-diffusion run: 48 components on 128^3
        {"name": "rcd_128_m48", "kind": "rcd", "dims": "128x128x128", "block": 4, "components": 48, "precision": 0,
         "steps": 10, "mode": 1, "threshold": 1e-4},
        # batched 1-D transforms longer than one tile, forward and back
        {"name": "fft_1d_2e18_b32", "kind": "fft", "dims": "262144", "batch": 32, "precision": 0},
        # the scan and classification of a 256^3 spectrum as separate calls
        {"name": "assess_256", "kind": "assess", "dims": "256x256x256", "block": 8, "precision": 0,
         "threshold": 1e-6},
        # the block predictor on the 48^3 map: inference and one training gradient over two maps
        {"name": "predictor_48", "kind": "predictor", "side": 48, "maps": 2},
    ]


def draw(rng):
    kind = rng.choice(["ch", "ch", "ch", "ensemble", "nls", "rcd", "fft", "assess", "predictor"])
    if kind == "ch":
        nd = rng.choice([2, 3, 3])
        if nd == 2:
            dims = [rng.choice([64, 128, 192, 256, 384, 512]) for _ in range(2)]
            block, half, precision = rng.choice([8, 16]), 0, rng.choice([0, 1])
        else:
            # at most the largest listed grid; unequal sides as often as not
            while True:
                dims = [rng.choice([64, 128, 192, 256, 384]) for _ in range(3)]
                if dims[0] * dims[1] * dims[2] <= 256 * 256 * 384:
                    break
            block, half, precision = rng.choice([4, 8, 8]), rng.choice([0, 1]), 0
        return {"kind": "ch", "dims": "x".join(map(str, dims)), "block": block, "precision": precision,
                "half": half, "steps": rng.choice([10, 15, 20]), "mode": rng.choice([0, 1, 1]),
                "measure": rng.choice([0, 0, 1]), "threshold": round(10.0 ** rng.uniform(-7, -4), 9),
                "tuned": False}
    if kind == "ensemble":
        return {"kind": "ensemble", "runs": rng.randint(3, 48), "largest": rng.choice([192, 256, 384, 512]),
                "block": rng.choice([8, 16]), "steps": rng.choice([10, 20, 33]),
                "threshold": round(10.0 ** rng.uniform(-7, -5), 9)}
    if kind == "nls":
        emin = rng.randint(9, 15)
        return {"kind": "nls", "signals": int(round(2 ** rng.uniform(0, 5.5))), "emin": emin,
                "emax": rng.randint(emin, 18), "precision": rng.choice([0, 0, 1]), "steps": rng.choice([10, 20, 33]),
                "mode": rng.choice([0, 1])}
    if kind == "rcd":
        nd = rng.choice([2, 3, 3])
        dims = [rng.choice([64, 128, 256] if nd == 2 else [32, 64, 128]) for _ in range(nd)]
        return {"kind": "rcd", "dims": "x".join(map(str, dims)), "block": rng.choice([4, 8]),
                "components": rng.choice([1, 2, 3, 5, 8, 13, 24, 32]), "precision": 0,
                "steps": rng.choice([5, 10]), "mode": rng.choice([0, 1, 1]),
                "threshold": round(10.0 ** rng.uniform(-5, -3), 9)}
    if kind == "fft":
        nd = rng.choice([1, 1, 2, 3])
        if nd == 1:
            dims = [2 ** rng.randint(6, 18)]
        else:
            dims = [rng.choice([16, 32, 64, 128, 192, 256, 384]) for _ in range(nd)]
        n = 1
        for d in dims:
            n *= d
        batch = max(1, int(2.0 ** rng.uniform(0, max(0.0, math.log2(2 ** 23 / n))))) if n < 2 ** 23 else 1
        return {"kind": "fft", "dims": "x".join(map(str, dims)), "batch": batch, "precision": rng.choice([0, 0, 1])}
    if kind == "assess":
        nd = rng.choice([2, 3])
        dims = [rng.choice([128, 192, 256, 384, 512] if nd == 2 else [64, 128, 192, 256]) for _ in range(nd)]
        return {"kind": "assess", "dims": "x".join(map(str, dims)), "block": rng.choice([4, 8, 16]),
                "precision": rng.choice([0, 0, 1]), "threshold": round(10.0 ** rng.uniform(-7, -4), 9)}
    return {"kind": "predictor", "side": rng.randint(8, 48), "maps": rng.randint(1, 3)}


# ------------------------------------------------------------------ inputs
def _dims(case):
    return tuple(int(d) for d in case["dims"].split("x"))


def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(shape, g, dtype=torch.float32):
    return 2.0 * torch.rand(shape, generator=g, device="cuda", dtype=dtype) - 1.0


def _k2(dims, dx, half, dtype):
    """|k|^2 on the grid's frequencies (the last axis 0 .. N/2 with `half`)."""
    out = None
    for a, n in enumerate(dims):
        f = torch.fft.fftfreq(n, device="cuda", dtype=torch.float64)
        if half and a == len(dims) - 1:
            f = torch.fft.rfftfreq(n, device="cuda", dtype=torch.float64)
        k = (2.0 * math.pi * f / dx) ** 2
        k = k.reshape([-1 if b == a else 1 for b in range(len(dims))])
        out = k if out is None else out + k
    return out.to(dtype)


def _ch_fields(dims, means, g):
    """Mid-run Cahn-Hilliard fields: seeded noise about each mean, taken to time 5 (500 steps of
    0.01; here with larger steps of the same scheme), when the high wavenumbers have decayed."""
    means = torch.tensor(means, device="cuda", dtype=torch.float32).reshape((-1,) + (1,) * len(dims))
    c = means + 0.05 * _uniform((len(means),) + tuple(dims), g)
    k2 = _k2(dims, 1.0, True, torch.float32)
    dt, axes = 0.1, tuple(range(1, len(dims) + 1))
    den = 1.0 + dt * CH_KAPPA * k2 * k2
    h = torch.fft.rfftn(c, dim=axes)
    for _ in range(50):
        h -= (dt * k2) * torch.fft.rfftn(c * c * c - c, dim=axes)
        h /= den
        c = torch.fft.irfftn(h, s=tuple(dims), dim=axes)
    return c


def _ensemble(case, seed):
    """(side, mean) of every run."""
    g = torch.Generator()
    g.manual_seed(int(case["runs"]) * 1000 + int(case["largest"]))   # the sizes belong to the case, not the seed
    sides = [s for s in ENSEMBLE_SIDES if s <= case["largest"]]
    pick = torch.randint(0, len(sides), (case["runs"],), generator=g).tolist()
    g.manual_seed(int(seed))
    means = (0.2 * (2.0 * torch.rand(case["runs"], generator=g) - 1.0)).tolist()
    return [(sides[i], m) for i, m in zip(pick, means)]


def _ensemble_fields(case, seed):
    members, g = _ensemble(case, seed), _rng(seed)
    out = [None] * len(members)
    for side in sorted({s for s, _ in members}):
        at = [i for i, (s, _) in enumerate(members) if s == side]
        c = _ch_fields((side, side), [members[i][1] for i in at], g)
        for j, i in enumerate(at):
            out[i] = c[j].contiguous()
    return out


def _nls_lengths(case):
    g = torch.Generator()
    g.manual_seed(int(case["signals"]) * 10000 + int(case["emin"]) * 100 + int(case["emax"]))
    e = torch.randint(case["emin"], case["emax"] + 1, (case["signals"],), generator=g).tolist()
    return [1 << x for x in e]


def _nls_signals(case, seed):
    """Sums of 8 QPSK channels with Gaussian shapes in distinct slots (1/32 of the band), 10 mW peak each."""
    cpu, g = torch.Generator(), _rng(seed)
    cpu.manual_seed(int(seed))
    out = []
    for n in _nls_lengths(case):
        w = n // 32
        slots = torch.randperm(32, generator=cpu)[:8].cuda()
        bits = torch.randint(0, 2, (8, w, 2), generator=g, device="cuda")
        sym = torch.view_as_complex((2.0 * bits - 1.0).to(torch.float64)) / math.sqrt(2.0)
        f = torch.arange(w, device="cuda", dtype=torch.float64) - (w - 1) / 2.0
        local = torch.fft.fftshift(torch.fft.fft(sym, dim=1), dim=1) * torch.exp(-f * f / (2.0 * (w / 6.0) ** 2))
        spec = torch.zeros((8, 32, w), device="cuda", dtype=torch.complex128)
        spec[torch.arange(8, device="cuda"), slots] = local
        e = torch.fft.ifft(spec.reshape(8, n), dim=1)
        peak = (e.real ** 2 + e.imag ** 2).amax(dim=1, keepdim=True)
        e = (e * torch.sqrt(0.01 / peak)).sum(dim=0)
        out.append(e.to(torch.complex64 if case["precision"] == 0 else torch.complex128))
    return out


def _rcd_fields(case, seed):
    """Concentrations near the homogeneous state, the perturbation smoothed as diffusion to time 4 leaves it."""
    dims, m, g = _dims(case), case["components"], _rng(seed)
    off = 0.0 if m <= 1 else RCD_BETA + RCD_ALPHA if m == 2 else 2.0 * (RCD_BETA + RCD_ALPHA) + (m - 3) * RCD_BETA
    base = RCD_R / (RCD_A + off)
    smooth = torch.exp(-4.0 * RCD_D * _k2(dims, RCD_DX, True, torch.float32))
    axes = tuple(range(1, len(dims) + 1))
    out = torch.empty((m,) + dims, device="cuda", dtype=torch.float32)
    for i in range(0, m, 8):
        u = _uniform((min(8, m - i),) + dims, g)
        out[i:i + 8] = base * (1.0 + 0.1 * torch.fft.irfftn(torch.fft.rfftn(u, dim=axes) * smooth, s=dims, dim=axes))
    return out


def _assess_input(case, seed):
    """A spectrum that falls off as a mid-run field's does, with random phases."""
    dims, g = _dims(case), _rng(seed)
    cdt = torch.complex64 if case["precision"] == 0 else torch.complex128
    q = torch.randn(dims + (2,), generator=g, device="cuda", dtype=torch.float64 if case["precision"] else
                    torch.float32)
    k2 = _k2(dims, 1.0, False, q.dtype)
    q *= (1e3 * k2 * torch.exp(-3.0 * k2) + 1e-4).unsqueeze(-1)
    return torch.view_as_complex(q).to(cdt).contiguous()


def _predictor_input(case, seed):
    side, maps, g = case["side"], case["maps"], _rng(seed)
    x = torch.randn((maps, side, side, side, 2), generator=g, device="cuda").to(torch.bfloat16).contiguous()
    y = (torch.rand((maps, side, side, side), generator=g, device="cuda") < 0.35).to(torch.float32)
    params = spdba.predictor_init_params(int(seed) % (1 << 31))
    return x, y, params


# ------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": dict(case)}
    if kind in ("ch", "ensemble", "nls", "rcd"):
        # plans replay their steps as graphs on a stream of their own, as the benchmark's do
        s["stream"] = torch.cuda.Stream()
        st = s["stream"].cuda_stream
    if kind == "ch":
        dims = _dims(case)
        rdt = torch.float32 if case["precision"] == 0 else torch.float64
        s["x"] = [_ch_fields(dims, [0.1 if len(dims) == 3 else 0.0], _rng(seed))[0].to(rdt).contiguous()]
        s["plan"] = spdba.Plan(dims, (case["block"],) * len(dims), threshold=case["threshold"], reassess=10,
                               stream=st, precision=case["precision"], half_storage=case["half"],
                               mode=case["mode"], measure=case["measure"], dt=CH_DT, kappa=CH_KAPPA)
    elif kind == "ensemble":
        s["x"] = _ensemble_fields(case, seed)
        s["plan"] = spdba.Plan(None, (case["block"],) * 2, threshold=case["threshold"], reassess=10, stream=st,
                               batch_dims=[tuple(x.shape) for x in s["x"]], precision=0, dt=CH_DT, kappa=CH_KAPPA)
    elif kind == "nls":
        s["x"] = _nls_signals(case, seed)
        s["plan"] = spdba.Plan(None, (-64,), threshold=1e-6, reassess=10, stream=st,
                               batch_dims=[tuple(x.shape) for x in s["x"]], model=spdba.SPDBA_MODEL_NLS,
                               precision=case["precision"], mode=case["mode"], beta2=NLS_BETA2, gamma=NLS_GAMMA,
                               h=NLS_H)
    elif kind == "rcd":
        dims = _dims(case)
        s["x"] = [_rcd_fields(case, seed)]
        s["plan"] = spdba.Plan(dims, (case["block"],) * len(dims), threshold=case["threshold"], reassess=10,
                               stream=st, precision=case["precision"], model=spdba.SPDBA_MODEL_RCD,
                               components=case["components"], mode=case["mode"], dx=RCD_DX, dt=RCD_DT,
                               rcd_d_diag=RCD_D, rcd_d_cross=RCD_CROSS, rcd_alpha=RCD_ALPHA, rcd_beta=RCD_BETA)
    elif kind == "fft":
        dims = _dims(case)
        cdt = torch.complex64 if case["precision"] == 0 else torch.complex128
        s["x"] = torch.randn((case["batch"],) + dims, generator=_rng(seed), device="cuda", dtype=cdt)
        s["y"], s["z"] = torch.empty_like(s["x"]), torch.empty_like(s["x"])
        s["plan"] = spdba.FFTPlan(dims, batch=case["batch"], precision=case["precision"])
    elif kind == "assess":
        dims = _dims(case)
        s["x"] = _assess_input(case, seed)
        nb = tuple(d // case["block"] for d in dims)
        n = math.prod(nb)
        s["nb"] = nb
        s["maxsq"] = torch.zeros(nb, dtype=torch.float64, device="cuda")
        s["gmax"] = torch.zeros(2, dtype=torch.float64, device="cuda")
        s["states"] = torch.zeros(nb, dtype=torch.uint8, device="cuda")
        s["chi"] = torch.zeros(nb, dtype=torch.uint8, device="cuda")
        s["list"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        s["count"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        s["scratch"] = torch.zeros(spdba.classify_scratch_bytes(n), dtype=torch.uint8, device="cuda")
    elif kind == "predictor":
        s["x"], s["y"], params = _predictor_input(case, seed)
        s["prob"] = torch.empty(s["y"].shape, dtype=torch.float32, device="cuda")
        s["net"] = spdba.Predictor((case["side"],) * 3, max_batch=case["maps"], params=params)
    if "stream" in s:
        s["out"] = [torch.empty_like(x) for x in s["x"]]
        torch.cuda.synchronize()   # the inputs were made on another stream than the plan's
        if case.get("tuned"):
            s["plan"].set_field(s["x"][0])
            s["plan"].autotune(20)
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind in ("ch", "ensemble", "nls", "rcd"):
        plan = s["plan"]
        for r, x in enumerate(s["x"]):
            plan.set_field(x, run=r)
        plan.step(case["steps"])
        return [plan.get_field(out, run=r) for r, out in enumerate(s["out"])]
    if kind == "fft":
        s["plan"].exec(s["x"], s["y"], spdba.SPDBA_FORWARD)
        s["plan"].exec(s["y"], s["z"], spdba.SPDBA_INVERSE)
        return [s["y"], s["z"]]
    if kind == "assess":
        spdba.block_activity(s["x"], (case["block"],) * s["x"].dim(), s["maxsq"], None, s["gmax"],
                             precision=case["precision"])
        tau = case["threshold"] * torch.sqrt(s["gmax"][1:])
        spdba.classify(s["nb"], torch.sqrt(s["maxsq"]), tau, 1, 1, s["states"], s["chi"], s["list"], s["count"],
                       s["scratch"])
        return [s["maxsq"], s["gmax"], s["states"], s["chi"], s["list"], s["count"]]
    s["net"].forward(s["x"], s["prob"], nmaps=case["maps"])
    loss, grads = s["net"].gradients(s["x"], s["y"], nmaps=case["maps"])
    return [s["prob"], loss, grads]


# ------------------------------------------------------------------ the work of a pass
def work(case):
    """Bytes: the solver state read and written once a step (the half spectrum of a real field, the
    spectrum of a signal), the field in and out once; transforms: the array in and out, each way.
    Flops: 5 n log2 n a complex transform, half of it for real data, plus the pointwise terms."""
    kind = case["kind"]
    if kind in ("ch", "rcd"):
        dims = _dims(case)
        n, m = math.prod(dims), case.get("components", 1)
        es = 8 if case["precision"] == 0 else 16
        half = n // dims[-1] * (dims[-1] // 2 + 1)
        steps = case["steps"]
        flops = 2 * 2.5 * n * math.log2(n) + 20.0 * half + 4.0 * n
        if kind == "rcd":
            share = 1.0 if case["mode"] == 0 else 0.05
            flops += share * half * 8.0 * m
        return {"bytes": m * (2.0 * es * half * steps + es * n), "flops": m * flops * steps}
    if kind == "ensemble":
        n = [s * s for s, _ in _ensemble(case, 0)]
        half = [s * (s // 2 + 1) for s, _ in _ensemble(case, 0)]
        return {"bytes": 16.0 * sum(half) * case["steps"] + 8.0 * sum(n),
                "flops": case["steps"] * sum(2 * 2.5 * a * math.log2(a) + 14.0 * a for a in n)}
    if kind == "nls":
        n = _nls_lengths(case)
        es = 8 if case["precision"] == 0 else 16
        return {"bytes": 2.0 * es * sum(n) * (case["steps"] + 1),
                "flops": case["steps"] * sum(2 * 5.0 * a * math.log2(a) + 50.0 * a for a in n)}
    if kind == "fft":
        n, es = math.prod(_dims(case)), 8 if case["precision"] == 0 else 16
        return {"bytes": 4.0 * es * n * case["batch"], "flops": 2 * 5.0 * n * math.log2(n) * case["batch"]}
    if kind == "assess":
        n, es = math.prod(_dims(case)), 8 if case["precision"] == 0 else 16
        nb = n // case["block"] ** len(_dims(case))
        return {"bytes": float(es) * n + 14.0 * nb, "flops": 4.0 * n}
    v = case["side"] ** 3 * case["maps"]
    macs = 27 * (2 * 8 + 8 * 16 + 16 * 8)
    # inference, then forward and backward of the gradient (no input gradient for the first layer)
    return {"bytes": 2 * 8.0 * v + 4.0 * 8000, "flops": 2.0 * v * (4 * macs - 27 * 2 * 8)}


# ------------------------------------------------------------------ 64-bit values
def _block_max(a, block):
    shape = []
    for n, b in zip(a.shape, block):
        shape += [n // b, b]
    return a.reshape(shape).amax(dim=tuple(range(1, 2 * len(block), 2)))


def _block_sum(a, block):
    shape = []
    for n, b in zip(a.shape, block):
        shape += [n // b, b]
    return a.reshape(shape).sum(dim=tuple(range(1, 2 * len(block), 2)))


def _across(f, axis, d, half):
    """Values of the block across each block's face (axis, d): periodic, or on a half map's last axis the
    conjugate counterpart of a neighbour in the omitted half."""
    last = f.dim() - 1
    out = torch.roll(f, -d, dims=axis)
    if half and axis == last:
        other = tuple(range(last))
        out = out.clone()
        if d < 0:
            out[..., 0] = torch.flip(f[..., 0], dims=other)
        else:
            out[..., -1] = torch.flip(f[..., -2], dims=other)
    return out


def _classify(measure, tau, half, force_dc):
    """(states, sigma builder) of a block map."""
    active = measure >= tau
    if force_dc:
        active.view(-1)[0] = True
    near = torch.zeros_like(active)
    last = active.dim() - 1
    for axis in range(active.dim()):
        if half and axis == last:
            other = tuple(range(last))
            near[..., 1:] |= active[..., :-1]
            near[..., :-1] |= active[..., 1:]
            near[..., 0] |= torch.flip(active[..., 0], dims=other)
            near[..., -2] |= torch.flip(active[..., -1], dims=other)
        else:
            near |= torch.roll(active, 1, dims=axis) | torch.roll(active, -1, dims=axis)
    return active, near & ~active


def _expand(f, block):
    for a, b in enumerate(block):
        f = f.repeat_interleave(b, dim=a)
    return f


def _sigma(active, trans, block, half):
    """Per-mode weight: 1 on active blocks, 0 on frozen ones, the taper product on transition blocks."""
    frozen = ~(active | trans)
    w = _expand((active | trans).to(torch.float64), block)
    for a, b in enumerate(block):
        i = torch.arange(b, device=w.device, dtype=torch.float64)
        t = 0.5 * (1.0 - torch.cos(math.pi * i / (b - 1)))
        shape = [-1 if c == a else 1 for c in range(len(block))]
        reps = w.shape[a] // b
        for d, tt in ((-1, t), (1, torch.flip(t, dims=(0,)))):
            face = _expand(_across(frozen, a, d, half) & trans, block)
            w = torch.where(face, w * tt.repeat(reps).reshape(shape), w)
    return w


def _states_sigma(q, sq, case, block, half, exclude_dc, force_dc):
    """Per-mode weight from a spectrum's squared amplitudes sq."""
    full = sq
    if half:
        pad = -sq.shape[-1] % block[-1]
        full = torch.nn.functional.pad(sq, (0, pad))
    m = torch.sqrt(_block_sum(full, block) if case.get("measure") else _block_max(full, block))
    flat = sq.reshape(-1)
    top = flat[1:].max() if exclude_dc else flat.max()
    active, trans = _classify(m, case["threshold"] * torch.sqrt(top), half, force_dc)
    w = _sigma(active, trans, block, half)
    return w[..., : sq.shape[-1]]


def _blend(old, new, w):
    return torch.where(w == 1.0, new, old + w * (new - old))


def _exact_ch(c0, case, block):
    dims, half = tuple(c0.shape), bool(case.get("half", 0))
    k2 = _k2(dims, 1.0, half, torch.float64)
    den = 1.0 + CH_DT * CH_KAPPA * k2 * k2
    fwd = torch.fft.rfftn if half else torch.fft.fftn

    def real(h):
        if not half:
            return torch.fft.ifftn(h).real
        # the last axis alone as a complex-to-real transform: it keeps the Hermitian part of the
        # kx = 0 and N/2 planes, which need not be symmetric once some of their blocks are frozen
        t = torch.fft.ifftn(h, dim=tuple(range(len(dims) - 1)))
        return torch.fft.irfft(t, n=dims[-1], dim=-1)

    q = fwd(c0.double())
    w = None
    for n in range(case["steps"]):
        if case.get("mode", 1) and n % 10 == 0:
            w = _states_sigma(q, q.real ** 2 + q.imag ** 2, case, block, half, True, True)
        c = real(q)
        new = (q - CH_DT * k2 * fwd(c * c * c - c)) / den
        q = new if w is None else _blend(q, new, w)
    return real(q)


def _exact_nls(e0, case):
    n = e0.numel()
    om = 2.0 * math.pi * torch.fft.fftfreq(n, device="cuda", dtype=torch.float64)
    hf = torch.exp(1j * NLS_BETA2 * om * om * NLS_H / 4.0)
    block, w = (n // 64,), None
    q = torch.fft.fft(e0.to(torch.complex128))
    for s in range(case["steps"]):
        if case["mode"] and s % 10 == 0:
            w = _states_sigma(q, q.real ** 2 + q.imag ** 2, {"threshold": 1e-6}, block, False, False, False)
        q = q * hf if w is None else _blend(q, q * hf, w)
        e = torch.fft.ifft(q)
        e = e * torch.exp(1j * NLS_GAMMA * NLS_H * (e.real ** 2 + e.imag ** 2))
        q = torch.fft.fft(e)
        q = q * hf if w is None else _blend(q, q * hf, w)
    return torch.fft.ifft(q)


def _exact_rcd(u0, case):
    m, dims = u0.shape[0], tuple(u0.shape[1:])
    axes = tuple(range(1, len(dims) + 1))
    k2 = _k2(dims, RCD_DX, False, torch.float64)
    d = torch.zeros((m, m), dtype=torch.float64)
    for i in range(m):
        d[i, i] = RCD_D + 2.0 * RCD_CROSS
        if m > 1:
            d[i, (i + 1) % m] = d[i, (i - 1) % m] = -RCD_CROSS
    lam, v = torch.linalg.eigh(d)
    lam, v = lam.cuda(), v.cuda()
    den = 1.0 + RCD_DT * k2 * lam.reshape((m,) + (1,) * len(dims))
    vc = v.to(torch.complex128)
    q, w = torch.fft.fftn(u0.double(), dim=axes), None
    for n in range(case["steps"]):
        if case["mode"] and n % 10 == 0:
            sq = torch.zeros(dims, dtype=torch.float64, device="cuda")
            for i in range(m):
                sq += q[i].real ** 2 + q[i].imag ** 2
            w = _states_sigma(None, sq / m, {"threshold": case["threshold"]}, (case["block"],) * len(dims), False,
                              True, True)
        u = torch.fft.ifftn(q, dim=axes).real
        s = u.sum(dim=0, keepdim=True)
        if m >= 3:
            inter = RCD_BETA * (s - u) + RCD_ALPHA * (torch.roll(u, 1, 0) + torch.roll(u, -1, 0))
        else:
            inter = (RCD_BETA + RCD_ALPHA) * (s - u)
        b = torch.fft.fftn(u * (RCD_R - RCD_A * u - inter), dim=axes)
        del u, s, inter
        b.mul_(RCD_DT).add_(q)
        y = (vc.T @ b.reshape(m, -1)).reshape(b.shape)
        y /= den
        b = (vc @ y.reshape(m, -1)).reshape(b.shape)
        del y
        q = b if w is None else _blend(q, b, w)
    return torch.fft.ifftn(q, dim=axes).real


def _exact_predictor(x, y, params):
    p = torch.from_numpy(params).double().cuda().requires_grad_(True)
    h, o = x.double().permute(0, 4, 1, 2, 3), 0
    for ci, co in ((2, 8), (8, 16), (16, 8)):
        wt = p[o:o + co * 27 * ci].reshape(co, 3, 3, 3, ci).permute(0, 4, 1, 2, 3)
        o += co * 27 * ci
        h = torch.nn.functional.pad(h, (1, 1, 1, 1, 1, 1), mode="circular")
        h = torch.relu(torch.nn.functional.conv3d(h, wt, p[o:o + co]))
        o += co
    z = (h * p[o:o + 8].reshape(1, 8, 1, 1, 1)).sum(dim=1) + p[o + 8]
    loss = torch.nn.functional.binary_cross_entropy_with_logits(z, y.double())
    loss.backward()
    return [torch.sigmoid(z).detach(), loss.detach(), p.grad]


def exact(case, seed):
    kind = case["kind"]
    if kind == "ch":
        dims = _dims(case)
        x = _ch_fields(dims, [0.1 if len(dims) == 3 else 0.0], _rng(seed))[0]
        return [_exact_ch(x, case, (case["block"],) * len(dims))]
    if kind == "ensemble":
        return [_exact_ch(x, case, (case["block"],) * 2) for x in _ensemble_fields(case, seed)]
    if kind == "nls":
        return [_exact_nls(x, case) for x in _nls_signals(case, seed)]
    if kind == "rcd":
        return [_exact_rcd(_rcd_fields(case, seed), case)]
    if kind == "fft":
        cdt = torch.complex64 if case["precision"] == 0 else torch.complex128
        x = torch.randn((case["batch"],) + _dims(case), generator=_rng(seed), device="cuda", dtype=cdt)
        x = x.to(torch.complex128)
        return [torch.fft.fftn(x, dim=tuple(range(1, x.dim()))), x]
    if kind == "assess":
        q = _assess_input(case, seed).to(torch.complex128)
        sq = q.real * q.real + q.imag * q.imag
        top = torch.stack([sq.max(), sq.reshape(-1)[1:].max()])
        return [_block_max(sq, (case["block"],) * q.dim()), top, None, None, None, None]
    x, y, params = _predictor_input(case, seed)
    return _exact_predictor(x, y, params)
