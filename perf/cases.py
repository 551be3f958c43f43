"""The work that users of this framework have it do, as cases to be timed.

Every case is one pass through a public entry point: ``Plan.run`` (search of a
recorded filterbank), ``Plan.run_window`` (the streaming server's step),
``BatchRunner.run`` (many beams), ``autograd.dedisperse`` with its backward
(fitting), ``Plan.run_host`` (host buffers end to end) and ``transpose`` (the
time-major front end).  Bands, sampling times and DM plans are those of this
repository's workloads, tests and benchmark.

A case names its band (``f_high``, ``band`` in MHz, ``n_chan`` equal channels,
channel 0 highest), ``t_samp`` in seconds, ``n_samp`` samples and its DM plan:
``n_dm`` trials from 0 in steps of ``dm_step`` at time bin ``bin``, or
``plan`` = "adaptive" (``dm_ranges`` up to ``dm_max``) or "stream" (the
four-range plan with bins 1 to 8).
"""
import math

import numpy as np
import torch

import paper_2311_05341_gb300 as dd
from paper_2311_05341_gb300 import autograd, batch, stream

C_DM = 4148.808  # MHz^2 s per unit DM
STREAM_RANGES = [(0.0, 150.0, 0.1, 1), (150.0, 300.0, 0.2, 2), (300.0, 1000.0, 0.5, 4),
                 (1000.0, 2000.0, 1.0, 8)]


def _case(kind, dtype, n_chan, n_samp, f_high, band, t_samp, **more):
    return dict(kind=kind, dtype=dtype, n_chan=n_chan, n_samp=n_samp, f_high=f_high, band=band,
                t_samp=t_samp, **more)


def listed():
    named = [
        # The smallest call: one short observation of 64 channels, 128 trials
        # (steps of 8 samples in the lowest channel); launch latency counts.
        ("tiny_u8", _case("run", "u8", 64, 8192, 1500.0, 300.0, 64e-6, n_dm=128, dm_step=0.5, bin=1)),
        # An ordinary beam of an L-band survey: 1024 channels, 8 s of 8-bit data.
        ("beam_u8", _case("run", "u8", 1024, 131072, 1520.0, 310.0, 64e-6, n_dm=2048, dm_step=0.1, bin=1)),
        # The largest: 8192 channels, 17 s, 4096 trials (the 8-bit headline).
        ("paper_u8", _case("run", "u8", 8192, 262144, 1670.0, 320.0, 64e-6, n_dm=4096, dm_step=0.1, bin=1)),
        # 16-bit data of a wide-band backend, 3072 trials.
        ("beam_u16", _case("run", "u16", 4096, 65536, 1670.0, 320.0, 54.6e-6, n_dm=3072, dm_step=0.2, bin=1)),
        # 4-bit recordings, two samples a byte.
        ("search_u4", _case("run", "u4", 8192, 131072, 1670.0, 320.0, 64e-6, n_dm=2048, dm_step=0.1, bin=1)),
        # A search over a plan made from a smearing tolerance: several ranges,
        # binned as DM grows, with ragged channel and sample counts.
        ("adaptive_u8", _case("run", "u8", 1001, 200003, 1500.0, 300.0, 64e-6, plan="adaptive", dm_max=1000.0)),
        # A low-frequency float beam: many samples of delay between trials.
        ("lowfreq_f32", _case("run", "f32", 336, 32768, 400.0, 100.0, 327.68e-6, n_dm=1024, dm_step=0.2, bin=1)),
        # One gradient step through the transform: forward and adjoint.
        ("train_f32", _case("train", "f32", 1024, 65536, 1500.0, 300.0, 128e-6, n_dm=1024, dm_step=0.2, bin=1)),
        # One chunk of one beam in the streaming server: a window of overlap
        # and chunk on the packed tiles, the chunk's new outputs of 4 ranges.
        ("stream_step_u8", _case("window", "u8", 4096, 65536, 1670.0, 320.0, 64e-6, plan="stream")),
        # Beams of three telescopes in one batch, captured in a CUDA graph.
        ("batch_mixed", _case("batch", "mixed", 1024, 65536, 1520.0, 310.0, 64e-6, n_dm=1024, dm_step=0.1, bin=1,
                              n_u8=6, n_u16=2, n_f32=2)),
        # From pinned host memory to host memory, copies included.
        ("host_u8", _case("host", "u8", 1024, 131072, 1520.0, 310.0, 64e-6, n_dm=512, dm_step=0.4, bin=1)),
        # The front end: time-major samples of a recorder to channel-major rows.
        ("transpose_u8", _case("transpose", "u8", 4096, 131072, 1670.0, 320.0, 64e-6)),
    ]
    return [dict(case, name=name) for name, case in named]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same paths: sizes over their whole range, odd ones
    among them, and delays from a fraction of a sample to a dozen per trial."""
    kind, dtype = rng.choice([("run", "u8"), ("run", "u8"), ("run", "u8"), ("run", "u16"), ("run", "u4"),
                              ("run", "f32"), ("train", "f32"), ("window", "u8"), ("batch", "mixed"),
                              ("host", "u8"), ("transpose", rng.choice(["u8", "u16", "f32"]))])
    f_high = rng.choice([400.0, 1500.0, 1520.0, 1670.0])
    band = rng.uniform(0.18, 0.25) * f_high
    t_samp = rng.choice([54.6e-6, 64e-6, 128e-6, 327.68e-6])
    n_samp = _log_int(rng, 4096, 262144 if kind == "run" else 65536)
    if kind == "transpose":
        return _case(kind, dtype, _log_int(rng, 60, 8192), n_samp, f_high, band, t_samp)
    n_chan = _log_int(rng, 48, {"run": 8192, "window": 2048, "batch": 512}.get(kind, 1024))
    if kind == "window":
        return _case(kind, dtype, n_chan, 32768, 1670.0, 320.0, 64e-6, plan="stream")
    if kind == "run" and dtype == "u8" and rng.random() < 0.3:
        return _case(kind, dtype, min(n_chan, 2048), max(n_samp, 65536), 1500.0, 300.0, 64e-6, plan="adaptive",
                     dm_max=rng.uniform(100.0, 800.0))
    steep = rng.random() < 0.15
    slope = rng.uniform(4.0, 12.0) if steep else math.exp(rng.uniform(math.log(0.2), math.log(2.5)))
    bin_ = rng.choice([1, 1, 1, 2, 4]) if dtype in ("u8", "u4") and kind == "run" else 1
    most = max(33, min(4096, int(0.6 * n_samp / bin_ / slope)))
    n_dm = _log_int(rng, 32, most)
    k_low = C_DM * (1.0 / (f_high - band) ** 2 - 1.0 / f_high ** 2)
    case = _case(kind, dtype, n_chan, n_samp, f_high, band, t_samp, n_dm=n_dm,
                 dm_step=slope * bin_ * t_samp / k_low, bin=bin_)
    if kind == "batch":
        case.update(n_u8=rng.randint(1, 5), n_u16=rng.randint(0, 2), n_f32=rng.randint(0, 2))
    return case


# -- plans, in plain numpy ---------------------------------------------------
def _freqs(case):
    df = case["band"] / case["n_chan"]
    return case["f_high"] - (np.arange(case["n_chan"]) + 0.5) * df


def _ranges(case):
    if case.get("plan") == "stream":
        return list(STREAM_RANGES)
    if case.get("plan") == "adaptive":
        return dd.dm_ranges(_freqs(case), case["t_samp"], case["dm_max"], tol=1.25, max_bin=8)
    return [(0.0, case["n_dm"] * case["dm_step"], case["dm_step"], case["bin"])]


def _shifts(case, rng_):
    lo, hi, step, b = rng_
    f = _freqs(case)
    k = C_DM * (1.0 / (f * f) - 1.0 / (case["f_high"] * case["f_high"]))
    n_dm = int(math.floor((hi - lo) / step + 0.5))
    dm = lo + np.arange(n_dm, dtype=np.float64) * step
    return np.floor(dm[:, None] * k[None, :] / (b * case["t_samp"]) + 0.5).astype(np.int64)


def _smax(case, rng_):
    lo, hi, step, b = rng_
    last = dict(case, n_chan=case["n_chan"])
    f = _freqs(last)[-1]
    k = C_DM * (1.0 / (f * f) - 1.0 / (case["f_high"] * case["f_high"]))
    n_dm = int(math.floor((hi - lo) / step + 0.5))
    return n_dm, int(math.floor((lo + (n_dm - 1) * step) * k / (b * case["t_samp"]) + 0.5))


def _overlap(case):
    """Raw samples a streamed window keeps so that each chunk gives chunk / bin outputs."""
    need = max(r[3] * _smax(case, r)[1] for r in _ranges(case))
    return (need + 15) // 16 * 16


def _length(case):
    return case["n_samp"] + _overlap(case) if case["kind"] == "window" else case["n_samp"]


def _outputs(case):
    """(n_dm, n_out) of every range."""
    out = []
    for r in _ranges(case):
        n_dm, s = _smax(case, r)
        out.append((n_dm, case["n_samp"] // r[3] if case["kind"] == "window" else case["n_samp"] // r[3] - s))
    return out


def _beams(case):
    """The batch's beams, as cases: 8-bit L-band, 16-bit wide-band, float low-frequency."""
    one = {"n_dm": case["n_dm"], "bin": 1}
    n, c = case["n_samp"], case["n_chan"]
    beams = [dict(case, kind="run", dtype="u8")] * case["n_u8"]
    beams += [_case("run", "u16", 2 * c, n // 2, 1670.0, 320.0, 54.6e-6, dm_step=0.2, **one)] * case["n_u16"]
    beams += [_case("run", "f32", c // 3, n // 2, 400.0, 100.0, 327.68e-6, dm_step=0.1, **one)] * case["n_f32"]
    fit = []
    for b in beams:  # no more trials than the beam's length allows
        s = _smax(b, _ranges(b)[0])[1]
        most = int(b["n_dm"] * min(1.0, 0.6 * b["n_samp"] / max(s, 1)))
        fit.append(dict(b, n_dm=max(most, 1)))
    return fit


# -- inputs --------------------------------------------------------------------
def _noise(case, seed, device="cuda"):
    """Receiver noise as the digitiser leaves it, rows padded to 16 bytes: 8-bit
    N(128, 16), 16-bit N(32768, 256), 4-bit N(8, 2) packed two a byte, N(0, 1)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    dtype, c, n = case["dtype"], case["n_chan"], _length(case)
    per = {"u8": 16, "u16": 8, "f32": 4, "u4": 32}[dtype]
    stride = (n + per - 1) // per * per
    mean, sd, top = {"u8": (128.0, 16.0, 255), "u16": (32768.0, 256.0, 65535), "u4": (8.0, 2.0, 15),
                     "f32": (0.0, 1.0, 0)}[dtype]
    tdt = {"u8": torch.uint8, "u16": torch.uint16, "u4": torch.uint8, "f32": torch.float32}[dtype]
    x = torch.zeros((c, stride // 2 if dtype == "u4" else stride), dtype=tdt, device="cuda")
    rows = max(1, (1 << 27) // stride)
    for c0 in range(0, c, rows):
        c1 = min(c, c0 + rows)
        v = torch.randn((c1 - c0, stride), generator=g, device="cuda")
        if dtype == "f32":
            x[c0:c1] = v
            x[c0:c1, n:] = 0
            continue
        v = v.mul_(sd).add_(mean).round_().clamp_(0, top)
        v[:, n:] = 0
        if dtype == "u4":
            w = v.to(torch.uint8)
            x[c0:c1] = w[:, 0::2] | (w[:, 1::2] << 4)
        elif dtype == "u16":
            x[c0:c1] = v.to(torch.int32).to(torch.uint16)
        else:
            x[c0:c1] = v.to(torch.uint8)
    return x


def _plan(case):
    return dd.Plan(_freqs(case), case["f_high"], case["t_samp"], _ranges(case), case["dtype"])


def _cotangent(case, seed):
    n_dm, n_out = _outputs(case)[0]
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    return torch.randn((n_dm, n_out), generator=g, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        beams = _beams(case)
        runner = batch.BatchRunner(
            [batch.BeamSpec(_freqs(b), b["f_high"], b["t_samp"], _ranges(b), b["dtype"], b["n_samp"]) for b in beams],
            autotune=False)
        for i, b in enumerate(beams):
            runner.inputs[i].copy_(_noise(b, seed * 1000 + i))
        return {"kind": kind, "runner": runner}
    if kind == "transpose":
        g = torch.Generator(device="cuda").manual_seed(seed)
        per = {"u8": 16, "u16": 8, "f32": 4}[case["dtype"]]
        shape = (case["n_samp"], (case["n_chan"] + per - 1) // per * per)
        if case["dtype"] == "f32":
            x = torch.randn(shape, generator=g, device="cuda")
        else:
            top = 256 if case["dtype"] == "u8" else 65536
            x = torch.randint(0, top, shape, generator=g, device="cuda", dtype=torch.int32)
            x = x.to(torch.uint8 if case["dtype"] == "u8" else torch.uint16)
        return {"kind": kind, "x": x, "n_chan": case["n_chan"]}
    plan = _plan(case)
    x = _noise(case, seed)
    st = {"kind": kind, "plan": plan, "x": x, "n": _length(case)}
    if kind == "train":
        st["x"] = x[:, :case["n_samp"]].requires_grad_(True)
        st["w"] = _cotangent(case, seed)
    elif kind == "window":  # as the server sets a beam up
        for r in range(len(plan.ranges)):
            try:
                plan.set_tile(r, "packed")
            except dd.DDError:
                pass
        assert stream.overlap_for(plan, plan.ranges) == _overlap(case)
        st["keep"] = [n for _, n in _outputs(case)]
        need = plan.input_scratch_bytes(st["n"])
        st["scratch"] = torch.empty(need, dtype=torch.uint8, device="cuda") if need else None
        st["out"] = torch.empty(sum(a * b for a, b in _outputs(case)), dtype=plan.out_dtype(), device="cuda")
    elif kind == "host":
        st["x"] = x.cpu().pin_memory()
        st["d_in"] = torch.empty_like(x)
        st["d_out"] = plan.empty_output(st["n"])
        st["out"] = torch.zeros(st["d_out"].shape, dtype=st["d_out"].dtype).pin_memory()
    return st


def run(st):
    kind = st["kind"]
    if kind == "run":
        return st["plan"].run(st["x"], n_samp=st["n"])
    if kind == "train":
        y = autograd.dedisperse(st["x"], st["plan"])
        (grad,) = torch.autograd.grad(y[0], st["x"], st["w"])
        return {"y": y[0].detach(), "grad": grad}
    if kind == "window":
        return st["plan"].run_window(st["x"], st["keep"], out=st["out"], n_samp=st["n"], scratch=st["scratch"])
    if kind == "batch":
        st["runner"].run()
        return [p for i in range(len(st["runner"].plans)) for p in st["runner"].planes(i)]
    if kind == "host":
        st["plan"].run_host(st["x"], st["out"], st["d_in"], st["d_out"], n_samp=st["n"])
        torch.cuda.current_stream().synchronize()  # the caller reads its host buffer next
        return st["plan"].split(st["out"], st["n"])
    return dd.transpose(st["x"], st["n_chan"])


# -- what a pass cannot do without ---------------------------------------------
def work(case):
    """Input and output bytes, each once, and one add per (trial, output sample,
    channel): the direct sum's count, by which dedispersion rates are quoted
    (sums shared between trials take fewer)."""
    if case["kind"] == "batch":
        each = [work(b) for b in _beams(case)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    bits = {"u8": 8, "u16": 16, "u4": 4, "f32": 32}[case["dtype"]]
    in_bytes = case["n_chan"] * _length(case) * bits // 8
    if case["kind"] == "transpose":
        return {"bytes": 2 * in_bytes, "flops": 0}
    outs = sum(a * b for a, b in _outputs(case))
    adds, size = outs * case["n_chan"], in_bytes + outs * 4
    return {"bytes": 2 * size, "flops": 2 * adds} if case["kind"] == "train" else {"bytes": size, "flops": adds}


# -- the same outputs in 64 bits -----------------------------------------------
def _rows64(case, x):
    """Samples of every channel row, 64-bit, decimation not yet applied."""
    if case["dtype"] == "u4":
        return lambda c: torch.stack((x[c] & 15, x[c] >> 4), 1).flatten()[:_length(case)].to(torch.int64)
    if case["dtype"] == "u16":
        return lambda c: x[c].view(torch.int16)[:_length(case)].to(torch.int64) & 65535
    wide = torch.float64 if case["dtype"] == "f32" else torch.int64
    return lambda c: x[c, :_length(case)].to(wide)


def _forward64(case, x):
    planes, row = [], _rows64(case, x)
    for r, (n_dm, n_out) in zip(_ranges(case), _outputs(case)):
        b, sh = r[3], torch.from_numpy(_shifts(case, r)).cuda()
        y = None
        for c in range(case["n_chan"]):
            v = row(c)
            v = v[:v.numel() // b * b].view(-1, b).sum(1)
            part = v.unfold(0, n_out, 1).index_select(0, sh[:, c])
            y = part if y is None else y.add_(part)
        planes.append(y)
    return planes


def _adjoint64(case, w):
    (r,), n = _ranges(case), case["n_samp"]
    sh = torch.from_numpy(_shifts(case, r)).cuda()
    n_dm, n_out = w.shape
    pad = n - n_out
    rows = torch.zeros((n_dm, pad + n), dtype=torch.float64, device="cuda")
    rows[:, pad:pad + n_out] = w
    flat, grad = rows.view(-1), torch.empty((case["n_chan"], n), dtype=torch.float64, device="cuda")
    windows = flat.unfold(0, n, 1)
    base = torch.arange(n_dm, device="cuda") * (pad + n) + pad
    for c in range(case["n_chan"]):
        grad[c] = windows.index_select(0, base - sh[:, c]).sum(0)
    return grad


def exact(case, seed):
    kind = case["kind"]
    if kind == "transpose":
        return prepare(case, seed)["x"][:, :case["n_chan"]].t()
    if kind == "batch":
        beams = _beams(case)
        if sum(_cost64(b) for b in beams) > 4e12:
            return None
        return [p for i, b in enumerate(beams) for p in _forward64(b, _noise(b, seed * 1000 + i))]
    if _cost64(case) > 4e12 or max(a * b for a, b in _outputs(case)) > 4e9:
        return None
    x = _noise(case, seed)
    if kind == "train":
        return {"y": _forward64(case, x)[0], "grad": _adjoint64(case, _cotangent(case, seed))}
    return _forward64(case, x)


def _cost64(case):
    return sum(a * b for a, b in _outputs(case)) * case["n_chan"] * (2 if case["kind"] == "train" else 1)
