"""The workloads this library's speed is judged by: what a search program has it do, through its
public entry points, from one small beam to the 4096-channel low-frequency beam.

A case is a dict of plain values; its "op" names the entry point:
  search      Plan.execute on device buffers (uint8, float16 or float32 filterbank rows)
  batch       Batch.execute: uneven uint8 beams in one launch
  host        Plan.execute_host: pinned host rows in, host plane out
  detect      detect: the boxcar search of a (DM,t) plane
  unpack      unpack: sigproc spectra to channel rows
  frontend    frontend: dual-polarisation voltages to the uint8 filterbank
  channelise  channelise: subband voltages to finer channels
"""
import math
import random

import numpy as np
import torch

import paper_1111_6399_gb300 as dd

#: Bands: highest channel centre (MHz), bandwidth (MHz), sampling time (s).
BANDS = {"lband": (1500.0, 300.0, 64e-6), "narrow": (1500.0, 64.0, 64e-6),
         "low": (150.0, 30.0, 327.68e-6)}
DTYPES = {"u8": torch.uint8, "f16": torch.float16, "f32": torch.float32}
#: Adds of the largest listed search; drawn cases stay below it.
MAX_ADDS = 4096 * 2000 * 262144


def listed():
    return [
        # One small beam: launches and latency count (a monitoring tool, a unit of a larger scan).
        dict(name="search-small-u8", op="search", band="narrow", dtype="u8", nchan=64, ndm=64,
             dm_step=1.0, nsamp=8192),
        # A ragged mid-size beam: odd channel count, odd DM count, odd length, DMs out of order.
        dict(name="search-ragged-u8", op="search", band="lband", dtype="u8", nchan=333, ndm=301,
             dm_step=1.7, nsamp=50021, shuffled=True),
        # The ordinary real-time search: an L-band beam, 8.4 s of data.
        dict(name="search-lband-u8", op="search", band="lband", dtype="u8", nchan=1024, ndm=1024,
             dm_step=1.0, nsamp=131072),
        # The largest search: the low-frequency beam of 4096 channels and 2000 DMs, 86 s of data.
        dict(name="search-lowfreq-u8", op="search", band="low", dtype="u8", nchan=4096, ndm=2000,
             dm_step=0.05, nsamp=262144),
        # The low-frequency beam kept in half precision, a 21 s block.
        dict(name="search-lowfreq-f16", op="search", band="low", dtype="f16", nchan=4096,
             ndm=2000, dm_step=0.05, nsamp=65536),
        # An L-band block as calibrated single-precision power.
        dict(name="search-lband-f32", op="search", band="lband", dtype="f32", nchan=1024,
             ndm=1024, dm_step=1.0, nsamp=65536),
        # Many beams of a multi-beam receiver, each with its own channels, DMs and length.
        dict(name="batch-uneven-u8", op="batch", beams=16, mix=4),
        # End to end from host memory: copies in, search, plane copied back.
        dict(name="host-lband-u8", op="host", band="lband", dtype="u8", nchan=1024, ndm=1024,
             dm_step=1.0, nsamp=131072),
        # Searching the L-band plane for pulses of widths 1..256.
        dict(name="detect-lband", op="detect", ndm=1024, nsamp=131072, nlevels=9, integer=True),
        # The corner turn of an 8-bit L-band file block into channel rows.
        dict(name="unpack-lband-8bit", op="unpack", nbits=8, nchan=1024, nsamp=147628),
        # Voltages of a quarter of the L-band channels to the filterbank: three clipping passes.
        dict(name="frontend-lband", op="frontend", nchan=256, nraw=147628 * 16, nint=16, niter=3,
             k=4.0),
        # Station subbands split into 16 channels each, int8 codes for the front end.
        dict(name="channelise-16ch", op="channelise", nsub=64, m=16, taps=8, nspec=295256,
             kind="ci8", scale=0.25),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["search"] * 6 + ["batch", "host", "detect", "detect", "unpack", "frontend",
                                      "channelise", "channelise"])
    if op in ("search", "host"):
        c = dict(op=op, band=rng.choice(list(BANDS)), dtype=rng.choice(["u8", "u8", "f16", "f32"]))
        low = c["band"] == "low"
        # Low-frequency beams have many narrow channels.
        c["nchan"] = _log(rng, 1024, 4096) if low else _log(rng, 64, 4096)
        c["ndm"] = _log(rng, 32, 2000)
        c["dm_step"] = round(rng.uniform(0.02, 0.06) if low else rng.uniform(0.1, 2.0), 4)
        c["nsamp"] = _log(rng, 4096, 131072)
        if rng.random() < 0.5:  # round sizes are as common as odd ones
            c["nchan"] = max(64, c["nchan"] // 64 * 64)
            c["nsamp"] = max(4096, c["nsamp"] // 4096 * 4096)
        limit = MAX_ADDS // (8 if op == "host" or c["dtype"] != "u8" else 4)
        while c["nchan"] * c["ndm"] * c["nsamp"] > limit:
            c["nsamp"] = max(4096, c["nsamp"] // 2)
            c["ndm"] = max(32, c["ndm"] * 3 // 4)
        return c
    if op == "batch":
        return dict(op=op, beams=rng.randrange(2, 17), mix=rng.randrange(1 << 30))
    if op == "detect":
        return dict(op=op, ndm=_log(rng, 16, 1500), nsamp=_log(rng, 1000, 80000),
                    nlevels=rng.choice([4, 7, 9, 9]), integer=rng.random() < 0.75)
    if op == "unpack":
        nchan = rng.choice([128, 256, 512, 1024, 2048, 8 * _log(rng, 8, 300)])
        return dict(op=op, nbits=rng.choice([8, 8, 4, 2, 1]), nchan=nchan,
                    nsamp=_log(rng, 4096, 1 << 26) // nchan + 1000)
    if op == "frontend":
        nint = rng.choice([1, 2, 4, 8, 16, 16, 32, 64])
        nraw = min(_log(rng, 1 << 15, 1 << 20) + nint, nint << 19)  # at most 2^19 outputs a row
        return dict(op=op, nchan=_log(rng, 16, 512), nraw=nraw, nint=nint,
                    niter=rng.choice([1, 3, 3, 5]), k=4.0)
    m = rng.choice([16, 16, 32, 64, 128, 256])
    kind = rng.choice(["ci8", "ci8", "cf32"])
    return dict(op=op, nsub=_log(rng, 1, 64), m=m, taps=rng.choice([4, 8, 8, 12, 16]),
                nspec=_log(rng, 1 << 16, 1 << 22) // m, kind=kind,
                scale=round(1.0 / math.sqrt(m), 6))


# --- shapes ------------------------------------------------------------------


def _dms(case):
    d = (np.arange(case["ndm"], dtype=np.float64) * case["dm_step"]).astype(np.float32)
    if case.get("shuffled"):
        order = list(range(len(d)))
        random.Random(case["ndm"]).shuffle(order)
        d = d[order]
    return d


def _beam(case):
    """nchan, fch1, foff, tsamp, DM list of a beam."""
    f_top, width, tsamp = BANDS[case["band"]]
    return case["nchan"], f_top, -width / case["nchan"], tsamp, _dms(case)


def _table(nchan, fch1, foff, tsamp):
    """The delay of each channel in samples at DM 1: FP64, rounded once."""
    f = fch1 + np.arange(nchan, dtype=np.float64) * foff
    top = f.max()
    return (4148.808 * (1.0 / (f * f) - 1.0 / (top * top)) / tsamp).astype(np.float32)


def _shifts(case):
    """s(c,d) as int64 [nchan][ndm]."""
    nchan, fch1, foff, tsamp, dms = _beam(case)
    return (dms[None, :] * _table(nchan, fch1, foff, tsamp)[:, None]).astype(np.int64)


def _beams_of(case):
    """The uneven beams of a batch: channels, DMs and lengths as in the 64-beam workload, at a
    quarter of its lengths."""
    r = random.Random(case["mix"])
    out = []
    for _ in range(case["beams"]):
        out.append(dict(op="search", dtype="u8", band=r.choice(["lband", "narrow"]),
                        nchan=r.choice([256, 512, 1024, 4096]), ndm=_log(r, 128, 2048),
                        dm_step=1.0, nsamp=_log(r, 1 << 14, 1 << 16)))
    out[0].update(nchan=1024, ndm=1024)
    budget = MAX_ADDS // 2
    for b in out:  # a batch stays below half of the largest search
        while b["nchan"] * b["ndm"] * b["nsamp"] > budget // len(out):
            b["ndm"] = b["ndm"] * 3 // 4
    return out


def _maxshift(case):
    nchan, fch1, foff, tsamp, dms = _beam(case)
    return int((dms.max() * _table(nchan, fch1, foff, tsamp)).astype(np.int64).max())


def _round(n, k):
    return (n + k - 1) // k * k


# --- inputs ------------------------------------------------------------------


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _filterbank(case, seed):
    """Noise of mean 128 and spread 16 with a few dispersed pulses, as the receiver delivers it."""
    g = _gen(seed)
    nin = case["nsamp"] + _maxshift(case)
    dtype = DTYPES[case["dtype"]]
    x = torch.empty((case["nchan"], _round(nin, 16)), dtype=dtype, device="cuda")
    rows = max(1, (1 << 27) // x.shape[1])
    for c in range(0, x.shape[0], rows):
        v = torch.randn((min(rows, x.shape[0] - c), x.shape[1]), generator=g, device="cuda")
        v = v.mul_(16).add_(128).clamp_(0, 255)
        x[c:c + rows] = v.round_() if case["dtype"] == "u8" else v
    nchan, fch1, foff, tsamp, dms = _beam(case)
    rng = random.Random(seed)
    rows = torch.arange(nchan, device="cuda")
    for _ in range(4):
        s = dms[rng.randrange(len(dms))] * _table(nchan, fch1, foff, tsamp)
        t0 = torch.from_numpy(s.astype(np.int64)).cuda() + rng.randrange(case["nsamp"] - 16)
        for k in range(rng.randrange(1, 17)):
            x[rows, t0 + k] = (x[rows, t0 + k].float() + 40).clamp(0, 255).to(dtype)
    return x, nin


def _voltages(nrow, nraw, seed, rfi):
    """Receiver noise of four levels as int8 (Xre, Xim, Yre, Yim), with tones and impulses where
    they are to be excised."""
    g = _gen(seed)
    rng = random.Random(seed)
    v = torch.empty((nrow, nraw, 4), dtype=torch.int8, device="cuda")
    step = 1 << 24
    for r in range(nrow):
        sigma = rng.choice((8.0, 12.0, 18.0, 27.0))
        for a in range(0, nraw, step):
            n = min(step, nraw - a)
            z = torch.randn((n, 4), generator=g, device="cuda")
            v[r, a:a + n] = z.mul_(sigma).round_().clamp_(-128, 127).to(torch.int8)
    if rfi:
        tone = torch.tensor([100, 0, 100, 0], dtype=torch.int8, device="cuda")
        for _ in range(max(1, nrow // 64)):
            n = max(1, nraw // rng.randrange(25, 200))
            a = rng.randrange(nraw - n + 1)
            v[rng.randrange(nrow), a:a + n] = tone
        for _ in range(2):
            n = max(1, nraw // 1000)
            a = rng.randrange(nraw - n + 1)
            v[:, a:a + n] = 50
    return v


def _prototype(m, taps):
    """The channeliser's filter: a windowed sinc of m * taps coefficients."""
    n = m * taps
    k = np.arange(n, dtype=np.float64)
    return (np.sinc((k - (n - 1) / 2) / m) * np.hamming(n)).astype(np.float32)


def _plane(case, seed):
    """A de-dispersed plane: sums over 1024 channels of 8-bit noise, with pulses."""
    g = _gen(seed)
    n, nsamp = case["ndm"], case["nsamp"]
    x = torch.empty((n, _round(nsamp, 4)), dtype=torch.float32, device="cuda")
    x.normal_(131072.0, 512.0, generator=g)
    rng = random.Random(seed)
    for _ in range(8):
        w = min(nsamp, 1 << rng.randrange(9))
        t = rng.randrange(nsamp - w + 1)
        x[rng.randrange(n), t:t + w] += 4000.0
    return x.round_() if case["integer"] else x.div_(1024.0)


def prepare(case, seed):
    op = case["op"]
    if op in ("search", "host"):
        x, nin = _filterbank(case, seed)
        plan = dd.Plan(*_beam(case))
        s = dict(op=op, plan=plan, x=x, nin=nin, nsamp=case["nsamp"])
        if op == "search":
            s["out"] = torch.zeros((case["ndm"], _round(case["nsamp"], 4)), dtype=torch.float32,
                                   device="cuda")
        else:
            s["x"] = torch.empty(x.shape, dtype=x.dtype, pin_memory=True).copy_(x)
            s["out"] = torch.zeros((case["ndm"], case["nsamp"]), dtype=torch.float32,
                                   pin_memory=True)
        return s
    if op == "batch":
        beams = _beams_of(case)
        plans = [dd.Plan(*_beam(b)) for b in beams]
        batch = dd.Batch(plans, "u8")
        outs = []
        for i, b in enumerate(beams):
            x, nin = _filterbank(b, seed * 64 + i)
            out = torch.zeros((b["ndm"], _round(b["nsamp"], 4)), dtype=torch.float32,
                              device="cuda")
            batch.set_io(i, x, out, nsamp_in=nin, nsamp_out=b["nsamp"])
            outs.append(out[:, :b["nsamp"]])
        return dict(op=op, batch=batch, outs=outs)
    if op == "detect":
        return dict(op=op, plane=_plane(case, seed), nsamp=case["nsamp"],
                    nlevels=case["nlevels"], integer=case["integer"])
    if op == "unpack":
        n = case["nchan"] * case["nbits"] // 8 * case["nsamp"]
        raw = torch.randint(0, 256, (n,), dtype=torch.uint8, device="cuda", generator=_gen(seed))
        out = torch.zeros((case["nchan"], _round(case["nsamp"], 16)), dtype=torch.uint8,
                          device="cuda")
        return dict(op=op, raw=raw, out=out, case=dict(case))
    if op == "frontend":
        v = _voltages(case["nchan"], case["nraw"], seed, True)
        n = case["nraw"] // case["nint"]
        out = torch.zeros((case["nchan"], _round(n, 16)), dtype=torch.uint8, device="cuda")
        work = torch.empty(max(16, dd.frontend_work_bytes(case["nchan"], case["nraw"],
                                                          case["nint"], case["niter"])),
                           dtype=torch.uint8, device="cuda")
        return dict(op=op, v=v, out=out, work=work, n=n, case=dict(case))
    nraw = (case["nspec"] + case["taps"] - 1) * case["m"]
    v = _voltages(case["nsub"], nraw, seed, False)
    h = torch.from_numpy(_prototype(case["m"], case["taps"])).cuda()
    ci8 = case["kind"] == "ci8"
    out = torch.zeros((case["nsub"] * case["m"], _round(case["nspec"], 4) if ci8
                       else case["nspec"], 4), dtype=torch.int8 if ci8 else torch.float32,
                      device="cuda")
    return dict(op=op, v=v, h=h, out=out, case=dict(case))


def run(s):
    op = s["op"]
    if op == "search":
        s["plan"].execute(s["x"], s["out"], nsamp_in=s["nin"], nsamp_out=s["nsamp"])
        return s["out"][:, :s["nsamp"]]
    if op == "host":
        s["plan"].execute_host(s["x"], s["out"], nsamp_in=s["nin"], nsamp_out=s["nsamp"])
        return s["out"]
    if op == "batch":
        s["batch"].execute()
        return s["outs"]
    if op == "detect":
        return dd.detect(s["plane"], nsamp=s["nsamp"], nlevels=s["nlevels"],
                         integer_valued=s["integer"])
    c = s["case"]
    if op == "unpack":
        dd.unpack(s["raw"], c["nbits"], c["nchan"], c["nsamp"], s["out"])
        return s["out"][:, :c["nsamp"]]
    if op == "frontend":
        out, mean, std = dd.frontend(s["v"], c["nint"], c["k"], c["niter"], out=s["out"],
                                     work=s["work"])
        return out[:, :s["n"]], mean, std
    dd.channelise(s["v"], c["m"], c["taps"], s["h"], kind=c["kind"], scale=c["scale"],
                  out=s["out"])
    return s["out"][:, :c["nspec"]]


def work(case):
    """Each input read once, each output written once, and the operations of the definition."""
    op = case["op"]
    if op in ("search", "host"):
        size = DTYPES[case["dtype"]].itemsize
        nin = case["nsamp"] + _maxshift(case)
        return dict(bytes=case["nchan"] * nin * size + case["ndm"] * case["nsamp"] * 4,
                    flops=case["nchan"] * case["ndm"] * case["nsamp"])
    if op == "batch":
        each = [work(b) for b in _beams_of(case)]
        return dict(bytes=sum(w["bytes"] for w in each), flops=sum(w["flops"] for w in each))
    if op == "detect":
        n = case["ndm"] * case["nsamp"]
        # per sample: one add per boxcar width, the two row sums
        return dict(bytes=4 * n + case["ndm"] * (16 + 16 * case["nlevels"]),
                    flops=n * (case["nlevels"] - 1 + 3))
    if op == "unpack":
        n = case["nchan"] * case["nsamp"]
        return dict(bytes=n * case["nbits"] // 8 + n, flops=0)
    if op == "frontend":
        n = case["nchan"] * case["nraw"]
        return dict(bytes=4 * n + n // case["nint"] + 16 * case["nchan"], flops=8 * n)
    m, t = case["m"], case["taps"]
    spectra = case["nsub"] * case["nspec"]
    element = 4 if case["kind"] == "ci8" else 16
    return dict(bytes=4 * case["nsub"] * (case["nspec"] + t - 1) * m + spectra * m * element,
                flops=spectra * 2 * (4 * m * t + 5 * m * math.log2(m)))


# --- what the definitions give in 64 bits -------------------------------------


def _exact_search(case, seed):
    x, _ = _filterbank(case, seed)
    shifts = torch.from_numpy(_shifts(case)).cuda()
    n = case["nsamp"]
    out = torch.zeros((case["ndm"], n), dtype=torch.float64, device="cuda")
    rows = max(1, (1 << 28) // n)
    for c in range(case["nchan"]):
        windows = x[c].double().unfold(0, n, 1)
        for d in range(0, case["ndm"], rows):
            out[d:d + rows] += windows[shifts[c, d:d + rows]]
    return out


def _exact_detect(case, seed):
    x = _plane(case, seed)[:, :case["nsamp"]].double()
    n = case["nsamp"]
    mean = x.mean(1)
    std = ((x * x).mean(1) - mean * mean).clamp_min(0).sqrt()
    total = torch.cat([torch.zeros_like(x[:, :1]), x.cumsum(1)], 1)
    snr = torch.full((case["ndm"], case["nlevels"]), -math.inf, dtype=torch.float64,
                     device="cuda")
    for level in range(case["nlevels"]):
        w = 1 << level
        if w <= n:
            best = (total[:, w:] - total[:, :-w]).max(1).values
            snr[:, level] = (best - w * mean) / (std * math.sqrt(w))
    return mean, std, snr, None


def _exact_frontend(case, seed):
    v = _voltages(case["nchan"], case["nraw"], seed, True)
    n = case["nraw"] // case["nint"]
    means, stds = [], []
    for row in v:
        p = row[:n * case["nint"]].double().square().sum(1).view(n, case["nint"]).sum(1)
        keep = torch.ones_like(p)
        for _ in range(case["niter"]):
            count = keep.sum()
            mean = (p * keep).sum() / count
            std = ((p * p * keep).sum() / count - mean * mean).clamp_min(0).sqrt()
            keep = (p <= (mean + case["k"] * std).floor()).double()
        means.append(mean)
        stds.append(std)
    return None, torch.stack(means), torch.stack(stds)


def _exact_channelise(case, seed):
    m, t, nspec = case["m"], case["taps"], case["nspec"]
    v = _voltages(case["nsub"], (nspec + t - 1) * m, seed, False)
    h = torch.from_numpy(_prototype(m, t)).cuda().double().view(t, m)
    out = torch.empty((case["nsub"], m, nspec, 4), dtype=torch.float64, device="cuda")
    for s in range(case["nsub"]):
        blocks = v[s].double().view(nspec + t - 1, m, 4)
        z = sum(h[k, :, None] * blocks[k:k + nspec] for k in range(t))
        y = torch.fft.fft(torch.view_as_complex(z.view(nspec, m, 2, 2)), dim=1)
        y = torch.view_as_real(torch.fft.fftshift(y, dim=1)).reshape(nspec, m, 4)
        out[s] = y.permute(1, 0, 2)
    return out.view(case["nsub"] * m, nspec, 4)


def exact(case, seed):
    op = case["op"]
    if op in ("search", "host"):
        if case["nchan"] * case["ndm"] * case["nsamp"] > MAX_ADDS // 2:
            return None
        out = _exact_search(case, seed)
        return out.cpu() if op == "host" else out
    if op == "batch":
        if work(case)["flops"] > MAX_ADDS // 2:
            return None
        return [_exact_search(b, seed * 64 + i) for i, b in enumerate(_beams_of(case))]
    if op == "detect":
        return _exact_detect(case, seed)
    if op == "frontend":
        return _exact_frontend(case, seed)
    if op == "channelise" and case["kind"] == "cf32":
        return _exact_channelise(case, seed)
    return None  # whole numbers: compared as they are
