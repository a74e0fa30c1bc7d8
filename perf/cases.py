"""The work that users of the package have it do, as timed cases.

Eight kinds of call, each through the package's public entry points:

  step        Plan.execute + Plan.search on device-resident input: one beam
  buffer      dd_channelise + Plan.execute + Plan.search: one buffer of the
              real-time pipeline, from baseband voltages to candidates
  serve       Server.submit / poll / candidates: one chunk of a streaming beam,
              from host memory
  batch       Batch.launch (captured graph) + Batch.results: uneven small beams
  subband     SubbandPlan.execute + search: the two-stage approximation
  survey      SurveyPlan.execute + search of every pass
  channelise  dd_channelise alone
  search      Plan.search alone, on a buffer that the caller has

Sizes are those of the repository's workloads (synth/), of bench.py's modes
and of the tests, or lie between them.  Inputs are unit-variance noise with
dispersed pulses in it (uint8: mean 128, standard deviation 16; float16: the
same noise rounded), drawn on the GPU from the seed.  Outputs come whole: the
de-dispersed buffer, the candidates' fields, the buffer's mean and deviation.
Candidate values and statistics of floating-point beams are given as float32:
they are formed from float32 sums.
"""
import math

import numpy as np
import torch

import paper_1107_2516_gb300 as dd

DTYPES = {"f32": dd.DD_F32, "u8": dd.DD_U8, "f16": dd.DD_F16}
ELEM = {"f32": 4, "u8": 1, "f16": 2}
OK, OVERFLOW = 0, 4      # dd_status
SIGMA = 6.0
POW2 = "1,2,4,8,16,32"
CAPACITY = 1 << 15      # candidates a search may return; a search of a quiet buffer finds far fewer


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest search (synth's small_f32): launches and read-backs count, not the sums
        {"name": "small_f32", "kind": "step", "dtype": "f32", "nchans": 128, "fch1": 150.0, "foff": -0.1953125,
         "tsamp": 327.68e-6, "nsamp": 8192, "pad": 0, "ndm": 64, "dm_step": 0.1, "widths": "1,2,4,8", "capacity": 4096},
        # the headline beam (synth's lofar_f32, bench.py's step): 2000 trials over 2^20 samples of 1024 channels
        {"name": "lofar_f32", "kind": "step", "dtype": "f32", "nchans": 1024, "fch1": 150.0, "foff": -0.01171875,
         "tsamp": 163.84e-6, "nsamp": 1 << 20, "pad": 0, "ndm": 2000, "dm_step": 0.05, "widths": POW2, "capacity": CAPACITY},
        # the same band from an 8-bit digitiser, a shorter buffer
        {"name": "lofar_u8", "kind": "step", "dtype": "u8", "nchans": 1024, "fch1": 150.0, "foff": -0.01171875,
         "tsamp": 163.84e-6, "nsamp": 1 << 18, "pad": 0, "ndm": 2000, "dm_step": 0.05, "widths": POW2, "capacity": CAPACITY},
        # the same band stored as half floats, fewer trials
        {"name": "lofar_f16", "kind": "step", "dtype": "f16", "nchans": 1024, "fch1": 150.0, "foff": -0.01171875,
         "tsamp": 163.84e-6, "nsamp": 1 << 17, "pad": 0, "ndm": 1000, "dm_step": 0.05, "widths": POW2, "capacity": CAPACITY},
        # a cut of a recording: an odd number of samples in a plain contiguous array, so rows start anywhere
        {"name": "ragged_f32", "kind": "step", "dtype": "f32", "nchans": 200, "fch1": 400.0, "foff": -0.09,
         "tsamp": 256e-6, "nsamp": 150001, "pad": 0, "ndm": 301, "dm_step": 0.2, "widths": POW2, "capacity": CAPACITY},
        # one buffer of the real-time pipeline (bench.py --mode realtime): 256 subbands x 8 channels, 2^19 spectra
        {"name": "realtime_buffer", "kind": "buffer", "npol": 1, "nsub": 256, "nfft": 8, "spectra": 1 << 19,
         "ftop": 620.0, "bw": 20.0, "tv": 12.8e-6, "ndm": 500, "dm_step": 0.12, "widths": POW2, "capacity": CAPACITY},
        # one chunk of a streaming 8-bit beam (synth's serving recipe: 4096 channels, 65536 samples, DM to 500)
        {"name": "serve_chunk_u8", "kind": "serve", "dtype": "u8", "nchans": 4096, "fch1": 1200.0, "foff": -0.048828125,
         "tsamp": 81.92e-6, "chunk": 65536, "ndm": 1500, "dm_step": 500.0 / 1500, "widths": POW2, "capacity": CAPACITY},
        # uneven small beams in one captured batch (synth's batch recipe at its small sizes)
        {"name": "batch_small", "kind": "batch", "beams": 8, "beam_seed": 5, "lo_nsamp": 13, "lo_ndm": 40, "hi_ndm": 200,
         "widths": "1,2,4,8,16", "capacity": 8192},
        # the two-stage approximation of the headline beam (bench.py --mode subband)
        {"name": "subband_f32", "kind": "subband", "dtype": "f32", "nchans": 1024, "fch1": 150.0, "foff": -0.01171875,
         "tsamp": 163.84e-6, "nsamp": 1 << 20, "ndm": 2000, "dm_step": 0.05, "group": 24, "nsub": 32, "widths": POW2, "capacity": CAPACITY},
        # a survey plan of three binned passes over a 60 s beam (bench.py --mode survey)
        {"name": "survey_f32", "kind": "survey", "dtype": "f32", "nchans": 1024, "fch1": 307.9921875, "foff": -0.015625,
         "tsamp": 64e-6, "nsamp": 937500, "scale": 1.0, "nsub": 32, "widths": POW2, "capacity": CAPACITY},
        # the front end alone, two polarisations, its longest transform
        {"name": "channelise_2pol", "kind": "channelise", "npol": 2, "nsub": 64, "nfft": 32, "nsamp": 1 << 19},
        # a search of a buffer that the caller has: widths that are no powers of two, each row by its own statistics
        {"name": "search_rows", "kind": "search", "ndm": 600, "nsamp": 262147, "widths": "1,3,7,20,50", "rows": True,
         "capacity": CAPACITY},
    ]


def _odd(rng, lo, hi):
    """A size between lo and hi, spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "buffer", "serve", "batch", "subband", "survey", "channelise", "search"])
    tsamp = rng.choice([64e-6, 81.92e-6, 163.84e-6, 327.68e-6])
    widths = rng.choice([POW2, POW2, "1,2,4,8", "1,2,4,8,16,32,64", "1,3,7,20,50", "2,5,9"])
    if kind in ("step", "serve", "subband"):
        # a band whose lowest channel stays above 0.6 of its highest, and trials
        # whose largest delay stays below a third of the samples
        nch = _odd(rng, 64, 4096) if kind == "step" else rng.choice([512, 1024, 2048, 4096])
        if kind == "subband":
            nch = rng.choice([256, 512, 1024])
        fch1 = rng.uniform(120.0, 1500.0)
        foff = -min(rng.uniform(6.0, 300.0), 0.4 * fch1) / nch
        ndm = _odd(rng, 32, 2000) if kind == "step" else _odd(rng, 500, 2000)
        nsamp = _odd(rng, 1 << 13, 1 << 18) if kind != "serve" else 65536
        # at most a twentieth of the largest case's adds
        while nch * ndm * nsamp > 1e11:
            ndm, nsamp = (ndm * 3 // 4, nsamp) if kind == "serve" or ndm > 500 else (ndm, nsamp * 3 // 4)
        span = _delays(nch, fch1, foff, tsamp, [1.0]).max() + 1.0      # samples per unit of DM
        step = float(min(rng.choice([0.05, 0.1, 0.2, 0.5]), nsamp / (3.0 * span * ndm)))
        case = {"kind": kind, "nchans": nch, "fch1": fch1, "foff": foff, "tsamp": tsamp, "ndm": ndm, "dm_step": step,
                "widths": widths, "capacity": CAPACITY}
        if kind == "step":
            dtype = rng.choice(["f32", "f32", "u8", "f16"])
            return {**case, "dtype": dtype, "nsamp": nsamp, "pad": -nsamp % 16 if rng.random() < 0.75 else rng.randrange(0, 8)}
        if kind == "serve":
            return {**case, "dtype": rng.choice(["u8", "u8", "f32"]), "chunk": nsamp}
        return {**case, "dtype": rng.choice(["f32", "u8"]), "nsamp": nsamp // 16 * 16, "group": rng.randrange(8, 41),
                "nsub": rng.choice([16, 32])}
    if kind == "buffer":
        nfft = rng.choice([4, 8, 16])
        return {"kind": kind, "npol": rng.choice([1, 2]), "nsub": rng.choice([64, 128, 256]), "nfft": nfft,
                "spectra": rng.randrange(1 << 12, 1 << 15) * nfft, "ftop": 620.0, "bw": rng.uniform(5.0, 20.0),
                "tv": 12.8e-6, "ndm": _odd(rng, 50, 500), "dm_step": 0.12, "widths": widths, "capacity": CAPACITY}
    if kind == "batch":
        return {"kind": kind, "beams": rng.randrange(3, 11), "beam_seed": rng.randrange(1000), "lo_nsamp": rng.choice([12, 13, 14]),
                "lo_ndm": 30, "hi_ndm": rng.randrange(100, 400), "widths": widths, "capacity": CAPACITY}
    if kind == "survey":
        return {"kind": kind, "dtype": rng.choice(["f32", "u8"]), "nchans": rng.choice([256, 512, 1024]), "fch1": 307.9921875,
                "foff": -0.015625, "tsamp": 64e-6, "nsamp": rng.randrange(12000, 56000) * 16, "scale": rng.uniform(0.1, 0.5),
                "nsub": rng.choice([16, 32]), "widths": widths, "capacity": CAPACITY}
    if kind == "channelise":
        nfft = rng.choice([2, 4, 8, 16, 32])
        return {"kind": kind, "npol": rng.choice([1, 2]), "nsub": _odd(rng, 4, 256), "nfft": nfft,
                "nsamp": _odd(rng, 1 << 12, 1 << 19) // 2 * 2}
    return {"kind": kind, "ndm": _odd(rng, 16, 1500), "nsamp": _odd(rng, 10000, 500000), "widths": widths, "capacity": CAPACITY,
            "rows": rng.random() < 0.5}


# ------------------------------------------------------------------ inputs

def _delays(nchans, fch1, foff, tsamp, dms):
    """Dispersion delays in samples (4.15e6 ms, MHz), [trials][channels], relative to the top of the band."""
    f = fch1 + np.arange(nchans) * foff
    u = 1.0 / (f * f) - 1.0 / (f.max() * f.max())
    x = (4.15e6 * np.asarray(dms, np.float64))[:, None] * u[None, :] / (tsamp * 1e3)
    return np.floor(x + 0.5).astype(np.int64)


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 1)
    return g


def _pulses(rng, n, dm_max, t_max, nchans):
    """n pulses (DM, sample, width, height per channel) of a boxcar signal-to-noise ratio between 8 and 20."""
    return [(rng.uniform(0.0, dm_max), int(rng.integers(0, max(1, t_max))), w, rng.uniform(8.0, 20.0) / math.sqrt(nchans * w))
            for w in rng.integers(1, 17, n)]


def _inject(x, nsamp, band, pulses):
    for dm, t0, w, amp in pulses:
        off = torch.from_numpy(_delays(*band, [dm])[0]).to(x.device)
        for j in range(int(w)):
            t = off + t0 + j
            c = torch.nonzero(t < nsamp).flatten()
            x[c, t[c]] += amp


def _beam(seed, dtype, nchans, nsamp, pad, band, dm_max):
    """One beam's input [nchans][nsamp + pad] on the GPU: a pulse in every 65536 samples, two at least."""
    g, rng = _generator(seed), np.random.default_rng(seed)
    x = torch.randn(nchans, nsamp + pad, device="cuda", generator=g)
    maxshift = int(_delays(*band, [dm_max]).max())
    _inject(x, nsamp, band, _pulses(rng, max(2, nsamp >> 16), dm_max, nsamp - maxshift - 32, nchans))
    if dtype == "u8":
        x = x.mul_(16.0).add_(128.0).round_().clamp_(0, 255).to(torch.uint8)
    elif dtype == "f16":
        x = x.to(torch.float16)
    return x


def _widths(case):
    return tuple(int(w) for w in case["widths"].split(","))


def _dms(case):
    return np.arange(case["ndm"], dtype=np.float64) * case["dm_step"]


def _band(case):
    return case["nchans"], case["fch1"], case["foff"], case["tsamp"]


def _out(ndm, nout, dtype):
    return torch.empty(ndm, nout, device="cuda", dtype=torch.int32 if dtype == "u8" else torch.float32)


def _batch_beams(case):
    """Plan parameters of the batch's beams: channels cycle 64..512, lengths and trials uneven, every other beam uint8."""
    rng = np.random.default_rng(case["beam_seed"])
    beams = []
    for i in range(case["beams"]):
        nch, nsamp = (64, 128, 256, 512)[i % 4], 1 << (case["lo_nsamp"] + 7 * i % 3)
        fch1 = rng.uniform(120.0, 1500.0)
        foff = -min(rng.uniform(6.0, 300.0), 0.5 * fch1) / nch
        tsamp = (64e-6, 81.92e-6, 163.84e-6, 327.68e-6)[int(rng.integers(0, 4))]
        ndm = int(rng.integers(case["lo_ndm"], case["hi_ndm"] + 1))
        step = math.exp(rng.uniform(math.log(0.01), math.log(0.5)))
        while _delays(nch, fch1, foff, tsamp, [(ndm - 1) * step]).max() > nsamp // 2:
            step *= 0.8
        beams.append((nch, fch1, foff, tsamp, nsamp, ndm, step, "f32" if i % 2 == 0 else "u8"))
    return beams


def _survey_passes(case):
    """The three passes of the survey table (low, high, step, bin, subband step), their DM ranges scaled."""
    k = case["scale"]
    a, b, c = 0.66 * round(53.46 * k / 0.66), 1.2 * round(34.8 * k / 1.2), 2.4 * round(62.4 * k / 2.4)
    return [(0.0, a, 0.03, 1, 0.66), (a, a + b, 0.05, 2, 1.2), (a + b, a + b + c, 0.10, 4, 2.4)]


def _buffer_plan(case):
    """(channels, top channel, channel width, sampling time, samples) of the filterbank that the channeliser makes."""
    nch = case["nsub"] * case["nfft"]
    cw = case["bw"] / nch
    return nch, case["ftop"] - 0.5 * cw, -cw, case["nfft"] * case["tv"], case["spectra"] // case["nfft"]


def prepare(case, seed):
    kind, st = case["kind"], {"case": case}
    if kind == "step":
        st["x"] = _beam(seed, case["dtype"], case["nchans"], case["nsamp"], case["pad"], _band(case), _dms(case)[-1])
        st["plan"] = dd.Plan(*_band(case), _dms(case), _widths(case), SIGMA, DTYPES[case["dtype"]], case["nsamp"])
        st["out"] = _out(case["ndm"], st["plan"].nsamp_out, case["dtype"])
    elif kind == "buffer":
        nch, fch1, foff, ts, nsamp = _buffer_plan(case)
        st["volt"] = torch.randn(case["npol"], case["nsub"], case["spectra"], 2, device="cuda", generator=_generator(seed))
        st["fil"] = torch.empty(nch, nsamp, device="cuda")
        st["plan"] = dd.Plan(nch, fch1, foff, ts, _dms(case), _widths(case), SIGMA, dd.DD_F32, nsamp)
        st["out"] = _out(case["ndm"], st["plan"].nsamp_out, "f32")
    elif kind == "serve":
        x = _beam(seed, case["dtype"], case["nchans"], case["chunk"], 0, _band(case), _dms(case)[-1])
        st["chunk"] = torch.empty(x.shape, dtype=x.dtype, pin_memory=True)
        st["chunk"].copy_(x)
        st["server"] = dd.Server(64 << 30, 2, 1 << 16)
        st["beam"] = st["server"].add_beam(*_band(case), _dms(case), _widths(case), SIGMA, DTYPES[case["dtype"]], case["chunk"])
        info = st["server"].beam_info(st["beam"])
        typ = "<i4" if case["dtype"] == "u8" else "<f4"
        st["out"] = torch.as_tensor(_DeviceBuffer(info["out_dev"], (case["ndm"], case["chunk"]), typ), device="cuda")
        # the stream's history: chunks until the beam has seen maxshift samples
        st["seq"] = 0
        for _ in range(-(-info["maxshift"] // case["chunk"])):
            _serve_one(st)
    elif kind == "batch":
        st["plans"], st["ins"], st["outs"], st["pitches"] = [], [], [], []
        for i, (nch, fch1, foff, ts, nsamp, ndm, step, dtype) in enumerate(_batch_beams(case)):
            st["ins"].append(_beam(seed * 100 + i, dtype, nch, nsamp, 0, (nch, fch1, foff, ts), (ndm - 1) * step))
            st["plans"].append(dd.Plan(nch, fch1, foff, ts, np.arange(ndm) * step, _widths(case), SIGMA, DTYPES[dtype], nsamp))
            st["outs"].append(_out(ndm, st["plans"][-1].nsamp_out, dtype))
            st["pitches"].append(nsamp)
        st["stream"] = torch.cuda.Stream()
        st["batch"] = dd.Batch(st["plans"])
        st["batch"].capture(st["ins"], st["pitches"], st["outs"], st["stream"])
    elif kind == "subband":
        st["x"] = _beam(seed, case["dtype"], case["nchans"], case["nsamp"], 0, _band(case), _dms(case)[-1])
        st["plan"] = dd.SubbandPlan(*_band(case), _dms(case), case["group"], case["nsub"], _widths(case), SIGMA,
                                    DTYPES[case["dtype"]], case["nsamp"])
        st["out"] = _out(case["ndm"], st["plan"].nsamp_out, case["dtype"])
    elif kind == "survey":
        passes = _survey_passes(case)
        st["x"] = _beam(seed, case["dtype"], case["nchans"], case["nsamp"], 0, _band(case), passes[-1][1])
        st["plan"] = dd.SurveyPlan(*_band(case), passes, case["nsub"], _widths(case), SIGMA, DTYPES[case["dtype"]], case["nsamp"])
        st["outs"] = [_out(p[0], p[4], case["dtype"] if p[1] == 1 else "f32") for p in st["plan"].passes]
    elif kind == "channelise":
        st["volt"] = torch.randn(case["npol"], case["nsub"], case["nsamp"], 2, device="cuda", generator=_generator(seed))
        st["fil"] = torch.empty(case["nsub"] * case["nfft"], case["nsamp"] // case["nfft"], device="cuda")
    elif kind == "search":
        # a buffer of 64 summed channels: rows of noise, their levels apart, a few pulses
        g, rng = _generator(seed), np.random.default_rng(seed)
        st["plan"] = dd.Plan(64, 150.0, -0.001, 1e-3, np.arange(case["ndm"]) * 0.01, _widths(case), SIGMA, dd.DD_F32, case["nsamp"])
        st["plan"].set_search_stats(bool(case["rows"]))
        x = torch.randn(case["ndm"], st["plan"].nsamp_out, device="cuda", generator=g).mul_(8.0)
        if case["rows"]:
            x += torch.randn(case["ndm"], 1, device="cuda", generator=g)
        for _ in range(16):
            r, t, w = int(rng.integers(0, case["ndm"])), int(rng.integers(0, x.shape[1] - 64)), int(rng.integers(1, 33))
            x[r, t:t + w] += 8.0 * rng.uniform(8.0, 20.0) / math.sqrt(w)
        st["out"] = x
    else:
        raise ValueError(kind)
    return st


class _DeviceBuffer:
    """A library-owned device buffer, for torch.as_tensor."""

    def __init__(self, ptr, shape, typestr):
        self.__cuda_array_interface__ = {"shape": shape, "typestr": typestr, "data": (ptr, False), "version": 3}


# ------------------------------------------------------------------ one pass

def _found(case, cands, whole, total):
    """The candidates' fields in tables of one length.  A search with more hits than its capacity returns an
    unspecified part of them: then only their number is a result."""
    n = 0 if total > case["capacity"] else len(cands)
    table = {"dm_idx": np.int32, "width_idx": np.int32, "t": np.int64, "snr": np.float32, "value": np.int64 if whole else np.float32}
    for field, typ in table.items():
        table[field] = np.zeros(case["capacity"], typ)
        table[field][:n] = cands[field][:n]
    return {**table, "total": int(total)}


def _search(case, plan, out, whole):
    cands, total = plan.search(out, capacity=case["capacity"], allow_overflow=True)
    return {**_found(case, cands, whole, total), "stats": np.float32(plan.stats())}


def _serve_one(st):
    server, seq = st["server"], st["seq"]
    server.submit(st["beam"], st["chunk"], st["chunk"].shape[1], seq)
    st["seq"] += 1
    while True:
        done = server.poll(wait_ms=1000)
        if len(done):
            if done[0]["status"] not in (OK, OVERFLOW, dd.DD_PRIMING):
                raise RuntimeError("chunk status %d" % done[0]["status"])
            return done[0], server.candidates(st["beam"], seq)


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "step":
        st["plan"].execute(st["x"], case["nsamp"] + case["pad"], st["out"])
        return {"out": st["out"], **_search(case, st["plan"], st["out"], case["dtype"] == "u8")}
    if kind == "buffer":
        nsamp = st["fil"].shape[1]
        dd.dd_channelise(st["volt"], case["npol"], case["nsub"], case["spectra"], case["nfft"], st["fil"], nsamp)
        st["plan"].execute(st["fil"], nsamp, st["out"])
        return {"out": st["out"], "fil": st["fil"], **_search(case, st["plan"], st["out"], False)}
    if kind == "serve":
        r, cands = _serve_one(st)
        # the library's buffer is overwritten by the beam's next chunk and freed with the server
        return {"out": st["out"].clone(), **_found(case, cands, case["dtype"] == "u8", r["n_candidates"]),
                "stats": np.float32([r["mu"], r["sigma"]])}
    if kind == "batch":
        st["batch"].launch(st["stream"])
        found = []
        for i, plan in enumerate(st["plans"]):
            cands, total = st["batch"].results(i, capacity=case["capacity"], stream=st["stream"], allow_overflow=True)
            found.append(_found(case, cands, plan.out_is_int, total))
        return {"out": st["outs"], "found": found}
    if kind == "subband":
        st["plan"].execute(st["x"], case["nsamp"], st["out"])
        return {"out": st["out"], **_search(case, st["plan"], st["out"], case["dtype"] == "u8")}
    if kind == "survey":
        st["plan"].execute(st["x"], case["nsamp"], st["outs"])
        found = []
        for i, out in enumerate(st["outs"]):
            cands, total = st["plan"].search(i, out, capacity=case["capacity"], allow_overflow=True)
            found.append({**_found(case, cands, out.dtype == torch.int32, total), "stats": np.float32(st["plan"].stats(i))})
        return {"out": st["outs"], "found": found}
    if kind == "channelise":
        dd.dd_channelise(st["volt"], case["npol"], case["nsub"], case["nsamp"], case["nfft"], st["fil"], st["fil"].shape[1])
        return st["fil"]
    found = _search(case, st["plan"], st["out"], False)
    return {**found, "rows": np.float32(st["plan"].row_stats())} if case["rows"] else found


# ------------------------------------------------------------------ what a pass cannot do without

def _sum_work(nch, ndm, nsamp, nout, elem):
    """Brute force: the input read once, every output written once and read once by the search; an add per channel and output."""
    return {"bytes": nch * nsamp * elem + 8.0 * ndm * nout, "flops": float(nch) * ndm * nout}


def _subband_work(band, dms, group, nsub, nsamp, elem):
    nch, cs = band[0], band[0] // nsub
    k = -(-len(dms) // group)
    nout = nsamp - int(_delays(*band, [dms[-1]]).max())
    return {"bytes": nch * nsamp * elem + 8.0 * len(dms) * nout, "flops": float(nout) * (k * nsub * cs + len(dms) * nsub)}


def work(case):
    kind = case["kind"]
    if kind == "step":
        nout = case["nsamp"] - int(_delays(*_band(case), [_dms(case)[-1]]).max())
        return _sum_work(case["nchans"], case["ndm"], case["nsamp"], nout, ELEM[case["dtype"]])
    if kind == "serve":
        return _sum_work(case["nchans"], case["ndm"], case["chunk"], case["chunk"], ELEM[case["dtype"]])
    if kind == "buffer":
        nch, fch1, foff, ts, nsamp = _buffer_plan(case)
        w = _sum_work(nch, case["ndm"], nsamp, nsamp - int(_delays(nch, fch1, foff, ts, [_dms(case)[-1]]).max()), 4)
        w["bytes"] += 8.0 * case["npol"] * case["nsub"] * case["spectra"]
        return w
    if kind == "batch":
        ws = [_sum_work(nch, ndm, nsamp, nsamp - int(_delays(nch, fch1, foff, ts, [(ndm - 1) * step]).max()), ELEM[dtype])
              for nch, fch1, foff, ts, nsamp, ndm, step, dtype in _batch_beams(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    if kind == "subband":
        return _subband_work(_band(case), _dms(case), case["group"], case["nsub"], case["nsamp"], ELEM[case["dtype"]])
    if kind == "survey":
        total = {"bytes": 0.0, "flops": 0.0}
        for low, high, step, nb, sub in _survey_passes(case):
            dms = low + step * np.arange(round((high - low) / step))
            band = (case["nchans"], case["fch1"], case["foff"], case["tsamp"] * nb)
            w = _subband_work(band, dms, round(sub / step), case["nsub"], case["nsamp"] // nb, 4)
            total["flops"] += w["flops"]
            total["bytes"] += w["bytes"] - case["nchans"] * (case["nsamp"] // nb) * 4
        total["bytes"] += case["nchans"] * case["nsamp"] * ELEM[case["dtype"]]
        return total
    if kind == "channelise":
        n = case["nsub"] * case["nsamp"]
        return {"bytes": 8.0 * case["npol"] * n + 4.0 * n, "flops": case["npol"] * n * (5.0 * math.log2(case["nfft"]) + 3.0)}
    return {"bytes": 4.0 * case["ndm"] * case["nsamp"], "flops": float(len(_widths(case))) * case["ndm"] * case["nsamp"]}


# ------------------------------------------------------------------ the same in 64 bits

def _sum64(x, d, nout):
    """out[j][t] = sum_c x[c][t + d[j][c]] in 64 bits, some trials at a time."""
    dev = torch.from_numpy(np.ascontiguousarray(d)).to(x.device)
    out = torch.empty(d.shape[0], nout, dtype=torch.float64, device=x.device)
    at = max(1, min(d.shape[0], (1 << 28) // nout))
    for j in range(0, d.shape[0], at):
        acc = torch.zeros(min(at, d.shape[0] - j), nout, dtype=torch.float64, device=x.device)
        for c in range(x.shape[0]):
            acc += x[c].unfold(0, nout, 1).index_select(0, dev[j:j + at, c])
        out[j:j + at] = acc
    return out


def _stats64(out):
    mu = out.sum() / out.numel()
    var = sum(((row - mu) ** 2).sum() for row in out) / out.numel()
    return np.array([float(mu), math.sqrt(float(var))])


def _answer64(out):
    return {"out": out, "dm_idx": None, "width_idx": None, "t": None, "snr": None, "value": None, "total": None, "stats": _stats64(out)}


def _subband64(x, band, dms, group, nsub):
    """The two-stage sum: nominal-DM delays inside the subbands, each trial's own between them."""
    nch, foff = band[0], band[2]
    cs = nch // nsub
    ref = np.arange(nsub) * cs + (0 if foff < 0 else cs - 1)
    first = np.arange(0, len(dms), group)
    last = np.minimum(first + group, len(dms)) - 1
    dn = _delays(*band, 0.5 * (dms[first] + dms[last]))
    d1 = dn - np.repeat(dn[:, ref], cs, axis=1)
    d = _delays(*band, dms)[:, np.repeat(ref, cs)] + d1[np.arange(len(dms)) // group]
    nout = x.shape[1] - int(d.max())
    out = torch.empty(len(dms), nout, dtype=torch.float64, device=x.device)
    for k, j in enumerate(first):
        d2 = _delays(*band, dms[j:j + group])[:, ref]
        n = nout + int(d2.max())
        series = torch.zeros(nsub, n, dtype=torch.float64, device=x.device)
        for c in range(nch):
            seg = x[c, int(d1[k, c]):int(d1[k, c]) + n]
            series[c // cs, :seg.numel()] += seg
        out[j:j + group] = _sum64(series, d2, nout)
    return out


def _channelise64(volt, nsub, nfft):
    """Intensities of the nfft-point transforms, channel-major, each subband's channels from the top down."""
    n = volt.shape[2] // nfft
    fil = torch.empty(nsub * nfft, n, dtype=torch.float64, device=volt.device)
    order = [(nfft // 2 - 1 - j) % nfft for j in range(nfft)]
    for s in range(nsub):
        v = torch.view_as_complex(volt[:, s, :n * nfft].double())
        p = torch.fft.fft(v.reshape(v.shape[0], n, nfft), dim=2).abs().square().sum(0)
        fil[s * nfft:(s + 1) * nfft] = p[:, order].T
    return fil


def exact(case, seed):
    kind = case["kind"]
    if case.get("dtype") == "u8" and kind != "survey":
        return None                                     # whole numbers
    if kind in ("step", "serve"):
        if kind == "step":
            x = _beam(seed, case["dtype"], case["nchans"], case["nsamp"], case["pad"], _band(case), _dms(case)[-1])[:, :case["nsamp"]]
        else:
            x = _beam(seed, case["dtype"], case["nchans"], case["chunk"], 0, _band(case), _dms(case)[-1])
        d = _delays(*_band(case), _dms(case))
        if kind == "serve":                             # the same chunk again and again: its last samples before itself
            x = torch.cat([x] * (1 + -(-int(d.max()) // case["chunk"])), 1)[:, -(case["chunk"] + int(d.max())):]
        ans = _answer64(_sum64(x, d, x.shape[1] - int(d.max())))
        return ans
    if kind == "buffer":
        nch, fch1, foff, ts, nsamp = _buffer_plan(case)
        volt = torch.randn(case["npol"], case["nsub"], case["spectra"], 2, device="cuda", generator=_generator(seed))
        fil = _channelise64(volt, case["nsub"], case["nfft"])
        d = _delays(nch, fch1, foff, ts, _dms(case))
        return {**_answer64(_sum64(fil, d, nsamp - int(d.max()))), "fil": fil}
    if kind == "batch":
        outs = []
        for i, (nch, fch1, foff, ts, nsamp, ndm, step, dtype) in enumerate(_batch_beams(case)):
            x = _beam(seed * 100 + i, dtype, nch, nsamp, 0, (nch, fch1, foff, ts), (ndm - 1) * step)
            d = _delays(nch, fch1, foff, ts, np.arange(ndm) * step)
            outs.append(_sum64(x, d, nsamp - int(d.max())) if dtype == "f32" else None)
        return {"out": outs, "found": [None] * len(outs)}
    if kind == "subband":
        x = _beam(seed, case["dtype"], case["nchans"], case["nsamp"], 0, _band(case), _dms(case)[-1])
        return _answer64(_subband64(x, _band(case), _dms(case), case["group"], case["nsub"]))
    if kind == "survey":
        passes, outs, found = _survey_passes(case), [], []
        x = _beam(seed, case["dtype"], case["nchans"], case["nsamp"], 0, _band(case), passes[-1][1])
        for low, high, step, nb, sub in passes:
            n = case["nsamp"] // nb
            xb = x if nb == 1 else x[:, :n * nb].double().reshape(x.shape[0], n, nb).mean(2)
            dms = low + step * np.arange(round((high - low) / step))
            band = (case["nchans"], case["fch1"], case["foff"], case["tsamp"] * nb)
            ans = _answer64(_subband64(xb, band, dms, round(sub / step), case["nsub"]))
            outs.append(ans.pop("out"))
            found.append(ans)
        return {"out": outs, "found": found}
    if kind == "channelise":
        volt = torch.randn(case["npol"], case["nsub"], case["nsamp"], 2, device="cuda", generator=_generator(seed))
        return _channelise64(volt, case["nsub"], case["nfft"])
    ans = _answer64(prepare(case, seed)["out"].double())    # the buffer that is searched
    out = ans.pop("out")
    return {**ans, "rows": np.stack([out.mean(1).cpu(), out.std(1, correction=0).cpu()])} if case["rows"] else ans
