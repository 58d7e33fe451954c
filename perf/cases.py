"""The framework's performance cases: what its users have it do, through its public entry points.

Each case is a dict of plain values with a ``kind``:

``coherent``  one stream dedispersed coherently at one DM: push, flush, read the profile and the series
``batched``   one chunk dedispersed at many DM trials: push, flush, read the series block
``incoherent`` one buffer through the AID or CID filterbank mode, with the fold or the scintillation spectrum
``boxcar``    the single-pulse detector over a block of trial series
``classify``  candidate patches cut from a series block and scored by the network
``train``     the network's loss and gradient on one mini-batch
``stack``     a series folded with a phase model into a pulse stack

The split-BF16 precision options are left out: they demonstrate a precision form
that is both slower and less accurate than the FP32 one, so no user picks them.

``exact`` evaluates the same mathematics in 64 bits with torch and numpy.  The
folded profile and the fluctuation spectrum are FP64 accumulators of FP32
terms: ``run`` hands them back in FP32, the precision that their terms have.
"""
import math
from fractions import Fraction

import numpy as np
import torch

from paper_1503_01405_gb300 import learn, pond

F0, BW, FS = 326.5, 16.0, 32e6        # the band of every workload of this repository
K_DM = 1.0 / 2.41e-4                  # s MHz^2
ROWS, COLS, NCLS = 32, 256, 4         # the network's patch and classes


def listed():
    return [
        # a few segments of a short transform: latency, launches and the reads that end a stream
        {"name": "coherent_short", "kind": "coherent", "logn": 14, "nchan": 4, "dm": 0.05, "n": 100_003, "ch": 1,
         "bw": 16.0, "nbins": 64, "period": 0.0123, "t_dec": 61.44e-6, "host": False, "pdot": 0.0},
        # the single-channel workload (2^23 samples): every sub-channel sample kept at full time resolution
        {"name": "coherent_1ch", "kind": "coherent", "logn": 21, "nchan": 1, "dm": 3.0, "n": 1 << 23, "ch": 1,
         "bw": 16.0, "nbins": 256, "period": 0.253, "t_dec": 61.44e-6, "host": False, "pdot": 0.0},
        # the full-rate workload: 60 s of the band on the device, 64 sub-channels
        {"name": "coherent_full", "kind": "coherent", "logn": 24, "nchan": 64, "dm": 26.8, "n": 1_920_000_000, "ch": 1,
         "bw": 16.0, "nbins": 1024, "period": 0.7145, "t_dec": 61.44e-6, "host": False, "pdot": 0.0},
        # two halves added in phase, inverted band, folded with a spin-down model, pushed from pinned host memory
        {"name": "coherent_aip_host", "kind": "coherent", "logn": 23, "nchan": 32, "dm": 12.0, "n": 60_000_001, "ch": 2,
         "bw": -16.0, "nbins": 512, "period": 0.0893, "t_dec": 61.44e-6, "host": True, "pdot": 4e-6},
        # the transient search's dedispersion: 8 s, 128 trials on the uniform DM grid
        {"name": "batched_128", "kind": "batched", "logn": 24, "nchan": 64, "ndm": 128, "dm_lo": 0.0, "dm_hi": 60.0,
         "n": 256_000_000, "t_dec": 32e-6},
        # DM refinement around a known source: a few closely spaced trials off the uniform grid, medium transform
        {"name": "batched_refine", "kind": "batched", "logn": 20, "nchan": 16, "ndm": 21, "dm_lo": 2.41, "dm_hi": 2.67,
         "n": 20_000_003, "t_dec": 32e-6},
        # adding the halves and 1024-channel spectra at full time resolution (8 s)
        {"name": "incoherent_aid", "kind": "incoherent", "nchan": 1024, "nint": 1, "dm": 26.8, "mode": "aid", "ch": 2,
         "bw": 16.0, "nbins": 1024, "period": 0.7145, "n": 256_000_000, "ips": 0},
        # the scintillation mode: cross-power of the halves integrated to 0.256 ms, fluctuation spectrum (4 s)
        {"name": "incoherent_ips", "kind": "incoherent", "nchan": 256, "nint": 16, "dm": 0.0, "mode": "cid", "ch": 2,
         "bw": 16.0, "nbins": 64, "period": 0.5, "n": 128_000_077, "ips": 256},
        # single-pulse search over the 128-trial block of an 8 s chunk
        {"name": "boxcar_128", "kind": "boxcar", "ndm": 128, "n": 250_000},
        # the candidates of a chunk cut out and scored, one batch of the network
        {"name": "classify_512", "kind": "classify", "ndm": 128, "n": 50_000, "batch": 512},
        # one training mini-batch
        {"name": "train_256", "kind": "train", "batch": 256},
        # 60 s of the 61.44 us series folded into one row per rotation
        {"name": "stack_60s", "kind": "stack", "n": 976_562, "dt": 61.44e-6, "g0": 803, "period": 0.7145, "pdot": 4e-6,
         "nbins": 1024, "n_sub": 0},
    ]


# ---------------------------------------------------------------------------
# Drawn cases: the same ranges
# ---------------------------------------------------------------------------

def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _overlap(dm, nchan, bw=BW):
    """(n_past, n_fut) channel samples of the overlap at one DM."""
    dtc, half = 2.0 * nchan / FS, abs(bw) / 2
    lo, hi = F0 - half, F0 + half
    return (math.ceil(K_DM * dm * (F0 ** -2 - hi ** -2) / dtc), math.ceil(K_DM * dm * (lo ** -2 - F0 ** -2) / dtc))


def _dm_for(nchan, span):
    """The DM whose overlap covers `span` channel samples."""
    return span * (2.0 * nchan / FS) / (K_DM * ((F0 - BW / 2) ** -2 - (F0 + BW / 2) ** -2))


def draw(rng):
    kind = rng.choice(["coherent"] * 6 + ["batched"] * 3 + ["incoherent"] * 4 + ["boxcar", "classify", "train", "stack"] * 2)
    if kind == "coherent":
        logn = rng.randint(14, 24)
        nchan = 1 << rng.randint(0, min(7, logn - 10))
        ch = rng.choice([1, 1, 2])
        n = _log_int(rng, 2 << logn, min(48 << logn, 600_000_000))
        m = (1 << logn) // (2 * nchan)
        return {"kind": kind, "logn": logn, "nchan": nchan, "dm": round(_dm_for(nchan, m * rng.uniform(0.02, 0.5)), 6),
                "n": n, "ch": ch, "bw": rng.choice([16.0, -16.0]), "nbins": rng.choice([64, 100, 256, 1024]),
                "period": round(math.exp(rng.uniform(math.log(0.005), math.log(1.2))), 6), "t_dec": 61.44e-6,
                "host": rng.random() < 0.25 and n * ch < 300_000_000, "pdot": rng.choice([0.0, 0.0, 1e-6])}
    if kind == "batched":
        logn = rng.randint(18, 24)
        nchan = 1 << max(0, min(6, (logn - 1) // 2 - 5 + rng.choice([0, 0, -1])))
        ndm = _log_int(rng, 2, 64)
        n = _log_int(rng, 2 << logn, min(24 << logn, 8_000_000_000 // ndm, 256_000_000)) if (2 << logn) * ndm < 4_000_000_000 else 3 << logn
        m = (1 << logn) // (2 * nchan)
        hi = round(_dm_for(nchan, m * rng.uniform(0.1, 0.45)), 4)
        return {"kind": kind, "logn": logn, "nchan": nchan, "ndm": ndm, "dm_lo": rng.choice([0.0, round(0.9137 * hi, 4)]),
                "dm_hi": hi, "n": n, "t_dec": rng.choice([32e-6, 61.44e-6])}
    if kind == "incoherent":
        nchan, nint = 1 << rng.randint(6, 11), 1 << rng.randint(0, 7)
        mode = rng.choice(["aid", "aid", "cid"])
        n = _log_int(rng, 4_000_000, 400_000_000)
        ips = rng.choice([0, 0, 64, 256, 1024])
        return {"kind": kind, "nchan": nchan, "nint": nint, "dm": 0.0 if ips else round(rng.uniform(0.1, 0.2) * n / FS * 200, 3),
                "mode": mode, "ch": 2 if mode == "cid" else rng.choice([1, 2]), "bw": rng.choice([16.0, -16.0]),
                "nbins": rng.choice([64, 256, 1024]), "period": round(rng.uniform(0.03, 0.9), 5), "n": n, "ips": ips}
    if kind == "boxcar":
        return {"kind": kind, "ndm": _log_int(rng, 1, 200), "n": _log_int(rng, 20_000, 400_000)}
    if kind == "classify":
        return {"kind": kind, "ndm": rng.randint(32, 160), "n": _log_int(rng, 4_000, 200_000), "batch": _log_int(rng, 1, 4096)}
    if kind == "train":
        return {"kind": kind, "batch": _log_int(rng, 8, 1024)}
    n = _log_int(rng, 20_000, 4_000_000)
    return {"kind": kind, "n": n, "dt": rng.choice([61.44e-6, 32e-6, 0.256e-3]), "g0": rng.randint(0, 5000),
            "period": round(math.exp(rng.uniform(math.log(0.033), math.log(1.2))), 6), "pdot": rng.choice([0.0, 4e-6]),
            "nbins": rng.choice([64, 128, 256, 1000, 1024]), "n_sub": rng.choice([0, 0, max(1000, n // rng.randint(5, 60))])}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _voltages(n, seed, period, sigma=20.0):
    """int8 receiver noise with a pulsar's periodic excess and 1 % of impulsive interference."""
    g = _gen(seed)
    out = torch.empty(n, dtype=torch.int8, device="cuda")
    block = 1 << 27
    for b in range(0, n, block):
        k = min(block, n - b)
        v = torch.randn(k, generator=g, device="cuda")
        # amplitude per run of 256 samples (8 us): the pulse's variance excess, and 5 sigma bursts
        runs = -(-k // 256)
        t = (torch.arange(runs, device="cuda", dtype=torch.float64) * 256 + b) / FS
        d = torch.frac(t / period).float() - 0.5
        amp = torch.sqrt(1.0 + 0.5 * torch.exp(-4 * math.log(2.0) * (d / 0.05) ** 2))
        amp = torch.where(torch.rand(runs, generator=g, device="cuda") < 0.01, 5.0 * amp, amp)
        v *= amp.repeat_interleave(256)[:k]
        out[b:b + k] = v.mul_(sigma).round_().clamp_(-127, 127)
    return out


def _halves(n, seed, period):
    """N / S int8 pairs: a common component over each half's own noise."""
    common = _voltages(n, seed, period, 10.0)
    out = torch.empty((n, 2), dtype=torch.int8, device="cuda")
    g = _gen(seed + 7)
    block = 1 << 27
    for b in range(0, n, block):
        k = min(block, n - b)
        own = torch.randn((k, 2), generator=g, device="cuda").mul_(10.0).round_()
        out[b:b + k] = own.add_(common[b:b + k].float()[:, None]).clamp_(-127, 127)
    return out.reshape(-1)


def _samples(case, seed):
    period = case.get("period", 0.5)
    return _halves(case["n"], seed, period) if case.get("ch", 1) == 2 else _voltages(case["n"], seed, period)


def _series_block(ndm, n, seed):
    """FP32 trial series of detected power (about 1000 degrees of freedom) with single pulses across the trials."""
    g = _gen(seed)
    mean, sd = 4.0e5, 1.8e4
    x = torch.randn((ndm, n), generator=g, device="cuda").mul_(sd).add_(mean)
    r = np.random.default_rng(seed)
    for _ in range(10):
        d0, t0 = int(r.integers(ndm)), int(r.integers(200, n - 400))
        w, snr = int(2 ** r.uniform(0, 6)), r.uniform(9, 30)
        for d in range(max(0, d0 - 6), min(ndm, d0 + 7)):
            wd = w + 2 * abs(d - d0)          # off its DM a pulse is smeared and drifts
            a = snr * sd * math.sqrt(w) / wd / (1 + 0.3 * abs(d - d0))
            x[d, t0 + 2 * (d - d0): t0 + 2 * (d - d0) + wd] += a
    return x


def _trial_dms(case):
    lo, hi, m = case["dm_lo"], case["dm_hi"], case["ndm"]
    return [lo + (hi - lo) * d / (m - 1) for d in range(m)]


def _phase_model(case):
    """(t_ref, coefficients) of the spin-down model, epoch 1 s into the stream."""
    p = case["period"]
    return 1.0, [0.3, 1.0 / p, -case["pdot"] / (2 * p * p)]


def _series_samples(n, nchan, t_dec):
    return int(n / FS / t_dec) + 4


def prepare(case, seed):
    kind = case["kind"]
    if kind == "coherent":
        x = _samples(case, seed)
        e = pond.Engine(F0, case["bw"], FS, case["dm"], 1 << case["logn"], case["nchan"], case["nbins"], case["period"],
                        t_dec=case["t_dec"], input_channels=case["ch"],
                        phase_model=_phase_model(case) if case["pdot"] else None)
        cap = _series_samples(case["n"], case["nchan"], case["t_dec"])
        st = {"case": case, "engine": e, "T": torch.empty(cap, dtype=torch.float32, pin_memory=True).numpy(),
              "C": torch.empty(cap, dtype=torch.int32, pin_memory=True).numpy()}
        if case["host"]:
            h = torch.empty(x.numel(), dtype=torch.int8, pin_memory=True)
            h.copy_(x)
            st["x"] = h.numpy()
        else:
            st["x"] = x
        return st
    if kind == "batched":
        x = _samples(case, seed)
        e = pond.Engine(F0, BW, FS, 0.0, 1 << case["logn"], case["nchan"], 1, 1.0, t_dec=case["t_dec"], dms=_trial_dms(case))
        cap = _series_samples(case["n"], case["nchan"], case["t_dec"])
        return {"case": case, "engine": e, "x": x,
                "T": torch.empty((case["ndm"], cap), dtype=torch.float32, pin_memory=True).numpy(),
                "C": torch.empty(cap, dtype=torch.int32, pin_memory=True).numpy()}
    if kind == "incoherent":
        x = _samples(case, seed)
        e = pond.Incoherent(F0, case["bw"], FS, case["dm"], case["nchan"], case["nint"], case["nbins"], case["period"],
                            mode=pond.POND_INCOH_CID if case["mode"] == "cid" else pond.POND_INCOH_AID,
                            input_channels=case["ch"], ips_len=case["ips"])
        return {"case": case, "engine": e, "x": x}
    if kind == "boxcar":
        return {"case": case, "series": _series_block(case["ndm"], case["n"], seed)}
    if kind == "classify":
        series = _series_block(case["ndm"], case["n"], seed)
        return {"case": case, "series": series, "corners": _corners(case, seed),
                "net": pond.Classifier(learn.init_params(5), max_batch=case["batch"])}
    if kind == "train":
        x, y = _patch_batch(case, seed)
        return {"case": case, "x": x, "y": y, "net": pond.Classifier(learn.init_params(5), max_batch=case["batch"])}
    if kind == "stack":
        g = _gen(seed)
        return {"case": case, "series": torch.randn(case["n"], generator=g, device="cuda").mul_(3.0).add_(10.0)}
    raise ValueError(kind)


def _corners(case, seed):
    """(first trial, first sample) of each candidate's patch; a few hang over an edge of the block, as in a search."""
    r = np.random.default_rng(seed + 1)
    c = np.stack([r.integers(0, case["ndm"] - ROWS + 1, case["batch"]), r.integers(-100, case["n"] - 100, case["batch"])], 1)
    return torch.from_numpy(c.astype(np.int32)).cuda()


def _patch_batch(case, seed):
    """Normalised BF16 patches, a quarter each with a pulse, a burst, a sinusoid or noise alone, and their labels."""
    g, b = _gen(seed), case["batch"]
    y = torch.randint(0, NCLS, (b,), generator=g, device="cuda", dtype=torch.int32)
    x = torch.randn((b, ROWS, COLS), generator=g, device="cuda")
    t = torch.arange(COLS, device="cuda", dtype=torch.float32)[None, None, :]
    d = torch.arange(ROWS, device="cuda", dtype=torch.float32)[None, :, None]
    t0 = 64 + 128 * torch.rand((b, 1, 1), generator=g, device="cuda")
    w = 1 + 10 * torch.rand((b, 1, 1), generator=g, device="cuda")
    pulse = 4 * torch.exp(-((t - t0 - 2 * (d - 16)) / (w + (d - 16).abs())) ** 2)
    burst = 4 * torch.exp(-((t - t0) / w) ** 2) + 0 * d
    tone = 2 * torch.sin(t / (2 + w) + t0) * torch.exp(-((t - 128) / 80) ** 2) + 0 * d
    k = y[:, None, None]
    x = x + (k == 0) * pulse + (k == 1) * burst + (k == 2) * tone
    x = (x - x.mean((1, 2), keepdim=True)) / x.std((1, 2), keepdim=True)
    return x.to(torch.bfloat16), y


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def _candidate_table(rows):
    """The candidates (trial, index, width, S/N) in order, in a table that holds every search of these sizes."""
    where, snr = np.zeros((1024, 3), np.int64), np.zeros(1024)
    if rows:
        where[:len(rows)] = [r[:3] for r in rows]
        snr[:len(rows)] = [r[3] for r in rows]
    return {"found": len(rows), "where": where, "snr": snr}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("coherent", "batched"):
        e = state["engine"]
        e.reset()
        if case.get("host"):
            e.push(state["x"])
        else:
            e.push_tensor(state["x"])
        e.flush()
        out = {}
        if kind == "coherent":
            s, hits, _ = e.profile()
            out = {"profile": s.astype(np.float32), "hits": hits}
        n, first = e.timeseries_into(state["T"], state["C"])
        out.update(series=state["T"][..., :n], counts=state["C"][:n], first=first)
        return out
    if kind == "incoherent":
        e = state["engine"]
        e.run_tensor(state["x"])
        d, first = e.series()
        s, hits = e.profile()
        out = {"series": d, "first": first, "profile": s.astype(np.float32), "hits": hits}
        if case["ips"]:
            a, chunks = e.ips()
            out.update(spectrum=a.astype(np.float32), chunks=chunks)
        return out
    if kind == "boxcar":
        x = state["series"]
        found = pond.boxcar(x.data_ptr(), x.shape[0], x.shape[1], x.stride(0))
        return _candidate_table([(c["trial"], c["index"], c["width"], c["snr"]) for c in found])
    if kind == "classify":
        p = pond.patches(state["series"], state["corners"])
        return {"patches": p, "prob": state["net"].forward(p)}
    if kind == "train":
        loss, grad = state["net"].gradient(state["x"], state["y"])
        return {"loss": np.float32(loss), "grad": grad}
    t_ref, coef = _phase_model(case)
    mode = pond.POND_STACK_SUBINT if case["n_sub"] else pond.POND_STACK_ROTATION
    s, hits, first = pond.fold_stack(state["series"], case["g0"], case["dt"], coef, t_ref, case["nbins"], mode=mode,
                                     n_sub=case["n_sub"])
    return {"sum": s, "hits": hits, "first": first}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind in ("coherent", "batched"):
        nchan, ch = case["nchan"], case.get("ch", 1)
        logl = case["logn"] - 1
        bins = 1 << logl
        m = bins // nchan
        past, fut = _overlap(case["dm"] if kind == "coherent" else case["dm_hi"], nchan)
        kept = m - past - fut
        out = case["n"] // (2 * nchan) - past - fut
        segs = -(-out // kept)
        trials = case.get("ndm", 1)
        # transforms 5 n log2 n, real-input split 10 and chirp 6 per bin, detection 4 per channel sample
        fwd = bins * (5 * logl + 10) + (case["n"] // segs if ch == 2 else 0)
        inv = bins * (6 + 5 * (m.bit_length() - 1)) + 4 * nchan * kept
        series = _series_samples(case["n"], nchan, case["t_dec"])
        return {"bytes": case["n"] * ch + trials * series * 4 + series * 4 + 16 * case.get("nbins", 0),
                "flops": segs * (fwd + trials * inv)}
    if kind == "incoherent":
        r = 2 * case["nchan"]
        spectra = case["n"] // r
        t = spectra // case["nint"]
        per = 5 * case["nchan"] * math.log2(case["nchan"]) + 10 * case["nchan"] + 4 * case["nchan"]
        return {"bytes": case["n"] * case["ch"] + 4 * t + 16 * case["nbins"] + 4 * case["ips"],
                "flops": spectra * per * (2 if case["mode"] == "cid" else 1) + t * case["nchan"]}
    if kind == "boxcar":
        return {"bytes": 4 * case["ndm"] * case["n"], "flops": case["ndm"] * case["n"] * 7 * 5}
    conv = 2 * ROWS * ROWS * 7 * (256 + 128 + 64)      # one forward pass of the three layers
    if kind == "classify":
        return {"bytes": case["batch"] * (ROWS * COLS * (4 + 2) + 4 * NCLS) + 2 * pond.CNN_NPARAM,
                "flops": case["batch"] * (conv + 6 * ROWS * COLS)}
    if kind == "train":
        return {"bytes": case["batch"] * (ROWS * COLS * 2 + 4) + 4 * 2 * pond.CNN_NPARAM,
                "flops": case["batch"] * (conv * 3 - 2 * ROWS * ROWS * 7 * 256)}    # no gradient of the input
    rows = -(-case["n"] // case["n_sub"]) if case["n_sub"] else case["n"] * case["dt"] / case["period"] + 1
    return {"bytes": 4 * case["n"] + 16 * rows * case["nbins"], "flops": 12 * case["n"]}


# ---------------------------------------------------------------------------
# The same results in 64 bits
# ---------------------------------------------------------------------------

def exact(case, seed):
    kind = case["kind"]
    if kind in ("coherent", "batched"):
        return _exact_coherent(case, seed)
    if kind == "incoherent":
        return _exact_incoherent(case, seed)
    if kind == "boxcar":
        return _exact_boxcar(_series_block(case["ndm"], case["n"], seed).double())
    if kind == "classify":
        raw, prob = _exact_classify(case, seed)
        return {"patches": raw, "prob": prob}
    if kind == "train":
        x, y = _patch_batch(case, seed)
        theta = _network(learn.init_params(5))
        for p in theta:
            p.requires_grad_(True)
        loss = torch.nn.functional.cross_entropy(_logits(theta, x.double()), y.long())
        loss.backward()
        return {"loss": loss.detach(), "grad": torch.cat([p.grad.reshape(-1) for p in theta])}
    return _exact_stack(case, seed)


def _add_pairs(x, ch):
    return x.double() if ch == 1 else x.reshape(-1, 2).double().sum(1)


def _exact_coherent(case, seed):
    single = case["kind"] == "coherent"
    nfft, nchan, bw = 1 << case["logn"], case["nchan"], case.get("bw", BW)
    ch, n = case.get("ch", 1), case["n"]
    bins, m = nfft // 2, nfft // 2 // nchan
    dms = [case["dm"]] if single else _trial_dms(case)
    past, fut = _overlap(max(dms), nchan, bw)
    kept, end = m - past - fut, n // (2 * nchan) - fut
    x = _samples(case, seed)
    k = torch.arange(bins, dtype=torch.float64, device="cuda") * (FS / nfft * 1e-6)
    f = k - abs(bw) / 2 if bw > 0 else abs(bw) / 2 - k
    unit = K_DM * 1e6 * f * f / (F0 * F0 * (F0 + f))    # cycles per unit of DM
    sign = 1.0 if bw > 0 else -1.0
    del k, f

    def chirp(dm):
        c = unit * dm
        return torch.polar(torch.ones_like(c), (c - torch.round(c)).mul_(-2 * math.pi * sign))

    power = torch.zeros((len(dms), end - past), dtype=torch.float64, device="cuda")
    s = 0
    one = chirp(dms[0]) if len(dms) == 1 else None
    while s * kept + past < end:
        seg = torch.zeros(nfft, dtype=torch.float64, device="cuda")
        a = s * kept * 2 * nchan
        part = _add_pairs(x[a * ch:(a + nfft) * ch], ch)
        seg[:part.numel()] = part
        spec = torch.fft.rfft(seg)[:bins]
        hi = min(m - fut, end - s * kept)
        for i, dm in enumerate(dms):
            v = torch.fft.ifft((spec * (one if one is not None else chirp(dm))).reshape(nchan, m), dim=1)[:, past:hi]
            power[i, s * kept:s * kept + hi - past] = torch.view_as_real(v).square().sum((0, 2))
        s += 1
    g = torch.arange(past, end, device="cuda")
    dec = Fraction(round(case["t_dec"] * 1e9)) * Fraction(int(FS)) / (Fraction(10 ** 9) * 2 * nchan)
    j = (g * dec.denominator) // dec.numerator
    first = int(j[0])
    nj = int(j[-1]) - first + 1
    series = torch.zeros((len(dms), nj), dtype=torch.float64, device="cuda").index_add_(1, j - first, power)
    counts = torch.bincount(j - first, minlength=nj).int()
    if not single:
        return {"series": series, "counts": counts, "first": first}
    dtc = 2.0 * nchan / FS
    if case["pdot"]:
        t_ref, c = _phase_model(case)
        tau = g.double() * dtc - t_ref
        phi = (c[2] * tau + c[1]) * tau + c[0]
    else:
        phi = g.double() * (dtc / case["period"])
    b = ((phi - torch.floor(phi)) * case["nbins"]).long().clamp_(max=case["nbins"] - 1)
    prof = torch.zeros(case["nbins"], dtype=torch.float64, device="cuda").index_add_(0, b, power[0])
    return {"profile": prof, "hits": torch.bincount(b, minlength=case["nbins"]), "series": series[0], "counts": counts,
            "first": first}


def _exact_incoherent(case, seed):
    nchan, nint, ch, bw = case["nchan"], case["nint"], case["ch"], case["bw"]
    r = 2 * nchan
    x = _samples(case, seed)
    t = case["n"] // r // nint
    ts = r * nint / FS
    df = abs(bw) / nchan
    k = np.arange(nchan)
    fk = F0 - abs(bw) / 2 + k * df if bw > 0 else F0 + abs(bw) / 2 - k * df
    delay = np.floor(K_DM * case["dm"] * (fk ** -2.0 - F0 ** -2.0) / ts + 0.5).astype(np.int64)
    bank = torch.empty((t, nchan), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 25) // (r * nint))
    for a in range(0, t, step):
        c = min(step, t - a)
        y = x[a * nint * r * ch:(a + c) * nint * r * ch]
        if case["mode"] == "cid":
            y = y.reshape(-1, r, 2).double()
            p = torch.fft.rfft(y[:, :, 0])[:, :nchan]
            q = torch.fft.rfft(y[:, :, 1])[:, :nchan]
            z = p.real * q.real + p.imag * q.imag
        else:
            p = torch.fft.rfft(_add_pairs(y, ch).reshape(-1, r))[:, :nchan]
            z = p.real.square() + p.imag.square()
        bank[a:a + c] = z.reshape(c, nint, nchan).sum(1)
    first = max(0, -int(delay.min()))
    n_out = max(0, t - max(0, int(delay.max())) - first)
    d = torch.zeros(n_out, dtype=torch.float64, device="cuda")
    for c in range(nchan):
        d += bank[first + delay[c]:first + delay[c] + n_out, c]
    g = torch.arange(first, first + n_out, device="cuda").double() * (ts / case["period"])
    b = ((g - torch.floor(g)) * case["nbins"]).long().clamp_(max=case["nbins"] - 1)
    out = {"series": d, "first": first,
           "profile": torch.zeros(case["nbins"], dtype=torch.float64, device="cuda").index_add_(0, b, d),
           "hits": torch.bincount(b, minlength=case["nbins"])}
    if case["ips"]:
        n = case["ips"]
        chunks = n_out // n
        spectrum = torch.zeros(n // 2 + 1, dtype=torch.float64, device="cuda")
        if chunks:
            z = torch.fft.rfft(d[:chunks * n].reshape(chunks, n))
            spectrum = (z.real.square() + z.imag.square()).sum(0)
        out.update(spectrum=spectrum, chunks=chunks)
    return out


def _exact_boxcar(x, threshold=6.0):
    ndm, n = x.shape

    def median(v):
        v = v.sort(1).values
        return (v[:, (n - 1) // 2] + v[:, n // 2])[:, None] / 2

    mu = median(x)
    sd = 1.4826 * median((x - mu).abs())
    best = torch.full_like(x, -math.inf)
    width = torch.zeros(x.shape, dtype=torch.int64, device=x.device)
    acc, w = x.clone(), 1
    while w <= 64:
        s = (acc - w * mu) / (sd * math.sqrt(w))
        s[:, n - w + 1:] = -math.inf
        width = torch.where(s > best, w, width)
        best = torch.maximum(best, s)
        acc = acc + torch.nn.functional.pad(acc, (0, w))[:, w:]
        w *= 2
    rows = []
    for d, t in (best >= threshold).nonzero().tolist():
        w = int(width[d, t])
        near = best[max(0, d - 2):d + 3, max(0, t - w):t + w + 1]
        if float(best[d, t]) >= float(near.max()):
            rows.append((d, t, w, float(best[d, t])))
    return _candidate_table(rows)


def _network(params):
    """The layers' weights in 64 bits: convolutions and head in BF16 values, biases as they are."""
    p = torch.from_numpy(params).cuda()
    out, o = [], 0
    for shape in ((ROWS, ROWS, 7), (ROWS,), (ROWS, ROWS, 7), (ROWS,), (ROWS, ROWS, 7), (ROWS,), (NCLS, ROWS), (NCLS,)):
        q = p[o:o + math.prod(shape)].reshape(shape)
        out.append((q.to(torch.bfloat16) if len(shape) > 1 else q).double())
        o += q.numel()
    return out


class _Bf16(torch.autograd.Function):
    """Activations are held in BF16; the gradient passes through."""

    @staticmethod
    def forward(ctx, x):
        return x.float().to(torch.bfloat16).double()

    @staticmethod
    def backward(ctx, g):
        return g


def _logits(theta, x):
    f = torch.nn.functional
    for layer in range(3):
        x = torch.relu(f.conv1d(x, theta[2 * layer], theta[2 * layer + 1], padding=3))
        x = _Bf16.apply(f.max_pool1d(x, 2)) if layer < 2 else x.mean(2)
    return f.linear(x, theta[6], theta[7])


def _exact_classify(case, seed):
    series, corners = _series_block(case["ndm"], case["n"], seed), _corners(case, seed).long()
    d = (corners[:, :1] + torch.arange(ROWS, device="cuda")).clamp_(0, case["ndm"] - 1)
    t = (corners[:, 1:] + torch.arange(COLS, device="cuda")).clamp_(0, case["n"] - 1)
    v = series[d[:, :, None], t[:, None, :]].double()
    v = v - v.mean((1, 2), keepdim=True)
    v = v / v.square().mean((1, 2), keepdim=True).sqrt()
    theta = _network(learn.init_params(5))
    prob = [torch.softmax(_logits(theta, p.float().to(torch.bfloat16).double()), 1) for p in v.split(256)]
    return v, torch.cat(prob)


def _exact_stack(case, seed):
    y = prepare(case, seed)["series"].cpu().numpy().astype(np.float64)
    t_ref, c = _phase_model(case)
    tau = (np.arange(case["n"]) + case["g0"]).astype(np.float64) * case["dt"] - t_ref
    phi = (c[2] * tau + c[1]) * tau + c[0]
    q = np.floor(phi)
    b = np.minimum(((phi - q) * case["nbins"]).astype(np.int64), case["nbins"] - 1)
    row = np.arange(case["n"]) // case["n_sub"] if case["n_sub"] else (q - q[0]).astype(np.int64)
    rows = int(row[-1]) + 1
    cell = row * case["nbins"] + b
    s = np.bincount(cell, weights=y, minlength=rows * case["nbins"]).reshape(rows, case["nbins"])
    hits = np.bincount(cell, minlength=rows * case["nbins"]).reshape(rows, case["nbins"])
    return {"sum": s, "hits": hits.astype(np.int64), "first": int(q[0])}
