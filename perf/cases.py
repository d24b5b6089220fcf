"""The work that a user of this library has it do, as cases that can be timed.

Each case is a dict of plain values.  ``prepare`` makes its inputs on the GPU
and what a program keeps between calls (output buffers, the workspace, a
captured batch, a beam's state); ``run`` is one pass through the public
calls; ``exact`` restates the same outputs in plain torch in 64 bits.

The lists of records come unordered, so ``run`` does what a program that
reads them does next: it orders them by (sample, dm).  Slots past the count
are zeroed before the call and sort to the front.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1611_09704_gb300 as spd
from paper_1611_09704_gb300 import binding

DEV = "cuda:0"
_TORCH = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
_SIGMA = {"sqrtn": spd.SIGMA_SQRTN, "linear": spd.SIGMA_LINEAR,
          "excess": spd.SIGMA_LINEAR_EXCESS}


def listed():
    return [
        # The smallest call: four seconds of 64 DM trials, plain noise and a
        # pulse or two.  Launches and host time count.
        {"name": "search_64x65536_w32", "kind": "search", "n_dm": 64, "n_samp": 65536,
         "dtype": "f32", "widths": "1-32", "thr": 6.0, "sigma": "sqrtn", "scope": "global",
         "mean": 0.0, "drift": 0.0, "drift_rows": 0, "pulses": 2, "snr_max": 16.0, "cap": 4096},
        # An odd row length in a plain contiguous tensor: rows that start at
        # no 16-byte boundary; one MSD per DM row.
        {"name": "search_333x100003_rows", "kind": "search", "n_dm": 333, "n_samp": 100003,
         "dtype": "f32", "widths": "1-16,24-256/8", "thr": 7.0, "sigma": "sqrtn", "scope": "row",
         "mean": 20.0, "drift": 0.0, "drift_rows": 0, "pulses": 2, "snr_max": 16.0, "cap": 4096},
        # The full survey chunk: 33.5 s of data at 64 us in 4096 DM trials,
        # the width list of the SKA-like configuration, flat baseline.
        {"name": "search_4096x524288_w46", "kind": "search", "n_dm": 4096, "n_samp": 524288,
         "dtype": "f32", "widths": "1-16,24-256/8", "thr": 7.0, "sigma": "sqrtn",
         "scope": "global", "mean": 100.0, "drift": 0.0, "drift_rows": 0, "pulses": 2,
         "snr_max": 16.0, "cap": 4096},
        # An eighth of a chunk in which some DM rows' baselines drift by two
        # sigma, so that those rows are full of candidates.
        {"name": "search_2048x131072_drift", "kind": "search", "n_dm": 2048, "n_samp": 131072,
         "dtype": "f32", "widths": "1-16,24-256/8", "thr": 7.0, "sigma": "sqrtn",
         "scope": "global", "mean": 100.0, "drift": 2.0, "drift_rows": 4, "pulses": 2,
         "snr_max": 16.0, "cap": 262144},
        # FP16 storage with a scale per row, drifting baseline, sigma of wide
        # boxcars measured (Eq. 5): the precision configuration.
        {"name": "search_2048x524288_f16_eq5", "kind": "search", "n_dm": 2048, "n_samp": 524288,
         "dtype": "f16", "widths": "1-16,24-256/8", "thr": 7.0, "sigma": "excess",
         "scope": "global", "mean": 100.0, "drift": 2.0, "drift_rows": 2048, "pulses": 6,
         "snr_max": 150.0, "cap": 4096},
        # Four DM ranges at time decimation 1, 2, 4 and 8 and widths up to
        # 64, 128, 256 and 512 in one captured call.
        {"name": "batched_4_ranges", "kind": "batched", "n_dm": 2048, "n_samp": 524288,
         "ranges": 4, "dtype": "f32", "wmax": 64, "thr": 7.0, "pulses": 1, "snr_max": 16.0, "cap": 16384},
        # One beam of the serving configuration: two chunks, then the end of
        # the stream.
        {"name": "stream_2048x32768_f16", "kind": "stream", "n_dm": 2048, "n_samp": 32768,
         "n_samp2": 20011, "dtype": "f16", "widths": "1-128", "thr": 7.0, "pulses": 2,
         "snr_max": 16.0, "cap": 4096},
        # Widths up to 512 by decimation in time, five levels.
        {"name": "decimated_1024x262144", "kind": "decimated", "n_dm": 1024, "n_samp": 262144,
         "dtype": "f32", "levels": 5, "thr": 7.0, "pulses": 1, "snr_max": 16.0, "cap": 8192},
        # Every sample's best SNR and width, thresholded in place: the plane
        # form of the search, here with a drifting baseline.
        {"name": "plane_512x262144_w46", "kind": "plane", "n_dm": 512, "n_samp": 262144,
         "dtype": "f32", "widths": "1-16,24-256/8", "thr": 7.0, "mean": 100.0, "drift": 2.0,
         "pulses": 16},
        # Clusters in time of the candidates of an SNR plane.
        {"name": "cluster_1024x262144", "kind": "cluster", "n_dm": 1024, "n_samp": 262144,
         "gap": 32, "thr": 6.0, "bursts": 2000, "cap": 4096},
        # The producer of the plane: a filterbank de-dispersed into 256 DM
        # trials.
        {"name": "dedisperse_256x256x262144", "kind": "dedisperse", "n_chan": 256, "n_dm": 256,
         "n_out": 262144, "dm_max": 100.0, "dtype": "f32", "out": "f32"},
        # Stored in 16 bits with a scale per channel, odd sizes, and trials
        # far apart.
        {"name": "dedisperse_200x117x60001_f16", "kind": "dedisperse", "n_chan": 200,
         "n_dm": 117, "n_out": 60001, "dm_max": 300.0, "dtype": "f16", "out": "f32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "search", "batched", "stream", "decimated", "plane",
                       "cluster", "dedisperse"])
    n_samp = _log(rng, 8192, 524288)
    if rng.random() < 0.5:
        n_samp = n_samp // 8 * 8
    dtype = rng.choice(["f32", "f32", "f16", "bf16"])
    if dtype != "f32" and n_samp % 8:
        n_samp |= 1         # rows of 16-bit samples: of whole 16-byte pieces, or odd
    wmax = rng.choice([32, 64, 128, 256, 512])
    widths = rng.choice(["1-%d" % wmax, "1-16,24-%d/8" % max(64, wmax),
                         "1-32,48-%d/16" % max(64, wmax)])
    thr = rng.choice([6.0, 6.5, 7.0, 8.0])
    if kind == "search":
        n_dm = min(_log(rng, 16, 4096), (1 << (31 if len(_widths(widths)) < 130 else 30)) // n_samp)
        drifting = rng.random() < 0.25
        sigma = rng.choice(["sqrtn", "sqrtn", "linear", "excess"])
        return {"kind": kind, "n_dm": n_dm, "n_samp": n_samp, "dtype": dtype, "widths": widths,
                "thr": thr, "sigma": sigma, "scope": rng.choice(["global", "global", "row"]),
                "mean": rng.choice([0.0, 20.0, 100.0]), "drift": 2.0 if drifting else 0.0,
                # at most half of a drifting row's samples are candidates
                "drift_rows": max(1, min(4, n_dm // 16, (1 << 19) // n_samp)) if drifting else 0,
                "pulses": 2, "snr_max": 16.0 if sigma == "sqrtn" else 60.0,
                "cap": 262144 if drifting else 8192}
    if kind == "batched":
        n_dm = min(_log(rng, 16, 2048), (1 << 30) // n_samp)
        return {"kind": kind, "n_dm": n_dm, "n_samp": n_samp // 64 * 64, "ranges": rng.randint(2, 4),
                "dtype": dtype, "wmax": rng.choice([32, 64]), "thr": thr, "pulses": 1,
                "snr_max": 16.0, "cap": 16384}
    if kind == "stream":
        n1 = _log(rng, 8192, 65536)
        return {"kind": kind, "n_dm": _log(rng, 64, 2048), "n_samp": n1,
                "n_samp2": _log(rng, 4096, 32768), "dtype": dtype,
                "widths": rng.choice(["1-64", "1-128", "1-16,24-256/8"]), "thr": thr,
                "pulses": 2, "snr_max": 16.0, "cap": 8192}
    if kind == "decimated":
        n_dm = min(_log(rng, 16, 2048), (1 << 28) // n_samp)
        return {"kind": kind, "n_dm": n_dm, "n_samp": n_samp, "dtype": dtype,
                "levels": rng.randint(2, 5), "thr": thr, "pulses": 1, "snr_max": 16.0, "cap": 16384}
    if kind == "plane":
        n_dm = min(_log(rng, 16, 2048), (1 << 32) // (n_samp * len(_widths(widths))) + 1)
        return {"kind": kind, "n_dm": n_dm, "n_samp": n_samp, "dtype": dtype, "widths": widths,
                "thr": thr, "mean": rng.choice([0.0, 100.0]), "drift": rng.choice([0.0, 2.0]),
                "pulses": 8}
    if kind == "cluster":
        n_dm = min(_log(rng, 16, 4096), (1 << 28) // n_samp)
        return {"kind": kind, "n_dm": n_dm, "n_samp": n_samp, "gap": rng.choice([1, 8, 32, 200]),
                "thr": thr, "bursts": max(1, min(4000, n_dm * n_samp // 65536)), "cap": 131072}
    n_chan, n_dm = _log(rng, 32, 512), _log(rng, 16, 256)
    return {"kind": kind, "n_chan": n_chan, "n_dm": n_dm,
            "n_out": min(n_samp, (1 << 34) // (n_chan * n_dm)),
            "dm_max": rng.choice([30.0, 100.0, 300.0, 1000.0]), "dtype": dtype,
            "out": rng.choice(["f32", "f32", "f16", "bf16"])}


# ------------------------------------------------------------------- inputs

def _widths(text):
    out = []
    for part in text.split(","):
        rng, _, step = part.partition("/")
        lo, _, hi = rng.partition("-")
        out += range(int(lo), int(hi or lo) + 1, int(step or 1))
    return out


def _generator(seed, k=0):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + k) & 0x7FFFFFFF)
    return g


def _noise(n_dm, n_samp, g, mean=0.0, sd=1.0):
    x = torch.empty((n_dm, n_samp), dtype=torch.float32, device=DEV)
    x.normal_(mean, sd, generator=g)
    return x


def _add_pulses(x, n, rs, sd=1.0, snr=(8.0, 30.0)):
    """Gaussian pulses over a few adjacent DM rows, tapering to the sides."""
    n_dm, n_samp = x.shape
    for _ in range(n):
        s = rs.uniform(1.0, 100.0) / 2.3548
        rows = min(int(rs.integers(1, 9)), n_dm)
        r0, tc = int(rs.integers(0, n_dm - rows + 1)), int(rs.integers(0, n_samp))
        half = int(math.ceil(4 * s)) + 1
        t = np.arange(max(0, tc - half), min(n_samp, tc + half + 1))
        prof = np.exp(-0.5 * ((t - tc) / s) ** 2)
        amp = rs.uniform(*snr) * sd / math.sqrt(float(np.sum(prof * prof)))
        taper = 1.0 - 0.5 * np.abs(np.arange(rows) - (rows - 1) / 2) / max(1, rows)
        p = torch.from_numpy((amp * taper[:, None] * prof[None, :]).astype(np.float32)).to(DEV)
        x[r0:r0 + rows, int(t[0]):int(t[-1]) + 1] += p


def _add_drift(x, amp, rows, g):
    """A slow sinusoid of period 65536 samples on every (n_dm // rows)-th row."""
    n_dm, n_samp = x.shape
    at = torch.arange(rows, device=DEV) * (n_dm // rows)
    ph = torch.rand(rows, generator=g, device=DEV) * (2 * math.pi)
    t = torch.arange(n_samp, device=DEV, dtype=torch.float32) * (2 * math.pi / 65536)
    for r0 in range(0, rows, 256):
        x[at[r0:r0 + 256]] += amp * torch.sin(t[None, :] + ph[r0:r0 + 256, None])


def _store(x, dtype):
    """(stored tensor, scale per row or None)."""
    if dtype == "f32":
        return x, None
    scale = torch.empty(x.shape[0], dtype=torch.float32, device=DEV)
    q = torch.empty(x.shape, dtype=_TORCH[dtype], device=DEV)
    for r0 in range(0, x.shape[0], 256):
        b = x[r0:r0 + 256]
        s = (b.abs().amax(dim=1) / 16384.0).clamp_min(1e-30)
        scale[r0:r0 + 256] = s
        q[r0:r0 + 256] = (b / s[:, None]).to(_TORCH[dtype])
    return q, scale


def _plane(case, seed, k=0, n_dm=None, n_samp=None):
    """Noise, drift and pulses, as stored."""
    n_dm, n_samp = n_dm or case["n_dm"], n_samp or case["n_samp"]
    mean = case.get("mean", 0.0)
    sd = 12.0 if mean else 1.0
    g = _generator(seed, k)
    x = _noise(n_dm, n_samp, g, mean, sd)
    if case.get("drift"):
        _add_drift(x, case["drift"] * sd, case.get("drift_rows") or n_dm, g)
    _add_pulses(x, case["pulses"], np.random.default_rng([int(seed), k, 7]), sd,
                (8.0, case.get("snr_max", 30.0)))
    return _store(x, case["dtype"])


def _ranges(case, seed):
    """The DM ranges of a batched search: fewer trials and fewer, longer
    samples from one to the next.  [(data, scale, widths, decimation)]"""
    out = []
    for k in range(case["ranges"]):
        n_dm = max(1, case["n_dm"] * (4 - k) // 4)
        x, sc = _plane(case, seed, k, n_dm, max(64, case["n_samp"] >> k))
        out.append((x, sc, list(range(1, (case["wmax"] << k) + 1)), 1 << k))
    return out


def _levels(case):
    return [(0, list(range(1, 33)))] + [(l, list(range(17, 33))) for l in range(1, case["levels"])]


def _chunks(case, seed):
    g = _generator(seed)
    n1, n2 = case["n_samp"], case["n_samp2"]
    x = _noise(case["n_dm"], n1 + n2, g)
    _add_pulses(x, case["pulses"], np.random.default_rng([int(seed), 0, 7]))
    x = x.to(_TORCH[case["dtype"]])
    return x, [x[:, :n1].contiguous(), x[:, n1:].contiguous()]


def _snr_plane(case, seed):
    """A best-SNR plane as the plane form writes it: most samples low, bursts
    of high ones, and the widths."""
    n_dm, n_samp = case["n_dm"], case["n_samp"]
    g = _generator(seed)
    snr = _noise(n_dm, n_samp, g, 2.0, 0.7)
    n = case["bursts"]
    row = torch.randint(0, n_dm, (n,), generator=g, device=DEV)
    t0 = torch.randint(0, n_samp, (n,), generator=g, device=DEV)
    ln = torch.randint(1, 300, (n,), generator=g, device=DEV)
    t = torch.arange(300, device=DEV)
    on = (t[None, :] < ln[:, None]) & (t0[:, None] + t[None, :] < n_samp)
    at = (row * n_samp + t0)[:, None] + t[None, :]
    snr.view(-1)[at[on]] += 7.0
    width = torch.randint(1, 257, (n_dm, n_samp), generator=g, device=DEV, dtype=torch.int16)
    return snr, width


def _delays(case):
    """Cold-plasma delays of channels from 1500 down to 1200 MHz at 64 us."""
    f = np.linspace(1500.0, 1200.0, case["n_chan"])
    dm = np.linspace(0.0, case["dm_max"], case["n_dm"])[:, None]
    return np.rint(4148.808 * dm * (f[None, :] ** -2 - 1500.0 ** -2) / 64e-6).astype(np.int32)


def _filterbank(case, seed):
    d = _delays(case)
    g = _generator(seed)
    x = _noise(case["n_chan"], case["n_out"] + int(d.max()), g)
    rs = np.random.default_rng([int(seed), 7])
    for _ in range(3):
        k, t0 = int(rs.integers(0, case["n_dm"])), int(rs.integers(0, case["n_out"]))
        w = int(rs.integers(1, 33))
        for c in range(case["n_chan"]):
            x[c, t0 + int(d[k, c]):t0 + int(d[k, c]) + w] += 0.8
    q, sc = _store(x, case["dtype"])
    return q, sc, torch.from_numpy(d).to(DEV)


# ---------------------------------------------------------------- the calls

def _records(cap):
    return torch.zeros((cap, 4), dtype=torch.int32, device=DEV)


def _result():
    return torch.zeros(binding.RESULT_BYTES, dtype=torch.uint8, device=DEV)


def _bytes(n):
    return torch.empty(max(int(n), 1), dtype=torch.uint8, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind, "case": case}
    if kind == "search":
        x, sc = _plane(case, seed)
        st["x"] = spd.Plane(x, scale=sc)
        scope = spd.MSD_PER_ROW if case["scope"] == "row" else spd.MSD_GLOBAL
        st["args"] = (_widths(case["widths"]), case["thr"], case["cap"], _SIGMA[case["sigma"]],
                      scope)
        st["out"], st["result"] = _records(case["cap"]), _result()
        st["msd"] = _bytes(binding.MSD_BYTES * (case["n_dm"] if case["scope"] == "row" else 1))
        st["ws"] = _bytes(binding.search_workspace_bytes(
            st["x"], st["args"][0], case["thr"], _SIGMA[case["sigma"]], scope))
    elif kind == "batched":
        specs = [spd.RangeSpec(spd.Plane(x, scale=sc), w, case["thr"], decimation=dec,
                               dm_offset=case["n_dm"] * k)
                 for k, (x, sc, w, dec) in enumerate(_ranges(case, seed))]
        st["batch"] = spd.BatchedSearch(specs, case["cap"])
    elif kind == "stream":
        st["chunks"] = _chunks(case, seed)[1]
        st["beam"] = binding.BeamStream(case["n_dm"], _TORCH[case["dtype"]],
                                        _widths(case["widths"]), case["thr"], device=DEV)
        st["out"] = _records(3 * case["cap"])
        st["results"] = [_result() for _ in range(3)]
        st["msd"] = _bytes(binding.MSD_BYTES)
        st["ws"] = _bytes(st["beam"].workspace_bytes(max(case["n_samp"], case["n_samp2"])))
    elif kind == "decimated":
        x, sc = _plane(case, seed)
        st["x"], st["levels"] = spd.Plane(x, scale=sc), _levels(case)
        st["out"], st["result"] = _records(case["cap"]), _result()
        st["msd"] = _bytes(binding.MSD_BYTES * case["levels"])
        st["ws"] = _bytes(binding.search_decimated_workspace_bytes(st["x"], st["levels"]))
    elif kind == "plane":
        x, sc = _plane(case, seed)
        st["x"], st["widths"] = spd.Plane(x, scale=sc), _widths(case["widths"])
        st["msd"] = _bytes(binding.MSD_BYTES)
        st["snr"] = torch.empty(x.shape, dtype=torch.float32, device=DEV)
        st["width"] = torch.empty(x.shape, dtype=torch.int16, device=DEV)
    elif kind == "cluster":
        st["snr"], st["width"] = _snr_plane(case, seed)
        st["out"] = torch.zeros((case["cap"], 8), dtype=torch.int32, device=DEV)
        st["result"] = _result()
    else:
        x, sc, st["delays"] = _filterbank(case, seed)
        st["x"] = spd.Plane(x, scale=sc)
        st["out"] = torch.empty((case["n_dm"], case["n_out"]), dtype=_TORCH[case["out"]],
                                device=DEV)
        st["result"] = _result()
    # the outcome and the statistics as a program reads them: views of the
    # buffers that the calls fill
    if kind == "batched":
        st["views"] = {**_outcome(st["batch"].result), **_stats(st["batch"].msd)}
    elif kind == "stream":
        st["views"] = {"outcome": [_outcome(r) for r in st["results"]], **_stats(st["msd"])}
    else:
        st["views"] = {**(_outcome(st["result"]) if "result" in st else {}),
                       **(_stats(st["msd"]) if "msd" in st else {})}
    return st


def _ordered(out, twice=False):
    """The records by (sample, dm): the first two words of a record as one
    number; `twice`: then by width, where a start may have several."""
    rec = out.view(torch.int64)
    key = rec[:, 0]
    if twice:    # sample, then dm (below 2^19) and width (below 2^12) in one word
        key = key + (key & 0xFFFFFFFF) * 4095 + (rec[:, 1] >> 32)
    rec = rec[key.sort().indices]
    ints = rec.view(torch.int32)
    return {"at": ints[:, :2], "snr": rec.view(torch.float32)[:, 2], "width": ints[:, 3]}


def _outcome(result):
    """Views of a result word: the count and the status."""
    return {"count": result[:8].view(torch.int64), "status": result[8:12].view(torch.int32)}


def _stats(msd):
    """Views of the MSD entries: mean, sd, sd_nmax and the counts of each."""
    return {"msd": msd.view(torch.float64).view(-1, 5)[:, :3],
            "n": msd.view(torch.int64).view(-1, 5)[:, 3],
            "nmax": msd.view(torch.int32).view(-1, 10)[:, 8:]}


def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "search":
        st["out"].zero_()
        spd.search(st["x"], *st["args"], out=st["out"], result=st["result"], msd_out=st["msd"],
                   workspace=st["ws"])
        return {**_ordered(st["out"]), **st["views"]}
    if kind == "batched":
        st["batch"].out.zero_()
        st["batch"].run()
        return {**_ordered(st["batch"].out), **st["views"]}
    if kind == "stream":
        beam, cap = st["beam"], case["cap"]
        st["out"].zero_()
        beam.reset()
        for k, chunk in enumerate(st["chunks"]):
            beam.push(chunk, st["out"][k * cap:(k + 1) * cap], cap, st["results"][k], st["ws"],
                      msd_out=st["msd"])
        beam.flush(st["out"][2 * cap:], cap, st["results"][2], st["ws"])
        return {**_ordered(st["out"]), **st["views"]}
    if kind == "decimated":
        st["out"].zero_()
        spd.search_decimated(st["x"], st["levels"], case["thr"], case["cap"], out=st["out"],
                             result=st["result"], msd_out=st["msd"], workspace=st["ws"])
        return {**_ordered(st["out"], True), **st["views"]}
    if kind == "plane":
        spd.msd(st["x"], out=st["msd"])
        spd.boxcar_snr(st["x"], st["msd"], st["widths"], snr_out=st["snr"],
                       width_out=st["width"])
        spd.threshold_plane(st["snr"], st["width"], case["thr"])
        return {"snr": st["snr"], "width": st["width"], **st["views"]}
    if kind == "cluster":
        st["out"].zero_()
        spd.cluster_rows(st["snr"], st["width"], case["thr"], case["gap"], case["cap"],
                         out=st["out"], result=st["result"])
        key = st["out"].view(torch.int64)[:, 0]     # (first sample, dm)
        rec = st["out"][key.sort().indices]
        return {"ints": rec[:, :4], "peak": rec.view(torch.float32)[:, 4], "more": rec[:, 5:7],
                **st["views"]}
    out = spd.dedisperse(st["x"], st["delays"], case["n_out"], out=st["out"],
                         status=st["result"])
    return {"plane": out}


def work(case):
    kind = case["kind"]
    b = {"f32": 4, "f16": 2, "bf16": 2}[case.get("dtype", "f32")]
    n = case.get("n_dm", 0) * case.get("n_samp", 0)
    if kind == "batched":
        n = sum(max(1, case["n_dm"] * (4 - k) // 4) * max(64, case["n_samp"] >> k)
                for k in range(case["ranges"]))
    if kind in ("search", "batched", "decimated"):
        # the statistics need the whole plane before the search can start
        return {"bytes": 2 * n * b, "flops": 8 * n}
    if kind == "stream":
        n = case["n_dm"] * (case["n_samp"] + case["n_samp2"])
        return {"bytes": 2 * n * b, "flops": 8 * n}
    if kind == "plane":
        # an add, a multiply and a max for each width and sample
        return {"bytes": 2 * n * b + 6 * n, "flops": 3 * len(_widths(case["widths"])) * n}
    if kind == "cluster":
        return {"bytes": 6 * n, "flops": n}
    out = case["n_dm"] * case["n_out"]
    return {"bytes": case["n_chan"] * case["n_out"] * b
            + out * {"f32": 4, "f16": 2, "bf16": 2}[case["out"]],
            "flops": case["n_chan"] * out}


# ------------------------------------------------------------ in 64 bits

def _values(x, sc, rows):
    v = x[rows].double()
    return v if sc is None else v * sc[rows].double()[:, None]


def _moments(x, sc, row_scope=False):
    """(mean, population sd) of the plane, or of each row."""
    n_dm, n = x.shape
    s = torch.zeros(n_dm, dtype=torch.float64, device=DEV)
    blocks = [slice(r, r + 64) for r in range(0, n_dm, 64)]
    for r in blocks:
        s[r] = _values(x, sc, r).sum(dim=1)
    mean = s / n if row_scope else (s.sum() / (n * n_dm)).expand(n_dm)
    q = torch.zeros(n_dm, dtype=torch.float64, device=DEV)
    for r in blocks:
        q[r] = (_values(x, sc, r) - mean[r, None]).square().sum(dim=1)
    var = q / n if row_scope else (q.sum() / (n * n_dm)).expand(n_dm)
    return mean, var.sqrt()


def _sd_nmax(x, sc, mean, nmax, row_scope):
    """The sd of the sums over nmax samples, pooled over the scope."""
    n_dm, n = x.shape
    k = n - nmax + 1
    t = torch.zeros(n_dm, dtype=torch.float64, device=DEV)
    q = torch.zeros(n_dm, dtype=torch.float64, device=DEV)
    if k < 1:
        return t
    for r0 in range(0, n_dm, 64):
        r = slice(r0, r0 + 64)
        c = torch.nn.functional.pad(_values(x, sc, r) - mean[r, None], (1, 0)).cumsum(1)
        b = c[:, nmax:] - c[:, :-nmax]
        t[r], q[r] = b.sum(dim=1), b.square().sum(dim=1)
    if row_scope:
        return (q / k - (t / k).square()).clamp_min(0).sqrt()
    m = t.sum() / (k * n_dm)
    return (q.sum() / (k * n_dm) - m * m).clamp_min(0).sqrt().expand(n_dm)


def _best(y, sig, widths):
    """Per start the highest SNR over the widths that fit; y: centred rows;
    sig: one sd of a boxcar per width, each a number or one per row."""
    n = y.shape[1]
    c = torch.nn.functional.pad(y, (1, 0)).cumsum(1)
    best = torch.full_like(y, -math.inf)
    for w, s in zip(widths, sig):
        if w > n:
            break
        v = (c[:, w:] - c[:, :n + 1 - w]) / s
        torch.maximum(best[:, :n + 1 - w], v, out=best[:, :n + 1 - w])
    return best


def _sigmas(widths, sd, sd_nmax, mode):
    out = []
    nm = widths[-1]
    for w in widths:
        s = math.sqrt(w) * sd
        if mode == "linear":
            s = s + (w - 1) * sd_nmax / (nm - 1)
        elif mode == "excess":
            s = s + (w - 1) * (sd_nmax - math.sqrt(nm) * sd) / (nm - 1)
        out.append(s)
    return out


def _found(best, thr, row0, found, base=0, shift=0):
    """Collects (sample, dm, snr) of best >= thr; False where a best is too
    near the threshold for the list to be defined at rounding level."""
    at = (best >= thr).nonzero()
    if bool(((best - thr).abs() < 2e-6 * thr).any()):
        return False
    found.append(torch.stack([((at[:, 1] + base) << shift).double(), (at[:, 0] + row0).double(),
                              best[at[:, 0], at[:, 1]]], dim=1))
    return True


def _listing(found, cap):
    """The SNRs as _ordered() lays them out; None where the list overflows."""
    rec = torch.cat(found)
    if rec.shape[0] > cap:
        return None
    # `found` holds the narrower widths of a start first
    order = (rec[:, 0].long() * (1 << 31) + rec[:, 1].long()).sort(stable=True).indices
    return torch.cat([torch.zeros(cap - rec.shape[0], dtype=torch.float64, device=DEV),
                      rec[order, 2]])


def _search64(x, sc, widths, thr, mode="sqrtn", row_scope=False, shift=0, evaluated=None):
    """(found or None, mean, sd, sd_nmax) of one plane."""
    mean, sd = _moments(x, sc, row_scope)
    snm = (_sd_nmax(x, sc, mean, widths[-1], row_scope) if mode != "sqrtn"
           else torch.zeros_like(sd))
    ev = evaluated or ([] if widths[0] == 1 else [1]) + widths
    found = []
    for r0 in range(0, x.shape[0], 64):
        r = slice(r0, r0 + 64)
        sig = _sigmas(widths, sd[r, None], snm[r, None], mode)
        sig = ([sd[r, None]] if len(ev) > len(widths) else []) + sig
        if not _found(_best(_values(x, sc, r) - mean[r, None], sig, ev), thr, r0, found,
                      shift=shift):
            return None, mean, sd, snm
    return found, mean, sd, snm


def exact(case, seed):
    kind = case["kind"]
    none = {"at": None, "width": None, "count": None, "status": None, "n": None, "nmax": None}
    if kind == "search":
        x, sc = _plane(case, seed)
        rows = case["scope"] == "row"
        found, mean, sd, snm = _search64(x, sc, _widths(case["widths"]), case["thr"],
                                         case["sigma"], rows)
        msd = torch.stack([mean, sd, snm], dim=1)
        return {**none, "snr": _listing(found, case["cap"]) if found else None,
                "msd": msd if rows else msd[:1]}
    if kind == "batched":
        found, msd = [], []
        for k, (x, sc, w, _) in enumerate(_ranges(case, seed)):
            f, mean, sd, snm = _search64(x, sc, w, case["thr"])
            msd.append(torch.stack([mean, sd, snm], dim=1)[:1])
            if f is None or found is None:
                found = None
            else:
                for rec in f:
                    rec[:, 1] += case["n_dm"] * k
                found += f
        return {**none, "snr": _listing(found, case["cap"]) if found else None,
                "msd": torch.cat(msd)}
    if kind == "decimated":
        x, sc = _plane(case, seed)
        found, msd = [], []
        for level, w in _levels(case):
            n = x.shape[1] >> level
            y, ysc = x, sc
            if level:
                y = torch.empty((x.shape[0], n), dtype=torch.float64, device=DEV)
                for r0 in range(0, x.shape[0], 64):
                    r = slice(r0, r0 + 64)
                    v = _values(x, sc, r)[:, :n << level]
                    y[r] = v.reshape(v.shape[0], n, 1 << level).sum(dim=2)
                ysc = None
            f, mean, sd, snm = _search64(y, ysc, w, case["thr"], shift=level, evaluated=w)
            msd.append(torch.stack([mean, sd, snm], dim=1)[:1])
            if f is None or found is None:
                found = None
            else:
                found += f
        return {**none, "snr": _listing(found, case["cap"]) if found else None,
                "msd": torch.cat(msd)}
    if kind == "stream":
        x, chunks = _chunks(case, seed)
        w = _widths(case["widths"])
        ev = ([] if w[0] == 1 else [1]) + w
        n1, hold = chunks[0].shape[1], w[-1] - 1
        cut = max(0, n1 - hold)
        found = []
        for part, base, last in ((chunks[0], 0, cut), (x, cut, x.shape[1])):
            mean, sd = _moments(part, None)
            for r0 in range(0, x.shape[0], 64):
                r = slice(r0, r0 + 64)
                y = part[r, base:].double() - mean[r, None]
                b = _best(y, [math.sqrt(v) * sd[r, None] for v in ev], ev)[:, :last - base]
                if found is not None and not _found(b, case["thr"], r0, found, base=base):
                    found = None
        msd = torch.stack([mean, sd, torch.zeros_like(sd)], dim=1)[:1]
        return {"at": None, "width": None, "outcome": None, "n": None, "nmax": None,
                "snr": _listing(found, 3 * case["cap"]) if found else None, "msd": msd}
    if kind == "plane":
        x, sc = _plane(case, seed)
        w = _widths(case["widths"])
        mean, sd = _moments(x, sc)
        snr = torch.empty(x.shape, dtype=torch.float64, device=DEV)
        for r0 in range(0, x.shape[0], 64):
            r = slice(r0, r0 + 64)
            b = _best(_values(x, sc, r) - mean[r, None], [math.sqrt(v) * sd[r, None] for v in w],
                      w)
            snr[r] = torch.where(b >= case["thr"], b, 0.0)
        msd = torch.stack([mean, sd, torch.zeros_like(sd)], dim=1)[:1]
        return {"snr": snr, "width": None, "msd": msd, "n": None, "nmax": None}
    if kind == "cluster":
        return None      # chosen from the inputs: nothing is computed in floating point
    x, sc, delays = _filterbank(case, seed)
    d = delays.cpu().numpy()
    out = torch.zeros((case["n_dm"], case["n_out"]), dtype=torch.float64, device=DEV)
    for c in range(case["n_chan"]):
        v = _values(x, sc, slice(c, c + 1))[0]
        for k in range(case["n_dm"]):
            out[k] += v[d[k, c]:d[k, c] + case["n_out"]]
    return {"plane": out}
