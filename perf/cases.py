"""Performance cases: what programs built on this framework spend their time on.

A case is one call (or one short burst of calls) of the public Python
interface.  The workloads are the framework's own (configs.py); the databases
of the two largest are built from fewer proteins where noted, which changes
how many peptides a precursor window holds but not how many index entries one
peptide adds, so the work per searched peptide is the workload's own.
"""
from __future__ import annotations

import dataclasses
import functools
import math

import numpy as np
import torch

from paper_2102_02286_gb300 import configs, synth
from paper_2102_02286_gb300 import hicops as hc

SAMPLES = 120          # bins of a sampled partial distribution (the library's default)
WATER, PROTON = 18.010565, 1.007276466812

# What a kind of case stands for, its workload, its proteins, the entry point
# and the range of spectra it is drawn from.
KINDS = {
    # a small closed search, every spectrum of a run in one call: launch latency
    "closed_tiny": dict(workload="tiny_closed", proteins=500, entry="device", lo=1, hi=2000),
    # an interactive open search of a few spectra that must not allocate
    "open_few": dict(workload="open_medium", proteins=20_000, entry="noalloc", lo=1, hi=64),
    # the open search of a run: the library's headline workload
    "open_batch": dict(workload="open_medium", proteins=20_000, entry="device", lo=500, hi=30_000),
    # a closed search of a modified database from and to host arrays
    "closed_host": dict(workload="open_medium", proteins=20_000, entry="host", lo=100, hi=4000, tol=10.0),
    # spectra of 50-500 peaks under mixed tolerances, a plan replayed as a graph
    "uneven_plan": dict(workload="uneven_batched", proteins=20_000, entry="plan", lo=200, hi=12_345),
    # the heavily modified database: charges 2-4, 150 peaks, top-10
    "open_dense": dict(workload="open_large", proteins=2_500, entry="device", lo=100, hi=6000),
    # fragment tolerance of one bin on the finer grid: 300 query bins a spectrum, in caller scratch
    "open_tol": dict(workload="open_medium_tol", proteins=20_000, entry="scratch", lo=100, hi=5000),
}


def listed():
    return [
        # one run's 1,000 spectra against an unmodified database, +-10 Da
        {"name": "closed_tiny_1000", "kind": "closed_tiny", "n": 1000, "proteins": 500},
        # the smallest call: one spectrum, +-500 Da
        {"name": "open_few_1", "kind": "open_few", "n": 1, "proteins": 20_000},
        # a handful of spectra, an odd number of them
        {"name": "open_few_37", "kind": "open_few", "n": 37, "proteins": 20_000},
        # a fraction of a run, less than fills the chip evenly
        {"name": "open_batch_1111", "kind": "open_batch", "n": 1111, "proteins": 20_000},
        # a run's spectra in one call
        {"name": "open_batch_30000", "kind": "open_batch", "n": 30_000, "proteins": 20_000},
        # what a search program with host arrays sees of a closed search
        {"name": "closed_host_2500", "kind": "closed_host", "n": 2500, "proteins": 20_000},
        # uneven spectra and tolerances in one graph replay
        {"name": "uneven_plan_12345", "kind": "uneven_plan", "n": 12_345, "proteins": 20_000},
        # a batch against the heavily modified database
        {"name": "open_dense_6000", "kind": "open_dense", "n": 6000, "proteins": 2_500},
        # fragment tolerance of one bin
        {"name": "open_tol_5000", "kind": "open_tol", "n": 5000, "proteins": 20_000},
        # a burst of requests of 1-512 spectra waiting at the server
        {"name": "serving_24", "kind": "serving", "requests": 24, "proteins": 2_500},
        # assembling eight ranks' partial results, their distributions sampled
        {"name": "merge_8x20000", "kind": "merge", "shards": 8, "n": 20_000, "top_k": 5, "s": SAMPLES},
        # a rank builds its eighth of the database and searches a first batch
        {"name": "shard_build_8", "kind": "shard_build", "shards": 8, "n": 64, "proteins": 20_000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(sorted(KINDS) + ["serving", "merge", "shard_build"])
    if kind == "serving":
        return {"kind": kind, "requests": rng.randint(3, 24), "proteins": 2_500}
    if kind == "merge":
        return {"kind": kind, "shards": rng.randint(2, 8), "n": _log(rng, 1000, 20_000), "top_k": rng.choice([5, 10]),
                "s": rng.choice([SAMPLES, rng.randint(16, SAMPLES)])}
    if kind == "shard_build":
        return {"kind": kind, "shards": rng.randint(8, 32), "n": rng.randint(16, 64), "proteins": 20_000}
    k = KINDS[kind]
    proteins = rng.randint(100, k["proteins"]) if kind == "closed_tiny" else k["proteins"]
    return {"kind": kind, "n": _log(rng, k["lo"], k["hi"]), "proteins": proteins}


# ---- inputs


def _workload(case):
    kind = case["kind"]
    name = {"serving": "serving_stream", "shard_build": "open_medium"}.get(kind) or KINDS[kind]["workload"]
    w = configs.BY_NAME[name].with_proteins(case["proteins"])
    tol = KINDS.get(kind, {}).get("tol")
    return w if tol is None else dataclasses.replace(w, spectra=dataclasses.replace(w.spectra, tol_da=(tol,)))


@functools.lru_cache(maxsize=4)
def _proteome(proteins, seed, length):
    return synth.make_proteome(proteins, seed, length)


@functools.lru_cache(maxsize=6)
def _index(proteins, seed, length, mods, params, upload=True):
    """The resident index a program builds once for its database."""
    prot = _proteome(proteins, seed, length)
    return hc.Index(prot.seq, prot.off, mods, params, upload=upload)


def _resident(w, upload=True):
    return _index(w.n_proteins, w.db_seed, w.protein_len, w.mods, w.params, upload)


def _spectra(w, n, seed):
    return synth.make_spectra(_proteome(w.n_proteins, w.db_seed, w.protein_len), w, n, seed=seed)


def _columns(psm, hist, n_scored):
    """The rows' fields as arrays (views of the buffers) beside the other outputs."""
    if isinstance(psm, np.ndarray):
        out = {f: psm[f] for f in ("query", "pid", "nb", "ny", "key", "hyperscore", "evalue")}
    else:
        i32 = psm.view(torch.int32).view(-1, 8)
        by = psm.view(-1, 32)
        out = {"query": i32[:, 0], "pid": i32[:, 1], "nb": by[:, 8], "ny": by[:, 9],
               "hyperscore": psm.view(torch.float32).view(-1, 8)[:, 3], "key": psm.view(torch.int64).view(-1, 4)[:, 2],
               "evalue": psm.view(torch.float64).view(-1, 4)[:, 3]}
    out["hist"], out["n_scored"] = hist, n_scored
    return out


def _partials(case, seed):
    """Partial results of a sharded search: each shard's rows in rank order
    (key descending, peptide ascending, the shard's own peptides, padding rows
    last) and its score distribution, a rising flank and a geometric tail."""
    rng = np.random.default_rng([seed, 7])
    S, n, k = case["shards"], case["n"], case["top_k"]
    psm = np.zeros((S, n, k), hc.PSM_DTYPE)
    psm["query"] = np.arange(n, dtype=np.uint32)[None, :, None]
    key = np.sort(rng.integers(12 << 32, 30 << 32, (S, n, k)), axis=2)[:, :, ::-1]
    pid = rng.integers(0, 1 << 20, (S, n, k)).astype(np.uint32) * np.uint32(S) + np.arange(S, dtype=np.uint32)[:, None, None]
    pad = np.arange(k)[None, None, :] >= rng.binomial(k, 0.97, (S, n, 1))
    psm["pid"] = np.where(pad, 0xFFFFFFFF, pid)
    psm["key"] = np.where(pad, np.iinfo(np.int64).min, key)
    psm["nb"] = np.where(pad, 0, rng.integers(1, 30, (S, n, k)))
    psm["ny"] = np.where(pad, 0, rng.integers(3, 30, (S, n, k)))
    psm["hyperscore"] = np.where(pad, 0.0, key * 2.0 ** -32)
    psm["evalue"] = np.where(pad, np.inf, 1.0)
    hist = np.zeros((S, n, 256), np.uint32)
    bins = np.arange(16, 60)
    mean = 400.0 * np.minimum(1.0, (bins - 14) / 8.0) * np.exp(-np.maximum(bins - 24, 0) / 3.0)
    hist[:, :, 16:60] = rng.poisson(mean[None, None, :] * rng.uniform(0.1, 1.0, (S, n, 1)))
    return psm, hist, hist.sum(2, dtype=np.uint32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "merge":
        psm, hist, ns = _partials(case, seed)
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
        return {"case": case, "psm": dev(psm.view(np.uint8).reshape(-1)), "hist": dev(hist.view(np.int32).reshape(-1)),
                "ns": dev(ns.view(np.int32).reshape(-1))}
    w = _workload(case)
    if kind == "serving":
        rng = np.random.default_rng(case["requests"])    # the burst's request sizes are the case's
        sizes = np.clip(np.exp(rng.uniform(0.0, math.log(513), case["requests"])).astype(np.int64), 1, 512)
        spec = _spectra(w, int(sizes.sum()), seed)
        ends = np.cumsum(sizes)
        return {"case": case, "requests": [spec.subset(np.arange(e - s, e)) for s, e in zip(sizes, ends)],
                "server": hc.Server(_resident(w), memory_budget=2 << 30)}
    spec = _spectra(w, case["n"], seed)
    if kind == "shard_build":
        # the digested database is on the host; the spectra are on the device
        return {"case": case, "base": _resident(w, upload=False), "rank": seed % case["shards"],
                "batch": hc.DeviceBatch.from_spectra(spec), "k": w.params.top_k}
    state = {"case": case, "entry": KINDS[kind]["entry"], "index": _resident(w), "n": case["n"]}
    if state["entry"] == "host":
        n, k = case["n"], w.params.top_k
        state["spec"] = spec
        state["out"] = hc.SearchResult(np.zeros((n, k), hc.PSM_DTYPE), np.zeros((n, hc.HIST_BINS), np.uint32),
                                       np.zeros(n, np.uint32))
        return state
    state["batch"] = hc.DeviceBatch.from_spectra(spec)
    state["out"] = o = hc.DeviceResult.alloc(case["n"], w.params.top_k)
    state["columns"] = _columns(o.psm, o.hist, o.n_scored)
    if state["entry"] == "plan":
        state["plan"] = state["index"].plan(case["n"])
        state["stream"] = torch.cuda.Stream()    # graphs are captured on a stream of the program's own
    elif state["entry"] == "scratch":
        nbytes = state["index"].search_scratch_bytes(case["n"])
        state["scratch"] = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    return state


def run(state):
    kind = state["case"]["kind"]
    if kind == "merge":
        c = state["case"]
        rec = hc.hist_sample(state["hist"], c["s"])
        hist = hc.hist_unsample(c["shards"], c["n"], rec, c["s"])
        ns = state["ns"].view(c["shards"], c["n"]).sum(0, dtype=torch.int32)
        out = hc.merge_shards(c["shards"], c["n"], c["top_k"], state["psm"], hist, ns, 1)
        return {**_columns(out.psm, out.hist, out.n_scored), "records": rec}
    if kind == "serving":
        srv = state["server"]
        tickets = [srv.submit(r) for r in state["requests"]]
        got = [srv.poll(t) for t in tickets]
        return _columns(*(np.concatenate([getattr(g, f) for g in got]) for f in ("psm", "hist", "n_scored")))
    if kind == "shard_build":
        part = state["base"].shard(state["case"]["shards"], state["rank"])
        out = hc.DeviceResult.alloc(state["batch"].n, state["k"])
        part.search_device(state["batch"], out)
        return _columns(out.psm, out.hist, out.n_scored)
    idx, entry, out = state["index"], state["entry"], state["out"]
    if entry == "host":
        idx.search(state["spec"], out)
        return _columns(out.psm, out.hist, out.n_scored)
    if entry == "plan":
        state["plan"].search(state["batch"], out, state["stream"])
    elif entry == "noalloc":
        idx.search_noalloc(state["batch"], out)
    elif entry == "scratch":
        idx.search_scratch(state["batch"], out, state["scratch"])
    else:
        idx.search_device(state["batch"], out)
    return state["columns"]


# ---- the work a pass cannot do without

# peptides a protein, index entries a peptide, entries of one query bin's
# bucket per peptide of the window (common fragments included), fraction of
# the database in a +-500 Da window: measured on the workloads' databases
_DB = {"tiny_closed": (62, 25.9, 4.0e-3), "open_medium": (652, 30.7, 2.3e-3), "uneven_batched": (652, 30.7, 2.3e-3),
       "open_medium_tol": (652, 30.7, 1.2e-3), "open_large": (4700, 32.2, 1.7e-3), "serving_stream": (4700, 32.2, 1.7e-3)}
_WINDOW = {10.0: 0.006, 100.0: 0.06, 500.0: 0.25}


def work(case):
    """Peaks, precursors and the index read once, rows and distributions
    written once.  The index is read once at most: the entries of the query
    bins' buckets inside the windows, or all of it where the spectra of a
    batch together need more than that.  One operation an entry in a window
    (the shared-peak count) and one an output value."""
    kind = case["kind"]
    if kind == "merge":
        n, S, k = case["n"], case["shards"], case["top_k"]
        read = S * n * (k * 32 + 1024 + 4)
        return {"bytes": read + n * (k * 32 + 1024 + 4) + 4 * S * n * (case["s"] + 1), "flops": S * n * (256 + k)}
    w = _workload(case)
    p, rec = w.params, w.spectra
    n = 82 * case["requests"] if kind == "serving" else case["n"]
    raw = sum(rec.target_peaks) / 2 if rec.target_peaks else 95
    bins = min(raw, p.top_n_peaks) * (2 * p.tol_bins + 1)
    per_protein, per_peptide, density = _DB[w.name]
    P = w.n_proteins * per_protein / (case["shards"] if kind == "shard_build" else 1)
    window = P * sum(_WINDOW[t] for t in rec.tol_da) / len(rec.tol_da)
    hits = n * bins * window * density
    entries = P * per_peptide
    io = n * (8 * raw + 33 + p.top_k * 32 + 1024 + 4)
    if kind == "shard_build":     # the peptide table in, the index out
        return {"bytes": io + 20 * P + 4 * entries, "flops": 2 * entries + hits}
    return {"bytes": io + 4 * min(hits, entries), "flops": hits + 256 * n}


# ---- 64-bit values


def exact(case, seed):
    """Hyperscores and e-values in 64 bits, where the database is unmodified
    (the modified ones take minutes without an index) and for merges."""
    if case["kind"] == "merge":
        psm, hist, _ = _partials(case, seed)
        if case["s"] < 64:      # the sample cuts the distribution: its own rule decides the e-value
            return None
        n, k = case["n"], case["top_k"]
        key = psm["key"].transpose(1, 0, 2).reshape(n, -1)
        pid = psm["pid"].transpose(1, 0, 2).reshape(n, -1)
        order = np.lexsort((pid, -key.astype(np.float64)), axis=1)[:, :k]
        key = np.take_along_axis(key, order, 1)
        pid = np.take_along_axis(pid, order, 1)
        return _scores(key, pid != 0xFFFFFFFF, hist.sum(0, dtype=np.int64), with_records=True)
    if case["kind"] != "closed_tiny":
        return None
    w = _workload(case)
    p = w.params
    residues, lens, masses = _digest(w)
    bins, isy, start = _ions(residues, lens, p)
    spec = _spectra(w, case["n"], seed)
    n, k = spec.n, p.top_k
    keys = np.full((n, k), np.iinfo(np.int64).min)
    hist = np.zeros((n, 256), np.int64)
    lf = np.cumsum(np.log10(np.maximum(np.arange(65), 1)))
    lf = np.floor(lf * 2.0 ** 32 + 0.5).astype(np.int64)
    for q in range(n):
        a, e = int(spec.peak_off[q]), int(spec.peak_off[q + 1])
        mz, inten = spec.mz[a:e].astype(np.float64), spec.intensity[a:e].astype(np.float64)
        ok = np.isfinite(mz) & np.isfinite(inten) & (inten > 0) & (mz >= p.frag_mz_min) & (mz < p.frag_mz_max)
        b, inten = np.floor(mz[ok] / p.bin_width_da).astype(np.int64), inten[ok]
        if not len(b):
            continue
        o = np.lexsort((-inten, b))
        b, inten = b[o], inten[o]
        first = np.concatenate([[True], b[1:] != b[:-1]])
        b, inten = b[first], inten[first]
        top = np.lexsort((b, -inten))[:p.top_n_peaks]
        iq = np.maximum(1, np.floor(inten[top] * p.intensity_scale / inten[top][0])).astype(np.int64)
        b = b[top]
        o = np.argsort(b)
        b, iq = b[o], iq[o]
        m = (spec.prec_mz[q] - PROTON) * float(spec.charge[q])
        lo = np.searchsorted(masses, m - spec.tol_da[q], "left")
        hi = np.searchsorted(masses, m + spec.tol_da[q], "right")
        if lo >= hi:
            continue
        s0, s1 = start[lo], start[hi]
        at = np.minimum(np.searchsorted(b, bins[s0:s1]), len(b) - 1)
        hit = b[at] == bins[s0:s1]
        pep = np.repeat(np.arange(hi - lo), np.diff(start[lo:hi + 1]))[hit]
        y = isy[s0:s1][hit]
        ny = np.bincount(pep[y], minlength=hi - lo)
        nb = np.bincount(pep[~y], minlength=hi - lo)
        tot = np.bincount(pep, weights=iq[at[hit]], minlength=hi - lo).astype(np.int64)
        c = np.flatnonzero(nb + ny >= p.min_shared)
        key = lf[nb[c]] + lf[ny[c]] + np.floor(np.log10(tot[c]) * 2.0 ** 32 + 0.5).astype(np.int64)
        hist[q] = np.bincount(np.minimum(key >> 31, 255), minlength=256)
        top = np.sort(key)[::-1][:k]
        keys[q, :len(top)] = top
    return _scores(keys, keys != np.iinfo(np.int64).min, hist)


def _digest(w):
    """Unmodified tryptic peptides (fixed modifications in the masses), by mass, sequence."""
    p, prot = w.params, _proteome(w.n_proteins, w.db_seed, w.protein_len)
    seqs = set()
    for i in range(prot.n):
        s = prot.protein(i)
        cut = [0] + [j + 1 for j in range(len(s) - 1) if s[j] in "KR" and s[j + 1] != "P"] + [len(s)]
        for a in range(len(cut) - 1):
            for b in range(a + 1, min(a + 2 + p.missed_cleavages, len(cut))):
                if p.min_len <= cut[b] - cut[a] <= p.max_len:
                    seqs.add(s[cut[a]:cut[b]])
    seqs = sorted(seqs)
    lens = np.array([len(s) for s in seqs])
    mono = {"G": 57.021464, "A": 71.037114, "S": 87.032028, "P": 97.052764, "V": 99.068414, "T": 101.047679,
            "C": 103.009185, "L": 113.084064, "I": 113.084064, "N": 114.042927, "D": 115.026943, "Q": 128.058578,
            "K": 128.094963, "E": 129.042593, "M": 131.040485, "H": 137.058912, "F": 147.068414, "R": 156.101111,
            "Y": 163.063329, "W": 186.079313}
    for m in w.mods:
        for r in m.residues:
            mono[r] = mono[r] + m.delta_da
    res = np.zeros((len(seqs), p.max_len))
    for i, s in enumerate(seqs):
        res[i, :len(s)] = [mono[c] for c in s]
    mass = np.cumsum(res, axis=1)[:, -1] + WATER
    keep = np.flatnonzero((mass >= p.min_mass) & (mass <= p.max_mass))
    keep = keep[np.argsort(mass[keep], kind="stable")]
    return res[keep], lens[keep], mass[keep]


def _ions(res, lens, p):
    """Distinct b/y bins of every peptide, concatenated; a bin of both kinds counts as b."""
    out_b, out_y, start = [], [], [0]
    for r, n in zip(res, lens):
        b = np.cumsum(r[:n - 1]) + PROTON
        y = (np.cumsum(r[n - 1:0:-1]) + WATER) + PROTON
        b = np.unique(np.floor(b[(b >= p.frag_mz_min) & (b < p.frag_mz_max)] / p.bin_width_da).astype(np.int64))
        y = np.unique(np.floor(y[(y >= p.frag_mz_min) & (y < p.frag_mz_max)] / p.bin_width_da).astype(np.int64))
        y = y[~np.isin(y, b)]
        out_b.append(np.concatenate([b, y]))
        out_y.append(np.repeat([False, True], [len(b), len(y)]))
        start.append(start[-1] + len(b) + len(y))
    return np.concatenate(out_b), np.concatenate(out_y), np.array(start)


def _scores(key, real, hist, with_records=False):
    """Hyperscores and e-values of ranked keys: the 5-point smoothed score
    distribution's survival tail, fitted by least squares between its mode
    and the top score's bin."""
    n, k = key.shape
    N = hist.sum(1)
    pad = np.pad(hist, ((0, 0), (2, 2)))
    g = sum(c * pad[:, i:i + 256] for i, c in enumerate((-3, 12, 17, 12, -3)))
    G = np.cumsum(g[:, ::-1], axis=1)[:, ::-1]
    ev = np.full((n, k), np.inf)
    for q in range(n):
        if not real[q, 0]:
            continue
        j = np.arange(int(np.argmax(g[q])) + 1, min(int(key[q, 0]) >> 31, 255))
        j = j[G[q, j] > 0]
        x = key[q, real[q]] * 2.0 ** -31
        ev[q, real[q]] = N[q]
        if len(j) >= 3:
            y = np.log10(G[q, j] / G[q, 0])
            slope = ((j - j.mean()) * (y - y.mean())).sum() / ((j - j.mean()) ** 2).sum()
            ev[q, real[q]] = N[q] * 10.0 ** (slope * x + (y.mean() - slope * j.mean()))
    hs = np.where(real, key * 2.0 ** -32, 0.0)
    out = {"query": None, "pid": None, "nb": None, "ny": None, "key": None, "hyperscore": hs.reshape(-1),
           "evalue": ev.reshape(-1), "hist": None, "n_scored": None}
    if with_records:
        out["records"] = None
    return out
