"""What this library is timed on: short-read alignment as a sequencing pipeline
uses it, through the public calls of ``paper_1805_00106_gb300.sr``.

Four kinds of call, over the sizes they are made with:

align     reads and candidate windows in host memory -> sr_align_batch -> scores,
          winners and CIGARs in host memory (requests of a service, whole read sets)
find      the device CAL finder: reads -> candidate windows (in host or device
          memory), for uniform and for repeat-rich references
pipeline  reads in device memory -> device CAL finder -> windows kept on the
          device -> sr_align_batch with classification -> results on the host
report    a staged batch, scored, with the tracker's N-best or all-tied report

References and their indexes are made once per process, as a program loads its
genome once.  Each case has its set of reads (and windows); the seed gives the
order in which the call gets them, so that every seed asks for other output
arrays of the same sizes (windows and CIGAR words depend on the reads).
"""
import functools
import json
import zlib

import numpy as np
import torch

from paper_1805_00106_gb300 import sr, synth

# References: "genome" one uniform reference at 41% GC; "pair" a reference and a
# diverged copy (15% substitutions, 2% indels, block moves), as reads of a
# xenograft are told apart; "repeats" 30% tandem and interspersed repeats.
GENOME, PAIR, REPEATS = 20_000_000, 16_000_000, 40_000_000
N_REFS = {"genome": 1, "pair": 2, "repeats": 1}

# Score sets: the library's default, BWA-MEM's and a wider one.
SCORES = {"default": (2, 3, 5, 2), "bwa": (1, 4, 6, 1), "wide": (5, 4, 10, 1)}

# Mean windows per read of the window-count distributions, and CALs and windows
# per read that the finder meets (measured with the host stage).
MEAN_WINDOWS = {"fixed": 4.0, "poisson": 6.0, "uniform": 32.0, "pareto": 4.9}
MEAN_CALS = {("pair", 1024): (68.0, 1.3), ("repeats", 0): (5100.0, 28.7), ("repeats", 1024): (3200.0, 28.7)}


def _align(name, reads, lo, hi, ref, windows, pad=32, scores="default", mode=0, cigar=True, classify=False):
    return dict(name=name, kind="align", reads=reads, lo=lo, hi=hi, ref=ref, windows=windows, pad=pad, scores=scores,
                mode=mode, cigar=cigar, classify=classify)


def _find(name, reads, lo, hi, ref, limit, k=20, stride=1, max_cands=0, device=True):
    return dict(name=name, kind="find", reads=reads, lo=lo, hi=hi, ref=ref, limit=limit, k=k, stride=stride,
                max_cands=max_cands, device=device)


def listed():
    return [
        # an interactive lookup of a few reads
        _align("align 9 reads", 9, 75, 250, "genome", "poisson"),
        # a service's request against a reference pair, classified
        _align("align request", 2049, 75, 250, "pair", "uniform", classify=True),
        # the batched, uneven workload the library is quoted on: mixed lengths, both strands
        _align("align mixed", 150_000, 75, 250, "genome", "poisson"),
        # a large call, which runs in parts that overlap one another's copies
        _align("align large", 600_000, 75, 250, "genome", "poisson"),
        # long reads with heavy-tailed window counts, under BWA-MEM's scores
        _align("align repeats", 40_001, 250, 250, "repeats", "pareto", scores="bwa"),
        # the array's own readout (best cell of the final row), scores only: a filter pass
        _align("align final row", 60_000, 151, 151, "genome", "fixed", pad=16, mode=1, cigar=False),
        # the finder on device reads, list kept on the device: the xenograft's read set
        _find("find pair", 1_000_000, 100, 100, "pair", 1024),
        # the finder for one request's reads, host reads and list
        _find("find request", 500, 75, 150, "pair", 1024, device=False),
        # repeats without a CAL limit: some reads meet hundreds of thousands of CALs
        _find("find repeats unlimited", 10_000, 250, 250, "repeats", 0),
        # repeats with the usual limit, host reads and list, at most 64 windows a read
        _find("find repeats limited", 20_001, 250, 250, "repeats", 1024, max_cands=64, device=False),
        # the whole pipeline with classification
        dict(name="pipeline pair", kind="pipeline", reads=300_000, lo=100, hi=100, ref="pair", limit=1024, k=20, stride=1,
             max_cands=0),
        # all alignments tied for the best, over repeats
        dict(name="report tied", kind="report", reads=20_000, lo=150, hi=250, ref="repeats", windows="pareto", pad=32,
             scores="default", mode=0, cigar=True, classify=False, report="tied", n_best=1),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["align", "align", "align", "find", "find", "pipeline", "report"])
    if kind in ("align", "report"):
        ref = rng.choice(["genome", "pair", "repeats"])
        windows = rng.choice(["fixed", "poisson", "uniform", "pareto"])
        lo = rng.randint(36, 250)
        hi = rng.choice([lo, rng.randint(lo, 250)])
        # no more windows than the largest listed call has
        most = int(3_600_000 / MEAN_WINDOWS[windows])
        case = dict(kind=kind, reads=_log(rng, 8, most if kind == "align" else min(most, 100_000)), lo=lo, hi=hi, ref=ref,
                    windows=windows, pad=rng.choice([16, 32]), scores=rng.choice(["default", "default", "bwa", "wide"]),
                    mode=rng.choice([0, 0, 0, 1]), cigar=rng.random() < 0.8, classify=ref == "pair")
        if kind == "report":
            case.update(cigar=True, report=rng.choice(["best", "tied"]), n_best=rng.choice([1, 3, 10]))
        return case
    ref, limit = ("pair", 1024) if kind == "pipeline" else rng.choice([("pair", 1024), ("repeats", 0), ("repeats", 1024)])
    lo = rng.randint(50, 250)
    case = dict(kind=kind, reads=_log(rng, 8, 300_000 if ref == "pair" else 10_000), lo=lo,
                hi=rng.choice([lo, rng.randint(lo, 250)]), ref=ref, limit=limit, k=rng.choice([20, 20, 25]),
                stride=rng.choice([1, 1, 1, 2, 5]), max_cands=rng.choice([0, 0, 16, 64]))
    if kind == "find":
        case["device"] = rng.random() < 0.5
    return case


# ------------------------------------------------------------------ inputs

@functools.lru_cache(maxsize=None)
def _refs(ref):
    if ref == "genome":
        return [synth.ref_iid(GENOME, 11, gc=0.41)], None
    if ref == "pair":
        a = synth.ref_iid(PAIR, 12)
        return [a, synth.mutate(a, 13, 0.15, 0.02, 12, 10_000, 800_000)], None
    r, mask = synth.ref_repeats(REPEATS, 14)
    return [r], mask


@functools.lru_cache(maxsize=None)
def _session(ref):
    return sr.Session.open(_refs(ref)[0])


@functools.lru_cache(maxsize=4)
def _finder(ref, k, limit):
    idx = [sr.Index.build(r.tobytes(), seed_len=k, address_bases=12, cal_limit=limit) for r in _refs(ref)[0]]
    s = sr.Session.from_indexes(idx)
    s.attach_index(idx)
    return s


def _pinned(a, dtype):
    a = np.ascontiguousarray(a, dtype)
    t = torch.empty(max(a.nbytes, 1), dtype=torch.uint8, pin_memory=torch.cuda.is_available())
    out = t.numpy()[: a.nbytes].view(dtype)
    out[:] = a
    return out


@functools.lru_cache(maxsize=2)
def _pool(key):
    """A case's reads (1% errors, both strands) and, for align and report, their
    windows, as (array, offsets) of the bases and of each window field."""
    case = json.loads(key)
    refs, mask = _refs(case["ref"])
    seed = zlib.crc32(key.encode())
    rd = synth.reads(refs, case["reads"], 2 * seed + 1, case["lo"], case["hi"], 0.009, 0.001, 0.5,
                     weights=[0.7, 0.3] if len(refs) == 2 else None)
    if "windows" not in case:
        return rd, None
    lens = [len(r) for r in refs]
    kind, p1, cap, p2 = {"fixed": (synth.COUNT_FIXED, 4, 4, 0.0), "poisson": (synth.COUNT_POISSON, 6.0, 64, 0.0),
                         "uniform": (synth.COUNT_UNIFORM, 64, 64, 0.0),
                         "pareto": (synth.COUNT_PARETO, 1.1, 256, 0.8 if mask is not None else 0.0)}[case["windows"]]
    return rd, synth.cands(rd, lens, 2 * seed + 2, kind, p1, case["pad"], cap_per_read=cap, p2=p2, rep_mask=mask)


def _inputs(case, seed):
    """The case's reads and windows in the seed's order: chunks of consecutive
    reads (single reads up to 1024 of them) shuffled."""
    rd, cd = _pool(json.dumps({k: v for k, v in case.items() if k != "name"}, sort_keys=True))
    n = case["reads"]
    chunks = min(n, 1024)
    cut = np.linspace(0, n, chunks + 1).astype(np.int64)
    order = np.random.default_rng(seed).permutation(chunks)

    def shuffled(off, *arrays):
        lens = np.diff(off)
        new = np.zeros(n + 1, np.int64)
        np.cumsum(np.concatenate([lens[cut[c]: cut[c + 1]] for c in order]), out=new[1:])
        return new, [np.concatenate([a[off[cut[c]]: off[cut[c + 1]]] for c in order]) for a in arrays]

    read_off, (bases,) = shuffled(rd["read_off"], rd["bases"])
    if cd is None:
        return dict(read_off=read_off, bases=bases), None
    fields = ("c_ref", "c_strand", "c_start", "c_len")
    cand_off, arrays = shuffled(cd["cand_off"], *[cd[f] for f in fields])
    return dict(read_off=read_off, bases=bases), dict(zip(fields, arrays), cand_off=cand_off)


def prepare(case, seed):
    rd, cd = _inputs(case, seed)
    st = dict(kind=case["kind"])
    if case["kind"] in ("align", "report"):
        st["session"] = _session(case["ref"])
        st["args"] = [_pinned(rd["bases"], np.uint8), _pinned(rd["read_off"], np.uint64), _pinned(cd["cand_off"], np.uint64),
                      _pinned(cd["c_ref"], np.uint8), _pinned(cd["c_strand"], np.uint8), _pinned(cd["c_start"], np.uint64),
                      _pinned(cd["c_len"], np.uint32)]
        st["scores"] = sr.score_params(*SCORES[case["scores"]])
        st["opts"] = sr.align_opts(mode=case["mode"], want_cigar=case["cigar"], classify=case["classify"])
        if case["kind"] == "report":
            st["report"] = (sr.REPORT_TIED if case["report"] == "tied" else sr.REPORT_BEST_N, case["n_best"])
        return st
    st["session"] = _finder(case["ref"], case["k"], case["limit"])
    st["find"] = dict(seed_stride=case["stride"], merge_dist=32, pad=32, max_cands=case["max_cands"])
    st["device"] = case.get("device", True)
    if st["device"]:
        st["reads"] = [torch.from_numpy(rd["bases"]).cuda(), torch.from_numpy(rd["read_off"]).cuda()]
    else:
        st["reads"] = [_pinned(rd["bases"], np.uint8), _pinned(rd["read_off"], np.uint64)]
    if case["kind"] == "pipeline":
        st["scores"] = sr.score_params()
        st["opts"] = sr.align_opts(classify=True)
    return st


# ------------------------------------------------------------------ the calls

_HIT_FIELDS = ("score", "second", "n_ties", "item", "ref_id", "strand", "read_start", "read_end", "ref_start", "ref_end",
               "cigar_off", "cigar_len")


def _records(h):
    """The record fields as arrays (views; unsigned words seen as signed ones)."""
    return [h[f].view({4: np.int32, 8: np.int64}.get(h.dtype[f].itemsize, np.uint8)) for f in _HIT_FIELDS]


def _results(r):
    out = dict(item_score=r["item_score"], item_end=r["item_end"].view(np.int32), best=_records(r["best"]),
               per_ref=_records(r["best_per_ref"]), cigar=r["cigar"].view(np.int32), cells=r["cells"])
    if r["read_class"] is not None:
        out["read_class"] = r["read_class"]
    return out


def _windows(c):
    if isinstance(c, sr.DeviceCandList):
        c = c.tensors()
        signed = {8: torch.int64, 4: torch.int32, 1: torch.uint8}
        return {k: v.view(signed[v.element_size()]) for k, v in c.items()}
    return {k: v.view({8: np.int64, 4: np.int32, 1: np.uint8}[v.itemsize]) for k, v in c.items()}


def run(st):
    s = st["session"]
    if st["kind"] == "align":
        return _results(s.align(*st["args"], st["scores"], st["opts"]))
    if st["kind"] == "report":
        b = s.stage(*st["args"])
        b.run(st["scores"], st["opts"])
        rep = b.report(*st["report"])
        res = _results(b.fetch())
        b.close()
        hits = rep["hits"]
        res["report"] = [rep["offsets"].view(np.int64), rep["n_truncated"]] + [
            hits[f].view({4: np.int32, 8: np.int64}.get(hits.dtype[f].itemsize, np.uint8))
            for f in ("score", "item", "ref_id", "strand", "end_col", "ref_end")]
        return res
    c = s.candidates(*st["reads"], out_device=st["device"], **st["find"])
    if st["kind"] == "find":
        return _windows(c)
    return _results(s.align_cands(*st["reads"], c, st["scores"], st["opts"]))


# ------------------------------------------------------------------ floors and values

def work(case):
    """Bytes: reads in, windows in or out, the packed windows of the reference,
    one 32-byte sector per seed lookup, one word per CAL, results out.
    Operations: six 16-bit operations per cell of the recurrence (three maxima of
    sums, the zero floor, the gap subtraction, the running maximum)."""
    n, m, nr = case["reads"], 0.5 * (case["lo"] + case["hi"]), N_REFS[case["ref"]]
    b, ops = n * (m + 8.0), 0.0
    if case["kind"] in ("align", "report"):
        w, pad = MEAN_WINDOWS[case["windows"]], case["pad"]
    else:
        cals, w = MEAN_CALS[(case["ref"], case["limit"])]
        w = min(w, case["max_cands"] or w)
        pad = 32
        seeds = max(0.0, m - case["k"]) // case["stride"] + 1
        b += n * (seeds * 32.0 + 4.0 * cals / case["stride"])
    b += n * (8.0 + w * 14.0)
    if case["kind"] != "find":
        cells = n * w * m * (m + 2 * pad)
        b += n * w * ((m + 2 * pad) / 4 + 8.0) + n * 56.0 * (1 + nr) + (n * 20.0 if case.get("cigar", True) else 0.0)
        ops = 6.0 * cells
    return dict(bytes=b, flops=ops)


def _scores64(refs, rd, cd, sp, mode):
    """Affine-gap scores of every window in 64 bits: row by row over all windows
    at once, the gaps along a row by a running maximum of H + j * extend (a gap
    opened from the end of another along the same row is never the better one)."""
    ma, mi, go, ge = sp
    m = np.diff(rd["read_off"]).astype(np.int64)
    item_read = np.repeat(np.arange(len(m)), np.diff(cd["cand_off"]))
    code = np.zeros(256, np.int8)
    code[[ord(c) for c in "ACGT"]] = range(4)
    n_items, mm, nn = len(item_read), int(m.max()), int(cd["c_len"].max(initial=1))
    q, t = np.full((n_items, mm), 4, np.int8), np.full((n_items, nn), 5, np.int8)
    for i, r in enumerate(item_read):
        x = code[rd["bases"][rd["read_off"][r]: rd["read_off"][r + 1]]]
        q[i, : len(x)] = 3 - x[::-1] if cd["c_strand"][i] else x
        s0 = int(cd["c_start"][i])
        t[i, : cd["c_len"][i]] = code[refs[cd["c_ref"][i]][s0: s0 + int(cd["c_len"][i])]]
    low = -(1 << 40)
    h = np.zeros((n_items, nn + 1), np.int64)
    f = np.full((n_items, nn + 1), low, np.int64)
    j = np.arange(nn + 1, dtype=np.int64) * ge
    inside = np.arange(nn) < cd["c_len"][:, None]
    best = np.zeros(n_items, np.int64)
    for i in range(mm):
        f = np.maximum(f, h - go) - ge
        g = np.maximum(0, f)
        g[:, 0] = 0
        g[:, 1:] = np.maximum(g[:, 1:], h[:, :-1] + np.where(q[:, i: i + 1] == t, ma, -mi))
        e = np.maximum.accumulate(g + j, axis=1)[:, :-1] - j[1:] - go
        g[:, 1:] = np.maximum(g[:, 1:], e)
        h = g
        row = np.where(inside, h[:, 1:], 0).max(axis=1)
        live = m[item_read] == i + 1 if mode else m[item_read] > i
        best = np.where(live, np.maximum(best, row), best)
    return best


def exact(case, seed):
    """The window scores in 64 bits, for calls of few windows.  The rest of the
    outputs (positions, CIGARs, windows, classes) are whole numbers with no
    rounding: they have no nearer value."""
    if case["kind"] != "align" or case["reads"] * MEAN_WINDOWS[case["windows"]] > 2000:
        return None
    rd, cd = _inputs(case, seed)
    if not len(cd["c_ref"]):
        return None
    score = _scores64(_refs(case["ref"])[0], rd, cd, SCORES[case["scores"]], case["mode"])
    out = dict(item_score=score, item_end=None, best=[None] * len(_HIT_FIELDS), per_ref=[None] * len(_HIT_FIELDS), cigar=None,
               cells=None)
    if case["classify"]:
        out["read_class"] = None
    return out
