"""The one-pass CAL finder's paths (warp, block tables, large reads) against the
host stage, at the edges of each: distinct CALs around what a warp (128 runs, 64
ranks), the two tables (768, 12288) and the large-read path take, every index form,
seeds that are their own reverse complement, and CALs off the reference's ends."""
import numpy as np
import pytest

from paper_1805_00106_gb300 import synth as S

pytestmark = pytest.mark.gpu

KEYS = ["cand_off", "c_ref", "c_strand", "c_start", "c_len", "c_hits"]
ACGT = np.frombuffer(b"ACGT", np.uint8)


@pytest.fixture(scope="module")
def sr():
    from paper_1805_00106_gb300 import sr as _sr
    _sr.lib()
    return _sr


def _check(sr, refs, bases, off, k, addr, limit=0, seeds=None, prms=({},)):
    idx = [sr.Index.build(bytes(r), seed_len=k, address_bases=addr, cal_limit=limit, hash_seed=h)
           for r, h in zip(refs, seeds or [0] * len(refs))]
    s = sr.Session.from_indexes(idx)
    s.attach_index(idx)
    out = []
    for prm in prms:
        h, d = sr.candidates(idx, bases, off, **prm), s.candidates(bases, off, **prm)
        for key in KEYS:
            assert np.array_equal(np.asarray(h[key], np.int64), np.asarray(d[key], np.int64)), (key, prm)
        out.append(h)
    return out


def _rc(x):
    return np.frombuffer(bytes(x)[::-1].translate(bytes.maketrans(b"ACGT", b"TGCA")), np.uint8)


PRMS = [dict(merge_dist=32, pad=32), dict(merge_dist=0, pad=4), dict(merge_dist=0, pad=4, max_cands=5),
        dict(seed_stride=7, merge_dist=200, pad=0, max_cands=1)]


@pytest.mark.parametrize("unit,copies", [(29, 62), (29, 65), (37, 127), (37, 130), (23, 760), (23, 770), (13, 6150),
                                         (7, 12150), (7, 12300)])
def test_distinct_cals_around_each_table(sr, unit, copies):
    """Reads inside, across the ends of and outside a tandem repeat: one inside
    has about one distinct CAL per copy (counted with merge_dist 0)."""
    rng = np.random.default_rng(unit * copies)
    u = rng.choice(ACGT, unit)
    ref = np.concatenate([rng.choice(ACGT, 700), np.tile(u, copies), rng.choice(ACGT, 700)])
    end = 700 + unit * copies
    cuts = [(700 + unit, 100), (700 + 3 * unit, 256), (650, 120), (end - 60, 120), (100, 100), (end - 200, 150)]
    reads = [ref[a: a + m] for a, m in cuts]
    reads += [_rc(x) for x in reads]
    off = np.cumsum([0] + [len(x) for x in reads])
    h = _check(sr, [ref], np.concatenate(reads), off, 20, 10, prms=PRMS)
    assert copies - 20 <= np.diff(h[1]["cand_off"]).max() <= copies + 300


@pytest.mark.parametrize("table", ["1", "3", "40", "1000000"])
@pytest.mark.parametrize("k,addr,seeds,heads", [(20, 12, (0, 0), "1"), (20, 12, (0, 0), "0"),
                                                (25, 12, (0, 0), "1"), (16, 8, (0, 0), "1"),
                                                (18, 7, (0, 0), "1"), (20, 10, (5, 9), "1"), (16, 8, (0, 0, 0), "1")])
def test_every_index_form_and_table_size(sr, monkeypatch, table, k, addr, seeds, heads):
    """The index forms (heads of both sizes, few or most of their buckets spilled,
    no heads, per reference, three references) with the tables held to few
    distinct CALs, so that reads go on to the next path, the large-read one
    included; its chunks cut small too."""
    monkeypatch.setenv("SR_CAL_TABLE", table)
    monkeypatch.setenv("SR_CAL_HEADS", heads)
    w = S.workload("c3", scale=0.0005, seed=31, rc_frac=0.5)
    refs = list(w["refs"]) + [w["refs"][0][5000:25000].copy()] * (len(seeds) - 2)
    _check(sr, refs, w["bases"], w["read_off"], k, addr, limit=1024, seeds=list(seeds), prms=PRMS)
    monkeypatch.setenv("SR_CAL_CHUNK_RECORDS", "9000")
    monkeypatch.setenv("SR_CAL_CHUNK_KEYS", "700")
    _check(sr, refs, w["bases"], w["read_off"], k, addr, limit=1024, seeds=list(seeds), prms=PRMS[:2])


@pytest.mark.parametrize("table", ["1", "1000000"])
def test_self_complementary_seeds_and_reference_ends(sr, monkeypatch, table):
    """Seeds of (AT)n and (ACGT)n are their own reverse complements (a '+' and a
    '-' CAL each); reads over the ends of the reference have CALs before its
    first base and windows cut at its last; reads shorter than a seed have none."""
    monkeypatch.setenv("SR_CAL_TABLE", table)
    rng = np.random.default_rng(8)
    body = rng.choice(ACGT, 900)
    ref = np.concatenate([body[:300], np.tile(ACGT[[0, 3]], 90), body[300:600], np.tile(ACGT, 60), body[600:]])
    junk = rng.choice(ACGT, 64)
    reads = [ref[310:420], ref[280:380], ref[790:900], ref[760:1000], np.concatenate([junk[:40], ref[:60]]),
             np.concatenate([ref[-70:], junk[:50]]), junk[:19], ref[:20], ref[-20:], ref[5:205]]
    reads += [_rc(x) for x in reads]
    off = np.cumsum([0] + [len(x) for x in reads])
    _check(sr, [ref], np.concatenate(reads), off, 20, 10, prms=PRMS)


def test_device_lists_in_turn(sr):
    """Freed device lists' memory is used again: earlier lists still held keep
    their windows, also past the session's close."""
    w = S.workload("c3", scale=0.001, seed=37, rc_frac=0.5)
    idx = [sr.Index.build(bytes(r), seed_len=20, address_bases=10) for r in w["refs"]]
    s = sr.Session.from_indexes(idx)
    s.attach_index(idx)
    off = np.asarray(w["read_off"])
    want, held = [], []
    for i in range(7):
        n = 250 * (i + 1)
        b, o = w["bases"][: off[n]], off[: n + 1]
        want.append(sr.candidates(idx, b, o))
        held.append(s.candidates(b, o, out_device=True))
        if i % 2:
            held[i - 1] = None  # its block goes to a later list
    s.close()
    for h, d in zip(want, held):
        if d is not None:
            got = d.to_numpy()
            assert all(np.array_equal(np.asarray(h[k], np.int64), np.asarray(got[k], np.int64)) for k in KEYS)
