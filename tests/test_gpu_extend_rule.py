"""How a batch's item pairs are spread over the chip is chosen by their number
and classes (every class in one launch, or a kernel per class):
on both sides of each line the scores are those of one forced shape, in both
readouts, and a small batch's those of the oracle."""
import numpy as np
import pytest

from paper_1805_00106_gb300 import synth as S
from tests.parity import compare, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


def _batch(n, lo, hi, windows, seed=5):
    ref = S.ref_iid(200_000, 9, gc=0.41)
    rd = S.reads([ref], n, seed, lo, hi, 0.02, 0.004, 0.5)
    return dict(refs=[ref], **rd, **S.cands(rd, [len(ref)], seed + 1, S.COUNT_FIXED, windows, 32))


@pytest.fixture(scope="module")
def sr():
    from paper_1805_00106_gb300 import sr as _sr
    _sr.lib()
    return _sr


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("n,lo,hi,windows", [(1, 256, 256, 1), (1, 1, 1, 2), (600, 1, 256, 3), (1024, 100, 100, 4),
                                             (1025, 100, 100, 4), (4000, 129, 256, 4), (4300, 129, 256, 4), (5000, 1, 256, 4),
                                             (6144, 90, 96, 4), (6145, 90, 96, 4), (8000, 30, 256, 4)])
def test_scores_do_not_depend_on_the_spread(sr, mode, n, lo, hi, windows):
    w = _batch(n, lo, hi, windows)
    s = sr.Session.open([bytes(r) for r in w["refs"]])
    a, b = gpu_run(s, w, mode=mode), gpu_run(s, w, mode=mode, lanes=32, rows=8)
    for k in ("item_score", "item_end", "best", "cigar"):
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("mode", [0, 1])
def test_every_row_count_against_the_oracle(sr, mode):
    """Reads at the edges of every class's rows on 32 and 16 lanes."""
    ref = S.ref_iid(60_000, 19)
    lens = sorted({m for g in (16, 32) for r in range(1, 256 // g + 1) for m in (g * r - 1, g * r, g * r + 1) if 1 <= m <= 256})
    rng = np.random.default_rng(3)
    pos = rng.integers(100, 59_000, len(lens))
    parts = [ref[p: p + m].copy() for p, m in zip(pos, lens)]
    for x in parts:
        x[rng.random(len(x)) < 0.03] = ord("A")
    off = np.concatenate([[0], np.cumsum(lens)])
    w = dict(refs=[ref], bases=np.concatenate(parts), read_off=off, cand_off=np.arange(len(lens) + 1),
             c_ref=np.zeros(len(lens), np.uint8), c_strand=np.zeros(len(lens), np.uint8), c_start=pos - 30,
             c_len=np.array(lens) + 60)
    s = sr.Session.open([bytes(ref)])
    o = oracle_run(w, mode=mode)
    few = gpu_run(s, w, mode=mode)  # one launch
    assert not compare(few, o)
    t = 400  # many pairs in 23 classes
    many = dict(w, bases=np.tile(w["bases"], t), read_off=np.concatenate([[0], np.cumsum(np.tile(lens, t))]),
                cand_off=np.arange(t * len(lens) + 1), **{k: np.tile(w[k], t) for k in ("c_ref", "c_strand", "c_start", "c_len")})
    got = gpu_run(s, many, mode=mode)
    for k in ("item_score", "item_end"):
        assert np.array_equal(got[k], np.tile(few[k], t)), k


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("sp", [(2, 7, 5, 2), (2, 8, 5, 2), (1, 20, 0, 1), (3, 1, 9, 3), (100, 127, 20, 7), (5, 100, 60, 30)])
@pytest.mark.parametrize("reads", [150, 9000])
def test_score_sets_on_both_sides_of_the_nonnegative_line(sr, mode, sp, reads):
    """Mismatch penalties up to and past go + ge (the recurrence with the plain
    diagonal add needs mismatch <= go + ge), low and high scores, small and large
    batches, and the one-launch engine, against the oracle."""
    w = _batch(150, 20, 256, 4, seed=11)
    o = oracle_run(w, sp=sp, mode=mode)
    s = sr.Session.open([bytes(r) for r in w["refs"]])
    if reads == 150:
        assert not compare(gpu_run(s, w, sp=sp, mode=mode), o)
        assert not compare(gpu_run(s, w, sp=sp, mode=mode, lanes=16, rows=16), o)
        if sp[0] * 256 < 31000:
            assert not compare(gpu_run(s, w, sp=sp, mode=mode, engine=1), o)
        return
    t = reads // 150
    lens, n = np.diff(w["read_off"]), np.diff(w["cand_off"])
    many = dict(w, bases=np.tile(w["bases"], t), read_off=np.concatenate([[0], np.cumsum(np.tile(lens, t))]),
                cand_off=np.concatenate([[0], np.cumsum(np.tile(n, t))]),
                **{k: np.tile(w[k], t) for k in ("c_ref", "c_strand", "c_start", "c_len")})
    g = gpu_run(s, many, sp=sp, mode=mode)
    assert np.array_equal(g["item_score"], np.tile(o["item_score"], t))
    assert np.array_equal(g["item_end"].astype(np.int64), np.tile(o["item_end_j"], t).astype(np.int64))


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("reads,lo,hi", [(512, 1, 128), (513, 1, 128), (1088, 250, 250), (1089, 250, 250), (2048, 129, 256),
                                         (2049, 129, 256)])
def test_both_sides_of_the_one_launch_line(sr, mode, reads, lo, hi):
    """2048 pairs of reads up to 128 bases; 4096 and 256 for each class of longer ones."""
    w = _batch(reads, lo, hi, 8)
    assert len(w["c_ref"]) // 2 in (2048, 2052, 4352, 4356, 8192, 8196)
    s = sr.Session.open([bytes(r) for r in w["refs"]])
    a, b = gpu_run(s, w, mode=mode), gpu_run(s, w, mode=mode, lanes=32, rows=8)
    for k in ("item_score", "item_end", "best", "cigar"):
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("mode", [0, 1])
def test_every_row_count_on_16_lanes(sr, mode):
    """A score set with mismatch > go + ge: reads at the edges of 16 lanes' rows."""
    lens = np.array(sorted({m for r in range(1, 17) for m in (16 * r - 1, 16 * r, 16 * r + 1) if m <= 256}))
    ref = S.ref_iid(60_000, 23)
    rng = np.random.default_rng(4)
    pos = rng.integers(100, 59_000, len(lens))
    parts = [ref[p: p + m].copy() for p, m in zip(pos, lens)]
    for x in parts:
        x[rng.random(len(x)) < 0.03] = ord("C")
    w = dict(refs=[ref], bases=np.concatenate(parts), read_off=np.concatenate([[0], np.cumsum(lens)]),
             cand_off=np.arange(len(lens) + 1), c_ref=np.zeros(len(lens), np.uint8),
             c_strand=np.zeros(len(lens), np.uint8), c_start=pos - 30, c_len=lens + 60)
    s = sr.Session.open([bytes(ref)])
    assert not compare(gpu_run(s, w, sp=(2, 8, 5, 2), mode=mode), oracle_run(w, sp=(2, 8, 5, 2), mode=mode))
