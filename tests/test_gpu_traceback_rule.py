"""Which kernel traces a band class is chosen by the class's read count (the
wavefront for few, two reads per thread for many): both sides of each line give
the oracle's alignments."""
import numpy as np
import pytest

from paper_1805_00106_gb300 import synth as S
from tests.parity import gpu_run, oracle_run
from tests.test_gpu_parity import _band_widths

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pool():
    """96 reads with errors and their oracle results, by band class."""
    from paper_1805_00106_gb300 import sr
    rng = np.random.default_rng(41)
    ref = rng.choice(np.frombuffer(b"ACGT", np.uint8), 60_000)
    rd = S.reads([ref], 400, 43, 60, 250, 0.03, 0.006, 0.5)
    cd = S.cands(rd, [len(ref)], 44, S.COUNT_FIXED, 2, 32)
    w = dict(refs=[ref], **rd, **cd)
    o = oracle_run(w)
    ok, width, _ = _band_widths(w, o)
    perfect = o["best"]["score"] == 2 * np.diff(w["read_off"])
    return sr, w, o, {16: np.nonzero(ok & (width <= 16) & ~perfect)[0], 32: np.nonzero(ok & (width > 16) & (width <= 32))[0]}


@pytest.mark.parametrize("cls,n", [(16, 16384), (16, 16385), (32, 4096), (32, 16384), (32, 16385)])
def test_both_sides_of_the_line(pool, cls, n):
    sr, w, o, classes = pool
    pick = np.resize(classes[cls][:48], n)
    assert len(classes[cls]) >= 20
    off, coff = np.asarray(w["read_off"]), np.asarray(w["cand_off"])
    t = dict(refs=w["refs"], bases=np.concatenate([w["bases"][off[r]:off[r + 1]] for r in pick]),
             read_off=np.concatenate([[0], np.cumsum(np.diff(off)[pick])]),
             cand_off=np.concatenate([[0], np.cumsum(np.diff(coff)[pick])]),
             **{k: np.concatenate([np.asarray(w[k])[coff[r]:coff[r + 1]] for r in pick])
                for k in ("c_ref", "c_strand", "c_start", "c_len")})
    s = sr.Session.open([bytes(r) for r in t["refs"]])
    g = gpu_run(s, t)
    for f in ("score", "second", "n_ties", "ref_end", "ref_start", "read_start", "read_end", "cigar_len"):
        assert np.array_equal(g["best"][f].astype(np.int64), o["best"][f].astype(np.int64)[pick]), f
    words = {int(r): o["cigar"][r][: int(o["best"]["cigar_len"][r])] for r in set(pick.tolist())}
    assert np.array_equal(g["cigar"], np.concatenate([words[int(r)] for r in pick]))
