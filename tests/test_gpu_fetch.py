"""Small results come back in one copy with room for six CIGAR words per read, and
inputs of at most 48 KB go out in one: calls on both sides of each give the
oracle's results, bad bases are still refused, and results outlive their batch."""
import numpy as np
import pytest

from paper_1805_00106_gb300 import synth as S
from tests.parity import compare, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reads,indel,refs,opts,past", [(1, 0.0, 1, {}, False), (40, 0.2, 1, {}, True),
                                                        (300, 0.25, 2, dict(classify=True), True),
                                                        (300, 0.001, 2, dict(want_cigar=False), False),
                                                        (1500, 0.002, 1, {}, False), (1500, 0.15, 1, {}, True)])
def test_copies_on_both_sides_of_their_sizes(reads, indel, refs, opts, past):
    from paper_1805_00106_gb300 import sr
    rs = [S.ref_iid(30_000, 60 + r) for r in range(refs)]
    rd = S.reads(rs, reads, 61, 120, 256, 0.01, indel, 0.5)
    w = dict(refs=rs, **rd, **S.cands(rd, [len(r) for r in rs], 62, S.COUNT_FIXED, 2, 48))
    o = oracle_run(w)
    words = int(o["best"]["cigar_len"].sum())
    assert (words > 6 * reads + 256) == past  # CIGARs past the room, or in it
    s = sr.Session.open([bytes(r) for r in rs])
    g = gpu_run(s, w, **opts)
    assert not compare(g, o, want_cigar=opts.get("want_cigar", True))
    again = gpu_run(s, w, **opts)
    s.close()
    for k in ("item_score", "item_end", "cigar"):
        assert np.array_equal(g[k], again[k])
    if opts.get("classify"):
        assert np.array_equal(g["read_class"], again["read_class"]) and len(g["read_class"]) == reads


@pytest.mark.parametrize("reads", [20, 2000])
def test_bad_bases_are_refused_and_the_session_goes_on(reads):
    from paper_1805_00106_gb300 import sr
    ref = S.ref_iid(30_000, 71)
    rd = S.reads([ref], reads, 72, 100, 100)
    w = dict(refs=[ref], **rd, **S.cands(rd, [len(ref)], 73, S.COUNT_FIXED, 3, 16))
    s = sr.Session.open([bytes(ref)])
    bad = dict(w, bases=w["bases"].copy())
    bad["bases"][777] = ord("N")
    with pytest.raises(sr.SrError) as e:
        gpu_run(s, bad)
    assert e.value.status == sr.SR_EBADBASE
    assert np.array_equal(gpu_run(s, w)["item_score"], oracle_run(w)["item_score"])
