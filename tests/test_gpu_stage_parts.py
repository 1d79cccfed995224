"""Calls of 2^19 reads or more are staged in parts, their offsets made part-relative
on the device: offsets that fall below a part's first are refused with the message of
an unsplit call."""
import numpy as np
import pytest

from paper_1805_00106_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("reads", [2_000, 600_000])
@pytest.mark.parametrize("which", ["read_off", "cand_off"])
def test_offsets_below_a_parts_first(reads, which):
    from paper_1805_00106_gb300 import sr
    ref = S.ref_iid(20_000, 3)
    s = sr.Session.open([bytes(ref)])
    rd = S.reads([ref], reads, 5, 20, 24)
    w = dict(**rd, **S.cands(rd, [len(ref)], 6, S.COUNT_FIXED, 3, 4))
    for at, to in ((reads // 2, 5), (reads // 2, 0), (reads - 1, 7)):
        args = {k: np.array(w[k]) for k in ("bases", "read_off", "cand_off", "c_ref", "c_strand", "c_start", "c_len")}
        args[which][at] = to
        with pytest.raises(sr.SrError) as e:
            s.align(*args.values(), sr.score_params(), sr.align_opts(want_cigar=False))
        assert e.value.status == sr.SR_EINVAL
        assert f"decreasing or out-of-range offsets at read {at - 1}" in str(e.value)
