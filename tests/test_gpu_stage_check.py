"""Host inputs are checked on the host for few windows and by a kernel for many:
both refuse the same inputs with the same status and message, naming the first bad
read or window by its index in the caller's arrays."""
import numpy as np
import pytest

from paper_1805_00106_gb300 import synth as S
from tests.parity import gpu_run, oracle_run

pytestmark = pytest.mark.gpu


def _bad(kind, w):
    w = {k: np.array(v) for k, v in w.items() if k != "refs"}
    n = len(w["read_off"]) - 1
    if kind == "window past its reference":
        w["c_start"][[40, 90]] = 19_990
    elif kind == "window length":
        w["c_len"][[41, 77]] = [0, 513]
    elif kind == "strand":
        w["c_strand"][43] = 2
    elif kind == "reference":
        w["c_ref"][45] = 1
    elif kind == "huge start":
        w["c_start"][46] = -5  # 2^64 - 5
    elif kind == "read length":
        w["read_off"][20:-1] = w["read_off"][19]  # reads 19 .. are empty
    elif kind == "read offsets":
        w["read_off"][12] = w["read_off"][10]
    else:
        w["cand_off"][9] = w["cand_off"][7]
    return w, n


@pytest.mark.parametrize("kind", ["window past its reference", "window length", "strand", "reference", "huge start",
                                  "read length", "read offsets", "window offsets"])
def test_few_and_many_windows_are_refused_alike(kind):
    from paper_1805_00106_gb300 import sr
    ref = S.ref_iid(20_000, 3)
    s = sr.Session.open([bytes(ref)])
    messages = set()
    for reads in (100, 2000):  # 400 and 8000 windows
        rd = S.reads([ref], reads, 5, 100, 100)
        w, _ = _bad(kind, dict(refs=[ref], **rd, **S.cands(rd, [len(ref)], 6, S.COUNT_FIXED, 4, 16)))
        with pytest.raises(sr.SrError) as e:
            s.align(w["bases"], w["read_off"], w["cand_off"], w["c_ref"], w["c_strand"], w["c_start"], w["c_len"])
        assert e.value.status == sr.SR_EINVAL
        messages.add(str(e.value))
    assert len(messages) == 1, messages
    good = S.reads([ref], 1100, 5, 60, 250)
    w = dict(refs=[ref], **good, **S.cands(good, [len(ref)], 6, S.COUNT_PARETO, 1.1, 16, cap_per_read=256))
    assert len(w["c_ref"]) > 4096
    g = gpu_run(s, w)
    assert np.array_equal(g["item_score"], oracle_run(w)["item_score"])
    assert g["cells"] == int(np.sum(np.repeat(np.diff(w["read_off"]), np.diff(w["cand_off"])) * w["c_len"].astype(np.int64)))
