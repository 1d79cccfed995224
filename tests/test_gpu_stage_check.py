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


@pytest.mark.parametrize("reads,windows", [(9000, 1), (320_001, 1), (160_001, 2), (40_001, 3)])
def test_more_reads_than_resident_groups(reads, windows):
    """One lane per read up to two windows on average, eight above; the blocks stride
    over the reads past 311,296 (38,912) of them.  Every read counts, the last too."""
    from paper_1805_00106_gb300 import sr
    ref = S.ref_iid(20_000, 3)
    s = sr.Session.open([bytes(ref)])
    rd = S.reads([ref], reads, 5, 20, 24)
    w = dict(refs=[ref], **rd, **S.cands(rd, [len(ref)], 6, S.COUNT_FIXED, windows, 4))
    args = [w[k] for k in ("bases", "read_off", "cand_off", "c_ref", "c_strand", "c_start", "c_len")]
    cells = int(np.sum(np.repeat(np.diff(w["read_off"]), windows) * w["c_len"].astype(np.int64)))
    g = gpu_run(s, w)
    assert g["cells"] == cells
    k = np.r_[0:200, reads - 200:reads]
    want = oracle_run(_reads(w, k))["item_score"]
    got = np.concatenate([g["item_score"][w["cand_off"][i]:w["cand_off"][i + 1]] for i in k])
    assert np.array_equal(got, want)
    args[6] = args[6].copy()
    args[6][-1] = 0
    with pytest.raises(sr.SrError) as e:
        s.align(*args)
    assert e.value.status == sr.SR_EINVAL and str(len(args[6]) - 1) in str(e.value)


def _reads(w, k):
    """the reads k of a workload, with their windows"""
    ro, co = w["read_off"], w["cand_off"]
    items = np.concatenate([np.arange(co[i], co[i + 1]) for i in k])
    return dict(refs=w["refs"], bases=np.concatenate([w["bases"][ro[i]:ro[i + 1]] for i in k]),
                read_off=np.r_[0, np.cumsum([ro[i + 1] - ro[i] for i in k])].astype(np.uint64),
                cand_off=np.r_[0, np.cumsum([co[i + 1] - co[i] for i in k])].astype(np.uint64),
                **{x: np.ascontiguousarray(w[x][items]) for x in ("c_ref", "c_strand", "c_start", "c_len")})
