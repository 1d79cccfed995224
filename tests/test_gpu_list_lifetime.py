"""A device candidate list outlives its session: it keeps its own arrays, while the
session's references, index and scratch are released as the session closes."""
import gc

import numpy as np
import pytest

from paper_1805_00106_gb300 import synth as S

pytestmark = pytest.mark.gpu

KEYS = ["cand_off", "c_ref", "c_strand", "c_start", "c_len", "c_hits"]


@pytest.mark.parametrize("lists", [1, 3])
def test_a_held_list_does_not_keep_its_session(lists):
    import torch
    from paper_1805_00106_gb300 import sr
    ref = S.ref_iid(4_000_000, 12)
    idx = [sr.Index.build(bytes(ref), seed_len=20, address_bases=12)]  # 2^24 bucket heads of 32 bytes
    rd = S.reads([ref], 2_000, 3, 80, 200, 0.01, 0.001, 0.5)
    want = sr.candidates(idx, rd["bases"], rd["read_off"])
    gc.collect()  # sessions of other tests go now or not at all
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    s = sr.Session.from_indexes(idx)
    s.attach_index(idx)
    held = [s.candidates(rd["bases"], rd["read_off"], out_device=True) for _ in range(lists)]
    freed = s.candidates(rd["bases"], rd["read_off"], out_device=True)
    del freed
    assert torch.cuda.mem_get_info()[0] < before - (500 << 20)
    s.close()
    assert torch.cuda.mem_get_info()[0] > before - (100 << 20)
    # the lists as they were, and another session's work with them
    t = sr.Session.open([bytes(ref)])
    for c in held:
        got = c.to_numpy()
        assert all(np.array_equal(np.asarray(want[k], np.int64), np.asarray(got[k], np.int64)) for k in KEYS)
    a = t.align_cands(rd["bases"], rd["read_off"], held[0])
    b = t.align(rd["bases"], rd["read_off"], *[want[k] for k in KEYS[:5]])
    assert np.array_equal(a["item_score"], b["item_score"])
    del held
    t.close()
    assert torch.cuda.mem_get_info()[0] > before - (100 << 20)
