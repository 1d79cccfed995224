"""Device memory that a session keeps for later calls (blocks of freed device lists,
arenas of freed batches) does not stand in the way of its own allocations, is bounded,
and a list that is still held keeps no more than its own arrays."""
import gc

import numpy as np
import pytest

from paper_1805_00106_gb300 import synth as S

pytestmark = pytest.mark.gpu

KEYS = ["cand_off", "c_ref", "c_strand", "c_start", "c_len", "c_hits"]
ACGT = np.frombuffer(b"ACGT", np.uint8)
MB = 1 << 20


def _free():
    import torch
    gc.collect()  # sessions of other tests go now or not at all
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


class _Repeat:
    """Reads inside a tandem repeat of 60 copies: some 60 windows of 18 bytes each."""

    def __init__(self, sr):
        rng = np.random.default_rng(5)
        unit = rng.choice(ACGT, 29)
        self.ref = np.concatenate([rng.choice(ACGT, 700), np.tile(unit, 60), rng.choice(ACGT, 700)])
        self.idx = [sr.Index.build(bytes(self.ref), seed_len=20, address_bases=10)]
        self.session = sr.Session.from_indexes(self.idx)
        self.session.attach_index(self.idx)

    def reads(self, n):
        import torch
        p = 700 + 29 * 2 + np.arange(n) % 1000
        bases = np.lib.stride_tricks.sliding_window_view(self.ref, 100)[p].reshape(-1).copy()
        return torch.from_numpy(bases).cuda(), torch.arange(n + 1, dtype=torch.int64).cuda() * 100

    def list(self, rd):
        return self.session.candidates(*rd, merge_dist=0, pad=4, out_device=True)


def test_large_lists_are_not_kept():
    from paper_1805_00106_gb300 import sr
    r = _Repeat(sr)
    rd = r.reads(400_000)
    c = r.list(rd)
    block = 18 * c.n_cands
    assert block > 256 * MB
    del c  # the scratch is sized now
    before = _free()
    c = r.list(rd)
    held = before - _free()
    assert held > 0.9 * block
    del c
    assert _free() > before - 32 * MB


def test_kept_blocks_make_room_for_the_sessions_own_allocations():
    """With almost all device memory taken, a batch and a host list that need more than
    is free and less than is free and kept."""
    import torch
    from paper_1805_00106_gb300 import sr
    r = _Repeat(sr)
    rd = r.reads(100_000)
    n = 10_000
    w = S.reads([r.ref], n, 5, 100, 100)
    args = [w["bases"], w["read_off"], np.arange(n + 1), np.zeros(n, np.uint8), np.zeros(n, np.uint8), np.full(n, 700),
            np.full(n, 150)]
    s2 = sr.Session.open([bytes(r.ref)])
    torch.cuda.empty_cache()
    before = _free()
    b = s2.stage(*args)
    need = (before - _free()) * 4 // 5  # an arena has a quarter of headroom
    b.close()
    s2.close()
    want = sr.candidates(r.idx, rd[0].cpu().numpy(), rd[1].cpu().numpy(), merge_dist=0, pad=4)
    for kind in ("batch", "list"):
        c = r.list(rd)
        block = 18 * c.n_cands
        need = need if kind == "batch" else block
        assert need < 256 * MB and block < 256 * MB
        left = need // 2
        assert block > need - left + 16 * MB
        del c  # kept: `left` below is what others may still have
        torch.cuda.empty_cache()
        hold = torch.empty(_free() - left, dtype=torch.uint8, device="cuda")
        try:
            assert _free() < need
            if kind == "batch":
                b = r.session.stage(*args)
                b.run(sr.score_params(), sr.align_opts())
                assert len(b.fetch()["item_score"]) == n
                b.close()
            else:
                got = r.session.candidates(*rd, merge_dist=0, pad=4)
                assert all(np.array_equal(np.asarray(want[k], np.int64), np.asarray(got[k], np.int64)) for k in KEYS)
        finally:
            del hold
            torch.cuda.empty_cache()
