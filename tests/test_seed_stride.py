"""Seed strides up to the largest of their type: past a read's last seed position
only the seed at 0 is taken, on the host and on the device."""
import numpy as np
import pytest

from paper_1805_00106_gb300 import synth as S

from .test_host_stage import oracle_cands, same

KEYS = ["cand_off", "c_ref", "c_strand", "c_start", "c_len", "c_hits"]
STRIDES = [255, 256, 257, 300, 1 << 26, 1 << 27, 3 << 27, (1 << 27) + 1, (1 << 31) - 1, 1 << 31, (1 << 32) - 256, (1 << 32) - 1]


@pytest.fixture(scope="module")
def sr():
    from paper_1805_00106_gb300 import sr as _sr
    _sr.lib()
    return _sr


def _workload():
    ref, _ = S.ref_repeats(30_000, seed=5, rep_frac=0.5, n_families=20)
    rd = S.reads([ref], 60, 7, 20, 256, 0.01, 0.0, 0.3)
    junk = S.reads([S.ref_iid(30_000, 77)], 8, 9, 250, 256)  # seeds that are found nowhere
    off = np.concatenate([rd["read_off"], rd["read_off"][-1] + junk["read_off"][1:]])
    return dict(refs=[ref], bases=np.concatenate([rd["bases"], junk["bases"]]), read_off=off)


@pytest.mark.parametrize("stride", STRIDES)
def test_host_stage_takes_any_stride(sr, stride):
    w = _workload()
    idx = [sr.Index.build(bytes(w["refs"][0]), seed_len=16, address_bases=8)]
    g = sr.candidates(idx, w["bases"], w["read_off"], seed_stride=stride, merge_dist=10, pad=8)
    # reads of at most 256 bases: one seed of 16 each
    same(g, oracle_cands(w["refs"], w, 16, min(stride, 256), 10, 8))


def test_host_stage_strides_through_longer_reads(sr):
    """The host stage's reads have no length limit: a stride past 256 bases counts there."""
    ref = S.ref_iid(5_000, 3)
    idx = [sr.Index.build(bytes(ref), seed_len=16, address_bases=8)]
    off = np.array([0, 2_000])
    hits = [int(sr.candidates(idx, ref[100:2_100], off, seed_stride=s)["c_hits"].sum()) for s in (300, 1_000, 1_984, 1_985)]
    assert hits == [7, 2, 2, 1]


@pytest.mark.gpu
@pytest.mark.parametrize("table", ["1", "1000000"])
@pytest.mark.parametrize("stride", STRIDES)
def test_device_finder_takes_any_stride(sr, monkeypatch, table, stride):
    """The warp's, the block's and the large-read path's seed loops."""
    monkeypatch.setenv("SR_CAL_TABLE", table)
    w = _workload()
    idx = [sr.Index.build(bytes(w["refs"][0]), seed_len=16, address_bases=8)]
    s = sr.Session.from_indexes(idx)
    s.attach_index(idx)
    for prm in (dict(merge_dist=0, pad=4), dict(merge_dist=32, pad=32, max_cands=3)):
        h, d = (f(w["bases"], w["read_off"], seed_stride=stride, **prm) for f in
                (lambda *a, **k: sr.candidates(idx, *a, **k), s.candidates))
        for key in KEYS:
            assert np.array_equal(np.asarray(h[key], np.int64), np.asarray(d[key], np.int64)), (key, prm)
