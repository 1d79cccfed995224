"""sr_batch_classify classifies the results of the batch's last run, whatever stream
that was enqueued on and however far it is."""
import numpy as np
import pytest

from paper_1805_00106_gb300 import synth as S

pytestmark = pytest.mark.gpu


def test_classify_follows_a_run_on_another_stream():
    import torch
    from paper_1805_00106_gb300 import sr
    a = S.ref_iid(50_000, 3)
    refs = [a, S.mutate(a, 4, 0.15, 0.02, 2, 1_000, 5_000)]
    s = sr.Session.open([bytes(r) for r in refs])
    rd = S.reads(refs, 3_000, 5, 30, 60, 0.01, 0.001, 0.5, weights=[0.5, 0.5])
    w = dict(**rd, **S.cands(rd, [len(r) for r in refs], 6, S.COUNT_UNIFORM, 8, 32, cap_per_read=8))
    args = [w[k] for k in ("bases", "read_off", "cand_off", "c_ref", "c_strand", "c_start", "c_len")]
    b = s.stage(*args)
    b.run(sr.score_params(), sr.align_opts(want_cigar=False))
    want = b.classify()
    b.run(sr.score_params(1, 3, 5, 2), sr.align_opts(want_cigar=False))  # scores of at most 60, the least is 40
    assert (b.classify() != want).mean() > 0.1
    b.close()
    for _ in range(3):
        st = torch.cuda.Stream()
        b = s.stage(*args)
        b.run(sr.score_params(1, 3, 5, 2), sr.align_opts(want_cigar=False))  # other records in the arena
        with torch.cuda.stream(st):
            torch.cuda._sleep(60_000_000)
        b.run_async(sr.score_params(), sr.align_opts(want_cigar=False, stream=st.cuda_stream))
        got = b.classify()
        b.sync()
        b.close()
        assert np.array_equal(got, want)
