"""A batch may be staged on one stream and run on another: sr_batch_stage returns
when its arrays are complete, however few they are and whatever its stream still has
to do before them."""
import numpy as np
import pytest

from paper_1805_00106_gb300 import synth as S
from tests.parity import compare, oracle_run

pytestmark = pytest.mark.gpu

KEYS = ("bases", "read_off", "cand_off", "c_ref", "c_strand", "c_start", "c_len")
BUSY = 60_000_000  # device clocks: some 30 ms


def _batch(ref, reads, windows, seed):
    rd = S.reads([ref], reads, seed, 30, 250, 0.02, 0.004, 0.5)
    return dict(refs=[ref], **rd, **S.cands(rd, [len(ref)], seed + 1, S.COUNT_FIXED, windows, 32))


# one copy up to 48 KB; the host check up to 4096 windows, a kernel above
SIZES = [(1, 1), (9, 6), (100, 4), (1500, 1), (1024, 4), (1100, 4), (20_000, 1)]


@pytest.mark.parametrize("reads,windows", SIZES)
def test_staging_is_complete_on_return(reads, windows):
    import torch
    from paper_1805_00106_gb300 import sr
    ref = S.ref_iid(50_000, 3)
    s = sr.Session.open([bytes(ref)])
    w = _batch(ref, reads, windows, 7)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        torch.cuda._sleep(BUSY)
    b = s.stage(*[w[k] for k in KEYS], stream=st.cuda_stream)
    assert st.query()
    b.close()


@pytest.mark.parametrize("reads,windows", SIZES[:5])
def test_staged_on_one_stream_run_on_another(reads, windows):
    """The arena is an earlier batch's; a run that did not wait would read its offsets."""
    import torch
    from paper_1805_00106_gb300 import sr
    ref = S.ref_iid(50_000, 3)
    s = sr.Session.open([bytes(ref)])
    old, w = _batch(ref, 3 * reads, windows + 1, 17), _batch(ref, reads, windows, 7)
    b = s.stage(*[old[k] for k in KEYS])
    b.run(sr.score_params(), sr.align_opts())
    b.close()
    st, run = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(st):
        torch.cuda._sleep(BUSY)
    b = s.stage(*[w[k] for k in KEYS], stream=st.cuda_stream)
    b.run(sr.score_params(), sr.align_opts(stream=run.cuda_stream))
    got = b.fetch()
    b.close()
    assert not compare(got, oracle_run(w))
    # and staged on the session's stream
    b = s.stage(*[w[k] for k in KEYS])
    b.run_async(sr.score_params(), sr.align_opts(stream=run.cuda_stream))
    again = b.fetch()
    b.close()
    assert all(np.array_equal(got[k], again[k]) for k in ("item_score", "item_end", "best", "cigar"))
