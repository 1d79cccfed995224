"""Score sets with mismatch > gap open + gap extend (linear gaps among them) run the
kernels, shapes and launch rule that every other score set runs."""
import numpy as np
import pytest

from paper_1805_00106_gb300 import synth as S
from tests.parity import compare, gpu_run, oracle_run

pytestmark = pytest.mark.gpu

KEYS = ("bases", "read_off", "cand_off", "c_ref", "c_strand", "c_start", "c_len")
SHAPES = ([(4, r) for r in range(16, 33, 4)] + [(8, r) for r in [8, 10, *range(12, 33)]] + [(16, r) for r in range(5, 17)] +
          [(32, r) for r in range(4, 9)])


def _batch(n, lo, hi, windows, seed=5):
    ref = S.ref_iid(100_000, 9, gc=0.41)
    rd = S.reads([ref], n, seed, lo, hi, 0.02, 0.004, 0.5)
    return dict(refs=[ref], **rd, **S.cands(rd, [len(ref)], seed + 1, S.COUNT_FIXED, windows, 32))


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("n,lo,hi", [(9, 75, 250), (2000, 75, 250), (4000, 100, 100), (20_000, 75, 250)])
@pytest.mark.parametrize("shape", [{}, dict(lanes=16, rows=16)])
def test_the_launches_of_other_score_sets(mode, n, lo, hi, shape):
    """One launch for few pairs, a kernel per length class for many or for a given
    shape: as many kernels under 2/-3 with linear gaps of 2 as under 2/-3 with 5 + 2."""
    from paper_1805_00106_gb300 import sr
    w = _batch(n, lo, hi, 4)
    s = sr.Session.open([bytes(r) for r in w["refs"]])
    b = s.stage(*[w[k] for k in KEYS])
    kernels = []
    for sp in ((2, 3, 0, 2), (2, 3, 5, 2)):
        b.run(sr.score_params(*sp), sr.align_opts(mode=mode, want_cigar=False, **shape))
        kernels.append(b.stats()["kernels"])
    b.close()
    assert kernels[0] == kernels[1]


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("sp", [(2, 3, 0, 2), (2, 8, 5, 2)])
def test_every_shape_against_the_oracle(mode, sp):
    from paper_1805_00106_gb300 import sr
    s, done = None, {}
    for lanes, rows in SHAPES:
        top = min(lanes * rows, 256)
        if top not in done:
            w = _batch(24, max(top - 60, 1), top, 3, seed=top)
            done[top] = w, oracle_run(w, sp=sp, mode=mode)
        w, o = done[top]
        s = s or sr.Session.open([bytes(r) for r in w["refs"]])
        assert not compare(gpu_run(s, w, sp=sp, mode=mode, lanes=lanes, rows=rows), o), (lanes, rows)
    for lanes, rows in ((16, 16), (32, 8)):  # and the one-launch-per-batch engine
        w = _batch(24, 100, 256, 3)
        assert not compare(gpu_run(s, w, sp=sp, mode=mode, engine=1, lanes=lanes, rows=rows), oracle_run(w, sp=sp, mode=mode))


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("sp", [(2, 3, 0, 2), (2, 8, 5, 2)])
def test_one_launch_and_a_kernel_per_class_agree(mode, sp):
    from paper_1805_00106_gb300 import sr
    w = _batch(300, 1, 256, 3)
    s = sr.Session.open([bytes(r) for r in w["refs"]])
    few = gpu_run(s, w, sp=sp, mode=mode)
    assert not compare(few, oracle_run(w, sp=sp, mode=mode))
    t, lens, n = 60, np.diff(w["read_off"]), np.diff(w["cand_off"])
    many = dict(w, bases=np.tile(w["bases"], t), read_off=np.concatenate([[0], np.cumsum(np.tile(lens, t))]),
                cand_off=np.concatenate([[0], np.cumsum(np.tile(n, t))]),
                **{k: np.tile(w[k], t) for k in ("c_ref", "c_strand", "c_start", "c_len")})
    got = gpu_run(s, many, sp=sp, mode=mode)
    for k in ("item_score", "item_end"):
        assert np.array_equal(got[k], np.tile(few[k], t)), k
