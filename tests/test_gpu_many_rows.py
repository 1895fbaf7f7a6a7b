"""Where a side has rows enough to keep every SM busy, long rows stay with a warp (or with the team of four) instead of a block: the
other side of the line that the boundary problems of a few hundred rows cover.  And fold-in on one context, call after call."""
import numpy as np
import pytest

from tests.test_gpu_edges import boundary_problem
from tests.test_gpu_parity import _epoch_checks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,storage,values,kw", [(16, "f32", True, {}), (32, "bf16", False, {}), (64, "bf16", True, {}),
                                                 (64, "f32", False, {}), (64, "f32", True, dict(solver=1)), (128, "f32", False, {}),
                                                 (64, "bf16", False, dict(dual_cond_limit=1.0)),
                                                 (128, "f32", True, dict(dual_cond_limit=1.0))])
def test_boundary_lengths_among_many_rows(d, storage, values, kw):
    # 24 000 short rows: above 148 x 20 x 8 and 148 x 12 x 8; rows of up to 1100 entries (every column)
    p = boundary_problem(f"many_d{d}_{storage}", d, storage, 1100, 0, values, seed=90 + d, repeat=2, extra_rows=24_000)
    # (conjugate gradients of fp32 tables stop at a relative residual of 1e-6: cond(A) of a few thousand times that)
    _epoch_checks(p, raw_gate=(p.emb_tol, 10 * p.emb_tol), **kw)


@pytest.mark.parametrize("d,storage", [(16, "f32"), (64, "bf16"), (64, "f32"), (128, "f32"), (128, "bf16")])
def test_fold_in_again_and_again_on_one_context(d, storage):
    """Buffers, the second stream and the context for new rows are kept between calls: sizes that grow and shrink, with and
    without labels, give what a context of its own gives for each."""
    from paper_2112_02194_b200 import Alx
    rng = np.random.default_rng(7 * d)
    m = 3001
    H = (0.1 * rng.standard_normal((m, d))).astype(np.float32)

    def fresh():
        a = Alx(10, m, d, 0.05, 0.002, storage=storage)
        a.set_embeddings(1, H)
        return a

    kept = fresh()
    for i, n_new in enumerate([3, 700, 1, 255, 256, 2500, 40]):
        deg = rng.integers(0, 70, n_new)
        deg[:: 37] = 1200
        ptr = np.zeros(n_new + 1, dtype=np.int64)
        ptr[1:] = np.cumsum(deg)
        idx = np.concatenate([np.sort(rng.choice(m, int(k), replace=False)) for k in deg]).astype(np.int32)
        vals = rng.uniform(0.5, 2.0, idx.size).astype(np.float32) if i % 2 else None
        if i == 4:      # a call that is refused leaves nothing behind
            with pytest.raises(Exception):
                kept.fold_in(ptr, np.full_like(idx, m), vals)
        one = fresh()
        np.testing.assert_array_equal(kept.fold_in(ptr, idx, vals), one.fold_in(ptr, idx, vals))
        one.destroy()
    kept.destroy()
