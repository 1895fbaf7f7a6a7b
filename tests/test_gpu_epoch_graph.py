"""Replayed epochs (a small matrix's third alx_epoch and later) against the same half-epochs launched one by one: the same bits, the
same counters, times that move; a new matrix on the same context starts over."""
import numpy as np
import pytest

from tests import problems

pytestmark = pytest.mark.gpu
ROWS, COLS = 0, 1


@pytest.mark.parametrize("index", [0, 1, 2, 4, 6, 9])
def test_replayed_epochs_are_the_half_epochs(index):
    from paper_2112_02194_b200 import Alx
    p = problems.small_suite()[index]()
    ctx = []
    for _ in range(2):
        a = Alx(p.n_rows, p.n_cols, p.d, p.lam, p.alpha, storage=p.storage, split=p.split)
        a.set_csr(p.rowptr, p.colidx, p.values)
        a.set_embeddings(ROWS, p.W0)
        a.set_embeddings(COLS, p.H0)
        ctx.append(a)
    a, b = ctx
    dt = "bf16" if p.storage == "bf16" else "f32"
    for epoch in range(6):
        a.epoch()
        b.half_epoch(ROWS)
        b.half_epoch(COLS)
        if epoch % 2:
            assert a.loss() == b.loss()
        for side in (ROWS, COLS):
            np.testing.assert_array_equal(a.get_embeddings(side, dtype=dt), b.get_embeddings(side, dtype=dt))
        s, t = a.get_stats(), b.get_stats()
        assert (s.kernel_launches, s.cg_rows, s.cg_products, s.dual_rows, list(s.kernel_path)) == \
               (t.kernel_launches, t.cg_rows, t.cg_products, t.dual_rows, list(t.kernel_path))
        assert 0.0 < s.ms_half_epoch < 1000.0 and s.ms_gramian > 0.0
    # another matrix on the same context: half of the rows
    keep = p.rowptr[: p.n_rows + 1].copy()
    half = p.n_rows // 2
    keep[half:] = keep[half]
    for c in ctx:
        c.set_csr(keep, p.colidx[: keep[-1]], None if p.values is None else p.values[: keep[-1]])
    for _ in range(4):
        a.epoch()
        b.half_epoch(ROWS)
        b.half_epoch(COLS)
    for side in (ROWS, COLS):
        np.testing.assert_array_equal(a.get_embeddings(side, dtype=dt), b.get_embeddings(side, dtype=dt))
    a.destroy()
    b.destroy()
