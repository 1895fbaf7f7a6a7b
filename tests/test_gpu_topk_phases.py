"""Top-K where its selection can go wrong: item counts around the single-phase limit and around tiles, every kernel's range of
query counts, items in the unlucky order (every item better than all before it: candidate lists overflow and are cut back
in place), equal scores everywhere, exclusion lists that hold the best items.  Scores are exact integers in fp32 (every partial
sum below 2^24), so ids and scores must be the full sort's; no tolerance."""
import numpy as np
import pytest

from oracle import evaluation as ev
from synth import graphs

pytestmark = pytest.mark.gpu
COLS = 1


def _tables(order, n, m, d, seed):
    rng = np.random.default_rng(seed)
    H, Q = np.zeros((n, d)), np.zeros((m, d))
    i = np.arange(n)
    if order == "random":
        return rng.integers(-4, 5, (n, d)).astype(np.float64), rng.integers(-4, 5, (m, d)).astype(np.float64)
    if order == "ascending":          # score = id
        H[:, 0], H[:, d - 1] = i // 256, i % 256
        Q[:, 0], Q[:, d - 1] = 256, 1
    else:                             # "equal": two scores only
        H[:, 3] = i % 2
        Q[:, 3] = 1
    return H, Q


@pytest.mark.parametrize("d,storage", [(16, "bf16"), (32, "f32"), (64, "bf16"), (128, "f32"), (128, "bf16")])
@pytest.mark.parametrize("order,n,m,k", [("random", 16384, 4, 20), ("random", 16385, 8, 50), ("random", 40001, 17, 256),
                                         ("ascending", 33000, 3, 10), ("ascending", 33000, 130, 64), ("equal", 30000, 65, 40),
                                         ("equal", 20000, 9, 256), ("random", 511, 129, 1)])
def test_topk_is_the_full_sort(order, n, m, k, d, storage):
    from paper_2112_02194_b200 import Alx
    H, Q = _tables(order, n, m, d, 31 * d + n)
    a = Alx(10, n, d, 0.05, 0.01, storage=storage)
    a.set_embeddings(COLS, graphs.to_storage_bits(H, storage))
    best = ev.topk(Q, H, k)[0]
    some = [np.sort(best[q, : (q * 7) % (k + 1)]) for q in range(m)]
    ptr = np.concatenate([[0], np.cumsum([s.size for s in some])]).astype(np.int64)
    for exclude in (None, (ptr, np.concatenate(some).astype(np.int32))):
        ids, sc = a.topk(COLS, Q, k, exclude=exclude)
        o_ids, o_sc = ev.topk(Q, H, k, exclude=exclude)
        np.testing.assert_array_equal(ids, o_ids)
        np.testing.assert_array_equal(sc.astype(np.float64), o_sc)
    a.destroy()
