"""The objective by tensor-core products (bfloat16 tables of 128 features, rows of 16 entries or more on average) and on the other
side of that line: rows that begin and end at every place of a 16-entry step, rows without entries, a last step that is not full."""
import numpy as np
import pytest

from oracle import ials
from tests import problems
from tests.test_gpu_parity import COLS, ROWS, make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("labels", [False, True])
@pytest.mark.parametrize("degrees", [[16], [1, 31, 2, 30, 15, 17], [0, 0, 48, 0, 1, 33], [500, 3, 0, 1, 1, 1, 700], [15] * 33 + [1], [3, 1, 0, 7]],
                         ids=["16", "odd", "empty", "long", "15", "short"])
@pytest.mark.parametrize("repeat", [1, 40])
def test_observed_term_matches_the_oracle(degrees, repeat, labels):
    rng = np.random.Generator(np.random.PCG64(len(degrees) + repeat))
    deg = np.asarray(degrees * repeat, dtype=np.int64)
    n_cols = 901
    rowptr = np.zeros(deg.size + 1, dtype=np.int64)
    rowptr[1:] = np.cumsum(deg)
    colidx = np.concatenate([np.sort(rng.choice(n_cols, int(k), replace=False)) for k in deg]).astype(np.int32)
    vals = rng.uniform(0.25, 2.0, colidx.size).astype(np.float32) if labels else None
    W0, H0 = problems._tables(deg.size, n_cols, 128, 5, "bf16")
    p = problems.Problem("loss", deg.size, n_cols, 128, 0.05, 0.003, "bf16", rowptr, colidx, vals, W0, H0)
    a = make_ctx(p)
    total, parts = a.loss()
    ref, ref_parts = ials.loss(rowptr, colidx, None if vals is None else vals.astype(np.float64), p.f64(W0), p.f64(H0), p.alpha, p.lam)
    # a dot product of 128 exact products is off by at most 128 x 2^-24 of the sum of their sizes; as the suite's gate
    np.testing.assert_allclose(parts, ref_parts, rtol=1e-6, atol=1e-12 * ref)
    assert a.loss()[0] == total      # a fixed order of sums
    a.destroy()
