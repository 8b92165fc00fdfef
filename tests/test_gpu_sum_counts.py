"""Sums of imported matrices whose packets, added up, pass the 62 bits in which
a matrix's packets are counted: the sums' other quantities and values stay
exact (32-bit counts may be taken only for sums below 2^32)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _matrix(rows, vals):
    """One link per row, (r, 7 + r)."""
    n = len(rows)
    return oracle.DCSR(np.array(rows, dtype=np.uint32), np.arange(n + 1, dtype=np.uint64),
                       np.array(rows, dtype=np.uint32) + np.uint32(7), np.array(vals, dtype=np.uint64))


BIG = 1 << 61


@pytest.mark.parametrize("tuning", [{}, {"sum_path": 1}, {"col_hash": 0}])
@pytest.mark.parametrize("vals", [(BIG, BIG), (BIG, BIG, 5), (BIG - 1, BIG - 1, 2), (1 << 60,) * 4,
                                  (BIG - 1, BIG - 1, 7), (3, 4), ((1 << 32) - 1, 1), (1 << 40, 2)])
def test_sums_and_combinations(vals, tuning):
    from paper_2510_14050_gb300 import ans
    a, b = _matrix(range(len(vals)), vals), _matrix([100, 101], [1, 2])
    ctx = ans.Context(0)
    ctx.set_tuning(**tuning)
    ma, mb = ctx.import_matrix(*a), ctx.import_matrix(*b)
    for x in (ma, mb):
        x.view()  # computed: its packets are known
    exp = oracle.sum_matrices([a, b])
    eq = oracle.network_quantities(exp)
    both = ctx.sum_windows([ma, mb])
    results = [(both, exp, eq)]
    if max(vals) < BIG:  # signed combinations hold counts below 2^61
        results.append((ctx.combine([both, mb], [1, -1]), a, oracle.network_quantities(a)))
    for got, want, q in results:
        for x, y in zip(got.to_numpy(), want):
            np.testing.assert_array_equal(x, y)
        gq = got.quantities()
        assert gq.pop("valid_packets") == q.pop("valid_packets") % (1 << 62)
        assert gq == q
        got.free()
    for x in (ma, mb):
        x.free()
    ctx.close()
