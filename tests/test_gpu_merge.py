"""Merge rounds (csrc/ans_merge.cu) through sums of two and three matrices,
exact against the oracle: runs whose ends fall on and beside a thread's 8
outputs and a block's 2048 or 4096, empty and one-sided runs, equal links."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _links(n, rng, share):
    src = np.arange(n, dtype=np.uint32) * np.uint32(3 if share else 5)
    return src, rng.integers(0, 3, n, dtype=np.uint32)


@pytest.mark.parametrize("tile", [2048, 4096])
@pytest.mark.parametrize("sizes", [(1, 1), (8, 7), (9, 4095), (4096, 2048), (2047, 2049), (5000, 1, 4097),
                                   (12289, 12288, 8193), (70_000, 64)])
@pytest.mark.parametrize("share", [False, True])
def test_sum(sizes, tile, share):
    from paper_2510_14050_gb300 import ans
    rng = np.random.default_rng(sum(sizes) + share)
    pairs = [_links(n, rng, share and i == 0) for i, n in enumerate(sizes)]
    if share:
        pairs[-1] = tuple(x[:sizes[-1]] for x in _links(sizes[-1], np.random.default_rng(sum(sizes) + share), True))
    exp = oracle.traffic_matrix(*(np.concatenate(x) for x in zip(*pairs)))
    ctx = ans.Context(0)
    ctx.set_tuning(sum_path=0, merge_tile=tile)
    mats = [ctx.build_window(*(torch.from_numpy(x.view(np.int32)).cuda() for x in p)) for p in pairs]
    m = ctx.sum_windows(mats)
    for g, e in zip(m.to_numpy(), exp):
        np.testing.assert_array_equal(np.asarray(g), np.asarray(e))
    assert m.quantities() == oracle.network_quantities(exp)
    for x in [*mats, m]:
        x.free()
    ctx.close()
