"""Batches that end in, or consist of, empty windows: nothing is written past
the plan's last tile, and results that no tile writes are still written."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TILE = 8192


def _packets(n, seed):
    rng = np.random.default_rng(seed)
    return rng.zipf(1.3, n).astype(np.uint32), rng.integers(0, 5000, n, dtype=np.uint32)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()


def _check(ans, ctx, src, dst, offs, flags, device=False):
    o = torch.from_numpy(offs.astype(np.int64)).cuda() if device else offs
    out = torch.full((len(offs) - 1, 9), -1, dtype=torch.int64, device="cuda")
    mats, summ, tk = ctx.batch_submit(_dev(src), _dev(dst), o, flags, out=out)
    assert ctx.wait_status(tk) == ans.OK
    emats, eq, esum = oracle.batch(src, dst, offs)
    assert ans.quantities_from_tensor(out) == eq
    for m, e in [*zip(mats or [], emats), *([(summ, esum)] if summ else [])]:
        for x, y in zip(m.to_numpy(), e):
            np.testing.assert_array_equal(x, y)
        assert m.quantities() == oracle.network_quantities(e)
        m.free()


# 32 full tiles: the regions of the sort's bucket counts end without padding
@pytest.mark.parametrize("tuning", [{}, {"sum_path": 2}, {"agg_path": 3}])
@pytest.mark.parametrize("lens", [(32 * TILE, 0), (0, 32 * TILE, 0, 0), (TILE,) * 32 + (0,), (5, 0), (0, 2 * TILE + 1, 0)])
def test_nothing_is_written_behind_the_last_tile(lens, tuning, monkeypatch):
    from paper_2510_14050_gb300 import ans
    offs = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    src, dst = _packets(int(offs[-1]), len(lens))
    monkeypatch.setenv("ANS_SCRATCH_GUARDS", "1")
    ctx = ans.Context(0)
    ctx.set_tuning(**tuning)
    for flags in (0, ans.BATCH_MATRICES, ans.BATCH_SUM):
        for device in (False, True):
            _check(ans, ctx, src, dst, offs, flags, device)
    ctx.close()


class _Dirty:
    """Allocator hooks whose blocks come filled with 0x55."""

    def __init__(self, ans):
        self.live = {}

        def _alloc(nbytes, stream, user):
            t = torch.full((int(nbytes),), 0x55, dtype=torch.uint8, device="cuda")
            torch.cuda.synchronize()
            self.live[t.data_ptr()] = t
            return t.data_ptr()

        def _free(ptr, stream, user):
            if ptr:
                torch.cuda.synchronize()
                del self.live[ptr]

        self.alloc_fn = ans.ALLOC_FN(_alloc)
        self.free_fn = ans.FREE_FN(_free)


@pytest.mark.parametrize("tuning", [{}, {"sum_path": 1}, {"sum_path": 2}, {"agg_path": 1}, {"agg_path": 3}])
@pytest.mark.parametrize("lens", [(0,), (0, 0, 0)])
def test_only_empty_windows(lens, tuning):
    from paper_2510_14050_gb300 import ans
    offs = np.full(len(lens) + 1, 3, dtype=np.uint64)
    src, dst = _packets(5, 1)
    ctx = ans.Context(0, allocator=_Dirty(ans))
    ctx.set_tuning(**tuning)
    for cap in (0, 2 * TILE):
        ctx.set_batch_capacity(cap)
        for device in (False, True):
            for flags in (ans.BATCH_SUM, ans.BATCH_MATRICES | ans.BATCH_SUM):
                _check(ans, ctx, src, dst, offs, flags, device)
    ctx.close()
