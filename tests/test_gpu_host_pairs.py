"""Batches whose pairs lie in page-locked host memory (run_pairs in
csrc/ans_abi.cu): copied to the device by a kernel where the sorts read them
more than once, read in place otherwise and where the copy does not fit; exact
against the oracle and equal errors, with offsets on the host and on the
device."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CHIP = 1 << 17  # largest window sorted on chip
PIECE = 1 << 14  # packets of a copied piece


def _pinned(n, seed):
    rng = np.random.default_rng(seed)
    src, dst = rng.zipf(1.4, n).astype(np.uint32), rng.integers(0, 300, n, dtype=np.uint32)
    return src, dst, *(torch.from_numpy(x.view(np.int32)).pin_memory() for x in (src, dst))


def _check(ans, ctx, src, dst, ps, pd, offs, device):
    o = torch.from_numpy(offs.astype(np.int64)).cuda() if device else offs
    out = torch.zeros((len(offs) - 1, 9), dtype=torch.int64, device="cuda")
    mats, summ, tk = ctx.batch_submit(ps, pd, o, ans.BATCH_MATRICES | ans.BATCH_SUM, out=out)
    ctx.wait(tk)
    a, b = int(offs[0]), int(offs[-1])
    emats, eq, esum = oracle.batch(src[a:b], dst[a:b], offs - offs[0])
    assert ans.quantities_from_tensor(out) == eq
    for m, e in [*zip(mats, emats), (summ, esum)]:
        for x, y in zip(m.to_numpy(), e):
            np.testing.assert_array_equal(x, y)
        m.free()


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("tuning", [{}, {"sum_path": 2}, {"agg_path": 3, "sum_path": 2}, {"agg_path": 1}])
@pytest.mark.parametrize("lens", [(1,), (PIECE - 1, 0, 2), (PIECE, PIECE), (CHIP,), (5, CHIP + 1), (3 * PIECE + 7,) * 5])
def test_batches(lens, tuning, device):
    from paper_2510_14050_gb300 import ans
    offs = np.concatenate([[3], 3 + np.cumsum(lens)]).astype(np.uint64)  # an odd first packet
    src, dst, ps, pd = _pinned(int(offs[-1]) + 2, len(lens))
    ctx = ans.Context(0)
    ctx.set_tuning(**tuning)
    _check(ans, ctx, src, dst, ps, pd, offs, device)
    if device:  # a capacity above the batch, then one below it
        ctx.set_batch_capacity(2 * int(offs[-1]))
        _check(ans, ctx, src, dst, ps, pd, offs, device)
        if lens[0] > 1:
            ctx.set_batch_capacity(int(offs[-1] - offs[0]) - 1)
            with pytest.raises(ans.AnsError):
                _check(ans, ctx, src, dst, ps, pd, offs, device)
    ctx.close()


@pytest.mark.parametrize("tuning", [{}, {"sum_path": 2}])
@pytest.mark.parametrize("lens", [(1,), (0, PIECE - 1, 0, 2), (PIECE, PIECE + 1, 5), (3 * PIECE + 7,) * 3, (7, CHIP + 1)])
@pytest.mark.parametrize("mixed", [False, True])
def test_windows_in_their_own_arrays(lens, tuning, mixed):
    from paper_2510_14050_gb300 import ans
    offs = np.concatenate([[3], 3 + np.cumsum(lens)]).astype(np.uint64)
    src, dst, ps, pd = _pinned(int(offs[-1]), len(lens))
    wins = [(ps[int(a):int(b)], pd[int(a):int(b)]) for a, b in zip(offs[:-1], offs[1:])]
    if mixed:  # every second window on the device
        wins = [(s.cuda(), d.cuda()) if i % 2 else (s, d) for i, (s, d) in enumerate(wins)]
    emats, eq, esum = oracle.batch(src[3:], dst[3:], offs - offs[0])
    ctx = ans.Context(0)
    ctx.set_tuning(**tuning)
    for budget in (0, 1):
        out = torch.zeros((len(lens), 9), dtype=torch.int64, device="cuda")
        mats, summ, tk = ctx.batch_submit_windows(wins, ans.BATCH_MATRICES | ans.BATCH_SUM, out=out)
        ctx.wait(tk)
        assert ans.quantities_from_tensor(out) == eq
        for m, e in [*zip(mats, emats), (summ, esum)]:
            for x, y in zip(m.to_numpy(), e):
                np.testing.assert_array_equal(x, y)
            m.free()
        if budget == 0:  # again without room for a copy beside the batch
            ctx.close()
            probe = ans.Context(0)
            need = probe.batch_bytes(offs, ans.BATCH_MATRICES | ans.BATCH_SUM)
            probe.close()
            ctx = ans.Context(0, budget_bytes=need + 4096)
    ctx.close()


@pytest.mark.parametrize("device", [False, True])
def test_decreasing_offsets_stay_refused(device):
    from paper_2510_14050_gb300 import ans
    src, dst, ps, pd = _pinned(1000, 1)
    ctx = ans.Context(0)
    ctx.set_tuning(sum_path=2)
    for bad in ([0, 10, 5, 1000], [7, 3, 900]):
        with pytest.raises(ans.AnsError):
            _check(ans, ctx, src, dst, ps, pd, np.array(bad, dtype=np.uint64), device)
    ctx.close()


@pytest.mark.parametrize("device", [False, True])
def test_budget_without_room_for_the_copy(device):
    """A budget that holds the batch and not the copy beside it."""
    from paper_2510_14050_gb300 import ans
    n = 1 << 19
    src, dst, ps, pd = _pinned(n, 2)
    offs = np.array([0, n // 2, n], dtype=np.uint64)
    probe = ans.Context(0)
    probe.set_tuning(sum_path=2)
    if device:
        dev = [x.cuda() for x in (ps, pd)]
        o = torch.from_numpy(offs.astype(np.int64)).cuda()
        mats, summ, tk = probe.batch_submit(*dev, o, ans.BATCH_MATRICES | ans.BATCH_SUM)
        probe.wait(tk)
        need = probe.memory()[0]
        for m in [*mats, summ]:
            m.free()
    else:
        need = probe.batch_bytes(offs, ans.BATCH_MATRICES | ans.BATCH_SUM)
    probe.close()
    ctx = ans.Context(0, budget_bytes=need + (1 << 20))
    ctx.set_tuning(sum_path=2)
    _check(ans, ctx, src, dst, ps, pd, offs, device)
    ctx.close()


@pytest.mark.parametrize("where", ["device", "pinned", "pageable"])
@pytest.mark.parametrize("shift", [0, 1, 4, 8])
def test_quantities_at_any_address(where, shift):
    """The array of quantities is written byte by byte where its address is
    no multiple of a word."""
    from paper_2510_14050_gb300 import ans
    lens = (20_000, 0, 3)
    offs = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    src, dst, ps, pd = _pinned(int(offs[-1]), 4)
    room = torch.full((len(lens) * 72 + 16,), 7, dtype=torch.uint8)
    room = room.cuda() if where == "device" else room.pin_memory() if where == "pinned" else room
    ctx = ans.Context(0)
    out = room[shift:shift + len(lens) * 72]
    _, _, tk = ctx.batch_submit(ps.cuda(), pd.cuda(), offs, out=out)
    ctx.wait(tk)
    got = np.frombuffer(bytes(out.cpu().numpy()), dtype=np.int64)
    assert ans.quantities_from_tensor(got) == oracle.batch(src, dst, offs, want_sum=False)[1]
    assert bool((room[:shift].cpu() == 7).all()) and bool((room[shift + len(lens) * 72:].cpu() == 7).all())
    ctx.close()


@pytest.mark.parametrize("call", ["host", "device", "windows", "windows_one_segment"])
def test_a_refused_batch_reads_nothing(call):
    """A budget that holds the copy of the pairs and not the batch: refused
    with nothing on the stream that reads them (their copy alone would take 2.5
    ms over the host link)."""
    from paper_2510_14050_gb300 import ans
    n = 1 << 26
    ps, pd = (torch.zeros(n, dtype=torch.int32).pin_memory() for _ in range(2))
    offs = np.array([0, n // 2, n], dtype=np.uint64)
    o = torch.from_numpy(offs.astype(np.int64)).cuda() if call == "device" else offs
    ctx = ans.Context(0, budget_bytes=9 * n)
    if call == "windows_one_segment":
        ctx.set_tuning(sum_path=2)
    if call == "device":
        ctx.set_batch_capacity(n)  # (its offsets are not read back)

    def refused():
        with pytest.raises(ans.AnsError) as e:
            if call.startswith("windows"):
                ctx.batch_submit_windows([(ps[:n // 2], pd[:n // 2]), (ps[n // 2:], pd[n // 2:])], ans.BATCH_SUM)
            else:
                ctx.batch_submit(ps, pd, o, ans.BATCH_SUM)
        assert e.value.code == ans.ERR_BUDGET

    refused()  # (its memory is mapped now)
    before, after = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    torch.cuda._sleep(100_000_000)  # about 50 ms of device time: the host's is hidden behind it
    before.record()
    refused()
    after.record()
    torch.cuda.synchronize()
    assert before.elapsed_time(after) < 1.0
    ctx.close()


class _RefuseOnce:
    """Allocator hooks that refuse the first allocation once armed."""

    def __init__(self, ans):
        self.live, self.armed, self.refused = {}, False, []

        def _alloc(nbytes, stream, user):
            if self.armed:
                self.armed = False
                self.refused.append(int(nbytes))
                return None
            t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
            self.live[t.data_ptr()] = t
            return t.data_ptr()

        def _free(ptr, stream, user):
            if ptr:
                torch.cuda.synchronize()
                del self.live[ptr]

        self.alloc_fn = ans.ALLOC_FN(_alloc)
        self.free_fn = ans.FREE_FN(_free)


@pytest.mark.parametrize("tuning", [{}, {"sum_path": 2}, {"sum_path": 1, "agg_path": 2}, {"agg_path": 3}])
@pytest.mark.parametrize("lens", [(1,), (0, PIECE - 1, 0, 2), (3 * PIECE + 7,) * 3, (7, CHIP + 1)])
def test_windows_in_place_when_their_copy_is_refused(lens, tuning):
    """The tuning is kept on the way to the fallback, which is seen to run: a
    sum by re-sorting the packets is merged instead when they lie apart."""
    from paper_2510_14050_gb300 import ans
    offs = np.concatenate([[3], 3 + np.cumsum(lens)]).astype(np.uint64)
    src, dst, ps, pd = _pinned(int(offs[-1]), len(lens))
    wins = [(ps[int(a):int(b)], pd[int(a):int(b)]) for a, b in zip(offs[:-1], offs[1:])]
    emats, eq, esum = oracle.batch(src[3:], dst[3:], offs - offs[0])
    hooks = _RefuseOnce(ans)
    ctx = ans.Context(0, allocator=hooks)
    ctx.set_tuning(**tuning)
    for refuse in (False, True, False):
        hooks.armed = refuse
        ctx.profile(True)
        out = torch.zeros((len(lens), 9), dtype=torch.int64, device="cuda")
        mats, summ, tk = ctx.batch_submit_windows(wins, ans.BATCH_MATRICES | ans.BATCH_SUM, out=out)
        ctx.wait(tk)
        ran = set(ctx.profile_read())
        ctx.profile(False)
        assert ans.quantities_from_tensor(out) == eq
        for m, e in [*zip(mats, emats), (summ, esum)]:
            for x, y in zip(m.to_numpy(), e):
                np.testing.assert_array_equal(x, y)
            m.free()
        if len(lens) > 1 and tuning in ({"sum_path": 2}, {"agg_path": 3}):
            assert ("merge" in ran) == refuse
        if refuse:  # the copy: the call's first allocation where no larger one is kept
            assert hooks.refused and hooks.refused[-1] >= 8 * int(offs[-1] - offs[0])
        if not refuse and tuning:  # the next copy is asked for again
            ctx.close()
            ctx = ans.Context(0, allocator=hooks)
            ctx.set_tuning(**tuning)
    ctx.close()
    assert not hooks.live
