"""Device memory of a batch: no more than when the packets were sorted by
digit passes, so that a budget that held a batch then still does; signed
combinations, whose scratch shares those regions, stay exact."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (window lengths, sum, matrices, tuning): bytes with the digit passes
SHAPES = [
    ((131_072,), False, True, {}, 10_639_104),
    ((262_145,), False, True, {}, 21_920_768),
    ((1 << 21,), False, True, {}, 169_905_408),
    ((131_072,) * 64, True, False, {}, 1_083_076_864),
    ((131_072,) * 64, True, False, {"sum_path": 2, "agg_path": 3}, 1_099_854_592),
    ((131_072,) * 64, False, False, {"agg_path": 1}, 1_116_625_408),
    ((40_000,) * 3, True, False, {}, 15_904_512),
    ((131_072,) * 128, True, False, {}, 2_205_028_608),
]


@pytest.mark.parametrize("lens,want_sum,mats,tuning,before", SHAPES)
def test_a_batch_fits_the_memory_it_took(lens, want_sum, mats, tuning, before):
    from paper_2510_14050_gb300 import ans
    offs = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    flags = (ans.BATCH_SUM if want_sum else 0) | (ans.BATCH_MATRICES if mats else 0)
    probe = ans.Context(0)
    probe.set_tuning(**tuning)
    assert probe.batch_bytes(offs, flags) <= before
    held = probe.memory()[0]
    probe.close()
    src, dst = (torch.randint(0, 1 << 20, (int(offs[-1]),), dtype=torch.int32, device="cuda") for _ in range(2))
    tables = sum(12 << max(13, (2 * n - 1).bit_length()) for n in lens) if tuning.get("agg_path") == 1 else 0
    ctx = ans.Context(0, budget_bytes=held + before + tables)
    ctx.set_tuning(**tuning)
    _, _, tk = ctx.batch_submit(src, dst, offs, flags)
    ctx.wait(tk)
    ctx.close()


@pytest.mark.parametrize("n", [1, 8192, 8193, 100_000])
def test_signed_combinations(n):
    from paper_2510_14050_gb300 import ans
    rng = np.random.default_rng(n)
    parts = [(rng.integers(0, 500, n, dtype=np.uint32), rng.integers(0, 500, n, dtype=np.uint32)) for _ in range(3)]
    ctx = ans.Context(0)
    ms = [ctx.build_window(*(torch.from_numpy(x.view(np.int32)).cuda() for x in p)) for p in parts]
    total = ctx.sum_windows(ms)
    got = ctx.combine([total, ms[0], ms[2]], [1, -1, -1])  # only the middle one is left
    exp = oracle.traffic_matrix(*parts[1])
    for x, y in zip(got.to_numpy(), exp):
        np.testing.assert_array_equal(x, y)
    assert got.quantities() == oracle.network_quantities(exp)
    for x in (*ms, total, got):
        x.free()
    ctx.close()


@pytest.mark.parametrize("guards", ["0", "1"])
@pytest.mark.parametrize("lens", [(1,), (5000, 0, 9000)])
def test_batch_bytes_is_what_a_batch_takes(lens, guards, monkeypatch):
    """In the debug mode too, whose guards take memory of their own."""
    from paper_2510_14050_gb300 import ans
    monkeypatch.setenv("ANS_SCRATCH_GUARDS", guards)
    offs = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    src, dst = (torch.randint(0, 99, (int(offs[-1]),), dtype=torch.int32, device="cuda") for _ in range(2))
    ctx = ans.Context(0)
    need, held = ctx.batch_bytes(offs, ans.BATCH_MATRICES | ans.BATCH_SUM), ctx.memory()[0]
    mats, summ, tk = ctx.batch_submit(src, dst, offs, ans.BATCH_MATRICES | ans.BATCH_SUM)
    ctx.wait(tk)
    assert ctx.memory()[0] - held == need
    for m in [*mats, summ]:
        m.free()
    ctx.close()
