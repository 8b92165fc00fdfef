"""Partitions of the column statistics with more destinations than a table
holds (csrc/ans_cols.cu): read in classes, or, in batches planned on the device
for more than 2^25 packets, cut into parts in memory; exact against the oracle
in both widths of the counts."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PART = 2731      # links of a partition aimed at
FILL = 3072      # destinations a table takes
SUBS = 512       # most parts of a partition
PARTS = 2048     # most partitions of a segment
ONES = 0xFFFFFFFF


def _unfmix32(h):
    """Inverse of MurmurHash3's 32-bit finalizer."""
    m = np.uint64(0xFFFFFFFF)

    def unxor(x, s):
        y = x.copy()
        for _ in range(32 // s + 1):
            y = x ^ (y >> np.uint64(s))
        return y & m

    x = unxor(np.asarray(h, dtype=np.uint64) & m, 16)
    x = x * np.uint64(pow(0xC2B2AE35, -1, 1 << 32)) & m
    x = unxor(x, 13)
    x = x * np.uint64(pow(0x85EBCA6B, -1, 1 << 32)) & m
    return unxor(x, 16).astype(np.uint32)


def _crowd(n, links, rng):
    """n destinations (all-ones among them) of the partition of the all-ones
    destination, in a segment of `links` links."""
    parts = min(PARTS, -(-links // PART))
    mixed = 0x81F16F39  # of the all-ones destination
    assert int(_unfmix32([mixed])[0]) == ONES
    p = mixed * parts >> 32
    lo, hi = -(-(p << 32) // parts), -(-((p + 1) << 32) // parts)
    step = (hi - lo) // n
    assert step >= 1
    return np.append(_unfmix32(lo + step * np.arange(n - 1, dtype=np.uint64)), np.uint32(ONES))


def _case(kind, n, rng):
    """Links (src, dst), all different, of about n destinations."""
    src = np.arange(n, dtype=np.uint32)
    if kind == "distinct":     # more destinations than all tables together hold
        return src, src * np.uint32(2654435761)
    if kind == "crowded":      # all of them in one partition
        return src, rng.permutation(_crowd(n, n, rng))
    # "late": the first links, nine of ten, meet few destinations of the
    # crowded partition: far fewer parts than the rest would need
    d = _crowd(n // 10, n, rng)
    return src, np.concatenate([d[src[:n - n // 10] % 3000], d])


@pytest.mark.parametrize("kind,n", [("distinct", 9_000_000), ("crowded", FILL + 1), ("crowded", 20_000),
                                    ("crowded", (1 << 18) + 5), ("crowded", SUBS * FILL // 4), ("crowded", 2_000_000),
                                    ("late", 200_000), ("late", 3_000_000)])
def test_window_and_import(kind, n):
    from paper_2510_14050_gb300 import ans
    rng = np.random.default_rng(n)
    src, dst = _case(kind, n, rng)
    exp = oracle.traffic_matrix(src, dst)
    eq = oracle.network_quantities(exp)
    ctx = ans.Context(0)
    m = ctx.build_window(*(torch.from_numpy(x.view(np.int32)).cuda() for x in (src, dst)))
    assert m.quantities() == eq
    big = exp._replace(vals=rng.integers(1, 1 << 40, len(exp[3]), dtype=np.uint64))
    mi = ctx.import_matrix(*big)
    bq = oracle.network_quantities(big)
    bq["valid_packets"] %= 1 << 62  # the width of a matrix's packet count
    assert mi.quantities() == bq
    assert ctx.network_quantities(mi) == bq
    for x in (m, mi):
        x.free()
    ctx.close()


@pytest.mark.parametrize("cap", [0, 1 << 26])
@pytest.mark.parametrize("kind,n", [("distinct", 8_500_000), ("crowded", 8 * FILL), ("crowded", 70_000),
                                    ("crowded", 2_000_000), ("late", 3_000_000)])
def test_device_planned_batch(kind, n, cap):
    """A long window between short ones; the capacity decides whether its
    partitions may be cut."""
    from paper_2510_14050_gb300 import ans
    rng = np.random.default_rng(n)
    lens = (5000, n, 0, 70_000)
    offs = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    parts = [rng.integers(0, 1 << 32, (2, 5000), dtype=np.uint32), np.stack(_case(kind, n, rng)),
             rng.integers(0, 1 << 12, (2, 70_000), dtype=np.uint32)]
    src, dst = np.concatenate(parts, axis=1)
    ctx = ans.Context(0)
    ctx.set_batch_capacity(cap)
    out = torch.zeros((len(lens), 9), dtype=torch.int64, device="cuda")
    ds, dd = (torch.from_numpy(x.view(np.int32)).cuda() for x in (src, dst))
    _, summ, tk = ctx.batch_submit(ds, dd, torch.from_numpy(offs.astype(np.int64)).cuda(), ans.BATCH_SUM, out=out)
    ctx.wait(tk)
    _, eq, esum = oracle.batch(src, dst, offs)
    assert ans.quantities_from_tensor(out) == eq
    assert summ.quantities() == oracle.network_quantities(esum)
    summ.free()
    ctx.close()
