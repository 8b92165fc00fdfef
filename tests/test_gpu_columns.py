"""Column statistics by hash partitions (csrc/ans_cols.cu) through the ABI,
exact against the oracle: partition and heavy-table limits, one destination
holding most links, the all-ones destination, 64-bit counts, and a partition
with more destinations than its table."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PART = 2731          # links of a partition aimed at
HEAVY = 1 << 18      # segments with a table of heavy destinations
SLOTS = 4096         # table slots


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


def _links(kind, n, rng):
    """About n distinct links (src, dst)."""
    src = np.arange(n, dtype=np.uint32) * np.uint32(2654435761)
    dst = rng.integers(0, 1 << 32, n, dtype=np.uint32)
    if kind == "heavy":  # a few destinations hold most links, one of them all-ones
        few = np.array([0xFFFFFFFF, 5, 6, 7], dtype=np.uint32)
        dst = np.where(rng.random(n) < 0.8, few[rng.integers(0, 4, n)], dst)
    elif kind == "one":
        dst[:] = 0xFFFFFFFF
    elif kind == "crowded":  # every destination's mix in the lowest partition
        parts = max(2, -(-n // PART))
        mixed = np.unique(rng.integers(0, (1 << 32) // parts, 2 * n))
        dst = _unfmix32(rng.permutation(mixed)[:n])
    return src, dst


@pytest.mark.parametrize("kind", ["random", "heavy", "one"])
@pytest.mark.parametrize("n", [1, PART, PART + 1, 8193, 100_000, HEAVY - 1, HEAVY, HEAVY + 8191, 1 << 20])
def test_window_and_import(kind, n):
    from paper_2510_14050_gb300 import ans
    rng = np.random.default_rng(n)
    src, dst = _links(kind, n, rng)
    exp = oracle.traffic_matrix(src, dst)
    eq = oracle.network_quantities(exp)
    ctx = ans.Context(0)
    m = ctx.build_window(*(torch.from_numpy(x.view(np.int32)).cuda() for x in (src, dst)))
    assert m.quantities() == eq
    # the same structure with counts beyond 32 bits: the 64-bit form
    vals = rng.integers(1, 1 << 40, len(exp[3]), dtype=np.uint64)
    big = exp._replace(vals=vals)
    mi = ctx.import_matrix(*big)
    assert mi.quantities() == oracle.network_quantities(big)
    assert ctx.network_quantities(mi) == oracle.network_quantities(big)
    for x in (m, mi):
        x.free()
    ctx.close()


@pytest.mark.parametrize("n", [SLOTS + 500, 20_000, HEAVY + 5])
def test_partition_with_too_many_destinations(n):
    from paper_2510_14050_gb300 import ans
    src, dst = _links("crowded", n, np.random.default_rng(n))
    ctx = ans.Context(0)
    m = ctx.build_window(*(torch.from_numpy(x.view(np.int32)).cuda() for x in (src, dst)))
    assert m.quantities() == oracle.network_quantities(oracle.traffic_matrix(src, dst))
    m.free()
    ctx.close()
