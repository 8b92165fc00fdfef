"""The packets' sample sort (csrc/ans_ssort.cu) through the ABI, exact against
the oracle: sizes around the on-chip sort, the bucket and tile edges and the
two-split limit, keys that fill whole buckets, and samples that misjudge."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LOCAL = 2048          # keys one CTA sorts on chip
BUCKET = 1366         # keys of a bucket aimed at
ONE_LEVEL = 1 << 18   # longest segment of one split (plans below 2^24 keys)


def _mix32(h):
    h = h.astype(np.uint64)
    h ^= h >> np.uint64(16)
    h = h * np.uint64(0x85EBCA6B) & np.uint64(0xFFFFFFFF)
    h ^= h >> np.uint64(13)
    h = h * np.uint64(0xC2B2AE35) & np.uint64(0xFFFFFFFF)
    return h ^ (h >> np.uint64(16))


def _sampled(n, samples):
    """The packets a segment of n is sampled at."""
    i = np.arange(samples, dtype=np.uint64)
    frac = _mix32(i + np.uint64(1)) & np.uint64(0xFFFF)
    return ((i << np.uint64(16) | frac) * np.uint64(n)) >> np.uint64(16 + samples.bit_length() - 1)


def _window(kind, n, rng):
    src = rng.integers(0, 1 << 32, n, dtype=np.uint32)
    dst = rng.integers(0, 1 << 32, n, dtype=np.uint32)
    if kind == "few":        # three sources, a handful of links: buckets of one value
        src, dst = (src % 3) * np.uint32(0x7FFFFFFF), dst % 5
    elif kind == "ones":     # the largest key fills most buckets, its neighbours the rest
        src = np.where(rng.random(n) < 0.9, np.uint32(0xFFFFFFFF), src)
        dst = np.where(rng.random(n) < 0.9, np.uint32(0xFFFFFFFF), np.uint32(0xFFFFFFFE))
    elif kind == "zero":     # keys 0 and 1 and their neighbourhood
        src, dst = np.zeros_like(src), dst % np.uint32(3)
    elif kind == "sorted":
        o = np.lexsort((dst, src))
        src, dst = src[o], dst[o]
    elif kind == "misjudged":  # small keys wherever the sample looks
        src |= np.uint32(0x80000000)
        for s in (1024, 2048, 4096, 8192):
            src[_sampled(n, s).astype(np.int64)] = 7
    return src, dst


def _check(wins, flags_sum=True, path=0):
    from paper_2510_14050_gb300 import ans
    src = np.concatenate([w[0] for w in wins])
    dst = np.concatenate([w[1] for w in wins])
    offs = np.concatenate([[0], np.cumsum([len(w[0]) for w in wins])]).astype(np.uint64)
    ds, dd = (torch.from_numpy(x.view(np.int32)).cuda() for x in (src, dst))
    ctx = ans.Context(0)
    ctx.set_tuning(sum_path=2, agg_path=path)
    out = torch.zeros((len(wins), 9), dtype=torch.int64, device="cuda")
    mats, summ, tk = ctx.batch_submit(ds, dd, offs, ans.BATCH_MATRICES | ans.BATCH_SUM, out=out)
    ctx.wait(tk)
    em, eq, es = oracle.batch(src, dst, offs)
    assert ans.quantities_from_tensor(out) == eq
    for m, e in zip(mats + [summ], em + [es]):
        for a, b in zip(m.to_numpy(), e):
            assert np.array_equal(a, b)
    assert summ.quantities() == oracle.network_quantities(es)
    for m in mats + [summ]:
        m.free()
    ctx.close()


@pytest.mark.parametrize("kind", ["random", "few", "ones", "zero", "sorted", "misjudged"])
@pytest.mark.parametrize("n", [1, 2, BUCKET, LOCAL, LOCAL + 1, 2 * LOCAL, 8191, 8193, 20011, 131072, ONE_LEVEL, ONE_LEVEL + 1])
def test_one_window(kind, n):
    if kind == "misjudged" and n <= LOCAL:
        n += 4 * LOCAL
    _check([_window(kind, n, np.random.default_rng(n))])


@pytest.mark.parametrize("path", [0, 3])
def test_mixed_windows(path):
    rng = np.random.default_rng(5)
    sizes = [0, 1, LOCAL, LOCAL + 1, 0, 100003, ONE_LEVEL, ONE_LEVEL + 12345, 3 * ONE_LEVEL + 1, 8192]
    kinds = ["random", "few", "ones", "misjudged"]
    _check([_window(kinds[i % 4] if n > 4 * LOCAL else "random", n, rng) for i, n in enumerate(sizes)], path=path)


def test_long_windows_of_a_large_batch():
    # 2^24 packets and more: one split takes windows of up to 2^21
    rng = np.random.default_rng(6)
    _check([_window("random", n, rng) for n in ((1 << 21), (1 << 21) + 1, (1 << 23) + (1 << 22) + 7, 5000)])
