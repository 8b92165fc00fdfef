"""Column statistics of large sums of given matrices: hash partitions up to
2^25 links, the column sort up to 2^26, hash groups from there; exact against
plain 64-bit torch, signed combinations too."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

MASK = 0xFFFFFFFF


def _packets(n, seed):
    """Sources in a few thousand rows, destinations with a heavy head."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    src = torch.randint(0, 1 << 31, (n,), generator=gen, device="cuda", dtype=torch.int32)
    dst = torch.randint(0, 1 << 31, (n,), generator=gen, device="cuda", dtype=torch.int32)
    dst = torch.where(torch.arange(n, device="cuda") % 8 == 0, dst % 1000, dst)
    return src, dst


def _quantities(key, count):
    def side(x):
        ids, inv, links = torch.unique(x, return_inverse=True, return_counts=True)
        packets = torch.zeros(ids.numel(), dtype=torch.int64, device="cuda").index_add_(0, inv, count)
        return [ids.numel(), int(packets.max()), int(links.max())]

    return [int(count.sum()), key.numel(), int(count.max())] + side(key >> 32) + side(key & MASK)


@pytest.mark.parametrize("links,kernels", [((1 << 24) + 50_000, {"col_count"}), ((1 << 25) + 50_000, {"colstat"}),
                                           ((1 << 26) + 50_000, {"hgroup"})])
def test_sum_and_combination(links, kernels):
    from paper_2510_14050_gb300 import ans
    ctx = ans.Context(0)
    n = links // 2
    src, dst = _packets(2 * n, links)
    a, b = (ctx.build_window(src[i * n:(i + 1) * n], dst[i * n:(i + 1) * n]) for i in range(2))
    assert a.nnz + b.nnz > links - 50_000  # (next to no packet twice)
    key = src.to(torch.int64) << 32 | dst.to(torch.int64)
    ctx.profile(True)
    both = ctx.sum_windows([a, b])
    got = list(both.quantities().values())
    ran = set(ctx.profile_read())
    ctx.profile(False)
    assert got == _quantities(*torch.unique(key, return_counts=True))
    assert kernels == ran & {"col_count", "colstat", "hgroup"} - ({"colstat"} if "hgroup" in ran else set())
    back = ctx.combine([both, b], [1, -1])
    assert list(back.quantities().values()) == _quantities(*torch.unique(key[:n], return_counts=True))
    for x in (a, b, both, back):
        x.free()
    ctx.close()
