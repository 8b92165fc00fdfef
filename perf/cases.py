"""The work a user of the library has it do, as measurable cases.

Each case is one pass through a public entry point of ``ans.Context`` (or of
the C ABI where the binding has no method of its own), on the traffic models
the package's generator describes: Zipf sources and destinations, bursts of
one link, a heavy hitter and scanners.  Inputs are made on the GPU; window
sizes follow from the case alone.  Where matrices are returned, the traffic's
pattern does too and the seed is the key of the anonymisation (addresses
xor'ed with two words, which keeps common prefixes as prefix-preserving
anonymisation does): every seed gives other matrices of the same shape.
Elsewhere the seed draws the traffic itself as well.

A program keeps one context per kind of work, so all states of one kind share
a context while any of them lives.  ``TUNINGS`` holds what ``Context.autotune``
chose for each kind, as a program that saves its tuning sets it at start-up.
"""
import ctypes
import math
import random
import weakref

import torch

from paper_2510_14050_gb300 import ans

DEV = "cuda:0"
MASK = 0xFFFFFFFF
SIGN = -(1 << 63)  # int64 order of (key ^ SIGN) is the unsigned order of key
GOLDEN = 0x9E3779B1

# Chosen by Context.autotune for batches of each kind: key and column passes
# over 4096-key sub-tiles or two blocks per SM, and the paths of window sorts
# and time sums.
_SHAPES = dict(key_threads=256, key_rank=0, key_blocks=4, kv_threads=512, kv_rank=2, kv_blocks=1,
               col_threads=512, col_rank=1, col_blocks=2)
TUNINGS = {
    "default": {},
    # up to about a hundred windows: window sorts, time sums by merge rounds
    "merge": dict(_SHAPES, sum_path=0, agg_path=0, merge_tile=2048),
    # large batches: windows and time sum from one sort of the packets
    "packets": dict(_SHAPES, sum_path=2, agg_path=3),
    # quantities alone: links, sources and destinations counted on chip
    "hash": dict(_SHAPES, sum_path=2, agg_path=2),
}

# Zipf exponent and ranks of sources and destinations, share of packets in
# bursts, share of a heavy hitter, share of scanners.
TRAFFIC = {
    "small_pool": dict(src=(1.2, 1 << 16), dst=(1.2, 1 << 16), burst=0.0, heavy=0.0, scan=0.0),
    "bursty": dict(src=(1.1, 1 << 20), dst=(1.3, 1 << 22), burst=0.05, heavy=0.0, scan=0.0),
    "scanned": dict(src=(1.1, 1 << 24), dst=(1.1, 1 << 24), burst=0.0, heavy=0.10, scan=0.10),
    "wide": dict(src=(1.05, 1 << 32), dst=(1.05, 1 << 32), burst=0.0, heavy=0.0, scan=0.0),
}
# Distinct links per packet within a window of 2^17 packets (used by work()).
LINKS = {"small_pool": 0.38, "bursty": 0.55, "scanned": 0.80, "wide": 0.89}


def listed():
    return [
        # the smallest call: one ragged window inside a capture loop that may not allocate
        dict(name="noalloc_20k", kind="noalloc", packets=20_011, traffic="bursty"),
        # one window at a time, the plain entry point, its matrix read back
        dict(name="window_128k", kind="window", packets=1 << 17, traffic="small_pool"),
        # a monitor's tick: many short ragged windows, quantities only
        dict(name="ticks_256", kind="batch", windows=256, low=1 << 10, high=1 << 14, traffic="bursty",
             tuning="hash", matrices=False, sum=False, offsets="host"),
        # a few ragged windows whose matrices and time sum the program goes on with
        dict(name="matrices_6", kind="batch", windows=6, low=1 << 12, high=1 << 17, traffic="bursty",
             tuning="merge", matrices=True, sum=True, offsets="host"),
        # a serving step: windows that arrived in their own pinned buffers, and their time sum
        dict(name="serving_100", kind="serving", windows=100, low=1 << 12, high=1 << 17, traffic="bursty",
             tuning="packets"),
        # the 64-window batch: quantities and the time sum
        dict(name="batch_64", kind="batch", windows=64, low=1 << 17, high=1 << 17, traffic="bursty",
             tuning="merge", matrices=False, sum=True, offsets="device"),
        # an hour's sum out of matrices already at hand
        dict(name="sum_16", kind="sum", matrices=16, low=1 << 18, high=1 << 21, traffic="wide"),
        # a sliding sum: one matrix enters, one leaves
        dict(name="slide", kind="slide", matrices=8, low=1 << 17, high=1 << 19, traffic="bursty"),
        # quantities of a matrix that came as DCSR
        dict(name="stats_3m", kind="stats", packets=3_400_007, traffic="wide"),
        # a thousand windows from a thousand to a million packets, a heavy hitter and scanners
        dict(name="windows_1024", kind="batch", windows=1024, low=1 << 10, high=1 << 20, traffic="scanned",
             tuning="packets", matrices=False, sum=True, offsets="host"),
        # the data set's 2^30 packets in 8192 windows, planned on the device
        dict(name="packets_2e30", kind="batch", windows=8192, low=1 << 17, high=1 << 17, traffic="wide",
             tuning="packets", matrices=False, sum=True, offsets="device"),
    ]


def _log_int(rng, low, high):
    return min(high, max(low, int(math.exp(rng.uniform(math.log(low), math.log(high + 1))))))


def draw(rng):
    kind = rng.choice(["noalloc", "window", "batch", "batch", "batch", "serving", "sum", "slide", "stats"])
    traffic = rng.choice(sorted(TRAFFIC))
    if kind == "noalloc":
        return dict(kind=kind, packets=_log_int(rng, 1, 65536), traffic=traffic)
    if kind == "window":
        return dict(kind=kind, packets=_log_int(rng, 1, 1 << 22), traffic=traffic)
    if kind == "stats":
        return dict(kind=kind, packets=_log_int(rng, 1000, 1 << 24), traffic=traffic)
    if kind in ("sum", "slide"):
        k = rng.randint(2, 24)
        high = _log_int(rng, 1 << 12, (1 << 24) // k)
        return dict(kind=kind, matrices=k, low=max(1, high // rng.choice([1, 4, 32])), high=high, traffic=traffic)
    if kind == "serving":
        return dict(kind=kind, windows=rng.randint(2, 256), low=1 << 12, high=_log_int(rng, 1 << 13, 1 << 17),
                    traffic=traffic, tuning="packets")
    tuning = rng.choice(["merge", "packets", "packets", "hash"])
    offsets = rng.choice(["host", "device"])
    if tuning == "merge":
        windows = rng.randint(1, 100)
        high = _log_int(rng, 1 << 10, 1 << 17)
        return dict(kind=kind, windows=windows, low=max(1, high // rng.choice([1, 8, 64])), high=high,
                    traffic=traffic, tuning=tuning, matrices=windows <= 10, sum=True, offsets=offsets)
    windows = _log_int(rng, 2, 4096)
    high = max(1024, min(1 << 20, _log_int(rng, 1 << 16, 1 << 28) // windows))
    return dict(kind=kind, windows=windows, low=max(1, high // rng.choice([1, 16, 1024])), high=high,
                traffic=traffic, tuning=tuning, matrices=False, sum=tuning == "packets", offsets=offsets)


# ---- inputs -----------------------------------------------------------------

def _sizes(case):
    """Packets of each window: one size, or log-uniform over [low, high]."""
    if "packets" in case:
        return [case["packets"]]
    n = case.get("windows") or case["matrices"]
    if case["low"] == case["high"]:
        return [case["high"]] * n
    rng = random.Random(n * 1_000_003 + case["low"] * 31 + case["high"])
    return [_log_int(rng, case["low"], case["high"]) for _ in range(n)]


def _zipf(gen, n, s, ranks):
    """n int64 ranks 1..ranks with P(k) about k^-s (the continuous inverse)."""
    h0 = (0.5 ** (1.0 - s)) / (1.0 - s)
    h1 = ((ranks + 0.5) ** (1.0 - s)) / (1.0 - s)
    u = torch.rand(n, generator=gen, device=DEV, dtype=torch.float64).mul_(h1 - h0).add_(h0)
    k = u.mul_(1.0 - s).pow_(1.0 / (1.0 - s)).round_().to(torch.int64)
    return k.clamp_(1, ranks)


def _addr(rank):
    """Addresses of ranks, as int32 bit patterns."""
    return (((rank - 1) * GOLDEN) & MASK).view(torch.int32)[::2].contiguous()


def _chunk(gen, n, t):
    """n packets of traffic t."""
    src, dst = _addr(_zipf(gen, n, *t["src"])), _addr(_zipf(gen, n, *t["dst"]))
    at = torch.arange(n, device=DEV)
    if t["burst"]:  # in some slots of 128 packets the first L in 2..100 are one link
        slots = (n + 127) // 128
        length = torch.randint(2, 101, (slots,), generator=gen, device=DEV)
        on = torch.rand(slots, generator=gen, device=DEV) < t["burst"] * 128 / 51
        slot = at // 128
        first = torch.where(on[slot] & (at % 128 < length[slot]), slot * 128, at)
        src, dst = src[first], dst[first]
    if t["heavy"] or t["scan"]:
        u = torch.rand(n, generator=gen, device=DEV)
        heavy = torch.tensor(0xC0A80001 - (1 << 32), device=DEV, dtype=torch.int32)
        src = torch.where(u < t["heavy"], heavy, src)
        # scanners: one source of 16,777 per 4096 packets, its destinations consecutive
        scan = u > 1.0 - t["scan"]
        groups = (n + 4095) // 4096
        who = _addr(torch.randint(1, 16_778, (groups,), generator=gen, device=DEV) * 997)
        base = torch.randint(0, 1 << 31, (groups,), generator=gen, device=DEV)
        src = torch.where(scan, who[at // 4096], src)
        dst = torch.where(scan, ((base[at // 4096] + at % 4096) & 0x7FFFFFFF).to(torch.int32), dst)
    return src, dst


def _packets(case, seed):
    """(src, dst) int32 tensors of all the case's windows back to back."""
    total = sum(_sizes(case))
    returns_matrix = case["kind"] in ("window", "sum", "slide", "serving") or case.get("sum") or case.get("matrices")
    gen = torch.Generator(device=DEV).manual_seed(17 if returns_matrix else seed * 7919 + 17)
    key = random.Random(seed)
    xs, xd = (key.getrandbits(32) - (1 << 31) for _ in range(2))
    src = torch.empty(total, dtype=torch.int32, device=DEV)
    dst = torch.empty_like(src)
    step = 1 << 25
    for a in range(0, total, step):
        b = min(total, a + step)
        cs, cd = _chunk(gen, b - a, TRAFFIC[case["traffic"]])
        torch.bitwise_xor(cs, xs, out=src[a:b])
        torch.bitwise_xor(cd, xd, out=dst[a:b])
    return src, dst


def _offsets(sizes):
    offs = [0]
    for n in sizes:
        offs.append(offs[-1] + n)
    return offs


# ---- what a program keeps -----------------------------------------------------

_contexts = weakref.WeakValueDictionary()


def _context(tuning, capacity=0):
    ctx = _contexts.get((tuning, capacity))
    if ctx is None:
        ctx = ans.Context(0)
        if TUNINGS[tuning]:
            ctx.set_tuning(**TUNINGS[tuning])
        if capacity:
            ctx.set_batch_capacity(capacity)
        _contexts[(tuning, capacity)] = ctx
    return ctx


def prepare(case, seed):
    kind = case["kind"]
    sizes = _sizes(case)
    src, dst = _packets(case, seed)
    s = {"kind": kind, "src": src, "dst": dst}
    if kind == "noalloc":
        s["lib"] = ans.load()
        s["out"] = torch.zeros(9, dtype=torch.int64, device=DEV)
        s["status"] = torch.zeros(1, dtype=torch.int32, device=DEV)
        return s
    offs = _offsets(sizes)
    if kind == "batch":
        device = case["offsets"] == "device"
        s["ctx"] = _context(case["tuning"], offs[-1] if device else 0)
        s["offsets"] = torch.tensor(offs, dtype=torch.int64, device=DEV if device else "cpu")
        if not device:
            s["offsets"] = s["offsets"].numpy().astype("uint64")
        s["flags"] = (ans.BATCH_MATRICES if case["matrices"] else 0) | (ans.BATCH_SUM if case["sum"] else 0)
        s["out"] = torch.zeros((len(sizes), 9), dtype=torch.int64, device=DEV)
        return s
    s["ctx"] = _context(case.get("tuning", "default"))
    if kind == "serving":
        hs, hd = src.cpu().pin_memory(), dst.cpu().pin_memory()
        s["windows"] = [(hs[a:b], hd[a:b]) for a, b in zip(offs, offs[1:])]
        s["src"], s["dst"] = hs, hd
        s["out"] = torch.zeros((len(sizes), 9), dtype=torch.int64).pin_memory()
        return s
    if kind in ("sum", "slide"):
        s["mats"] = [s["ctx"].build_window(src[a:b], dst[a:b]) for a, b in zip(offs, offs[1:])]
        if kind == "slide":  # the sum of all but the newest; the oldest leaves
            s["total"] = s["ctx"].sum_windows(s["mats"][:-1])
            s["total"].view()
    if kind == "stats":
        m = s["ctx"].build_window(src, dst)
        s["matrix"] = s["ctx"].import_matrix(*m.device_arrays())
        s["out"] = torch.zeros(9, dtype=torch.int64, device=DEV)
    return s


# ---- one pass -------------------------------------------------------------------

def _views(m):
    """The matrix's four arrays as tensors (zero-copy views that keep it)."""
    arrays = m.device_arrays()
    for a in arrays:
        a.matrix = m
    return list(arrays)


def _arrays(m):
    return {**dict(zip(("row_ids", "row_ptr", "col_ids", "vals"), _views(m))),
            "quantities": torch.tensor(list(m.quantities().values()), dtype=torch.int64)}


def run(s):
    kind = s["kind"]
    if kind == "noalloc":
        p = ctypes.c_void_p
        rc = s["lib"].ans_window_quantities_noalloc(p(s["src"].data_ptr()), p(s["dst"].data_ptr()),
                                                    s["src"].numel(), p(s["out"].data_ptr()),
                                                    p(s["status"].data_ptr()),
                                                    p(torch.cuda.current_stream().cuda_stream))
        if rc:
            raise RuntimeError(ans.status_string(rc))
        return {"quantities": s["out"], "status": s["status"]}
    ctx = s["ctx"]
    if kind == "window":
        return _arrays(ctx.build_window(s["src"], s["dst"]))
    if kind == "sum":
        return _arrays(ctx.sum_windows(s["mats"]))
    if kind == "slide":
        return _arrays(ctx.combine([s["total"], s["mats"][-1], s["mats"][0]], [1, 1, -1]))
    if kind == "stats":
        ctx.network_quantities(s["matrix"], out=s["out"])
        return {"quantities": s["out"]}
    if kind == "serving":
        _, total, ticket = ctx.batch_submit_windows(s["windows"], ans.BATCH_SUM, out=s["out"])
        ctx.wait(ticket)  # the quantities are read on the host
        return {"quantities": s["out"], "sum": _arrays(total)}
    mats, total, _ = ctx.batch_submit(s["src"], s["dst"], s["offsets"], s["flags"], out=s["out"])
    got = {"quantities": s["out"]}
    if mats is not None:
        got["matrices"] = [_views(m) for m in mats]
    if total is not None:
        got["sum"] = _arrays(total)
    return got


# ---- the same in 64-bit torch ----------------------------------------------------

def _links(src, dst):
    """Distinct links (src << 32 | dst, sign bit flipped, ascending) and counts."""
    key = (src.to(torch.int64) << 32 | dst.to(torch.int64) & MASK) ^ SIGN
    return torch.unique(key, return_counts=True)


def _low(x):
    """The low 32 bits of int64 words as int32."""
    return x.view(torch.int32)[::2].contiguous()


def _quantities(key, count):
    """The nine quantities of a matrix given by its links, as a list."""
    if key.numel() == 0:
        return [0] * 9

    def side(x):
        ids, inv, links = torch.unique(x, return_inverse=True, return_counts=True)
        packets = torch.zeros(ids.numel(), dtype=torch.int64, device=x.device).index_add_(0, inv, count)
        return torch.stack([torch.tensor(ids.numel(), device=x.device), packets.max(), links.max()])

    head = torch.stack([count.sum(), torch.tensor(key.numel(), device=key.device), count.max()])
    return torch.cat([head, side(key >> 32), side(key & MASK)]).tolist()


def _exact_arrays(key, count):
    key, count = key[count != 0], count[count != 0]
    rows, fan = torch.unique_consecutive(key >> 32, return_counts=True)
    ptr = torch.zeros(rows.numel() + 1, dtype=torch.int64, device=key.device)
    torch.cumsum(fan, 0, out=ptr[1:])
    return {"row_ids": _low(rows ^ (SIGN >> 32)), "row_ptr": ptr, "col_ids": _low(key), "vals": count,
            "quantities": torch.tensor(_quantities(key, count), dtype=torch.int64)}


def exact(case, seed):
    kind = case["kind"]
    sizes = _sizes(case)
    if sum(sizes) > 1 << 28 or len(sizes) > 4096:
        return None  # thousands of windows one by one: over 20 seconds
    src, dst = _packets(case, seed)
    offs = _offsets(sizes)
    whole = _links(src, dst)
    if kind == "noalloc":
        return {"quantities": torch.tensor(_quantities(*whole), dtype=torch.int64),
                "status": torch.zeros(1, dtype=torch.int32)}
    if kind in ("window", "sum"):
        return _exact_arrays(*whole)
    if kind == "slide":  # everything but the first matrix
        return _exact_arrays(*_links(src[offs[1]:], dst[offs[1]:]))
    if kind == "stats":
        return {"quantities": torch.tensor(_quantities(*whole), dtype=torch.int64)}
    parts = [_links(src[a:b], dst[a:b]) for a, b in zip(offs, offs[1:])]
    got = {"quantities": torch.tensor([_quantities(*p) for p in parts], dtype=torch.int64)}
    if kind == "batch" and case["matrices"]:
        got["matrices"] = [list(_exact_arrays(*p).values())[:4] for p in parts]
    if kind == "serving" or case["sum"]:
        got["sum"] = _exact_arrays(*whole)
    return got


def work(case):
    """Bytes of one pass: packets or stored links read once, quantities and
    returned matrices written once (links estimated from the traffic); nothing
    is computed in floating point."""
    sizes = _sizes(case)
    total = sum(sizes)
    links = total * LINKS[case["traffic"]]
    matrix = 16.0 * links  # 12 bytes a link and 12 a row, a row for every three links
    kind = case["kind"]
    if kind in ("sum", "slide"):
        moved = 2 * matrix
    elif kind == "stats":
        moved = matrix + 72
    else:
        moved = 8.0 * total + 72.0 * len(sizes)
        if kind == "window" or case.get("matrices"):
            moved += matrix
        if kind == "serving" or case.get("sum"):
            moved += matrix * 0.75
    return {"bytes": moved, "flops": 0}
