"""Stage c by counting (traces without runs) against the oracle's distances,
bit-exact, at sizes around the edges of its warps (1,024 positions), tiles
(8,192) and buckets (32,768 re-reads); the distances of runs by blocks of 512;
the fallback for a prev that takes a value twice; and stage d's bins where a CTA walks many tiles."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
NONE = np.uint32(0xFFFFFFFF)


@pytest.fixture(scope="module")
def ptc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_28870_gb300 as p
    p.lib()
    return p


def _prev(ids):
    at = np.argsort(ids, kind="stable")
    same = ids[at][1:] == ids[at][:-1]
    prev = np.full(len(ids), NONE, dtype=np.uint32)
    prev[at[1:][same]] = at[:-1][same]
    return prev


@pytest.mark.parametrize("n", [31, 1023, 1024, 1025, 8191, 8192, 8193, 32768, 40_001, 65_537, 120_000, 700_001])
@pytest.mark.parametrize("objects", [0.02, 0.6])
def test_counted_distances(ptc, n, objects):
    rng = np.random.default_rng(n)
    prev = _prev(rng.integers(0, max(2, int(n * objects)), n))
    got = ptc.u32(ptc.ptc_stack_distance(ptc.to_device_u32(prev)))
    assert np.array_equal(got, oracle.sd_fenwick(prev))


@pytest.mark.parametrize("rereads", [32_767, 32_768, 32_769, 65_536, 98_305])
def test_counted_distances_at_bucket_edges(ptc, rereads):
    """Exactly this many re-reads: every block of a first pass read again in another order."""
    rng = np.random.default_rng(rereads)
    ids = np.concatenate([np.arange(rereads), rng.permutation(rereads)])
    prev = _prev(ids)
    got = ptc.u32(ptc.ptc_stack_distance(ptc.to_device_u32(prev)))
    assert np.array_equal(got, oracle.sd_fenwick(prev))


@pytest.mark.parametrize("n", [1, 31, 511, 512, 513, 1023, 1025, 20_000, 262_145])
def test_runs_by_blocks(ptc, n):
    """The distances of runs around the edges of their blocks of 512: context
    re-reads of random stretches, so that runs of every length and rank order
    meet, and a trace without runs (every access its own)."""
    rng = np.random.default_rng(n)
    parts, size = [], 0
    while size < n:
        lo = int(rng.integers(0, max(1, n // 3)))
        parts.append(np.arange(lo, lo + int(rng.integers(1, 9))))
        size += len(parts[-1])
    for ids in (np.concatenate(parts)[:n], rng.integers(0, max(1, n // 2), n)):
        prev = _prev(ids)
        got = ptc.u32(ptc.ptc_stack_distance(ptc.to_device_u32(prev), method=ptc.PTC_SD_RUNS))
        assert np.array_equal(got, oracle.sd_fenwick(prev))


def test_more_runs_than_blocks_take(ptc):
    """Above 2^21 runs the forced run method builds its matrix level by level."""
    rng = np.random.default_rng(1)
    p = ptc.to_device_u32(_prev(rng.integers(0, 900_000, 2_300_000)))
    assert np.array_equal(ptc.u32(ptc.ptc_stack_distance(p, method=ptc.PTC_SD_RUNS)), ptc.u32(ptc.ptc_stack_distance(p)))


def test_prev_that_repeats_a_value_takes_the_matrix(ptc):
    rng = np.random.default_rng(5)
    prev = _prev(rng.integers(0, 900, 20_000))
    prev[15_000] = prev[14_000] if prev[14_000] != NONE else 3
    prev[15_001] = prev[15_000]
    p = ptc.to_device_u32(prev)
    assert np.array_equal(ptc.u32(ptc.ptc_stack_distance(p)), ptc.u32(ptc.ptc_stack_distance(p, method=ptc.PTC_SD_POINTS)))


@pytest.mark.parametrize("length", [3, 70_000])
@pytest.mark.parametrize("falls", [False, True])
def test_curves_over_many_tiles(ptc, length, falls):
    """20M distances: a CTA of stage d walks more tiles than its 32-bit depth
    sums hold, at depths below and above 2^16; with and without falls inside
    requests."""
    import torch
    n = 20_000_000
    g = torch.Generator(device="cuda").manual_seed(length)
    off = torch.arange(0, n + length, length, device="cuda").clamp_(max=n)
    depth = torch.arange(n, device="cuda") % length
    if falls:
        dist = torch.randint(1, 3_000_000, (n,), device="cuda", generator=g, dtype=torch.int32)
    else:
        dist = (1 + 40 * (depth // 3) + torch.arange(n, device="cuda") // length % 40).int()
    caps = np.unique(np.rint(64 * (2_000_000 / 64) ** (np.arange(65) / 64)).astype(np.uint64))
    got = ptc.ptc_curves(dist, off, 16, caps, ptc.PTC_COST_LINEAR, f_attn=1)
    d = dist.cpu().numpy().astype(np.int64)
    o = off.cpu().numpy()
    run = d.copy()
    if falls:  # running maximum per request
        full = n // length * length
        run[:full] = np.maximum.accumulate(d[:full].reshape(-1, length), axis=1).reshape(-1)
        run[full:] = np.maximum.accumulate(d[full:]) if full < n else run[full:]
    k = np.arange(n) - np.repeat(o[:-1], np.diff(o))
    bins = np.searchsorted(caps, run)
    hits = np.cumsum(np.bincount(bins, minlength=len(caps) + 1))[: len(caps)]
    ks = np.cumsum(np.bincount(bins, weights=k.astype(np.float64), minlength=len(caps) + 1))[: len(caps)]
    assert got["hits"] == hits.tolist()
    assert got["saved"] == [256 * int(s) + 136 * int(h) for s, h in zip(ks, hits)]  # sums below 2^53: exact
