"""The partitioned dedup where its kernels turn: partitions of as many records
as fit in shared memory at once, one more and one less, with repeats; and level
1's walk over the bitmap of the accesses to settle, with ranges of several
refills and rounds that a hint leaves mostly empty.  The ids are known by
construction (keys are an injection of them)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
NONE = 0xFFFFFFFF
FIT = 3072  # records of a partition that fit at once


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_28870_gb300 as ptc
    ptc.lib()


def _keys(ids, part=None):
    """An injection of ids below 2^27 into keys; with `part`, all of one
    partition (bits 45..60 of h0)."""
    x = ids.astype(np.uint64)
    h = (x * np.uint64(0x9E3779B97F4A7C15)) & np.uint64((1 << 61) - 1)
    if part is not None:
        h = (h & np.uint64((1 << 45) - 1)) | (part.astype(np.uint64) << np.uint64(45))
    return np.stack([h, x * np.uint64(0xC2B2AE3D27D4EB4F) & np.uint64((1 << 60) - 1)], axis=1)


def _check(keys, want, blk=None, prior=None):
    import torch
    import paper_2609_28870_gb300 as ptc
    dk = ptc.to_device_u64(np.ascontiguousarray(keys).reshape(-1)).view(-1, 2)
    args = (dk, ptc.PTC_IDS_PARTITIONED)
    if blk is not None:
        args += (ptc.to_device_u64(blk.astype(np.uint64)),
                 torch.from_numpy(np.ascontiguousarray(prior, dtype=np.uint32).view(np.int32)).cuda())
    ids, d = ptc.ptc_assign_ids_ex(*args)
    assert d == int(want.max()) + 1
    assert np.array_equal(ptc.u32(ids), want)


@pytest.mark.parametrize("apart", [3, 32])  # in 32 partitions settled together: eleven of them, or one
@pytest.mark.parametrize("distinct", [True, False])
@pytest.mark.parametrize("size", [1, 2, 33, 511, 512, 513, FIT - 1, FIT, FIT + 1, 2 * FIT - 1])
def test_partition_sizes(size, distinct, apart):
    rng = np.random.default_rng(size)
    parts = 40  # partitions of this size, next to each other and among empty ones
    which = np.repeat(np.arange(parts) * apart, size)
    own = np.arange(size) if distinct else rng.integers(0, max(size // 3, 1), parts * size) if size > 1 else np.zeros(1)
    label = (np.tile(own, parts) if len(own) == size else own).astype(np.int64) + which * 4 * FIT
    order = rng.permutation(len(label))
    label, which = label[order], which[order]
    _, first, inv = np.unique(label, return_index=True, return_inverse=True)
    rank = np.empty(len(first), np.int64)
    rank[np.argsort(first, kind="stable")] = np.arange(len(first))
    _check(_keys(label, which), rank[inv.ravel()].astype(np.uint32))


@pytest.mark.parametrize("n_req,longest,keep", [(3000, 8191, 0.98), (2000, 12000, 0.5), (40, 70, 0.9), (1, 5, 0)])
def test_walk_with_a_hint(n_req, longest, keep):
    """A chain of requests, each repeating most of the one before: their ids
    and the words of the bitmap that are not zero follow."""
    rng = np.random.default_rng(n_req)
    rows, prev, fresh = [], np.zeros(0, np.int64), 0
    for _ in range(n_req):
        size = int(rng.integers(1, longest + 1))
        lam = min(len(prev), size, int(round(keep * size)))
        row = np.concatenate([prev[:lam], np.arange(fresh, fresh + size - lam)])
        fresh += size - lam
        rows.append(row)
        prev = row
    ids = np.concatenate(rows)
    blk = np.concatenate([[0], np.cumsum([len(r) for r in rows])])
    prior = np.arange(-1, n_req - 1)
    prior = np.where(prior < 0, NONE, prior)
    keys = _keys(ids)
    _check(keys, ids.astype(np.uint32))
    _check(keys, ids.astype(np.uint32), blk, prior)


def test_more_keys_than_the_small_variant_takes():
    """180M accesses to settle, 2,747 to a partition: the variant with larger
    tables, with a key repeated 200,000 times and 4.8M others twice."""
    import torch
    import paper_2609_28870_gb300 as ptc
    n, once = 180_000_000, 175_000_000
    if torch.cuda.mem_get_info()[0] < 40 << 30:
        pytest.skip("needs 40 GB")
    gen = torch.Generator(device="cuda").manual_seed(3)
    ids = torch.arange(n, device="cuda", dtype=torch.int64)
    ids[once:] = torch.randint(0, once, (n - once,), device="cuda", generator=gen)
    ids[once:once + 200_000] = 7
    mask = (1 << 61) - 1
    keys = torch.empty((n, 2), device="cuda", dtype=torch.int64)
    keys[:, 0] = (ids * -0x61C8864680B583EB) & mask
    keys[:, 1] = (ids * -0x3D4D51C2D82B14B1) & mask
    got, d = ptc.ptc_assign_ids_ex(keys, ptc.PTC_IDS_PARTITIONED)
    assert d == once
    assert bool((got.view(torch.int32) == ids.to(torch.int32)).all())
