"""ptc_verify_ids at block sizes from one token to the largest: ids that hold,
and one token changed in a repeated block (its first, middle or last), which the
check must find wherever the block lies among the warp's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ptc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_28870_gb300 as p
    p.lib()
    return p


@pytest.mark.parametrize("B", [1, 2, 4, 5, 7, 24, 31, 32, 33, 100, 512])
def test_verify(ptc, B):
    rng = np.random.default_rng(B)
    doc = rng.integers(0, 150_000, 60 * B).astype(np.uint32)
    rows = [doc[:int(k)] for k in rng.integers(0, 60 * B + 1, 12)]  # with a ragged end each
    rows = [np.concatenate([r, rng.integers(0, 150_000, int(rng.integers(0, 3 * B))).astype(np.uint32)]) for r in rows]
    tokens = np.concatenate([doc] + rows)
    lens = np.array([len(doc)] + [len(r) for r in rows])
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    dt, do = ptc.to_device_u32(tokens), ptc.to_device_u64(off)
    keys, blk_off, n = ptc.ptc_hash_blocks(dt, do, None, B, 3)
    ids, d = ptc.ptc_assign_ids(keys)
    ptc.ptc_verify_ids(dt, do, blk_off, B, ids, d)
    i = ptc.u32(ids)
    bo = ptc.u64(blk_off)
    _, first = np.unique(i, return_index=True)
    repeats = np.setdiff1d(np.arange(n), first)
    assert len(repeats) > 0
    for a in rng.choice(repeats, min(6, len(repeats)), replace=False):
        r = int(np.searchsorted(bo, a, side="right") - 1)
        for o in {0, B // 2, B - 1}:
            at = int(off[r]) + B * int(a - bo[r]) + o
            bad = tokens.copy()
            bad[at] ^= 1
            with pytest.raises(ptc.PtcError) as e:
                ptc.ptc_verify_ids(ptc.to_device_u32(bad), do, blk_off, B, ids, d)
            assert e.value.name == "PTC_ERR_HASH_COLLISION"
