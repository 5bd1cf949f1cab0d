"""Block keys by units of 16, 12 and 8 tokens against the oracle's prefix
hash, bit-exact: block sizes of one to many units, token buffers that start at
any word, tiles of one request and of hundreds (many without a full block),
sizes around the 32 units of a round and the 256 of a tile, tokens that need
three limbs, and the carried keys that the pipeline hands to its id stage."""
import numpy as np
import pytest

import oracle
import tracegen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ptc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_28870_gb300 as p
    p.lib()
    return p


def _keys(ptc, tokens, off, B, lead, seed=3):
    import torch
    buf = torch.zeros(lead + len(tokens) + 1, dtype=torch.int32, device="cuda")
    buf[lead: lead + len(tokens)] = ptc.to_device_u32(tokens)
    keys, blk_off, n = ptc.ptc_hash_blocks(buf[lead: lead + len(tokens)], ptc.to_device_u64(off), None, B, seed)
    return ptc.u64(keys).reshape(-1, 2)[:n]


def _trace(rng, lens, vocab):
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.uint64)
    return rng.integers(0, vocab, int(off[-1])).astype(np.uint32), off


@pytest.mark.parametrize("B", [8, 12, 16, 24, 32, 36, 40, 48, 64, 80, 108, 144, 176, 264, 272, 280, 352, 496, 512])
@pytest.mark.parametrize("lead", [0, 1, 2, 3])
def test_block_sizes_and_alignments(ptc, B, lead):
    rng = np.random.default_rng(100 * B + lead)
    lens = np.concatenate([[0, B - 1, B, 33 * B + 5, 300 * B + 3], rng.integers(0, 9 * B, 70), [0, 0, 2 * B + 1]])
    tokens, off = _trace(rng, lens, 151_936)
    assert np.array_equal(_keys(ptc, tokens, off, B, lead), oracle.prefix_hash(tokens, off, B, 3))


@pytest.mark.parametrize("B", [8, 12, 16, 48])
def test_many_requests_per_tile(ptc, B):
    """Requests of zero to three blocks, most of them without one: more than a
    window of 32 meets a round."""
    rng = np.random.default_rng(B)
    lens = np.where(rng.random(9000) < 0.9, rng.integers(0, B, 9000), rng.integers(B, 4 * B, 9000))
    tokens, off = _trace(rng, lens, 50_000)
    assert np.array_equal(_keys(ptc, tokens, off, B, 1), oracle.prefix_hash(tokens, off, B, 3))


@pytest.mark.parametrize("blocks", [1, 31, 32, 33, 255, 256, 257, 2049])
@pytest.mark.parametrize("B", [16, 24])
def test_tile_edges(ptc, B, blocks):
    rng = np.random.default_rng(blocks)
    tokens, off = _trace(rng, [blocks * B, 0, 3 * B + 1, blocks * B + 7], 151_936)
    assert np.array_equal(_keys(ptc, tokens, off, B, 0), oracle.prefix_hash(tokens, off, B, 3))


@pytest.mark.parametrize("B", [12, 16, 40])
def test_wide_tokens(ptc, B):
    rng = np.random.default_rng(B)
    lens = rng.integers(0, 200 * B, 60)
    tokens, off = _trace(rng, lens, 151_936)
    at = rng.integers(0, len(tokens), 40)
    tokens[at] = rng.integers(2**27, 2**32, 40).astype(np.uint32)
    tokens[0] = tokens[-1] = 0xFFFFFFFF
    assert np.array_equal(_keys(ptc, tokens, off, B, 2), oracle.prefix_hash(tokens, off, B, 3))


@pytest.mark.parametrize("B", [8, 12, 24, 40, 48])
def test_pipeline_carries(ptc, B):
    tr = tracegen.make(0, max_requests=250)
    tok, off = ptc.to_device_u32(tr.tokens), ptc.to_device_u64(tr.req_tok_off)
    o = oracle.run(tr.tokens, tr.req_tok_off, B, np.asarray([10, 1000, 10**6], dtype=np.uint64))
    got = ptc.ptc_pipeline(tok, off, None, B, [10, 1000, 10**6])
    assert got["n_access"] == o["n_access"] and got["n_distinct"] == o["n_distinct"] and got["hits"] == o["hits"]


@pytest.mark.parametrize("lead", [0, 3])
@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("B", [40, 60, 80, 88, 108, 136, 144, 204, 272, 336])
def test_tiles_of_more_units(ptc, B, wide, lead):
    """9 or 11 units per lane, which token counts with many tiles take: a buffer
    of that length whose requests lie in its front."""
    import torch
    rng = np.random.default_rng(10 * B + lead)
    lens = np.concatenate([[0, B - 1, B, 33 * B + 5, 700 * B + 3], np.where(rng.random(900) < 0.7, rng.integers(0, B, 900),
                          rng.integers(B, 6 * B, 900)), rng.integers(0, 90 * B, 40), [0, 2 * B + 1]])
    tokens, off = _trace(rng, lens, 151_936)
    if wide:
        at = rng.integers(0, len(tokens), 9)
        tokens[at] = rng.integers(2**27, 2**32, 9).astype(np.uint32)
        tokens[0] = tokens[-1] = 0xFFFFFFFF
    n_tok = 16 * 152 * 64 * B + 7
    buf = torch.zeros(lead + n_tok, dtype=torch.int32, device="cuda")
    buf[lead: lead + len(tokens)] = ptc.to_device_u32(tokens)
    keys, _, n = ptc.ptc_hash_blocks(buf[lead:], ptc.to_device_u64(off), None, B, 3)
    assert np.array_equal(ptc.u64(keys).reshape(-1, 2)[:n], oracle.prefix_hash(tokens, off, B, 3))
