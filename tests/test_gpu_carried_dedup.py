"""Keys whose hash tiles' carries are added by the partitioned dedup's level 1
(the pipeline without returned keys, above the size where the id table leaves
L2): hash tiles of 4, 8 and 16 blocks, so that a word of 32 accesses lies in
8, 4 and 2 of them."""
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DRAM_SIZED = 12_700_000  # accesses: the id table would not fit in L2


def _tile_blocks(L, B, blocks=1 << 24):
    """Blocks per hash tile, from the 32 bytes that the workspace holds of each."""
    more = L.ptc_hash_blocks_workspace_bytes(1, 2 * blocks * B, B) - L.ptc_hash_blocks_workspace_bytes(1, blocks * B, B)
    return 1 << round(np.log2(32 * blocks / more))


def test_every_block_size_has_tiles_the_dedup_makes_room_for():
    import paper_2609_28870_gb300 as ptc
    from paper_2609_28870_gb300 import build
    build.build()
    tiles = {B: _tile_blocks(ptc.lib(), B) for B in range(1, ptc.MAX_BLOCK_SIZE + 1)}
    src = open(os.path.join(ROOT, "paper_2609_28870_gb300", "csrc", "ptc_internal.h")).read()
    room = re.search(r"constexpr uint32_t kCarryTileMin = (\d+);", src)
    assert room and min(tiles.values()) >= int(room.group(1))
    assert (tiles[488], tiles[504], tiles[136], tiles[16]) == (4, 8, 16, 256)


@pytest.mark.parametrize("B,U", [(56, 8), (104, 8), (488, 8)])
def test_units_only_while_their_exponents_fit(B, U):
    """A request of 2^32 units or more is hashed by blocks, in tiles of 256 chunks
    of 16 tokens (the routes differ in the blocks of a tile)."""
    import paper_2609_28870_gb300 as ptc
    from paper_2609_28870_gb300 import build
    build.build()
    chunks = 1 << int(np.ceil(np.log2((B + 15) // 16)))
    units = 1 << int(np.floor(np.log2(352 * U // B)))
    assert units != 256 // chunks
    assert _tile_blocks(ptc.lib(), B, 2**31 * U // B) == units           # 2^31 and (nearly) 2^32 units
    assert _tile_blocks(ptc.lib(), B, 2**32 * U // B + 1) == 256 // chunks


@pytest.mark.gpu
@pytest.mark.parametrize("sessions", [False, True])
@pytest.mark.parametrize("B", [488, 504, 136, 104])
def test_carried_keys(B, sessions):
    """The grids follow the token buffer's length, the work its requests': a
    few long requests at the front of a buffer that the id table of L2's size
    does not serve."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.mem_get_info()[0] < 60 << 30:
        pytest.skip("needs 60 GB")
    import oracle
    import paper_2609_28870_gb300 as ptc
    from tests import gpu_util as gu
    rng = np.random.default_rng(B)
    S, turns, ctx, rows, ses = 6, 5, {}, [], []
    prompt = rng.integers(0, 151_936, 150 * B)
    for _ in range(turns):
        for s in range(S):
            old = ctx.get(s, prompt)
            ctx[s] = np.concatenate([old, rng.integers(0, 151_936, int(rng.integers(20 * B, 400 * B)))])
            rows.append(ctx[s])
            ses.append(s)
    tokens = np.concatenate(rows).astype(np.uint32)
    off = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.uint64)
    n_tok = DRAM_SIZED * B
    tok = torch.zeros(n_tok, dtype=torch.int32, device="cuda")
    tok[: len(tokens)] = ptc.to_device_u32(tokens)
    caps = [1, 200, 3000, 10**6]
    o = oracle.run(tokens, off, B, caps)
    n = o["n_access"]
    assert n > 10_000
    buf = {k: torch.empty(DRAM_SIZED, dtype=torch.int32, device="cuda") for k in ("ids", "prev", "next", "dist")}
    buf["req_blk_off"] = torch.empty(len(off), dtype=torch.int64, device="cuda")
    kw = dict(req_session=ptc.to_device_u32(ses), n_session=S) if sessions else {}
    g = ptc.ptc_pipeline(tok, ptc.to_device_u64(off), None, B, caps, outputs=buf, **kw)
    for k in ("ids", "prev", "next", "dist"):
        g[k] = ptc.u32(buf[k])[:n]
    g["req_blk_off"] = ptc.u64(buf["req_blk_off"])
    gu.assert_same(g, o)
