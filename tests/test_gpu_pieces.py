"""The pipeline's stage c from stage b's pieces, against the separate call (whose
stage c reads prev), and stage b against the uses by definition: numbers of
pieces around a tile, below and above the bound up to which the pipeline does not
wait for the number of runs, and more runs than are counted by blocks; pieces
that start where a tile of accesses does."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_28870_gb300 as ptc
    ptc.lib()


@pytest.mark.parametrize("n_req", [1, 2, 300, 2047, 2048, 2049, 30000, 600000, 1300000, 2900000])
@pytest.mark.parametrize("follow", [0.0, 0.7])
def test_pieces(n_req, follow):
    """Requests of eight one-token blocks each re-read a document whole, now and
    then the one after the last request's (which makes runs of several pieces)."""
    import torch
    import paper_2609_28870_gb300 as ptc
    rng = np.random.default_rng(n_req)
    docs = n_req // 3 + 1
    pick = rng.integers(0, docs, n_req)
    for r in np.flatnonzero(rng.random(n_req) < follow):
        if r > 0:
            pick[r] = (pick[r - 1] + 1) % docs
    tok = (pick[:, None] * 8 + np.arange(8)).astype(np.uint32).ravel()
    off = np.arange(n_req + 1, dtype=np.uint64) * 8
    n = tok.size
    buf = {k: torch.zeros(n, dtype=torch.int32, device="cuda") for k in ("ids", "prev", "next", "dist")}
    caps = np.unique(np.linspace(1, max(n // 2, 1), 20).astype(np.uint64))
    dt = torch.from_numpy(tok.view(np.int32)).cuda()
    plan = ptc.PipelinePlan(dt, ptc.to_device_u64(off), None, 1, caps, ptc.PTC_COST_UNIFORM, outputs=buf)
    res = plan.run().result()
    order = np.argsort(tok, kind="stable")  # the accesses of every token together, in order
    again = tok[order[1:]] == tok[order[:-1]]
    prev, nxt = np.full(n, 0xFFFFFFFF, np.uint32), np.full(n, 0xFFFFFFFF, np.uint32)
    prev[order[1:][again]] = order[:-1][again]
    nxt[order[:-1][again]] = order[1:][again]
    assert res["n_access"] == n and res["n_distinct"] == 8 * len(np.unique(pick))
    assert np.array_equal(ptc.u32(buf["prev"]), prev) and np.array_equal(ptc.u32(buf["next"]), nxt)
    ids = torch.zeros(n + 1, dtype=torch.int32, device="cuda")  # not 16-byte aligned from its second entry on
    ids[1:] = buf["ids"]
    p1, n1 = ptc.ptc_reuse_indices(ids[1:], res["n_distinct"])
    assert np.array_equal(ptc.u32(p1), prev) and np.array_equal(ptc.u32(n1), nxt)
    dist = ptc.ptc_stack_distance(torch.from_numpy(prev.view(np.int32)).cuda())
    assert torch.equal(buf["dist"], dist.view(torch.int32))
    c = ptc.ptc_curves(dist, ptc.to_device_u64(off), 1, caps, ptc.PTC_COST_UNIFORM)
    assert res["hits"] == [int(x) for x in c["hits"]]
