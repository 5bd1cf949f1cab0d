"""The methods of the stack-distance stage (the wavelet matrix over every
access, the count over runs, the automatic choice) against the oracle's
distances, bit-exact, on traces with short and with long runs."""
import numpy as np
import pytest

import oracle
import tracegen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_28870_gb300 as ptc
    ptc.lib()


def _ids_prev(tr, B):
    ids, D = oracle.block_ids(tr.tokens, tr.req_tok_off, B)
    prev, _ = oracle.reuse(ids, D)
    return ids, prev


def _all_methods(prev):
    import paper_2609_28870_gb300 as ptc
    p = ptc.to_device_u32(prev)
    return {m: ptc.u32(ptc.ptc_stack_distance(p, method=m)) for m in
            (ptc.PTC_SD_AUTO, ptc.PTC_SD_POINTS, ptc.PTC_SD_RUNS)}


@pytest.mark.parametrize("seed", range(20))
def test_methods_agree_on_tiny_traces(seed):
    rng = np.random.default_rng(7000 + seed)
    B = int(rng.choice([1, 2, 3, 4, 16]))
    tr = tracegen.tiny(seed, n_sessions=int(rng.integers(1, 14)), max_turns=7, vocab=int(rng.integers(2, 6)),
                       max_seg=int(rng.integers(3, 50)))
    ids, prev = _ids_prev(tr, B)
    if prev.size == 0:
        pytest.skip("no blocks")
    want = oracle.sd_mattson(ids)
    for m, got in _all_methods(prev).items():
        assert np.array_equal(got, want), m


@pytest.mark.parametrize("workload,requests", [(0, None), (1, 3000), (2, 150)])
def test_methods_agree_on_workloads(workload, requests):
    tr = tracegen.make(workload, max_requests=requests)
    _, prev = _ids_prev(tr, 16)
    want = oracle.sd_fenwick(prev)
    for m, got in _all_methods(prev).items():
        assert np.array_equal(got, want), m


def test_runs_edge_cases():
    """Hand-made reuse arrays: one access; all first accesses; one long
    context run; a window that is empty (prev = i - 1); alternating runs that
    break every access; a run cut by the window start."""
    N = oracle.NONE
    cases = [
        [N],
        [N] * 40,
        [N] * 10 + list(range(10)),
        [N, 0, 1, 2],
        [N, N, 1, 0, 3, 2, 5, 4],
        [N] * 6 + [2, 3, 4, 5] + [N, N] + [0, 1],
        [N] * 5 + [0, 1, 2] + [6, 7] + [3, 4],
    ]
    for prev in cases:
        prev = np.asarray(prev, dtype=np.uint32)
        # each case must be a reuse array: prev[i] < i, each value used once
        fin = prev[prev != N]
        assert len(set(fin.tolist())) == fin.size
        assert all(p < i for i, p in enumerate(prev.tolist()) if p != N)
        want = oracle.sd_fenwick(prev)
        for m, got in _all_methods(prev).items():
            assert np.array_equal(got, want), (prev.tolist(), m, got.tolist(), want.tolist())


def test_forced_runs_with_a_small_workspace_is_refused():
    import torch
    import paper_2609_28870_gb300 as ptc
    prev = np.full(5000, oracle.NONE, dtype=np.uint32)
    prev[1::2] = np.arange(0, 4999, 2, dtype=np.uint32)  # every access starts a run
    want = oracle.sd_fenwick(prev)
    p = ptc.to_device_u32(prev)
    L = ptc.lib()
    ws = torch.empty(L.ptc_stack_distance_workspace_bytes(prev.size), dtype=torch.uint8, device="cuda")
    # the automatic choice counts over the accesses instead
    assert np.array_equal(ptc.u32(ptc.ptc_stack_distance(p, ws=ws)), want)
    dist = torch.empty(prev.size, dtype=torch.int32, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    rc = L.ptc_stack_distance_ex(p.data_ptr(), prev.size, dist.data_ptr(), ptc.PTC_SD_RUNS, ws.data_ptr(),
                                 ws.numel(), stream)
    assert ptc.STATUS[rc] == "PTC_ERR_WORKSPACE"
    big = torch.empty(L.ptc_stack_distance_ex_workspace_bytes(prev.size, ptc.PTC_SD_RUNS), dtype=torch.uint8,
                      device="cuda")
    rc = L.ptc_stack_distance_ex(p.data_ptr(), prev.size, dist.data_ptr(), ptc.PTC_SD_RUNS, big.data_ptr(),
                                 big.numel(), stream)
    assert rc == 0 and np.array_equal(ptc.u32(dist), want)
    rc = L.ptc_stack_distance_ex(p.data_ptr(), prev.size, dist.data_ptr(), 7, big.data_ptr(), big.numel(), stream)
    assert ptc.STATUS[rc] == "PTC_ERR_INVALID_ARG"


def test_many_runs_take_the_per_level_build():
    """A random reuse array with short runs, about as many as accesses, forced
    onto the count over runs (by blocks of pair sums; tests/test_gpu_pieces.py
    has more runs than those take, which go to the matrix level by level)."""
    import torch
    import paper_2609_28870_gb300 as ptc
    rng = np.random.default_rng(11)
    ids = rng.integers(0, 60000, size=300000).astype(np.uint32)
    _, first = np.unique(ids, return_index=True)
    order = np.argsort(np.argsort(first))
    dense = np.empty_like(ids)
    remap = np.empty(ids.max() + 1, dtype=np.uint32)
    remap[np.unique(ids)] = order.astype(np.uint32)
    dense = remap[ids]
    prev, _ = oracle.reuse(dense, int(dense.max()) + 1)
    want = oracle.sd_fenwick(prev)
    p = ptc.to_device_u32(prev)
    got = ptc.u32(ptc.ptc_stack_distance(p, method=ptc.PTC_SD_RUNS))
    assert np.array_equal(got, want)


@pytest.mark.parametrize("shift", [0, 1])  # 16-byte loads, and prev off their alignment
def test_previous_uses_that_do_not_lie_before(shift):
    """A previous use at or after its access is an error, whatever it is: the key
    of its run is not marked (the highest would lie 512 MB past the bitmap)."""
    import torch
    import paper_2609_28870_gb300 as ptc
    n = 50_000
    good = np.full(n, oracle.NONE, dtype=np.uint32)
    good[n // 2:] = np.arange(n - n // 2)  # few runs: pass 2 marks them
    want = oracle.sd_fenwick(good)
    buf = torch.zeros(n + shift, dtype=torch.int32, device="cuda")
    for at, value in ((n // 3, 0xFFFFFFFE), (n - 1, n - 1), (7, 0x80000000), (0, 0)):
        bad = good.copy()
        bad[at] = value
        buf[shift:] = ptc.to_device_u32(bad)
        for method in (None, ptc.PTC_SD_RUNS):
            with pytest.raises(ptc.PtcError) as e:
                ptc.ptc_stack_distance(buf[shift:], method=method)
            assert e.value.name == "PTC_ERR_INVALID_ARG"
    buf[shift:] = ptc.to_device_u32(good)
    assert np.array_equal(ptc.u32(ptc.ptc_stack_distance(buf[shift:])), want)


@pytest.mark.parametrize("order,residency", [(1, 0), (1, 1), (0, 1)])
def test_variants_with_malformed_offsets(order, residency):
    """Offsets that leave accesses to no request: leaf-first, their previous uses
    in touch order are never written, and hold what the workspace held."""
    import torch
    import paper_2609_28870_gb300 as ptc
    n = 50_000
    prev = np.full(n, oracle.NONE, dtype=np.uint32)
    prev[n // 2:] = np.arange(n - n // 2)
    p = ptc.to_device_u32(prev)
    L = ptc.lib()
    ws = torch.empty(L.ptc_stack_distance_variant_workspace_bytes(n, 3, order, residency), dtype=torch.uint8,
                     device="cuda")
    for off in ([0, 100, 200, n - 5000], [0, 30_000, 20_000, n], [10, 100, 200, n]):
        ws.fill_(0xFE)
        with pytest.raises(ptc.PtcError) as e:
            ptc.ptc_stack_distance_variant(p, ptc.to_device_u64(np.array(off, np.uint64)), order, residency, ws=ws)
        assert e.value.name == "PTC_ERR_INVALID_ARG"
    good = ptc.to_device_u64(np.array([0, n // 2, n // 2, n], np.uint64))
    a = ptc.ptc_stack_distance_variant(p, good, order, residency, ws=ws)
    b = ptc.ptc_stack_distance_variant(p, good, order, residency, method=ptc.PTC_SD_POINTS)
    assert torch.equal(a, b)
