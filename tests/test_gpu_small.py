"""Sorts that run as one launch (csrc/os_small.cu), bit-exact against the oracle.

The sizes are the edges of each form - one block, one cluster, a cooperative
grid, and the pass-by-pass kernels beyond - and of their tiles. Every
workspace starts as random bytes: the one-launch forms initialise what they
read.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2206_01784_gb300 import onesweep as osw  # noqa: E402
from paper_2206_01784_gb300 import workload  # noqa: E402

pytestmark = pytest.mark.gpu

KB = {"u32": 32, "u64": 64, "f32": 32, "f64": 64, "i32": 32, "i64": 64}
SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152
EDGES = sorted({1, 2, 31, 33, 3 * 2048 + 5}
               | {t + d for t in (1024, 4096) for d in (-1, 0, 1)}                      # one block
               | {16 * t + d for t in (2048, 4096, 8192) for d in (-1, 0, 1)}           # clusters
               | {SMS * t + d for t in (2048, 4096, 8192, 12288) for d in (0, 1)})      # grids


def _dev(a):
    return torch.from_numpy(a.view(np.int64 if a.dtype.itemsize == 8 else np.int32).copy()).cuda()


def _sort(kt, keys, pairs, begin=0, end=None, descending=False, stream=None):
    """(keys, values or None) on the device and the workspace's status."""
    end = KB[kt] if end is None else end
    k, v = _dev(keys), _dev(workload.iota_u32(keys.size))
    ws = osw.workspace(osw.KEY_TYPES[kt], keys.size, 4 if pairs else 0, begin, end, k.device).random_(0, 256)
    opts = dict(begin_bit=begin, end_bit=end, key_type=kt, ws=ws, descending=descending)
    out = osw.sort_pairs(k, v, **opts) if pairs else (osw.sort_keys(k, **opts), None)
    return out, osw.os_workspace_status(ws.data_ptr(), torch.cuda.current_stream().cuda_stream)


def _check(kt, keys, pairs, begin=0, end=None, descending=False):
    end = KB[kt] if end is None else end
    (ko, vo), status = _sort(kt, keys, pairs, begin, end, descending)
    assert status == osw.OS_OK
    vals = workload.iota_u32(keys.size) if pairs else None
    exp = oracle.sort(kt, keys, vals, begin, end, descending=descending)
    ek, ev = exp if pairs else (exp, None)
    assert np.array_equal(ko.cpu().numpy().view(ek.dtype), ek)
    assert not pairs or np.array_equal(vo.cpu().numpy().view(np.uint32), ev)


@pytest.mark.parametrize("kt,pairs", [("u32", True), ("u32", False), ("u64", True), ("u64", False)])
@pytest.mark.parametrize("n", EDGES)
def test_edges_of_every_form(n, kt, pairs):
    _check(kt, workload.keys(kt, "uniform" if n % 2 else "and2", n, seed=n % 89), pairs)


@pytest.mark.parametrize("n", [1000, 4000, 30_001, 60_000, 150_001, 1_200_007])
@pytest.mark.parametrize("kt,dist,begin,end,descending", [
    ("f32", "normal", 0, 32, True), ("f64", "normal", 0, 64, False), ("i32", "and3", 0, 32, False),
    ("i64", "uniform", 7, 64, True), ("u32", "const", 0, 32, False), ("u32", "and8", 3, 29, True),
    ("u64", "uniform", 0, 40, False), ("u32", "uniform", 4, 5, False), ("i32", "and16", 0, 31, True)])
def test_types_orders_and_bit_ranges(n, kt, dist, begin, end, descending):
    _check(kt, workload.keys(kt, dist, n, seed=n % 83), n % 2 == 1, begin, end, descending)


@pytest.mark.parametrize("n", [777, 20_000, 100_000, 700_000])
def test_unaligned_pointers_and_inputs_kept(n):
    keys = workload.keys("u32", "and2", n + 1, seed=5)
    k, v = _dev(keys)[1:], _dev(workload.iota_u32(n + 1))[1:]
    ko, vo = torch.empty(n + 1, dtype=torch.int32, device="cuda")[1:], torch.empty(n + 1, dtype=torch.int32, device="cuda")[1:]
    osw.sort_pairs(k, v, key_type="u32", keys_out=ko, values_out=vo)
    ek, ev = oracle.sort("u32", keys[1:], workload.iota_u32(n + 1)[1:])
    assert np.array_equal(ko.cpu().numpy().view(np.uint32), ek) and np.array_equal(vo.cpu().numpy().view(np.uint32), ev)
    assert np.array_equal(k.cpu().numpy().view(np.uint32), keys[1:])


@pytest.mark.parametrize("n", [900, 17_000, 120_000, 500_000])
def test_graph_replay_on_new_data(n):
    k, v = torch.empty(n, dtype=torch.int32, device="cuda"), _dev(workload.iota_u32(n))
    ko, vo = torch.empty_like(k), torch.empty_like(v)
    ws = osw.workspace(osw.OS_KEY_U32, n, 4, 0, 32, k.device)
    run = lambda: osw.sort_pairs(k, v, key_type="u32", keys_out=ko, values_out=vo, ws=ws)  # noqa: E731
    k.random_()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        run()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    for seed in (1, 2, 3):
        keys = workload.keys("u32", ("uniform", "and3", "const")[seed - 1], n, seed=seed)
        k.copy_(torch.from_numpy(keys.view(np.int32)))
        ws.random_(0, 256)
        graph.replay()
        torch.cuda.synchronize()
        ek, ev = oracle.sort("u32", keys, workload.iota_u32(n))
        assert np.array_equal(ko.cpu().numpy().view(np.uint32), ek)
        assert np.array_equal(vo.cpu().numpy().view(np.uint32), ev)


def test_sorts_on_several_streams_at_once():
    # grids and clusters of different sorts compete for the SMs
    sizes = (900_001, 50_000, 1_300_000, 3000, 400_000, 20_000)
    work = []
    for i, n in enumerate(sizes):
        keys = workload.keys("u32", "uniform", n, seed=i)
        work.append((keys, _dev(keys), _dev(workload.iota_u32(n)), torch.cuda.Stream(),
                     osw.workspace(osw.OS_KEY_U32, n, 4, 0, 32, "cuda")))
    torch.cuda.synchronize()
    # (outputs of every round are kept: the allocator knows nothing of the streams)
    outs = [[osw.sort_pairs(k, v, key_type="u32", ws=ws, stream=s) for _, k, v, s, ws in work] for _ in range(4)]
    torch.cuda.synchronize()
    for (keys, *_), (ko, vo) in zip(work * len(outs), sum(outs, [])):
        ek, ev = oracle.sort("u32", keys, workload.iota_u32(keys.size))
        assert np.array_equal(ko.cpu().numpy().view(np.uint32), ek)
        assert np.array_equal(vo.cpu().numpy().view(np.uint32), ev)


@pytest.mark.parametrize("cfg", range(12))
@pytest.mark.parametrize("kt", ["u32", "u64"])
def test_named_variants_still_run_pass_by_pass(cfg, kt):
    pairs = cfg % 2 == 0
    t = osw.os_tile_config_keys(KB[kt], 4 if pairs else 0, cfg)
    key_type = osw.KEY_TYPES[kt]
    for n in (t - 1, 2 * t, 5 * t + 3):
        keys = workload.keys(kt, "and2", n, seed=cfg)
        k, v = _dev(keys), _dev(workload.iota_u32(n))
        ko, vo = torch.empty_like(k), torch.empty_like(v)
        ws = osw.workspace(key_type, n, 4 if pairs else 0, 0, KB[kt], k.device)
        s = torch.cuda.current_stream().cuda_stream
        args = (n, 0, KB[kt], ws.data_ptr(), ws.numel(), s)
        if pairs:
            rc = osw.os_sort_pairs_ex(key_type, k.data_ptr(), ko.data_ptr(), v.data_ptr(), vo.data_ptr(), *args,
                                      tile_config=cfg)
        else:
            rc = osw.os_sort_keys_ex(key_type, k.data_ptr(), ko.data_ptr(), *args, tile_config=cfg)
        assert rc == osw.OS_OK and osw.os_workspace_status(ws.data_ptr(), s) == osw.OS_OK
        exp = oracle.sort(kt, keys, workload.iota_u32(n) if pairs else None)
        ek = exp[0] if pairs else exp
        assert np.array_equal(ko.cpu().numpy().view(ek.dtype), ek)
        assert not pairs or np.array_equal(vo.cpu().numpy().view(np.uint32), exp[1])
