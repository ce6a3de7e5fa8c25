"""Sorts by the route they take, bit-exact against the oracle.

A sort that names a tile variant runs pass by pass whatever its size, so the
variants' kernels are reached by naming them, with both payloads; the sizes of
the cluster form are those around its 8 and 16 blocks; and the default's tile
is asserted beside the sorts that rely on it.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2206_01784_gb300 import autotune  # noqa: E402
from paper_2206_01784_gb300 import onesweep as osw  # noqa: E402
from paper_2206_01784_gb300 import workload  # noqa: E402

pytestmark = pytest.mark.gpu

KB = {"u32": 32, "u64": 64, "f32": 32, "f64": 64, "i32": 32, "i64": 64}
DEFAULT = osw.OS_TILE_CONFIG_DEFAULT


def _dev(a, shift=0):
    """A copy on the device, `shift` elements past an aligned address."""
    t = torch.from_numpy(np.concatenate([np.zeros(shift, a.dtype), a]).view(np.int64 if a.dtype.itemsize == 8 else np.int32))
    return t.cuda()[shift:]


def _check(kt, keys, pairs, variant=None, begin=0, end=None, descending=False, shift=0, radix_bits=None):
    end = KB[kt] if end is None else end
    n = keys.size
    key_type = osw.KEY_TYPES[kt] | (osw.OS_SORT_DESCENDING if descending else 0)
    vals = workload.iota_u32(n)
    k, v = _dev(keys, shift), _dev(vals, shift)
    ko, vo = _dev(np.zeros_like(keys), shift), _dev(np.zeros_like(vals), shift)
    ws = osw.workspace(key_type, n, 4 if pairs else 0, begin, end, k.device).random_(0, 256)
    s = torch.cuda.current_stream().cuda_stream
    tail = (n, begin, end, ws.data_ptr(), ws.numel(), s)
    opts = dict(tile_config=variant, radix_bits=radix_bits)
    if pairs:
        rc = osw.os_sort_pairs_ex(key_type, k.data_ptr(), ko.data_ptr(), v.data_ptr(), vo.data_ptr(), *tail, **opts)
    else:
        rc = osw.os_sort_keys_ex(key_type, k.data_ptr(), ko.data_ptr(), *tail, **opts)
    assert rc == osw.OS_OK and osw.os_workspace_status(ws.data_ptr(), s) == osw.OS_OK
    exp = oracle.sort(kt, keys, vals if pairs else None, begin, end, descending=descending)
    ek = exp[0] if pairs else exp
    assert np.array_equal(ko.cpu().numpy().view(ek.dtype), ek)
    assert not pairs or np.array_equal(vo.cpu().numpy().view(np.uint32), exp[1])


def _keys(kt, dist, n, seed):
    return workload.keys(kt, "normal" if kt[0] == "f" else dist, n, seed=seed)


@pytest.mark.parametrize("pairs", [True, False])
@pytest.mark.parametrize("kt", ["u32", "u64", "f32", "i64"])
@pytest.mark.parametrize("cfg", range(12))
def test_every_variant_with_both_payloads(cfg, kt, pairs):
    t = osw.os_tile_config_keys(KB[kt], 4 if pairs else 0, cfg)
    for n in (t - 1, 2 * t, 5 * t + 3):
        _check(kt, _keys(kt, "and2", n, cfg * 7 + n), pairs, cfg)


@pytest.mark.parametrize("shift", [1, 2, 3])
@pytest.mark.parametrize("kt,pairs,cfg", [("u32", True, 4), ("u32", False, 4), ("u64", True, 4), ("u64", False, 6),
                                          ("f32", True, 5), ("u32", True, 7), ("u64", True, 7), ("f64", False, 3)])
def test_pass_by_pass_at_any_address(kt, pairs, cfg, shift):
    t = osw.os_tile_config_keys(KB[kt], 4 if pairs else 0, cfg)
    for n in (t + 1, 7 * t - 5):
        _check(kt, _keys(kt, "and2", n, n), pairs, cfg, shift=shift)


@pytest.mark.parametrize("seed", range(16))
def test_random_sorts_pass_by_pass(seed):
    rng = np.random.default_rng(1000 + seed)
    kt = str(rng.choice(list(KB)))
    n = int(np.exp(rng.uniform(np.log(1), np.log(400_000))))
    begin = int(rng.integers(0, KB[kt] - 1)) if kt[0] != "f" and rng.random() < 0.5 else 0
    end = int(rng.integers(begin + 1, KB[kt] + 1)) if kt[0] != "f" and rng.random() < 0.5 else KB[kt]
    dist = str(rng.choice(["uniform", "and2", "and3", "and8", "const"]))
    _check(kt, _keys(kt, dist, n, seed), bool(rng.integers(2)), int(rng.integers(12)), begin, end,
           bool(rng.integers(2)), int(rng.integers(4)))


CLUSTERS = [4097, 6000, 8191, 8192, 8193, 9 * 1024, 9 * 1024 + 1, 15 * 1024 + 1, 16383, 16384, 16385]


@pytest.mark.parametrize("n", CLUSTERS)
@pytest.mark.parametrize("kt,dist,begin,end,descending", [
    ("u32", "uniform", 0, 32, False), ("f32", "normal", 0, 32, True), ("i64", "and3", 7, 64, True),
    ("f64", "normal", 0, 64, False), ("u64", "const", 0, 40, False), ("i32", "and8", 0, 31, False)])
def test_clusters(n, kt, dist, begin, end, descending):
    for pairs in (True, False):
        _check(kt, _keys(kt, dist, n, n), pairs, None, begin, end, descending, shift=n % 4)


def test_clusters_on_several_streams_and_in_a_graph():
    sizes = (6000, 9217, 16384, 12_345, 16384, 5000)
    work = []
    for i, n in enumerate(sizes):
        keys = _keys("u32", "and2", n, i)
        work.append((keys, _dev(keys), _dev(workload.iota_u32(n)), torch.cuda.Stream(),
                     osw.workspace(osw.OS_KEY_U32, n, 4, 0, 32, "cuda")))
    torch.cuda.synchronize()
    # (outputs of every round are kept: the allocator knows nothing of the streams)
    outs = [[osw.sort_pairs(k, v, key_type="u32", ws=ws, stream=s) for _, k, v, s, ws in work] for _ in range(4)]
    torch.cuda.synchronize()
    for (keys, *_), (ko, vo) in zip(work * len(outs), sum(outs, [])):
        ek, ev = oracle.sort("u32", keys, workload.iota_u32(keys.size))
        assert np.array_equal(ko.cpu().numpy().view(np.uint32), ek) and np.array_equal(vo.cpu().numpy().view(np.uint32), ev)
    for _, k, v, _, ws in work:
        ko, vo = torch.empty_like(k), torch.empty_like(v)
        run = lambda: osw.sort_pairs(k, v, key_type="u32", keys_out=ko, values_out=vo, ws=ws)  # noqa: E731
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            run()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            run()
        keys = _keys("u32", "and3", k.numel(), 77)
        k.copy_(_dev(keys))
        ws.random_(0, 256)
        graph.replay()
        torch.cuda.synchronize()
        ek, ev = oracle.sort("u32", keys, workload.iota_u32(keys.size))
        assert np.array_equal(ko.cpu().numpy().view(np.uint32), ek) and np.array_equal(vo.cpu().numpy().view(np.uint32), ev)


@pytest.mark.parametrize("kt,pairs", [("u32", True), ("u64", False)])
def test_default_by_size_is_what_runs(kt, pairs):
    vb, saved = 4 if pairs else 0, autotune.current()
    tiles = [osw.os_tile_config_keys(KB[kt], vb, 4 + g) for g in range(3)]
    try:
        for variant in (None, DEFAULT):
            # (named for the call, the default holds whatever the process-wide variant)
            assert osw.os_set_tile_config(KB[kt], vb, DEFAULT if variant is None else 0) == osw.OS_OK
            for edge, below, above in ((152 * 4 * tiles[2], tiles[2], tiles[1]), (152 * 3 * tiles[1], tiles[1], tiles[0])):
                for n, tile in ((edge, below), (edge + 1, above)):
                    if variant is None:
                        assert osw.os_sort_workspace_layout(osw.KEY_TYPES[kt], n, vb, 0, 13).tile_keys == tile
                    _check(kt, _keys(kt, "and2", n, n % 97), pairs, variant, 0, 13)
        _check(kt, _keys(kt, "and2", 100_003, 3), pairs, DEFAULT, radix_bits=6)
    finally:
        autotune.apply(saved)



@pytest.mark.parametrize("cfg", [4, 5, 6, DEFAULT])
@pytest.mark.parametrize("by_call", [True, False])
def test_a_batch_runs_the_variant_that_was_set(cfg, by_call):
    # word 2 of the workspace: the tiles that the plan laid out
    sizes = [100_000, 50_001, 70_000]
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    keys, vals, n = _keys("u32", "and2", int(offs[-1]), 5), workload.iota_u32(int(offs[-1])), int(offs[-1])
    tile = osw.os_tile_config_keys(32, 4, 6 if cfg == DEFAULT else cfg)  # (by size: a small batch, small tiles)
    k, v, o = _dev(keys), _dev(vals), torch.from_numpy(offs).cuda()
    ko, vo = torch.empty_like(k), torch.empty_like(v)
    ws = osw.batch_workspace(osw.OS_KEY_U32, n, len(sizes), 4, 0, 32, "cuda")
    s = torch.cuda.current_stream().cuda_stream
    saved = autotune.current()
    try:
        assert osw.os_set_tile_config(32, 4, 0 if by_call else cfg) == osw.OS_OK
        assert osw.os_sort_batch_ex(osw.OS_KEY_U32, k.data_ptr(), ko.data_ptr(), v.data_ptr(), vo.data_ptr(),
                                    o.data_ptr(), len(sizes), n, 0, 32, ws.data_ptr(), ws.numel(), s,
                                    tile_config=cfg if by_call else None) == osw.OS_OK
        assert osw.os_workspace_status(ws.data_ptr(), s) == osw.OS_OK
    finally:
        autotune.apply(saved)
    assert int(ws[8:12].cpu().numpy().view(np.uint32)[0]) == sum((x + tile - 1) // tile for x in sizes)
    ek, ev = oracle.sort_segments("u32", keys, offs.astype(np.uint64), vals)
    assert np.array_equal(ko.cpu().numpy().view(np.uint32), ek) and np.array_equal(vo.cpu().numpy().view(np.uint32), ev)


@pytest.mark.parametrize("segments", [1, 100, 152, 153, 304, 305, 457, 700])
@pytest.mark.parametrize("kt,pairs,dist", [("u32", True, "and2"), ("u64", True, "uniform"), ("f32", False, "normal")])
def test_batches_by_blocks_an_sm(segments, kt, pairs, dist):
    # one to four blocks an SM, of 256 threads or (few long segments) of 1024
    cap = 4096 if KB[kt] == 32 else 2048
    for lo, hi in ((1, 200), (cap // 2, cap), (cap // 2, 4 * cap)):
        sizes = np.random.default_rng(segments).integers(lo, hi + 1, segments)
        offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        keys, vals = _keys(kt, dist, int(offs[-1]), segments), workload.iota_u32(int(offs[-1]))
        ws = osw.batch_workspace(osw.KEY_TYPES[kt], keys.size, segments, 4 if pairs else 0, 0, KB[kt], "cuda").random_(0, 256)
        out = osw.sort_batch(_dev(keys), torch.from_numpy(offs).cuda(), _dev(vals) if pairs else None, key_type=kt, ws=ws)
        assert osw.os_workspace_status(ws.data_ptr(), torch.cuda.current_stream().cuda_stream) == osw.OS_OK
        exp = oracle.sort_segments(kt, keys, offs.astype(np.uint64), vals if pairs else None)
        ko, ek = (out[0], exp[0]) if pairs else (out, exp)
        assert np.array_equal(ko.cpu().numpy().view(ek.dtype), ek)
        assert not pairs or np.array_equal(out[1].cpu().numpy().view(np.uint32), exp[1])


def _shared(kt, n, seed, live, odd):
    """Uniform words of which only the bits `live` vary; with `odd`, the last key alone differs in every bit."""
    keys = workload.keys("u64" if KB[kt] == 64 else "u32", "uniform", n, seed=seed)
    word = workload.keys("u64" if KB[kt] == 64 else "u32", "uniform", 1, seed=seed + 1)
    live = keys.dtype.type(live & ((1 << KB[kt]) - 1))
    out = (keys & live) | (word[0] & ~live)
    if odd and n:
        out[-1] = ~out[0]
    return out


@pytest.mark.parametrize("live", [0, 0xFF, 0xFFFF, 0xFF00FF00, 0x00FF0000, 1 << 31, 0xFFFF << 40, 0x0F0F0F0F0F0F0F0F])
@pytest.mark.parametrize("kt,pairs,begin,end,descending", [
    ("u32", True, 0, 32, False), ("i32", False, 0, 32, True), ("u32", True, 3, 29, False), ("u64", True, 0, 64, False),
    ("i64", False, 5, 61, True)])
def test_batch_rows_that_share_places(kt, pairs, begin, end, descending, live):
    # places that a whole segment shares are passed over, in each class, by few wide blocks or many narrow ones
    cap = 4096 if KB[kt] == 32 else 2048
    sizes = [1, 2, 31, 257, 300, 1000, cap - 1, cap, cap + 1, 2 * cap, 3 * cap + 5, 4 * cap]
    for sizes in (sizes, sizes + [700] * 300, sizes + [20] * 300):
        offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        keys = np.concatenate([_shared(kt, n, i, live, i % 3 == 2) for i, n in enumerate(sizes)])
        vals = workload.iota_u32(keys.size)
        key_type = osw.KEY_TYPES[kt]
        ws = osw.batch_workspace(key_type, keys.size, len(sizes), 4 if pairs else 0, begin, end, "cuda").random_(0, 256)
        out = osw.sort_batch(_dev(keys), torch.from_numpy(offs).cuda(), _dev(vals) if pairs else None, begin, end,
                             key_type=kt, ws=ws, descending=descending)
        assert osw.os_workspace_status(ws.data_ptr(), torch.cuda.current_stream().cuda_stream) == osw.OS_OK
        exp = oracle.sort_segments(kt, keys, offs.astype(np.uint64), vals if pairs else None, begin, end,
                                   descending=descending)
        ko, ek = (out[0], exp[0]) if pairs else (out, exp)
        assert np.array_equal(ko.cpu().numpy().view(ek.dtype), ek)
        assert not pairs or np.array_equal(out[1].cpu().numpy().view(np.uint32), exp[1])
