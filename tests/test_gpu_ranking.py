"""The binning kernel's rankings, ragged tiles and the classes of a batch, bit-exact against the oracle.

Every sort names tile variant 4 (the default geometry, adaptive ranking), so
that it runs pass by pass whatever its size. The keys make each place rank in
each way - counting atomics, the most frequent digit apart, ballots - and the
sizes end in ragged tiles, whose fill must never reach the output: bit ranges
that leave a narrow top place, signed, float and descending orders included.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2206_01784_gb300 import onesweep as osw  # noqa: E402
from paper_2206_01784_gb300 import workload  # noqa: E402

pytestmark = pytest.mark.gpu

KB = {"u32": 32, "u64": 64, "f32": 32, "f64": 64, "i32": 32, "i64": 64}
VARIANT = 4


def _dev(a):
    return torch.from_numpy(a.view(np.int64 if a.dtype.itemsize == 8 else np.int32).copy()).cuda()


def _check(kt, keys, pairs, begin=0, end=None, descending=False, variant=VARIANT):
    end = KB[kt] if end is None else end
    n = keys.size
    key_type = osw.KEY_TYPES[kt] | (osw.OS_SORT_DESCENDING if descending else 0)
    vals = workload.iota_u32(n)
    k, v = _dev(keys), _dev(vals)
    ko, vo = torch.zeros_like(k), torch.zeros_like(v)
    ws = osw.workspace(key_type, n, 4 if pairs else 0, begin, end, k.device).random_(0, 256)
    s = torch.cuda.current_stream().cuda_stream
    tail = (n, begin, end, ws.data_ptr(), ws.numel(), s)
    if pairs:
        rc = osw.os_sort_pairs_ex(key_type, k.data_ptr(), ko.data_ptr(), v.data_ptr(), vo.data_ptr(), *tail,
                                  tile_config=variant)
    else:
        rc = osw.os_sort_keys_ex(key_type, k.data_ptr(), ko.data_ptr(), *tail, tile_config=variant)
    assert rc == osw.OS_OK and osw.os_workspace_status(ws.data_ptr(), s) == osw.OS_OK
    exp = oracle.sort(kt, keys, vals if pairs else None, begin, end, descending=descending)
    ek = exp[0] if pairs else exp
    assert np.array_equal(ko.cpu().numpy().view(ek.dtype), ek)
    assert not pairs or np.array_equal(vo.cpu().numpy().view(np.uint32), exp[1])


def _digits(kt, n, seed, shares):
    """Keys whose every byte is drawn from the given shares of byte values (the rest uniform)."""
    rng = np.random.default_rng(seed)
    values = rng.permutation(256)[: len(shares)]
    p = np.full(256, (1.0 - sum(shares)) / (256 - len(shares)))
    p[values] = shares
    size = KB[kt] // 8
    return rng.choice(256, size=n * size, p=p).astype(np.uint8).view(np.uint32 if size == 4 else np.uint64)


def _tile(kt, pairs):
    return osw.os_tile_config_keys(KB[kt], 4 if pairs else 0, VARIANT)


# shares of the most frequent byte values: atomics, one digit apart (a little
# and mostly), ballots (several frequent digits, two digits, 16 digits alone)
SHARES = {"uniform": (), "tenth": (0.1,), "most": (0.9,), "all but few": (0.999,), "several": (0.3, 0.2, 0.1, 0.1),
          "two": (0.5, 0.499), "sixteen": (1 / 16 - 1e-6,) * 16}


@pytest.mark.parametrize("shares", SHARES)
@pytest.mark.parametrize("kt,pairs", [("u32", True), ("u32", False), ("u64", True), ("u64", False)])
def test_each_way_of_ranking(kt, pairs, shares):
    t = _tile(kt, pairs)
    for n in (t - 1, 3 * t, 5 * t + 33):
        _check(kt, _digits(kt, n, n % 97, SHARES[shares]), pairs)


@pytest.mark.parametrize("kt,dist,begin,end,descending", [
    ("i32", "uniform", 0, 32, False), ("i32", "and3", 3, 32, True), ("u32", "const", 0, 32, False),
    ("u32", "uniform", 5, 18, True), ("u32", "and8", 9, 12, False), ("f32", "normal", 0, 32, True),
    ("f64", "normal", 0, 64, False), ("i64", "and2", 0, 61, True), ("u64", "const", 3, 40, True)])
@pytest.mark.parametrize("pairs", [True, False])
def test_ragged_tiles(kt, dist, begin, end, descending, pairs):
    t = _tile(kt, pairs)
    for n in (1, 31, t - 1, t + 1, 2 * t + 4097):
        _check(kt, workload.keys(kt, dist, n, seed=n), pairs, begin, end, descending)


# ---------------------------------------------------------------- batches

def _batch(kt, sizes, pairs, dist, seed, descending=False, begin=0, end=None):
    end = KB[kt] if end is None else end
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(offs[-1])
    keys = workload.keys(kt, dist, n, seed)
    vals = workload.iota_u32(n)
    key_type = osw.KEY_TYPES[kt]
    ws = osw.batch_workspace(key_type, n, len(sizes), 4 if pairs else 0, begin, end, "cuda").random_(0, 256)
    out = osw.sort_batch(_dev(keys), torch.from_numpy(offs).cuda(), _dev(vals) if pairs else None, begin, end,
                         key_type=kt, ws=ws, descending=descending)
    assert osw.os_workspace_status(ws.data_ptr(), torch.cuda.current_stream().cuda_stream) == osw.OS_OK
    exp = oracle.sort_segments(kt, keys, offs.astype(np.uint64), vals if pairs else None, begin, end,
                               descending=descending)
    ko, ek = (out[0], exp[0]) if pairs else (out, exp)
    assert np.array_equal(ko.cpu().numpy().view(ek.dtype), ek)
    assert not pairs or np.array_equal(out[1].cpu().numpy().view(np.uint32), exp[1])


CLASSES = {32: (4096, 8192, 16384), 64: (2048, 4096, 8192)}


@pytest.mark.parametrize("kt,pairs,dist,descending", [
    ("u32", True, "uniform", False), ("u32", False, "and5", False), ("u64", True, "and2", True),
    ("f32", True, "normal", True), ("f64", False, "normal", False), ("i32", True, "const", False)])
@pytest.mark.parametrize("empty", [2, 400])  # few segments: one block of 1024 threads each
@pytest.mark.parametrize("longest", [0, 1, 60_001])
def test_batch_class_edges(kt, pairs, dist, descending, longest, empty):
    # longest: nothing above the last class, one key above it, or several tiles;
    # with a longer segment, only the first class is sorted in one block
    caps = CLASSES[KB[kt]]
    sizes = [c + d for c in caps for d in (-1, 0, 1)][:-1] + [0, 1, 33, 256, 257, 1000] + [0] * empty
    sizes += [caps[-1] + longest] if longest else []
    _batch(kt, sizes, pairs, dist, 7, descending)


@pytest.mark.parametrize("segments", [1023, 1024, 2500])
def test_batch_of_many_short_segments(segments):
    sizes = workload.segment_sizes(segments, seed=segments, median=90.0, sigma=1.3, lo=0, hi=5000)
    _batch("u32", [int(x) for x in sizes], True, "and2", 9)
    _batch("u32", [0] * segments + [17], False, "uniform", 10)


def test_batch_bit_ranges_of_each_class():
    for begin, end in ((0, 8), (3, 29), (31, 32)):
        _batch("u32", [100, 5000, 9000, 16384, 4096], True, "uniform", 11, begin=begin, end=end)
        _batch("u32", [100, 5000, 9000, 16385, 4096, 40_000], True, "and3", 12, True, begin, end)


@pytest.mark.parametrize("kt,pairs", [("u32", True), ("i32", False), ("u64", True), ("f64", False)])
def test_default_tiles_by_size(kt, pairs):
    # the default variant at the sizes where its tile changes
    keys = [osw.os_tile_config_keys(KB[kt], 4 if pairs else 0, VARIANT + g) for g in range(3)]
    for edge in (152 * 4 * keys[2], 152 * 3 * keys[1], 152 * 3 * keys[0]):
        for n in (edge, edge + 1):
            _check(kt, workload.keys(kt, "normal" if kt == "f64" else "and2", n, seed=n), pairs, 0, 13,
                   variant=None)
