"""The sorts that are timed: single arrays and batches through the package's public calls.

A case names a call (`sort_keys`, `sort_pairs` or `sort_batch`), a key type, an order, a bit range, the keys'
distribution and the sizes. Its state holds what a program that sorts repeatedly keeps: the inputs, the output
arrays and the workspace (for a batch also the captured CUDA graph, where the case says so).

Left out: the host-memory calls (bound by the host link), and the service loop and its cost model, which spend
their device time in the batched call that is here.
"""
import math

import numpy as np
import torch

from paper_2206_01784_gb300 import onesweep as osw

BITS = {"u32": 32, "i32": 32, "f32": 32, "u64": 64, "i64": 64, "f64": 64}
DTYPE = {"u32": torch.int32, "i32": torch.int32, "f32": torch.float32,
         "u64": torch.int64, "i64": torch.int64, "f64": torch.float64}
MAX_BYTES = 3 << 30  # inputs of the largest cases: 256M 32-bit pairs, 128M 64-bit pairs, 288M-key batches


def _single(name, key_type, n, pairs, dist="uniform", descending=False, begin_bit=0, end_bit=None):
    return {"name": name, "kind": "single", "key_type": key_type, "n": n, "pairs": pairs, "dist": dist,
            "descending": descending, "begin_bit": begin_bit,
            "end_bit": BITS[key_type] if end_bit is None else end_bit}


def _batch(name, key_type, segments, median, sigma, lo, hi, pairs, graph, dist="uniform"):
    return {"name": name, "kind": "batch", "key_type": key_type, "segments": segments, "median": median,
            "sigma": sigma, "lo": lo, "hi": hi, "pairs": pairs, "graph": graph, "dist": dist, "descending": False,
            "begin_bit": 0, "end_bit": BITS[key_type]}


def listed():
    return [
        # a short candidate list ordered by score, best first: the call's latency is all there is
        _single("f32_pairs_desc_1000", "f32", 1000, True, "normal", descending=True),
        # the smallest requests of the sort service
        _single("u32_pairs_16k", "u32", 16384, True),
        # composite 64-bit ids of which the low 40 bits vary, a ragged mid-size table column
        _single("u64_pairs_40bit_150k", "u64", 150_001, True, end_bit=40),
        # 1M uniform uint32 keys, the package's smallest named workload
        _single("u32_keys_1m", "u32", 1 << 20, False),
        # signed row ids with heavy duplication (AND of three words), a ragged size
        _single("i32_pairs_and3_5m", "i32", 5_000_011, True, "and3"),
        # double-precision values alone
        _single("f64_keys_12m", "f64", 12_345_678, False, "normal"),
        # N(0,1) float32 keys with signed zeros, with their row indices
        _single("f32_pairs_64m", "f32", 1 << 26, True, "normal"),
        # 256M uint32 keys alone: the size and shape the method is quoted on
        _single("u32_keys_256m", "u32", 1 << 28, False),
        # 256M uint32 keys with index values: the benchmark's default workload
        _single("u32_pairs_256m", "u32", 1 << 28, True),
        # 128M uint64 keys with index values, 8 passes
        _single("u64_pairs_128m", "u64", 1 << 27, True),
        # token routing: many short rows, each sorted by itself, the launch sequence captured once
        _batch("batch_u32_pairs_2048_short", "u32", 2048, 1500.0, 1.0, 16, 16384, True, True),
        # 4096 uneven arrays (lognormal lengths, 1K-4M keys, 288M in all) under a CUDA graph
        _batch("batch_u32_pairs_4096", "u32", 4096, 32768.0, 1.18, 1024, 4 << 20, True, True),
    ]


def _unnamed(case):
    return {k: v for k, v in case.items() if k != "name"}


def _log_size(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    # sizes that people write down are often round; the rest are whatever the data has
    return n if rng.random() < 0.75 else max(lo, n >> 8 << 8)


def draw(rng):
    key_type = rng.choice(["u32", "u32", "u32", "i32", "f32", "f32", "u64", "i64", "f64"])
    wide = BITS[key_type] == 64
    pairs = rng.random() < 0.65
    dist = "normal" if key_type in ("f32", "f64") else rng.choice(["uniform", "uniform", "and2", "and3", "and5", "const"])
    if rng.random() < 0.25:
        segments = _log_size(rng, 16, 4096)
        # a mean length of 32768 * exp(1.18^2 / 2) keys with 4096 segments is the largest listed batch
        median = float(_log_size(rng, 64, 32768 if not wide else 12000))
        return _unnamed(_batch("", key_type, segments, median, round(rng.uniform(0.3, 1.18), 2), 1, int(median * 64),
                               pairs, rng.random() < 0.5, dist))
    n = _log_size(rng, 500, 1 << (27 if wide else 28))
    begin, end = 0, BITS[key_type]
    if key_type[0] != "f" and rng.random() < 0.2:
        begin = rng.choice([0, 0, 3, 8])
        end = rng.randint(begin + 5, BITS[key_type])
    return _unnamed(_single("", key_type, n, pairs, dist, rng.random() < 0.25, begin, end))


def _lengths(case):
    """Segment lengths, the same multiset for every seed (so that outputs keep their shapes)."""
    z = np.random.RandomState(10).standard_normal(case["segments"])
    lengths = np.clip(np.rint(case["median"] * np.exp(case["sigma"] * z)), case["lo"], case["hi"]).astype(np.int64)
    most = MAX_BYTES // (BITS[case["key_type"]] // 8 + (4 if case["pairs"] else 0))
    while lengths.sum() > most:
        lengths = np.maximum(lengths * 3 // 4, 1)
    return lengths


def _offsets(case, seed):
    lengths = np.random.RandomState(seed % (1 << 31)).permutation(_lengths(case))
    return np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)


def _keys(case, n, gen):
    dtype, dist = DTYPE[case["key_type"]], case["dist"]
    if dist == "normal":
        k = torch.empty(n, dtype=dtype, device="cuda").normal_(generator=gen)
        spot = torch.empty(n, dtype=torch.uint8, device="cuda").random_(0, 200, generator=gen)
        k[spot == 0] = 0.0
        k[spot == 1] = -0.0
        return k
    lo, hi = torch.iinfo(dtype).min, torch.iinfo(dtype).max

    def word():
        # every bit uniform (random_ leaves out the largest value of a 64-bit type)
        return torch.empty(n, dtype=dtype, device="cuda").random_(lo, hi if dtype == torch.int64 else hi + 1,
                                                                  generator=gen)

    if dist == "const":
        return word()[:1].expand(n).contiguous()
    k = word()
    for _ in range(int(dist[3:]) - 1 if dist.startswith("and") else 0):
        k &= word()
    return k


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kt = osw.KEY_TYPES[case["key_type"]]
    begin, end = case["begin_bit"], case["end_bit"]
    vb = 4 if case["pairs"] else 0
    batch = case["kind"] == "batch"
    offsets = _offsets(case, seed) if batch else None
    n = int(offsets[-1]) if batch else case["n"]
    keys = _keys(case, n, gen)
    values = torch.arange(n, dtype=torch.int32, device="cuda") if case["pairs"] else None
    state = {"case": case, "keys": keys, "values": values, "keys_out": torch.empty_like(keys),
             "values_out": torch.empty_like(values) if case["pairs"] else None, "graph": None}
    if not batch:
        state["ws"] = osw.workspace(kt, n, vb, begin, end, keys.device)
        return state
    state["offsets"] = torch.from_numpy(offsets).cuda()
    state["ws"] = osw.batch_workspace(kt, n, case["segments"], vb, begin, end, keys.device)
    if case["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _call(state)
        torch.cuda.current_stream().wait_stream(side)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            _call(state)
        state["graph"] = graph
    return state


def _call(s):
    case = s["case"]
    opts = {"begin_bit": case["begin_bit"], "end_bit": case["end_bit"], "key_type": case["key_type"], "ws": s["ws"],
            "descending": case["descending"]}
    if case["kind"] == "batch":
        return osw.sort_batch(s["keys"], s["offsets"], s["values"], keys_out=s["keys_out"],
                              values_out=s["values_out"], **opts)
    if case["pairs"]:
        return osw.sort_pairs(s["keys"], s["values"], keys_out=s["keys_out"], values_out=s["values_out"], **opts)
    return osw.sort_keys(s["keys"], out=s["keys_out"], **opts)


def run(state):
    if state["graph"] is not None:
        state["graph"].replay()
        return (state["keys_out"], state["values_out"]) if state["values_out"] is not None else state["keys_out"]
    return _call(state)


def work(case):
    n = int(_lengths(case).sum()) if case["kind"] == "batch" else case["n"]
    return {"bytes": 2.0 * n * (BITS[case["key_type"]] // 8 + (4 if case["pairs"] else 0)), "flops": 0.0}


def exact(case, seed):
    """Sorted float keys as torch orders them in 64 bits; integer results are compared as they are."""
    if case["key_type"][0] != "f" or case["begin_bit"] != 0 or case["end_bit"] != BITS[case["key_type"]]:
        return None
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["kind"] == "batch":
        offsets = _offsets(case, seed)
        keys = _keys(case, int(offsets[-1]), gen).double()
        out = torch.cat([keys[a:b].sort(descending=case["descending"])[0]
                         for a, b in zip(offsets[:-1].tolist(), offsets[1:].tolist())])
    else:
        out = _keys(case, case["n"], gen).double().sort(descending=case["descending"])[0]
    return (out, None) if case["pairs"] else out
