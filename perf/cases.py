"""The plotting work that users of this package run, as cases that can be timed.

listed() names the cases and draw() gives more of the same kinds and ranges.
prepare() makes what a program holds before the call: the plot (its plan and
its bound device buffers) or the rows to hash.  run() is one pass through the
public calls.  work() is what a pass cannot do without.  exact() computes the
small cases in numpy, without this package.

Kinds:
  plot    vx_plot_run: both tables in one pass, then the sync that gives the
          Table-2 count (the call of the benchmark and of a plotting program)
  split   vx_table1, then vx_match (programs that use Table 1 by itself)
  cross   vx_plot_run with match_scope 1 (pairs across bucket edges)
  tiled   vx_plot_tiled: a plot built in 2^window_bits windows of less device
          memory, its Table 2 (what a plot file holds) copied to host memory
  sorted  a plot whose Table 2 is then ordered by its hash for lookups
  batch   vx_plot_batch of plots of mixed K
  rows    vx_hash_nonces of a run of nonces and vx_pair_hash of a list of
          pairs (a program that checks records and pairs it was handed)
"""
import math

import numpy as np
import torch

from paper_2606_14007_gb300 import vaultx as vx

# BLAKE3 compressions take 53 message-dependent G functions of 12 operations,
# less the 14 of the last round that reach no kept word, plus 2 output xors.
OPS_PER_HASH = 624


def listed():
    return [
        # smoke-sized plot: launches and latency are all of it
        {"name": "plot_k14", "kind": "plot", "K": 14},
        # the smallest plot of the batch mix, one scatter level
        {"name": "plot_k20", "kind": "plot", "K": 20},
        # the small single-plot configuration
        {"name": "plot_k22", "kind": "plot", "K": 22},
        # an ordinary plot of the batch mix, two scatter levels of odd widths,
        # with a match distance of its own
        {"name": "plot_k25_d", "kind": "plot", "K": 25, "dnum": 51},
        # the middle of the served range (22 to 29), working set beyond L2
        {"name": "plot_k28", "kind": "plot", "K": 28},
        # the headline plot
        {"name": "plot_k31", "kind": "plot", "K": 31},
        # Table 1 and Table 2 as two calls
        {"name": "split_k24", "kind": "split", "K": 24},
        # pairs across bucket edges
        {"name": "cross_k26", "kind": "cross", "K": 26},
        # a plot in quarters, Table 2 to pinned host memory
        {"name": "tiled_k26", "kind": "tiled", "K": 26, "window_bits": 2},
        # plot, then its Table 2 in hash order
        {"name": "sorted_k26", "kind": "sorted", "K": 26},
        # the head of the mixed batch: 20 plots, K 20 to 26
        {"name": "batch_20", "kind": "batch", "count": 20, "lo": 20, "hi": 26, "mix": 2026},
        # records and pairs checked outside a plot, counts that fill no tile
        {"name": "rows_20m", "kind": "rows", "count": 20000003, "pairs": 9000001},
    ]


def draw(rng):
    kind = rng.choice(["plot", "plot", "plot", "split", "cross", "tiled", "sorted", "batch", "rows"])
    if kind == "batch":
        lo = rng.randint(16, 22)
        return {"kind": kind, "count": rng.randint(2, 20), "lo": lo, "hi": lo + rng.randint(1, 4),
                "mix": rng.randrange(1 << 20)}
    if kind == "rows":
        return {"kind": kind, "count": int(2 ** rng.uniform(8, 26)) | 1, "pairs": int(2 ** rng.uniform(8, 25)) | 1}
    top = {"plot": 30, "split": 28, "cross": 28, "tiled": 27, "sorted": 28}[kind]
    case = {"kind": kind, "K": rng.randint(14 if kind == "tiled" else 12, top), "dnum": rng.randint(17, 79)}
    if kind == "tiled":
        case["window_bits"] = rng.randint(1, 3)
    return case


def _key(seed, i=0):
    return np.random.default_rng([seed, i]).bytes(32)


def _distance(case):
    """The match distance: dnum 64ths of the default 2^(64-K)."""
    return ((1 << 64) >> case["K"]) * case.get("dnum", 64) // 64


def _batch_ks(case):
    return [int(k) for k in np.random.default_rng(case["mix"]).integers(case["lo"], case["hi"] + 1, case["count"])]


class _Plot:
    """A plot and the buffers it was given.  Table 2's starts as zeros: what
    lies past the plot's pairs stays as it was."""

    def __init__(self, K, key, opts=None):
        self.handle = vx.vx_plot_create(K, key, opts)
        t1, t2, scratch = vx.vx_plot_required_bytes(K, opts)
        self.t1 = torch.empty(t1, dtype=torch.uint8, device="cuda")
        self.t2 = torch.zeros(t2, dtype=torch.uint8, device="cuda")
        self.scratch = torch.empty(scratch, dtype=torch.uint8, device="cuda")
        vx.vx_plot_bind(self.handle, self.t1.data_ptr(), self.t2.data_ptr(), self.scratch.data_ptr())
        self.n1 = 1 << K

    def sync(self):
        """Waits; the count of pairs, and both tables as the 32- and 64-bit
        words of their records."""
        vx.vx_sync(self.handle)
        n2 = vx.vx_table_info(self.handle, vx.VX_TABLE2)[1]
        return n2, self.t1[: 12 * self.n1].view(torch.int32), self.t2.view(torch.int64)

    def __del__(self):
        vx.vx_plot_destroy(self.handle)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "rows":
        n0 = int(np.random.default_rng([seed, 1]).integers(0, 2 ** 32 - case["count"]))
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        pairs = torch.randint(-(2 ** 31), 2 ** 31, (case["pairs"], 2), generator=g, device="cuda", dtype=torch.int32)
        return {"kind": kind, "key": _key(seed), "nonce0": n0, "count": case["count"], "pairs": pairs,
                "records": torch.empty((case["count"], 3), dtype=torch.int32, device="cuda"),
                "out": torch.empty((case["pairs"], 4), dtype=torch.int32, device="cuda")}
    if kind == "batch":
        return {"kind": kind, "plots": [_Plot(k, _key(seed, i)) for i, k in enumerate(_batch_ks(case))]}
    opts = {}
    if "dnum" in case:
        opts["match_distance"] = _distance(case)
    if kind == "cross":
        opts["match_scope"] = 1
    opts = vx.make_opts(**opts) if opts else None
    if kind == "tiled":
        bits = case["window_bits"]
        device, _, host = vx.vx_plot_tiled_bytes(case["K"], bits, opts)
        return {"kind": kind, "K": case["K"], "key": _key(seed), "bits": bits, "opts": opts,
                "t2": torch.zeros(host, dtype=torch.uint8, pin_memory=True),
                "work": torch.empty(device, dtype=torch.uint8, device="cuda")}
    return {"kind": kind, "plot": _Plot(case["K"], _key(seed), opts)}


def run(state):
    kind = state["kind"]
    if kind == "rows":
        vx.vx_hash_nonces(state["key"], state["nonce0"], state["count"], state["records"].data_ptr())
        vx.vx_pair_hash(state["key"], state["pairs"].data_ptr(), state["pairs"].shape[0], state["out"].data_ptr())
        return state["records"], state["out"]
    if kind == "batch":
        vx.vx_plot_batch([p.handle for p in state["plots"]])
        return [p.sync() for p in state["plots"]]
    if kind == "tiled":
        t2, space = state["t2"], state["work"]
        _, n1, n2 = vx.vx_plot_tiled(state["K"], state["key"], state["bits"], 0, 0, t2.data_ptr(), t2.numel(),
                                     state["opts"], d_work=space.data_ptr(), work_bytes=space.numel())
        return n1, n2, t2.view(torch.int64)
    plot = state["plot"]
    if kind == "split":
        vx.vx_table1(plot.handle)
        vx.vx_match(plot.handle)
    else:
        vx.vx_plot_run(plot.handle)
    if kind == "sorted":
        vx.vx_sync(plot.handle)
        need = vx.vx_sort_table2_work_bytes(plot.handle)
        space = torch.empty(need, dtype=torch.uint8, device="cuda")
        vx.vx_sort_table2(plot.handle, space.data_ptr(), need)
    return plot.sync()


def _expected_pairs(K, D, cross):
    n = 2.0 ** K
    if cross:
        return n * n / 2 * 2 * (D / 2.0 ** 64)
    u = min(1.0, D / 2.0 ** 40)
    lam = n / 2 ** 24
    return 2 ** 24 * lam * lam / 2 * (2 * u - u * u)


def work(case):
    kind = case["kind"]
    if kind == "rows":
        return {"bytes": 12 * case["count"] + 24 * case["pairs"], "flops": OPS_PER_HASH * (case["count"] + case["pairs"])}
    ks = _batch_ks(case) if kind == "batch" else [case["K"]]
    nbytes = ops = 0.0
    for K in ks:
        pairs = _expected_pairs(K, _distance(case) if kind != "batch" else (1 << 64) >> K, kind == "cross")
        nbytes += 32 + (0 if kind == "tiled" else 12 * 2.0 ** K) + 16 * pairs
        ops += OPS_PER_HASH * (2.0 ** K + pairs)
    return {"bytes": math.ceil(nbytes), "flops": math.ceil(ops)}


# ------------------------------------------------------------------- exact

_IV = (0x6A09E667, 0xBB67AE85, 0x3C6EF372, 0xA54FF53A)
_PERM = (2, 6, 3, 10, 7, 0, 4, 13, 1, 11, 12, 5, 9, 14, 15, 8)


def _blake3_words(key, words, block_len):
    """Output words 0 and 1 of keyed BLAKE3 of one short block per row."""
    n = words[0].shape[0]
    zero = np.zeros(n, np.uint32)
    m = list(words) + [zero] * (16 - len(words))
    v = [np.full(n, int(k), np.uint32) for k in np.frombuffer(key, "<u4")]
    v += [np.full(n, x, np.uint32) for x in (*_IV, 0, 0, block_len, 1 | 2 | 8 | 16)]

    def rot(x, r):
        return (x >> np.uint32(r)) | (x << np.uint32(32 - r))

    def g(a, b, c, d, x, y):
        v[a] = v[a] + v[b] + x
        v[d] = rot(v[d] ^ v[a], 16)
        v[c] = v[c] + v[d]
        v[b] = rot(v[b] ^ v[c], 12)
        v[a] = v[a] + v[b] + y
        v[d] = rot(v[d] ^ v[a], 8)
        v[c] = v[c] + v[d]
        v[b] = rot(v[b] ^ v[c], 7)

    for r in range(7):
        for i in range(4):
            g(i, 4 + i, 8 + i, 12 + i, m[2 * i], m[2 * i + 1])
        for i in range(4):
            g(i, 4 + (i + 1) % 4, 8 + (i + 2) % 4, 12 + (i + 3) % 4, m[8 + 2 * i], m[9 + 2 * i])
        m = [m[p] for p in _PERM]
    return v[0] ^ v[8], v[1] ^ v[9]


def _key64(h0, h1):
    return (h0.byteswap().astype(np.uint64) << np.uint64(32)) | h1.byteswap().astype(np.uint64)


def _exact_plot(K, key, D, words, cross=False, by_hash=False):
    """The count of pairs and both tables, Table 2 as `words` 64-bit words."""
    nonces = np.arange(1 << K, dtype=np.uint32)
    h0, h1 = _blake3_words(key, [nonces], 4)
    k = _key64(h0, h1)
    order = np.lexsort((nonces, k))
    nonces, h0, h1, k = nonces[order], h0[order], h1[order], k[order]
    t1 = np.stack([nonces, h0, h1], 1)
    at_i, at_j = [], []
    bucket = k >> np.uint64(40)
    for t in range(1, k.shape[0]):
        near = k[t:] - k[:-t] < np.uint64(D)
        if not cross:
            near &= bucket[t:] == bucket[:-t]
        i = np.nonzero(near)[0]
        if not i.size:
            break
        at_i.append(i)
        at_j.append(i + t)
    i, j = (np.concatenate(x) if x else np.zeros(0, np.int64) for x in (at_i, at_j))
    order = np.lexsort((j, i))
    a, b = nonces[i[order]], nonces[j[order]]
    g0, g1 = _blake3_words(key, [a, b], 8)
    t2 = np.stack([a, b, g0, g1], 1)
    if by_hash:
        t2 = t2[np.lexsort((b, a, _key64(g0, g1)))]
    whole = np.zeros(words, np.int64)
    whole[: 2 * t2.shape[0]] = np.ascontiguousarray(t2).reshape(-1).view(np.int64)
    return t2.shape[0], t1.reshape(-1).view(np.int32), whole


def exact(case, seed):
    kind = case["kind"]
    if kind == "rows":
        if max(case["count"], case["pairs"]) > 1 << 20:
            return None
        s = prepare(case, seed)
        nonces = np.arange(s["nonce0"], s["nonce0"] + case["count"], dtype=np.uint64).astype(np.uint32)
        records = np.stack([nonces, *_blake3_words(s["key"], [nonces], 4)], 1)
        p = s["pairs"].cpu().numpy().view(np.uint32)
        a, b = np.ascontiguousarray(p[:, 0]), np.ascontiguousarray(p[:, 1])
        return records.view(np.int32), np.stack([a, b, *_blake3_words(s["key"], [a, b], 8)], 1).view(np.int32)
    if (max(_batch_ks(case)) if kind == "batch" else case["K"]) > 18:
        return None
    s = prepare(case, seed)
    if kind == "batch":
        return [_exact_plot(K, _key(seed, i), (1 << 64) >> K, p.t2.numel() // 8)
                for i, (K, p) in enumerate(zip(_batch_ks(case), s["plots"]))]
    held = s["t2"] if kind == "tiled" else s["plot"].t2
    n2, t1, t2 = _exact_plot(case["K"], _key(seed), _distance(case), held.numel() // 8, kind == "cross", kind == "sorted")
    return (1 << case["K"], n2, t2) if kind == "tiled" else (n2, t1, t2)
