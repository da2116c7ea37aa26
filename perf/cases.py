"""The calls this library is measured by: what its users have it do, through
its public entry points, from the smallest sorts to the largest.

Every case is a dict of plain values; `kind` picks the entry point:

  sort     pgs_sort_copy on device buffers with a caller-kept workspace
  batch    a pgs_batch plan and its out-of-place sort (many instances, one call)
  host     pgs_sort_host on pinned host buffers, copies inside the call
  merge    pgs_merge_lists, the stable merge of sorted lists (the receiving step of the sharded sort)
  search   pgs_search on sorted keys, with the bucket of every query

Keys are drawn on the GPU from the distributions of the library's own
workloads (uniform, normal + lognormal, Zipf duplicates with signed zeros and
NaNs, exponential), the payload is the input index, and the outputs are
everything the call is asked to write: keys, payloads, bucket bounds, the cut
matrix and the splitters.
"""
import math

import numpy as np
import torch

from paper_1611_00463_gb300 import pgs

CHUNK = 1 << 26                 # keys drawn at a time (float64 temporaries stay small)
MAX_KEYS = 1 << 30


def listed():
    return [
        # A few thousand keys: the call itself (launches, latency) is what a user waits for.
        {"name": "tiny_u32", "kind": "sort", "n": 2000, "P": 4, "dtype": "u32", "dist": "uniform", "vals": True},
        # The small workload of the library's bench: one million uniform keys on 16 partitions.
        {"name": "small_u32", "kind": "sort", "n": 1 << 20, "P": 16, "dtype": "u32", "dist": "uniform", "vals": True},
        # Ordinary sizes, neither a power of two: duplicate-heavy floats, and wide keys without a
        # payload on a partition count that is no power of two.
        {"name": "mid_f32", "kind": "sort", "n": 16_777_259, "P": 64, "dtype": "f32", "dist": "zipf", "vals": True},
        {"name": "mid_u64_keys", "kind": "sort", "n": 20_000_003, "P": 100, "dtype": "u64", "dist": "normal_lognormal",
         "vals": False},
        # The three large workloads of the library's bench at their own sizes.
        {"name": "large_u64", "kind": "sort", "n": 1 << 28, "P": 128, "dtype": "u64", "dist": "normal_lognormal",
         "vals": True},
        {"name": "large_f32", "kind": "sort", "n": 1 << 29, "P": 256, "dtype": "f32", "dist": "zipf", "vals": True},
        {"name": "largest_u32", "kind": "sort", "n": 1 << 30, "P": 1024, "dtype": "u32", "dist": "exponential",
         "vals": True},
        # Learned splitters: the model is trained inside the call on the sort's own sample.
        {"name": "learned_u32", "kind": "sort", "n": 1 << 22, "P": 16, "dtype": "u32", "dist": "exponential",
         "vals": True, "splitters": "learned"},
        # Two thousand uneven instances (1K to 16M keys, lognormal sizes) in one call.
        {"name": "batch_u64", "kind": "batch", "instances": 2000, "lo": 1024, "hi": 1 << 24, "dtype": "u64",
         "vals": True},
        # Host buffers in and out, the size of an ordinary request.
        {"name": "host_u32", "kind": "host", "n": 4_194_319, "P": 32, "dtype": "u32", "dist": "uniform", "vals": True},
        # What one rank of a sharded sort does with the sixteen segments it received.
        {"name": "merge_u64", "kind": "merge", "n": 67_108_879, "lists": 16, "dtype": "u64", "dist": "normal_lognormal",
         "vals": True},
        # Lookups in sorted output.
        {"name": "search_u64", "kind": "search", "n": 1 << 26, "queries": 1 << 24, "P": 64, "dtype": "u64",
         "dist": "normal_lognormal"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sort", "sort", "sort", "sort", "batch", "host", "merge", "search"])
    dtype = rng.choice(["u32", "u64", "f32"])
    dist = "zipf" if dtype == "f32" else rng.choice(["uniform", "exponential"] +
                                                    (["normal_lognormal", "zipf"] if dtype == "u64" else []))
    if kind == "sort":
        n = _log_int(rng, 1000, 1 << 28)
        c = {"kind": kind, "n": n, "P": _log_int(rng, 1, min(1024, max(2, n // 500))), "dtype": dtype, "dist": dist,
             "vals": rng.random() < 0.8}
        if rng.random() < 0.25:
            c["guaranteed"] = True
        return c
    if kind == "batch":
        return {"kind": kind, "instances": _log_int(rng, 10, 2000), "lo": 64, "hi": _log_int(rng, 1 << 12, 1 << 20),
                "dtype": dtype, "vals": rng.random() < 0.8}
    if kind == "host":
        return {"kind": kind, "n": _log_int(rng, 1 << 12, 1 << 24), "P": _log_int(rng, 2, 64), "dtype": dtype,
                "dist": dist, "vals": rng.random() < 0.8}
    if kind == "merge":
        return {"kind": kind, "n": _log_int(rng, 1 << 12, 1 << 26), "lists": _log_int(rng, 2, 64), "dtype": dtype,
                "dist": dist, "vals": rng.random() < 0.8}
    return {"kind": kind, "n": _log_int(rng, 1 << 12, 1 << 26), "queries": _log_int(rng, 1 << 10, 1 << 24),
            "P": _log_int(rng, 2, 64), "dtype": dtype, "dist": dist}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _u64_from_double(x):
    """Rounds and clamps float64 into uint64, as int64 bits (values from 2^64 saturate)."""
    x = x.round().clamp_(min=0.0)
    hi = x >= 2.0 ** 63
    low = torch.where(hi, x - 2.0 ** 63, x).clamp_(max=2.0 ** 63 - 1024)
    bits = low.to(torch.int64)
    bits = torch.where(hi, bits ^ torch.iinfo(torch.int64).min, bits)
    return torch.where(x >= 2.0 ** 64, torch.full_like(bits, -1), bits)


def _zipf_table(dtype, g, distinct=1000):
    if dtype == "f32":
        t = torch.randn(4 * distinct, generator=g, device="cuda", dtype=torch.float32) * 1000.0
        t = t[t != 0]
        u = torch.unique(t)
        return u[torch.randperm(u.numel(), generator=g, device="cuda")[:distinct]].view(torch.int32)
    hi = torch.randint(0, 1 << 32, (distinct,), generator=g, device="cuda", dtype=torch.int64)
    lo = torch.randint(0, 1 << 32, (distinct,), generator=g, device="cuda", dtype=torch.int64)
    t = (hi << 32) | lo
    return t if dtype == "u64" else t.to(torch.int32)


def _zipf(out, dtype, g, s=1.1):
    table = _zipf_table(dtype, g)
    w = torch.arange(1, table.numel() + 1, device="cuda", dtype=torch.float64) ** (-s)
    cdf = torch.cumsum(w, 0)
    cdf /= cdf[-1].clone()
    special = torch.from_numpy(np.array([0, 0x80000000, 0x7FC00000, 0xFFC00000], dtype=np.uint32).view(np.int32)).cuda()
    for lo in range(0, out.numel(), CHUNK):
        m = min(CHUNK, out.numel() - lo)
        r = torch.searchsorted(cdf, torch.rand(m, generator=g, device="cuda", dtype=torch.float64), right=True)
        k = table[r.clamp_(max=table.numel() - 1)]
        if dtype == "f32":          # one key in twenty is a signed zero or a NaN
            pick = torch.randint(0, 80, (m,), generator=g, device="cuda")
            k = torch.where(pick < 4, special[pick.clamp(max=3)], k)
        out[lo:lo + m] = k


def _keys(n, dtype, dist, seed):
    """n keys as the bits the library takes (int64 for u64, else int32), on the GPU."""
    g = _gen(seed)
    out = torch.empty(n, dtype=pgs.KEY_TORCH[dtype], device="cuda")
    if dist == "zipf":
        _zipf(out, dtype, g)
        return out
    for lo in range(0, n, CHUNK):
        m = min(CHUNK, n - lo)
        part = out[lo:lo + m]
        if dist == "uniform":
            info = torch.iinfo(part.dtype)
            part.random_(info.min, info.max, generator=g)
        elif dist == "exponential":
            scale = 2.0 ** 40 if dtype == "u64" else 1e8
            x = torch.empty(m, device="cuda", dtype=torch.float64).exponential_(1.0 / scale, generator=g)
            if dtype == "u64":
                part.copy_(_u64_from_double(x))
            else:
                part.copy_(x.round_().clamp_(max=float(0xFFFFFFFF)).to(torch.int64).to(torch.int32))
        elif dist == "normal_lognormal":
            z = torch.randn(m, generator=g, device="cuda", dtype=torch.float64)
            heads = torch.rand(m, generator=g, device="cuda") < 0.5
            x = torch.where(heads, 2.0 ** 63 + 2.0 ** 60 * z, torch.exp(40.0 + 2.0 * z))
            part.copy_(_u64_from_double(x))
        else:
            raise ValueError(dist)
    return out


def _index(n):
    return torch.arange(n, dtype=torch.int32, device="cuda")


def _batch_sizes(case, seed):
    """Lognormal sizes between lo and hi (the median of the library's batched
    workload, or the middle of a smaller range)."""
    mid = min(math.exp(10.65), math.sqrt(case["lo"] * case["hi"]))
    sigma = 1.8 if case["hi"] > 1 << 20 else 1.0
    x = np.random.default_rng(case["instances"]).lognormal(math.log(mid), sigma, case["instances"])
    return np.clip(np.rint(x), case["lo"], case["hi"]).astype(np.int64)


def _order(keys, dtype):
    """Signed integers in the library's key order (totalOrder for floats)."""
    if dtype == "f32":
        return torch.where(keys < 0, keys ^ 0x7FFFFFFF, keys)
    return keys ^ torch.iinfo(keys.dtype).min


def _sorted_keys(keys, dtype):
    o = torch.sort(_order(keys, dtype))[0]
    return torch.where(o < 0, o ^ 0x7FFFFFFF, o) if dtype == "f32" else o ^ torch.iinfo(o.dtype).min


def prepare(case, seed):
    kind, dtype = case["kind"], case["dtype"]
    with_vals = case.get("vals", False)
    st = {"case": case}
    if kind == "batch":
        sizes = _batch_sizes(case, seed)
        off = np.zeros(len(sizes) + 1, dtype=np.uint64)
        off[1:] = np.cumsum(sizes)
        n = int(off[-1])
        kinds = ["zipf"] if dtype == "f32" else ["uniform", "exponential", "zipf"]
        kin = torch.empty(n, dtype=pgs.KEY_TORCH[dtype], device="cuda")
        groups = [int(off[len(sizes) * i // len(kinds)]) for i in range(len(kinds))] + [n]
        for i, d in enumerate(kinds):   # neighbouring instances share a distribution
            kin[groups[i]:groups[i + 1]] = _keys(groups[i + 1] - groups[i], dtype, d, seed * 7 + i)
        st["kin"], st["vin"] = kin, _index(n) if with_vals else None
        st["kout"], st["vout"] = torch.empty_like(kin), torch.empty_like(st["vin"]) if with_vals else None
        st["batch"] = pgs.Batch(off, None, dtype=dtype, with_vals=with_vals)
        st["cfg"] = st["batch"].config()
        return st
    n = case["n"]
    keys = _keys(n, dtype, case["dist"], seed)
    if kind in ("sort", "host"):
        P = case["P"]
        opts = {"splitters": case.get("splitters", "sampled"), "guaranteed": bool(case.get("guaranteed", False))}
        Pe = max(1, min(P, n))
        out = {"bounds": torch.zeros(Pe + 1, dtype=torch.int64, device="cuda"),
               "cuts": torch.zeros(Pe * (Pe + 1), dtype=torch.int64, device="cuda"),
               "splitters": torch.zeros(max(1, Pe - 1), dtype=keys.dtype, device="cuda")}
        st["model"] = torch.zeros(pgs.MLP_WORDS, dtype=torch.float32, device="cuda") \
            if opts["splitters"] == "learned" else None
        vals = _index(n) if with_vals else None
        base = pgs.make_config(dtype=dtype, **opts)
        if kind == "sort":
            st["kin"], st["vin"] = keys, vals
            st["kout"], st["vout"] = torch.empty_like(keys), torch.empty_like(vals) if with_vals else None
            ws = pgs.workspace(n, P, base)
        else:
            st["kin"] = keys.cpu().pin_memory()
            st["vin"] = vals.cpu().pin_memory() if with_vals else None
            st["kout"] = torch.empty(n, dtype=keys.dtype, pin_memory=True)
            st["vout"] = torch.empty(n, dtype=torch.int32, pin_memory=True) if with_vals else None
            ws = torch.empty(pgs.pgs_host_workspace_bytes(n, P, base), dtype=torch.uint8, device="cuda")
        st["cfg"] = pgs.make_config(dtype=dtype, workspace=ws, bucket_bounds=out["bounds"], cuts=out["cuts"],
                                    splitters_out=out["splitters"], model_out=st["model"], **opts)
        st["out"] = out
    elif kind == "merge":
        k = case["lists"]
        cut = np.sort(np.random.default_rng(seed).integers(0, n + 1, size=k - 1))
        st["off"] = np.concatenate([[0], cut, [n]]).astype(np.uint64)
        for j in range(k):
            a, b = int(st["off"][j]), int(st["off"][j + 1])
            if b > a:
                keys[a:b] = _sorted_keys(keys[a:b], dtype)
        st["kin"], st["vin"] = keys, _index(n) if with_vals else None
        st["kout"], st["vout"] = torch.empty_like(keys), torch.empty_like(st["vin"]) if with_vals else None
        base = pgs.make_config(dtype=dtype)
        st["ws"] = torch.empty(pgs.pgs_merge_workspace_bytes(n, k, base), dtype=torch.uint8, device="cuda")
        st["cfg"] = pgs.make_config(dtype=dtype, workspace=st["ws"])
    else:
        P = case["P"]
        st["kin"] = _sorted_keys(keys, dtype)
        st["queries"] = _keys(case["queries"], dtype, case["dist"], seed + 1)
        st["bounds"] = torch.tensor([b * n // P for b in range(P + 1)], dtype=torch.int64, device="cuda")
        m = case["queries"]
        st["pos"] = torch.empty(m, dtype=torch.int64, device="cuda")
        st["bucket"] = torch.empty(m, dtype=torch.int32, device="cuda")
        st["ws"] = torch.empty(max(256, pgs.pgs_search_workspace_bytes(n, dtype)), dtype=torch.uint8, device="cuda")
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "search":
        pgs.pgs_search(st["kin"], st["queries"], st["pos"], "left", case["dtype"], st["bounds"], st["bucket"], st["ws"])
        return {"pos": st["pos"], "bucket": st["bucket"]}
    if kind == "sort":
        pgs.pgs_sort_copy(st["kin"], st["vin"], st["kout"], st["vout"], case["P"], st["cfg"])
    elif kind == "host":
        pgs.pgs_sort_host(st["kin"], st["vin"], st["kout"], st["vout"], case["P"], st["cfg"])
    elif kind == "batch":
        st["batch"].sort_copy(st["kin"], st["vin"], st["kout"], st["vout"], cfg=st["cfg"])
    else:
        pgs.pgs_merge_lists(st["kin"], st["vin"], st["off"], st["kout"], st["vout"], st["cfg"])
    res = {"keys": st["kout"], "vals": st["vout"]}
    if kind in ("sort", "host"):
        res.update(st["out"])
        if st["model"] is not None:
            res["model"] = st["model"]
    return res


def work(case):
    w = 8 if case["dtype"] == "u64" else 4
    if case["kind"] == "search":
        m = case["queries"]
        # every query, its position and its bucket, and each key of the searched array once
        return {"bytes": m * (w + 8 + 4) + case["n"] * w, "flops": 0}
    n = int(_batch_sizes(case, 0).sum()) if case["kind"] == "batch" else case["n"]
    pair = w + (4 if case.get("vals", False) else 0)
    return {"bytes": 2 * n * pair, "flops": 0}


def exact(case, seed):
    """Every output but the learned model's weights is a whole number or a key's
    bits, compared as such; the trained weights have no closed 64-bit form."""
    return None
