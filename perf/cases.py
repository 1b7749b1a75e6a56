"""Work that users of the sort have it do, as cases that can be timed.

Each case is one call of a public entry point on arrays that are already
where the call wants them (device memory; pinned host memory for the host
entry).  The sizes run from the smallest calls, where launches and latency
count, to the 2^26 keys of the benchmark's headline, with odd sizes between;
the distributions are those of the repository's synthetic workloads, drawn
here on the GPU so that inputs are quick to make.
"""
import math

import numpy as np
import torch

import paper_cs_0004013_gb300 as rs

PARTS = 64  # output partitions, the paper's contract

# entry -> (bytes of a key, bytes of a value)
ENTRIES = {
    "sort": (4, 0),            # rs.sort: 32-bit keys
    "sort_pairs": (4, 4),      # rs.sort_pairs: 32-bit keys, 32-bit values, stable
    "sort_pairs64": (4, 8),    # rs.sort_pairs64: 32-bit keys, 64-bit values
    "sort64": (8, 0),          # rs.sort64: 64-bit keys
    "sort64_pairs": (8, 4),    # rs.sort64_pairs: 64-bit keys, 32-bit values
    "sort64_pairs64": (8, 8),  # rs.sort64_pairs: 64-bit keys, 64-bit values
    "segmented": (4, 0),       # rs.sort_segmented: many arrays in one call
    "segmented_pairs": (4, 4),
    "merge": (4, 0),           # rs.merge: two sorted runs
    "merge_pairs": (4, 4),
    "host": (4, 0),            # rs_sort_u32_host: pinned host arrays in and out
    "host_pairs": (4, 4),
}
KINDS = {"u32": rs.RS_KEY_U32, "i32": rs.RS_KEY_I32, "f32": rs.RS_KEY_F32}


def listed():
    return [
        # a short list sorted inside a larger step: launches and host work are all there is
        {"name": "keys_1000", "entry": "sort", "n": 1000, "kind": "u32", "dist": "uniform"},
        # the paper's first data set at the benchmark's small size: random keys, one million of them
        {"name": "keys_2p20", "entry": "sort", "n": 1 << 20, "kind": "u32", "dist": "uniform"},
        # an index sort of odd size with some clustering: values are input positions, order of equal keys kept
        {"name": "pairs_300001", "entry": "sort_pairs", "n": 300001, "kind": "u32", "dist": "gauss_mix"},
        # scores: binary32 keys of both signs, normally distributed, between the small and the large plans
        {"name": "floats_4m", "entry": "sort", "n": 4000003, "kind": "f32", "dist": "normal"},
        # the benchmark's headline: the contest's 64 million random keys
        {"name": "keys_2p26", "entry": "sort", "n": 1 << 26, "kind": "u32", "dist": "uniform"},
        # the same with a payload, the largest memory traffic of the 32-bit sorts
        {"name": "pairs_2p26", "entry": "sort_pairs", "n": 1 << 26, "kind": "u32", "dist": "uniform"},
        # the paper's fifth data set: clustered values, many duplicates, an odd size
        {"name": "clusters_2p24", "entry": "sort", "n": (1 << 24) + 1, "kind": "u32", "dist": "tight_clusters"},
        # hashes or ids: 64-bit keys over all words
        {"name": "keys64_2p24", "entry": "sort64", "n": 1 << 24, "kind": "u32", "dist": "uniform64"},
        # records by a 64-bit key with a pointer-sized value
        {"name": "records64_5m", "entry": "sort64_pairs64", "n": 5000011, "kind": "u32", "dist": "uniform64"},
        # the batched workload: many key+payload arrays of 2^10 to 2^20 keys sorted in one call
        {"name": "segmented_pairs", "entry": "segmented_pairs", "n": 1 << 25, "segs": 220, "kind": "u32",
         "dist": "uniform"},
        # two sorted runs joined, one shorter and of odd length
        {"name": "merge_21m", "entry": "merge", "n": (1 << 24) + 5000011, "left": 1 << 24, "kind": "u32",
         "dist": "uniform"},
        # a served request: pinned host keys in, sorted host keys out, copies included
        {"name": "host_2p24", "entry": "host", "n": 1 << 24, "kind": "u32", "dist": "uniform"},
    ]


def _log_size(rng, lo, hi):
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    """One more case: an entry point, a size over its range (by its logarithm) and a distribution of its keys."""
    entry = rng.choice(["sort", "sort", "sort_pairs", "sort_pairs", "sort_pairs64", "sort64", "sort64_pairs",
                        "sort64_pairs64", "segmented", "segmented_pairs", "merge", "merge_pairs", "host",
                        "host_pairs"])
    case = {"entry": entry, "kind": "u32"}
    if entry in ("sort", "sort_pairs"):
        case["n"] = _log_size(rng, 1000, 1 << 26)
        case["dist"] = rng.choice(["uniform", "uniform", "few_distinct", "gauss_mix", "tight_clusters", "normal",
                                   "signed"])
        case["kind"] = {"normal": "f32", "signed": "i32"}.get(case["dist"], "u32")
    elif entry == "sort_pairs64":
        case["n"] = _log_size(rng, 1000, 1 << 24)
        case["dist"] = rng.choice(["uniform", "gauss_mix"])
    elif entry in ("sort64", "sort64_pairs", "sort64_pairs64"):
        case["n"] = _log_size(rng, 1000, 1 << 24)
        case["dist"] = rng.choice(["uniform64", "uniform64", "stamps64"])
    elif entry in ("segmented", "segmented_pairs"):
        case["n"] = _log_size(rng, 1 << 20, 1 << 25)
        case["segs"] = _log_size(rng, 16, 4096)
        case["dist"] = rng.choice(["uniform", "gauss_mix"])
    elif entry in ("merge", "merge_pairs"):
        case["n"] = _log_size(rng, 2000, 1 << 25)
        case["left"] = rng.randint(case["n"] // 8, case["n"] // 2)
        case["dist"] = "uniform"
    else:
        case["n"] = _log_size(rng, 1 << 16, 1 << 24)
        case["dist"] = rng.choice(["uniform", "gauss_mix"])
    return case


def _sizes(case):
    """Segment lengths of a batch, by the case alone: log-uniform between 2^10 and 2^20 as in the repository's
    batched workload, scaled to add up to n."""
    r = np.random.default_rng(case["segs"])
    w = np.exp(r.uniform(math.log(1 << 10), math.log(1 << 20), case["segs"]))
    cut = np.floor(np.concatenate([[0.0], np.cumsum(w)]) * (case["n"] / w.sum()))
    cut[-1] = case["n"]
    return cut.astype(np.uint64)


def _keys(dist, n, g):
    """n keys on the GPU; unsigned ones as int32 / int64 storage of values below 2^31 / of any 64-bit word."""
    def below(bound, m=n):
        return torch.randint(0, bound, (m,), generator=g, device="cuda", dtype=torch.int64)

    if dist == "uniform":
        return below(1 << 31).to(torch.int32)
    if dist == "signed":
        return (below(1 << 32) - (1 << 31)).to(torch.int32)
    if dist == "normal":
        return torch.randn(n, generator=g, device="cuda", dtype=torch.float32)
    if dist == "few_distinct":  # 65,536 distinct values
        return below(1 << 31, 65536).to(torch.int32)[below(65536)]
    if dist == "tight_clusters":  # 8 clusters, 4,096 wide
        return (below((1 << 31) - 4096, 8)[below(8)] + below(4096)).to(torch.int32)
    if dist == "gauss_mix":  # 30 % in 16 clusters of sigma 2^20, the rest uniform
        u = below(1 << 31)
        c = below(1 << 31, 16)[below(16)].to(torch.float64)
        c = torch.round(c + float(1 << 20) * torch.randn(n, generator=g, device="cuda", dtype=torch.float64))
        c = c.clamp(0, (1 << 31) - 1).to(torch.int64)
        pick = torch.rand(n, generator=g, device="cuda") < 0.3
        return torch.where(pick, c, u).to(torch.int32)
    if dist == "uniform64":
        return (below(1 << 32) << 32) | below(1 << 32)
    if dist == "stamps64":  # microseconds within a day, late and early ones mixed
        return 1_600_000_000_000_000 + below(86_400_000_000)
    raise ValueError(dist)


def _values(n, nbytes, g):
    """Positions (32-bit values) or pointer-sized words."""
    if nbytes == 4:
        return torch.arange(n, device="cuda", dtype=torch.int32)
    return torch.randint(0, 1 << 62, (n,), generator=g, device="cuda", dtype=torch.int64)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    n, entry = case["n"], case["entry"]
    kb, vb = ENTRIES[entry]
    keys = _keys(case["dist"], n, g)
    vals = _values(n, vb, g) if vb else None
    s = {"entry": entry, "keys": keys, "vals": vals,
         "plan": None if case["kind"] == "u32" else {"key_kind": KINDS[case["kind"]]}}
    if entry.startswith("segmented"):
        s["offsets"] = _sizes(case)
    elif entry.startswith("merge"):
        left = case["left"]
        for name, part in (("a", slice(0, left)), ("b", slice(left, n))):
            s[name] = torch.sort(keys[part]).values
            s["v" + name] = None if vals is None else vals[part].clone()
    elif entry.startswith("host"):  # pinned arrays and the device scratch that a server keeps
        for name, t in (("keys", keys), ("vals", vals)):
            s[name] = None if t is None else t.cpu().pin_memory()
            s["out_" + name] = None if t is None else torch.empty_like(s[name], pin_memory=True)
        need = rs.rs_sort_u32_host(None, s["vals"], None, s["out_vals"], n, PARTS)
        s["temp"] = torch.empty(need, dtype=torch.uint8, device="cuda")
    return s


def run(s):
    entry, keys, vals, plan = s["entry"], s["keys"], s["vals"], s["plan"]
    if entry == "sort":
        return rs.sort(keys, PARTS, plan)
    if entry == "sort_pairs":
        return rs.sort_pairs(keys, vals, PARTS, plan)
    if entry == "sort_pairs64":
        return rs.sort_pairs64(keys, vals, PARTS, plan)
    if entry == "sort64":
        return rs.sort64(keys, PARTS, plan)
    if entry in ("sort64_pairs", "sort64_pairs64"):
        return rs.sort64_pairs(keys, vals, PARTS, plan)
    if entry.startswith("segmented"):
        return rs.sort_segmented(keys, vals, s["offsets"], PARTS, plan)
    if entry.startswith("merge"):
        return rs.merge(s["a"], s["b"], s["va"], s["vb"], PARTS, plan)
    offs = rs.rs_sort_u32_host(keys, vals, s["out_keys"], s["out_vals"], keys.numel(), PARTS, plan, s["temp"])
    return s["out_keys"], s["out_vals"], offs


def work(case):
    """Every key and value read once and written once; a sort has no floating-point work to speak of."""
    return {"bytes": 2 * case["n"] * sum(ENTRIES[case["entry"]]), "flops": 0}


def _offsets(n):
    q, r = divmod(n, PARTS)
    p = np.arange(PARTS + 1)
    return (p * q + np.minimum(p, r)).astype(np.uint64)


def _order(keys):
    """Stable ascending order of keys; 64-bit words as unsigned."""
    k = keys ^ torch.tensor(-(1 << 63), device=keys.device) if keys.dtype == torch.int64 else keys
    return torch.sort(k, stable=True).indices


def exact(case, seed):
    s = prepare(case, seed)
    entry, keys, vals, n = case["entry"], s["keys"], s["vals"], case["n"]
    if entry.startswith("merge"):
        keys = torch.cat([s["a"], s["b"]])
        vals = None if vals is None else torch.cat([s["va"], s["vb"]])
    if entry.startswith("segmented"):
        cut = s["offsets"].astype(np.int64)
        seg = torch.repeat_interleave(torch.arange(case["segs"], device="cuda"), torch.from_numpy(np.diff(cut)).cuda())
        order = torch.sort((seg << 32) | keys.to(torch.int64), stable=True).indices
        offs = torch.from_numpy(np.concatenate([a + _offsets(b - a).astype(np.int64) for a, b in zip(cut, cut[1:])]))
        return keys[order], None if vals is None else vals[order], offs
    order = _order(keys)
    out = keys[order]
    out = out.to(torch.float64) if out.is_floating_point() else out
    v = None if vals is None else vals[order]
    if entry in ("sort", "sort64"):
        return out, _offsets(n)
    return out, v, _offsets(n)
