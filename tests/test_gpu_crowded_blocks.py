"""One-block sorts of values that crowd into few bins, of every key and payload
width, against the oracle: few distinct values, clusters narrower than a bin,
densities that the second set of bins flattens, and crowds that only some bins
have (which the first keys of the threads do not show)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

KIND = {"u32": 0, "f32": 2, "u64": 0, "i64": 1}
DATA = ["eight", "mean20", "consecutive", "clusters", "log", "normal", "half", "hidden", "edges", "last_differs"]


def _words(bits, n, data):
    r = np.random.default_rng(n + bits)
    even = synth.splitmix64(n + bits, n) >> np.uint64(64 - bits)
    top = (1 << bits) - 1
    if data == "eight":
        w = even[r.integers(0, 8, n)]
    elif data == "mean20":  # about 20 keys per value
        w = even[r.integers(0, max(n // 20, 1), n)]
    elif data == "consecutive":  # a bin per value, 300 keys in each
        w = np.uint64(1 << 20) + r.integers(0, max(n // 300, 1), n).astype(np.uint64)
    elif data == "clusters":
        w = even[r.integers(0, 8, n)] // np.uint64(2) + r.integers(0, 4096, n).astype(np.uint64)
    elif data == "log":
        w = np.exp(r.uniform(0, 0.69 * bits, n)).astype(np.uint64)
    elif data == "normal":
        w = r.standard_normal(n).astype(np.float32 if bits == 32 else np.float64)
        return w.view(np.uint32 if bits == 32 else np.uint64)
    elif data == "half":
        w = np.where(r.random(n) < 0.5, even[0], even)
    elif data == "hidden":  # forty equal keys behind the first thousand
        w = even.copy()
        w[-40:] = even[1]
    elif data == "edges":
        w = np.where(r.random(n) < 0.1, np.uint64(0), np.where(r.random(n) < 0.1, np.uint64(top), even))
    else:  # equal but for one key at the end
        w = np.full(n, 77, np.uint64)
        w[-1] = top
    return w.astype(np.uint32 if bits == 32 else np.uint64)


CASES = ([(k, vb, n) for k, vb in (("u32", 0), ("u32", 4), ("f32", 4)) for n in (40, 1024, 1025, 4096, 16384)] +
         [(k, vb, n) for k, vb in (("u32", 8), ("u64", 0), ("u64", 4), ("i64", 8)) for n in (40, 1024, 1025, 8192)])


@pytest.mark.parametrize("data", DATA)
@pytest.mark.parametrize("kind,vb,n", CASES)
def test_crowded_block(kind, vb, n, data):
    import paper_cs_0004013_gb300 as rs
    import torch
    wide = kind.endswith("64")
    w = _words(64 if wide else 32, n, data)
    d = torch.from_numpy(w.view(np.int64 if wide else np.int32).copy()).cuda()
    vals = np.arange(n, dtype=np.uint32)
    plan = {"key_kind": KIND[kind]}
    if vb == 0:
        out = (rs.sort64 if wide else rs.sort)(d, plan=plan)[0]
    else:
        v = torch.from_numpy(vals.astype(np.int64 if vb == 8 else np.int32)).cuda()
        out, vo, _ = (rs.sort64_pairs if wide else rs.sort_pairs64 if vb == 8 else rs.sort_pairs)(d, v, plan=plan)
    torch.cuda.synchronize()
    rs.rs_check_device_error()
    wk, wv = oracle.sort_pairs(w, vals, kind) if vb else (oracle.sort_keys(w, kind), None)
    assert np.array_equal(out.cpu().numpy().view(w.dtype), wk)
    if vb:
        assert np.array_equal(vo.cpu().numpy().astype(np.uint32), wv)
