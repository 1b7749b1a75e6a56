"""The sorts by value buckets against the oracle, for every key and payload
width: evenly spread keys at the sizes where the route changes (one block, one
or two splits, a single launch), with groups of equal keys that crowd one bin of
a bucket or of the first and last one (ordered digit by digit), and with more
equal keys than a bucket takes (the radix passes take over)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

KIND = {"u32": 0, "i32": 1, "f32": 2, "u64": 0, "i64": 1, "f64": 2}


def _keys(bits, n, data):
    w = synth.splitmix64(n, n)
    if bits == 32:
        w = (w >> np.uint64(11)).astype(np.uint32)
    top = w.dtype.type(~w.dtype.type(0))
    if data == "overfull":
        w[5::7][:5000] = w[3]
    if data == "crowded":
        at = 0
        for g, value in ((30, w[1]), (33, w[2]), (64, w[3]), (400, w[4]), (40, w.dtype.type(0)), (40, top)):
            w[at + np.arange(g) * 19] = value  # spread over several tiles and warps
            at += g * 19
    return w


SIZES = {
    ("u32", 0): [8192, 16384, 16385, 300_001, 3_000_001], ("f32", 0): [3_000_001], ("i32", 4): [3_000_001],
    ("u32", 4): [16384, 16385, 300_001, 3_000_001],
    ("u32", 8): [8192, 8193, 256 * 1365, 256 * 1365 + 1, 3_000_001],
    ("u64", 0): [8192, 8193, 256 * 2048, 256 * 2048 + 1, 3_000_001], ("f64", 0): [3_000_001],
    ("u64", 4): [8192, 8193, 256 * 1365, 256 * 1365 + 1, 32768 * 1365 + 1], ("i64", 8): [8192, 8193, 256 * 1365, 3_000_001],
}


@pytest.mark.parametrize("data", ["even", "crowded", "overfull"])
@pytest.mark.parametrize("kind,vb,n", [(k, v, n) for (k, v), ns in SIZES.items() for n in ns])
def test_value_buckets(kind, vb, n, data):
    import paper_cs_0004013_gb300 as rs
    import torch
    if n < 5000 * 7 + 5 and data == "overfull":
        pytest.skip("fewer keys than the group")
    if n > 1 << 22 and data != "even":
        pytest.skip("the sizes above show it")
    wide = kind.endswith("64")
    w = _keys(64 if wide else 32, n, data if n > 16384 else "even")
    d = torch.from_numpy(w.view(np.int64 if wide else np.int32).copy()).cuda()
    vals = np.arange(n, dtype=np.uint32)
    plan = {"key_kind": KIND[kind]}
    if vb == 0:
        out = (rs.sort64 if wide else rs.sort)(d, plan=plan)[0]
    else:
        v = torch.from_numpy(vals.astype(np.int64 if vb == 8 else np.int32)).cuda()
        out, vo, _ = (rs.sort64_pairs if wide else rs.sort_pairs64 if vb == 8 else rs.sort_pairs)(d, v, plan=plan)
        vo = vo.cpu().numpy()
    torch.cuda.synchronize()
    rs.rs_check_device_error()
    wk, wv = oracle.sort_pairs(w, vals, kind) if vb else (oracle.sort_keys(w, kind), None)
    assert np.array_equal(out.cpu().numpy().view(w.dtype), wk)
    if vb:
        assert np.array_equal(vo.astype(np.uint32), wv)
