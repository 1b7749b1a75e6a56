"""Sorts of repeated values around the limits that the sample sets for value
buckets, and of pairs around the size from which they are offered, against the
oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,vb,n", [(32, 0, 20_000), (32, 0, 1 << 20), (32, 4, 50_000), (32, 4, 1 << 20), (32, 8, 50_000),
                                       (64, 0, 65_536), (64, 0, 65_537), (64, 4, 300_001), (64, 8, 65_536),
                                       (32, 4, (1 << 22) - 1), (32, 4, 1 << 22)])
@pytest.mark.parametrize("per_value", [1, 5, 9, 17, 50])
def test_repeats(bits, vb, n, per_value):
    import paper_cs_0004013_gb300 as rs
    import torch
    if n > 1 << 21 and per_value > 5:
        pytest.skip("smaller sizes show it")
    words = synth.splitmix64(n + per_value, n)
    pick = (synth.splitmix64(3, n) % np.uint64(max(n // per_value, 1))).astype(np.int64)
    w = (words[pick] if per_value > 1 else words) >> np.uint64(64 - bits)
    w = w.astype(np.uint32 if bits == 32 else np.uint64)
    d = torch.from_numpy(w.view(np.int32 if bits == 32 else np.int64).copy()).cuda()
    vals = np.arange(n, dtype=np.uint32)
    if vb == 0:
        out = (rs.sort if bits == 32 else rs.sort64)(d)[0]
    else:
        v = torch.from_numpy(vals.astype(np.int64 if vb == 8 else np.int32)).cuda()
        out, vo, _ = (rs.sort64_pairs if bits == 64 else rs.sort_pairs64 if vb == 8 else rs.sort_pairs)(d, v)
    torch.cuda.synchronize()
    rs.rs_check_device_error()
    wk, wv = oracle.sort_pairs(w, vals, "u32" if bits == 32 else "u64")
    assert np.array_equal(out.cpu().numpy().view(w.dtype), wk)
    if vb:
        assert np.array_equal(vo.cpu().numpy().astype(np.uint32), wv)
