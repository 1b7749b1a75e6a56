"""Merges around the sizes at which the default tile changes, and the largest
tile at its edges, against the oracle."""
import numpy as np
import pytest

import oracle
import synth
from tests._gpu import to_dev, to_host_u32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pairs", [False, True])
@pytest.mark.parametrize("n,left,tile", [(n + d, n // 3, 0) for n in (1 << 20, 1 << 22, 1 << 24) for d in (0, 1)] +
                         [(2816, 1, 0), (2817, 2000, 0), (5888, 5, 3), (5889, 5888, 3), (2 * 5888 + 5, 7000, 3)])
def test_merge_sizes(n, left, tile, pairs):
    import paper_cs_0004013_gb300 as rs
    import torch
    w = synth.splitmix64(n, n).astype(np.uint32) >> np.uint32(8)  # some equal keys
    a, b = np.sort(w[:left]), np.sort(w[left:])
    va, vb = np.arange(left, dtype=np.uint32), np.arange(left, n, dtype=np.uint32)
    out, vout, offs = rs.merge(to_dev(a), to_dev(b), to_dev(va) if pairs else None, to_dev(vb) if pairs else None,
                               plan={"tile": tile})
    torch.cuda.synchronize()
    rs.rs_check_device_error()
    wk, wv = oracle.merge(a, b, va, vb)
    assert np.array_equal(to_host_u32(out), wk)
    assert np.array_equal(offs, oracle.partition_offsets(n, 64))
    if pairs:
        assert np.array_equal(to_host_u32(vout), wv)
