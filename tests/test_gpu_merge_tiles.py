"""Merge tiles at their edges against the oracle: slices that start anywhere in
a 16-byte unit, runs shorter than one, tiles and threads that are not full, the
largest key, and each way of searching the tile boundaries (by their number)."""
import numpy as np
import pytest

import oracle
import synth
from tests._gpu import to_dev, to_host_u32

pytestmark = pytest.mark.gpu

TILE = 5888  # outputs per default tile


def _run(seed, n, kind, top):
    w = synth.splitmix64(seed, (n + 1) // 2).view(np.uint32)[:n].copy()
    w[: n // 3] |= np.uint32(top)  # many of the largest key with top = 0xffffffff
    return oracle.sort_keys(w, kind)


@pytest.mark.parametrize("kind", ["u32", "f32"])
@pytest.mark.parametrize("pairs", [False, True])
@pytest.mark.parametrize("na,nb,tile,shift", [
    (1, 2, 0, (1, 2, 3)), (22, 1, 0, (3, 3, 1)), (TILE - 2, 3, 0, (2, 1, 1)), (TILE, TILE, 0, (0, 0, 0)),
    (2 * TILE + 5, 9, 0, (1, 3, 2)), (40_001, 33_334, 4, (3, 0, 1)),
    (2_900_000, 2_867_167, 2, (1, 1, 1)), (2_900_000, 2_867_169, 2, (0, 2, 0)),  # 2048 and 2049 tiles
    (20_000_000, 3_068_673, 2, (2, 0, 3)),  # 8193 tiles
])
def test_tile_edges(na, nb, tile, shift, pairs, kind):
    import paper_cs_0004013_gb300 as rs
    import torch
    a, b = _run(3, na, kind, 0xFFFFFFFF), _run(4, nb, kind, 0)
    va, vb = np.arange(na, dtype=np.uint32), np.arange(na, na + nb, dtype=np.uint32)

    def dev(x, s):  # a buffer that starts s words after a 16-byte boundary
        t = torch.empty(x.size + 8, dtype=torch.int32, device="cuda")
        t[s:s + x.size] = to_dev(x).view(torch.int32)
        return t[s:s + x.size]

    out = dev(np.zeros(na + nb, np.uint32), shift[2])
    vout = dev(np.zeros(na + nb, np.uint32), shift[0])
    plan = {"key_kind": {"u32": 0, "f32": 2}[kind], "tile": tile}
    args = (dev(a, shift[0]), dev(va, shift[1]) if pairs else None, na, dev(b, shift[1]),
            dev(vb, shift[2]) if pairs else None, nb, out, vout if pairs else None, 64, plan)
    temp = torch.empty(rs.rs_merge_u32(*args), dtype=torch.uint8, device="cuda")
    rs.rs_merge_u32(*args, temp)
    torch.cuda.synchronize()
    rs.rs_check_device_error()
    wk, wv = oracle.merge(a, b, va, vb, kind)
    assert np.array_equal(to_host_u32(out), wk)
    if pairs:
        assert np.array_equal(to_host_u32(vout), wv)
