"""Segmented sorts whose segments are mostly empty, so that few blocks take the
short ones in turn, against the oracle: more short segments than blocks, each
class at its edges, and calls whose offsets change on the device between replays
of the captured launches (the host's copy only plans them)."""
import numpy as np
import pytest

import oracle
import synth
from tests._gpu import to_dev, to_host_u32

pytestmark = pytest.mark.gpu

EDGES = [1, 2, 4095, 4096, 4097, 16383, 16384, 16385, 40_000]


def _lengths(num_segs, short, edges, seed):
    r = np.random.default_rng(seed)
    m = np.zeros(num_segs, np.int64)
    at = r.permutation(num_segs)
    m[at[:short]] = r.integers(1, 65, short)
    m[at[short:short + len(edges)]] = edges
    return m


def _offsets(m):
    return np.concatenate([[0], np.cumsum(m)]).astype(np.uint64)


@pytest.mark.parametrize("pairs", [False, True])
@pytest.mark.parametrize("num_segs,short,edges", [(12_000, 1, []), (12_000, 5_000, EDGES), (100_001, 3, EDGES),
                                                  (12_000, 11_000, EDGES)])
def test_mostly_empty(num_segs, short, edges, pairs):
    import paper_cs_0004013_gb300 as rs
    import torch
    offs = _offsets(_lengths(num_segs, short, edges, 7))
    n = int(offs[-1])
    keys = synth.splitmix64(11, (n + 1) // 2).view(np.uint32)[:n].copy()
    vals = np.arange(n, dtype=np.uint32)
    ko, vo, _ = rs.sort_segmented(to_dev(keys), to_dev(vals) if pairs else None, offs)
    torch.cuda.synchronize()
    rs.rs_check_device_error()
    wk, wv, _ = oracle.sort_segmented(keys, vals, offs)
    assert np.array_equal(to_host_u32(ko), wk)
    if pairs:
        assert np.array_equal(to_host_u32(vo), wv)


def test_offsets_that_change_on_the_device():
    import paper_cs_0004013_gb300 as rs
    import torch
    few = _lengths(6_000, 100, EDGES, 1)
    n = int(few.sum())
    many = np.full(6_000, n // 6_000, np.int64)
    many[0] += n - many.sum()
    keys = synth.splitmix64(5, (n + 1) // 2).view(np.uint32)[:n].copy()
    h = _offsets(few)
    d = to_dev(h)
    dk = to_dev(keys)
    out = torch.empty_like(dk)
    args = (dk, None, out, None, d, h, 6_000, n, 64, None, None)
    temp = torch.empty(rs.rs_sort_u32_segmented(*args), dtype=torch.uint8, device="cuda")
    rs.rs_sort_u32_segmented(*args, temp)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        rs.rs_sort_u32_segmented(*args, temp)
    for m in (few, many, few[::-1]):
        d.copy_(to_dev(_offsets(m)))
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        rs.rs_check_device_error()
        assert np.array_equal(to_host_u32(out), oracle.sort_segmented(keys, None, _offsets(m))[0])
