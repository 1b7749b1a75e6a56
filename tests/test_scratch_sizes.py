"""Scratch sizes never fall as n grows: a workspace that a caller allocates for
its largest request takes every smaller one (automatic plans; size queries
only, no GPU)."""
import numpy as np
import pytest


def _sizes():
    """Every size class' edges: powers of two, value-bucket counts at which a split changes its digits or the
    buckets end, tiles of the status words, the word width of large sorts, and sizes between."""
    at = {0, 1, (1 << 30) - 65536, (1 << 32) - 2}
    at |= {1 << k for k in range(32)}
    for mean, cap in ((2048, 3072), (1365, 2048)):  # keys per bucket, aimed at and at most
        for k in range(5, 17):
            at |= {b * mean for b in (1 << k, (1 << k) + 1, 3 << (k - 1))}
        at |= {49152 * mean, 49152 * cap * 3 // 4}
    at |= {int(x) for x in np.exp(np.linspace(np.log(1000), np.log(4e9), 4000))}
    return sorted({n + d for n in at for d in (-1, 0, 1) if 0 <= n + d < 1 << 32})


def _queries():
    import paper_cs_0004013_gb300 as rs
    return {
        "sort": lambda n: rs.rs_sort_u32(None, None, n),
        "sort_pairs": lambda n: rs.rs_sort_u32_pairs(None, None, None, None, n),
        "sort_pairs64": lambda n: rs.rs_sort_u32_pairs64(None, None, None, None, n),
        "sort64": lambda n: rs.rs_sort_u64(None, None, n),
        "sort64_pairs": lambda n: rs.rs_sort_u64_pairs(None, None, None, None, n),
        "sort64_pairs64": lambda n: rs.rs_sort_u64_pairs64(None, None, None, None, n),
        "host": lambda n: rs.rs_sort_u32_host(None, None, None, None, n),
        "host_pairs": lambda n: rs.rs_sort_u32_host(None, 1, None, 2, n),
        "merge": lambda n: rs.rs_merge_u32(None, None, n // 3, None, None, n - n // 3, None, None),
        "merge_pairs": lambda n: rs.rs_merge_u32(None, 1, n // 3, None, 1, n - n // 3, None, 1),
    }


@pytest.mark.parametrize("entry", ["sort", "sort_pairs", "sort_pairs64", "sort64", "sort64_pairs", "sort64_pairs64",
                                   "host", "host_pairs", "merge", "merge_pairs"])
def test_scratch_never_falls(entry):
    query = _queries()[entry]
    at = _sizes()
    need = [query(n) for n in at]
    falls = [(a, b, x - y) for a, b, x, y in zip(at, at[1:], need, need[1:]) if y < x]
    assert not falls, f"{entry}: (n, next n, bytes fewer) {falls[:8]}"
