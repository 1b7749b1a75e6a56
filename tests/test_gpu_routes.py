"""Which way sorts with the automatic plan go, and that each way gives the
oracle's result: value buckets for even keys, the radix passes where the sample
finds clusters, and where a bucket turns out to hold too many keys; in the single
launch and in the launches of larger sorts, for every key and payload width.  Also
under capture and replay on other data, from addresses off a 16-byte boundary and
on two streams at once."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

# (key bits, payload bytes, n): the single launch's three tile shapes, then one and two splits
SINGLE = [(32, 0, 300_001), (32, 0, 900_001), (32, 0, 2_500_001), (32, 4, 300_001), (32, 4, 900_001)]
LARGE = [(32, 0, 3_000_001), (32, 4, (1 << 23) + 500_001), (32, 8, 300_001), (32, 8, 1_000_001), (64, 0, 300_001), (64, 0, 1_000_001),
         (64, 4, 300_001), (64, 4, 1_000_001), (64, 8, 300_001), (64, 8, 3_000_001)]


class Sort:
    """One sort's buffers (shift: words between a 16-byte boundary and the 32-bit arrays)."""

    def __init__(self, bits, vb, n, shift=0):
        import paper_cs_0004013_gb300 as rs
        import torch
        self.rs, self.torch, self.bits, self.vb, self.n = rs, torch, bits, vb, n
        self.call = {(32, 0): rs.rs_sort_u32, (32, 4): rs.rs_sort_u32_pairs, (32, 8): rs.rs_sort_u32_pairs64,
                     (64, 0): rs.rs_sort_u64, (64, 4): rs.rs_sort_u64_pairs, (64, 8): rs.rs_sort_u64_pairs64}[bits, vb]

        def buf(nbytes):
            t = torch.empty(n + 8, dtype=torch.int64 if nbytes == 8 else torch.int32, device="cuda")
            k = shift if nbytes == 4 else shift % 2
            return t[k:k + n]

        self.k, self.ko = buf(bits // 8), buf(bits // 8)
        self.v, self.vo = (buf(vb), buf(vb)) if vb else (None, None)
        self.args = (self.k, self.v, self.ko, self.vo, n) if vb else (self.k, self.ko, n)
        self.temp = torch.empty(self.call(*self.args), dtype=torch.uint8, device="cuda")

    def put(self, words):
        self.words = words
        self.k.copy_(self.torch.from_numpy(words.view(np.int32 if self.bits == 32 else np.int64).copy()))
        if self.vb:
            self.v.copy_(self.torch.arange(self.n, device="cuda"))
        return self

    def run(self, stream=None):
        self.call(*self.args, 64, None, self.temp, stream)
        return self

    def check(self, *routes):
        self.torch.cuda.synchronize()
        self.rs.rs_check_device_error()
        if routes:
            assert self.rs.rs_selftest_route(self.bits // 8, self.vb, self.n, self.temp) in routes
        vals = np.arange(self.n, dtype=np.uint32)
        wk, wv = oracle.sort_pairs(self.words, vals, f"u{self.bits}")
        assert np.array_equal(self.ko.cpu().numpy().view(self.words.dtype), wk)
        if self.vb:
            assert np.array_equal(self.vo.cpu().numpy().astype(np.uint32), wv)


def _words(bits, n, data, seed=0, vb=0):
    w = synth.splitmix64(n + seed, n)
    if data == "overfull":
        # equal keys, spread over the array: one bucket holds more than it takes with
        # them (mean and most keys of a bucket), but not so many that the sample minds
        single = bits == 32 and vb < 8 and n < 400_000
        mean, most = (4545, 6144) if single else (2048, 3072) if vb == 0 else (1365, 2048)
        extra = most - mean + 200
        w[np.arange(extra) * (n // extra)] = w[3]
    elif data == "clusters":
        w = w[:8][(synth.splitmix64(9, n) % np.uint64(8)).astype(np.int64)] // np.uint64(2) + (w & np.uint64(0xFFFFFFFFFF))
    return (w >> np.uint64(64 - bits)).astype(np.uint32 if bits == 32 else np.uint64)


@pytest.mark.parametrize("bits,vb,n", SINGLE + LARGE)
def test_even_keys_take_the_buckets(bits, vb, n):
    s = Sort(bits, vb, n).put(_words(bits, n, "even")).run()
    s.check(s.rs.RS_ROUTE_BUCKETS)


@pytest.mark.parametrize("bits,vb,n", SINGLE + LARGE)
def test_clusters_take_the_radix_passes(bits, vb, n):
    s = Sort(bits, vb, n).put(_words(bits, n, "clusters")).run()
    s.check(s.rs.RS_ROUTE_RADIX)


@pytest.mark.parametrize("bits,vb,n", [(32, 0, 300_001), (32, 4, 300_001), (32, 0, 3_000_001), (32, 8, 1_000_001), (64, 0, 1_000_001),
                                       (64, 4, 1_000_001), (64, 8, 3_000_001)])
def test_an_overfull_bucket_turns_to_the_radix_passes(bits, vb, n):
    s = Sort(bits, vb, n).put(_words(bits, n, "overfull", vb=vb)).run()
    s.check(s.rs.RS_ROUTE_OVERFULL)


@pytest.mark.parametrize("bits,vb,n", [(32, 0, 16_384), (32, 4, 16_384), (64, 0, 8192), (64, 8, 8192), (32, 4, 3_000_001)])
def test_sizes_without_a_choice(bits, vb, n):
    s = Sort(bits, vb, n).put(_words(bits, n, "even")).run()
    s.check(s.rs.RS_ROUTE_FIXED)


@pytest.mark.parametrize("shift", [1, 2, 3])
@pytest.mark.parametrize("bits,vb,n", [(32, 0, 300_001), (32, 4, 300_001), (32, 0, 3_000_001), (32, 4, (1 << 23) + 500_001), (32, 8, 300_001),
                                       (64, 0, 300_001), (64, 4, 300_001)])
def test_addresses_off_a_16_byte_boundary(bits, vb, n, shift):
    s = Sort(bits, vb, n, shift).put(_words(bits, n, "even")).run()
    s.check(s.rs.RS_ROUTE_BUCKETS)


@pytest.mark.parametrize("bits,vb,n", [(32, 0, 1000), (32, 4, 300_001), (32, 0, 3_000_001), (32, 4, (1 << 23) + 500_001), (32, 8, 1_000_001),
                                       (64, 0, 1_000_001), (64, 4, 300_001), (64, 8, 3_000_001)])
def test_capture_and_replay_on_other_data(bits, vb, n):
    s = Sort(bits, vb, n).put(_words(bits, n, "even")).run()
    s.torch.cuda.synchronize()
    g = s.torch.cuda.CUDAGraph()
    with s.torch.cuda.graph(g):
        s.run()
    for data in ("clusters", "even"):  # the route is chosen anew in each replay
        s.put(_words(bits, n, data, seed=1))
        s.ko.zero_()
        g.replay()
        s.check()
        if n > 16_384:
            assert s.rs.rs_selftest_route(bits // 8, vb, n, s.temp) == (
                s.rs.RS_ROUTE_BUCKETS if data == "even" else s.rs.RS_ROUTE_RADIX)


@pytest.mark.parametrize("pairs", [False, True])
def test_merge_capture_and_replay(pairs):
    import paper_cs_0004013_gb300 as rs
    import torch
    na, nb = 700_001, 400_003
    a, b = (torch.empty(n, dtype=torch.int32, device="cuda") for n in (na, nb))
    va = torch.arange(na, dtype=torch.int32, device="cuda") if pairs else None
    vb = torch.arange(na, na + nb, dtype=torch.int32, device="cuda") if pairs else None
    out = torch.empty(na + nb, dtype=torch.int32, device="cuda")
    vout = torch.empty_like(out) if pairs else None

    def put(seed):
        w = [np.sort(synth.splitmix64(seed + i, n).astype(np.uint32)) for i, n in enumerate((na, nb))]
        a.copy_(torch.from_numpy(w[0].view(np.int32)))
        b.copy_(torch.from_numpy(w[1].view(np.int32)))
        return w

    args = (a, va, na, b, vb, nb, out, vout)
    temp = torch.empty(rs.rs_merge_u32(*args), dtype=torch.uint8, device="cuda")
    put(1)
    rs.rs_merge_u32(*args, 64, None, temp)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        rs.rs_merge_u32(*args, 64, None, temp)
    for seed in (5, 9):
        w = put(seed)
        g.replay()
        torch.cuda.synchronize()
        rs.rs_check_device_error()
        wk, wv = oracle.merge(w[0], w[1], np.arange(na, dtype=np.uint32), np.arange(na, na + nb, dtype=np.uint32))
        assert np.array_equal(out.cpu().numpy().view(np.uint32), wk)
        if pairs:
            assert np.array_equal(vout.cpu().numpy().view(np.uint32), wv)


def test_two_streams_at_once():
    import torch
    sorts = [Sort(32, 0, 3_000_001).put(_words(32, 3_000_001, "even")), Sort(32, 0, 3_000_001).put(_words(32, 3_000_001, "clusters")),
             Sort(64, 8, 300_001).put(_words(64, 300_001, "even")), Sort(32, 4, 300_001).put(_words(32, 300_001, "even"))]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    for _ in range(5):
        for i, s in enumerate(sorts):
            s.run(streams[i % 2])
    for s, data in zip(sorts, ("even", "clusters", "even", "even")):
        s.check(s.rs.RS_ROUTE_RADIX if data == "clusters" else s.rs.RS_ROUTE_BUCKETS)


def _fill_one_bucket(w, bits, mean, count):
    """w with keys from elsewhere moved into a middle bucket until it holds `count`, as the sort will
    see it: the value map of a sample at fixed places, which stay as they are."""
    n = w.size
    S = 2304 if -(-n // mean) <= 768 else 8192
    q = np.arange(S, dtype=np.uint64)
    m32 = np.uint64(0xFFFFFFFF)
    h = (q * np.uint64(0x9E3779B1)) & m32
    h ^= h >> np.uint64(15)
    pos = q * np.uint64(n) // np.uint64(S)
    if n // S > 1:
        pos = pos + ((((h * np.uint64(0x85EBCA77)) & m32) * np.uint64(n // S)) >> np.uint64(32))
    pos = pos.astype(np.int64)
    buckets = -(-n // mean)
    lo, hi = int(w[pos].min()), int(w[pos].max())
    ext = (hi - lo) // (S // 8)
    lo, hi = max(lo - ext, 0), min(hi + ext, (1 << bits) - 1)
    sh = max((hi - lo).bit_length() - 32, 0)
    mult = (buckets << 32) // (((hi - lo) >> sh) + 1)
    x = np.clip(w.astype(np.uint64), np.uint64(lo), np.uint64(hi)) - np.uint64(lo)
    bucket = ((x >> np.uint64(sh)) * np.uint64(mult)) >> np.uint64(32)
    b = buckets // 2
    first, last = -(-(b << 32) // mult), -(-((b + 1) << 32) // mult)  # its offsets: [first, last)
    need = count - int((bucket == b).sum())
    free = np.ones(n, bool)
    free[pos] = False
    move = np.flatnonzero(free & (bucket != b))[:: 97][:need]
    assert 0 < need == move.size
    step = (synth.splitmix64(17, need) % np.uint64((last - first) << sh)) + np.uint64((first << sh) + lo)
    out = w.copy()
    out[move] = step.astype(w.dtype)
    return out


@pytest.mark.parametrize("over", [0, 1])
@pytest.mark.parametrize("bits,vb,n,mean,most", [(32, 0, 3_000_001, 2048, 3072), (32, 8, 1_000_001, 1365, 2048), (64, 0, 1_000_001, 2048, 3072),
                                                 (64, 4, 1_000_001, 1365, 2048), (64, 8, 3_000_001, 1365, 2048),
                                                 (32, 4, (1 << 23) + 500_001, 2048, 3072)])
def test_a_bucket_at_its_most_keys(bits, vb, n, mean, most, over):
    w = _fill_one_bucket(_words(bits, n, "even"), bits, mean, most + over)
    s = Sort(bits, vb, n).put(w).run()
    s.check(s.rs.RS_ROUTE_OVERFULL if over else s.rs.RS_ROUTE_BUCKETS)
