"""Per-vector grouping (Section 2, "Group-wise Quantization"; the KCVT backbone of Section 4): one key group per
channel over the whole segment, one value group per token, Filter_s (Eq. 4) on those whole vectors.  The CUDA path
(C ABI, group = GEAR_GROUP_PER_VECTOR) against the float64 oracle run with a group length no vector reaches:
bit-exact on codes, scales, zero-points and outlier sets / values, <= 1e-3 on the low-rank product and on attention."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture
def pair_factory():
    from tests.gear_harness import Pair
    made = []

    def make(*a, **k):
        p = Pair(*a, **k)
        made.append(p)
        return p
    yield make
    for p in made:
        if p.cache is not None:
            p.close()


def test_four_bit_prefill_of_4096_tokens_then_flushed_buffers(pair_factory):
    """The paper's 4-bit setting (s = 2 %, r = 4) at n = 4096: 41 entries per side leave every key channel."""
    from paper_2403_05527_b200 import binding as G
    p = pair_factory(2, 1, 4, 2, 4, 0, 2.0, 32, 2, 4096 + 128, r_max=4)
    p.compress(4096, 4)
    si = G.gear_segment_info_get(p.cache, 0)
    assert (si.g_k, si.k_k, si.g_v, si.k_v) == (4096, 41, 128, 2)
    p.check_segment(0)
    p.check_attention()
    assert p.append(40) == 1                      # one flushed 32-token segment (a key group = its 32 tokens), 8 buffered
    si = G.gear_segment_info_get(p.cache, 1)
    assert (si.g_k, si.k_k) == (32, 1)
    p.check_segment(1)
    p.check_attention(extra=1)


@pytest.mark.parametrize("bits,group,n,hq,r_flush", [(4, 0, 1024, 4, 2), (2, 64, 256, 4, 2), (4, 128, 128, 4, 2),
                                                     (4, 0, 1024, 2, 4), (2, 128, 256, 2, 4), (2, 64, 256, 2, 3)])
def test_buffer_of_twenty_tokens(pair_factory, bits, group, n, hq, r_flush):
    """n_b = 20 (Section 4, "Implementation details"): a flushed buffer is one block of 20 tokens, a key group its
    20 tokens of a channel; the record keeps two 16-token slabs, the second one partly empty."""
    from paper_2403_05527_b200 import binding as G
    p = pair_factory(2, 2, hq, 2, bits, group, 2.0, 20, r_flush, n + 100, r_max=4)     # hq = 2: the one-head kernel
    p.compress(n, 4)
    assert p.append(67) == 3                      # three flushed 20-token segments, seven tokens buffered
    for si in (1, 2, 3):
        info = G.gear_segment_info_get(p.cache, si)
        assert (info.n_c, info.g_k, info.k_k) == (20, 20, 1)
        p.check_segment(si)
    p.check_attention(extra=3)
    assert p.append(13) == 1                      # the buffer is empty right after a flush
    p.check_segment(4)
    p.check_attention(extra=4)


@pytest.mark.parametrize("bits,n,s,rank", [(2, 512, 2.0, 2), (4, 1024, 5.0, 0), (2, 192, 0.0, 4), (4, 8192, 1.0, 2)])
def test_other_shapes(pair_factory, bits, n, s, rank):
    p = pair_factory(3, 2, 2, 2, bits, 0, s, 64, 2, n + 128, r_max=max(rank, 2))
    p.compress(n, rank)
    p.check_segment(0)
    p.check_attention()
    p.append(70)
    p.check_segment(1)
    p.check_attention(extra=2)


def test_ties_go_to_the_lower_token(pair_factory):
    """Keys drawn from a handful of values: the thresholds of Filter_s sit inside long runs of equal entries, and a
    channel that is constant has its k largest and k smallest in the first 2k tokens."""
    import torch
    from oracle import gear_oracle as O
    from paper_2403_05527_b200 import binding as G, synth
    B, H, n = 1, 2, 512
    rng = np.random.default_rng(7)
    k16 = rng.choice(np.array([-1.5, -0.25, 0.0, 0.25, 2.0], np.float16), size=(B, H, n, 128))
    k16[:, :, :, 5] = np.float16(0.75)            # a constant channel
    k16[:, :, ::7, 9] = np.float16(-0.0)          # both zeros in one channel
    _, v16 = synth.make_kv(3, B, H, n, 128)
    p = pair_factory(3, B, H, H, 4, 0, 3.0, 64, 0, n + 64, r_max=0)
    p.oracle.compress(k16, v16, 0, None)
    dev = p.dev
    G.gear_compress(p.cache, None, torch.from_numpy(k16).to(dev), torch.from_numpy(v16).to(dev), n, 0, None)
    torch.cuda.synchronize()
    p.check_segment(0)
    p.check_attention()
    assert O.outlier_count(3.0, n) == 8


def test_limits_are_errors(pair_factory):
    import torch
    from paper_2403_05527_b200 import binding as G
    with pytest.raises(G.GearError):              # a buffer longer than one block of per-vector keys
        G.gear_create(G.make_config(1, 1, 1, 4, 0, 2.0, 256, 0, 1024))
    cfg = G.make_config(1, 1, 1, 4, 0, 2.0, 64, 0, 16384)
    cache = G.gear_create(cfg)
    try:
        x = torch.zeros(1, 1, 16384, 128, dtype=torch.float16, device="cuda:0")
        with pytest.raises(G.GearError):          # longer than the select kernel's shared memory holds
            G.gear_compress(cache, None, x, x, 16384, 0, None)
        with pytest.raises(G.GearError):          # not a multiple of the 64-token record block
            G.gear_compress(cache, None, x, x, 208, 0, None)
    finally:
        G.gear_free(cache)


def test_two_long_segments_a_short_one_and_a_buffer(pair_factory):
    """Two prefill calls of per-vector keys (each its own groups and outlier list), a 128-token segment that is a
    single ordinary block, then a flushed buffer and buffered tokens."""
    import torch
    from paper_2403_05527_b200 import binding as G, synth
    p = pair_factory(5, 2, 2, 2, 2, 0, 2.0, 32, 2, 2048, r_max=4)
    p.compress(512, 4)
    p.compress(256, 2, extra=1)
    p.compress(128, 3, extra=2)
    infos = [G.gear_segment_info_get(p.cache, i) for i in range(3)]
    assert [(i.n_c, i.g_k, i.k_k) for i in infos] == [(512, 512, 6), (256, 256, 3), (128, 128, 2)]
    for si in range(3):
        p.check_segment(si)
    p.append(37)
    p.check_segment(3)
    p.check_attention(extra=5)
    b = G.gear_cache_bytes(p.cache)
    assert b.stored_total >= b.codes + b.scale_zero + b.outliers + b.lowrank_a + b.lowrank_b + b.buffer


def test_capacity_of_the_arena_is_an_error_not_a_fault():
    import torch
    from paper_2403_05527_b200 import binding as G
    cfg = G.make_config(1, 1, 1, 4, 0, 2.0, 32, 0, 512)
    cache = G.gear_create(cfg)
    try:
        x = torch.randn(1, 1, 512, 128, device="cuda:0").half()
        G.gear_compress(cache, None, x, x, 512, 0, None)
        with pytest.raises(G.GearError):          # the cache was sized for 512 tokens
            G.gear_compress(cache, None, x, x, 192, 0, None)
        assert G.gear_last_device_status(cache) == 0
    finally:
        G.gear_free(cache)


@pytest.mark.parametrize("n,s", [(192, 2.0), (4096, 4.0), (4096, 2.0), (8192, 5.0), (4160, 2.0)])
def test_selection_of_the_outliers(pair_factory, n, s):
    """Counts of outliers on both sides of the select kernel's limits (one or two extremes per lane, the histograms), and
    channels whose extremes all lie with few lanes, that are sorted, rounded to few values or zeros of both signs."""
    import torch
    from paper_2403_05527_b200 import binding as G, synth
    k16, v16 = synth.make_kv(9, 1, 1, n, 128)
    t = np.arange(n)
    k16[0, 0, t % 256 < 8, 3] += np.float16(40.0)          # a lane's eight neighbours, every 256 tokens
    k16[0, 0, t % 256 < 8, 3] *= (1 + t[t % 256 < 8] / n).astype(np.float16)
    k16[0, 0, :, 4] = np.sort(k16[0, 0, :, 4])
    k16[0, 0, :, 5] = np.sort(k16[0, 0, :, 5])[::-1]
    k16[0, 0, :, 6] = np.round(k16[0, 0, :, 6] * 4) / 4    # ties at both thresholds
    k16[0, 0, :, 7] = np.sign(k16[0, 0, :, 7]) * np.float16(0.0) + (t == 11) - (t == 12)
    p = pair_factory(9, 1, 1, 1, 4, 0, s, 64, 0, n + 64, r_max=0)
    p.oracle.compress(k16, v16, 0, None)
    G.gear_compress(p.cache, None, torch.from_numpy(k16).to(p.dev), torch.from_numpy(v16).to(p.dev), n, 0, None)
    torch.cuda.synchronize()
    p.check_segment(0)


# Lets the kernel behind it start at once, and writes what that kernel reads some thirty microseconds later.
_LATE_COPY = r"""
extern "C" __global__ void late_copy(const uint4* src, uint4* dst, int n) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  for (int i = 0; i < 60; ++i) __nanosleep(500);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) dst[i] = src[i];
}
"""


@pytest.mark.parametrize("group,s,rank", [(0, 0.0, 0), (0, 1.0, 0), (0, 2.0, 0), (0, 2.0, 4), (64, 2.0, 0), (128, 2.0, 0)])
def test_keys_and_values_that_the_kernel_in_front_writes(pair_factory, group, s, rank):
    """The producer of a segment's rows may let its dependents start before it has written them: every kernel of the call has to
    wait for it, also the values' where no keys' kernel is in front of it.  The second segment: a new cache clears scratch first."""
    import torch
    from paper_2403_05527_b200 import binding as G, synth
    p = pair_factory(6, 1, 2, 2, 4, group, s, 64, 0, 1024, r_max=4)
    p.compress(256, 0)
    k16, v16 = synth.make_kv(6, 1, 2, 256, 128, extra=1)
    b0 = synth.make_b0(6, 1, 2, 128, rank, extra=1)
    p.oracle.compress(k16, v16, rank, b0)
    made = torch.from_numpy(np.stack([k16, v16])).to(p.dev)
    rows = torch.zeros_like(made)
    b0d = torch.from_numpy(np.ascontiguousarray(b0)).to(p.dev) if rank else None
    late_copy = torch.cuda._compile_kernel(_LATE_COPY, "late_copy")
    torch.cuda.synchronize()
    late_copy(grid=(8, 1, 1), block=(256, 1, 1), args=[made, rows, made.numel() // 8])
    G.gear_compress(p.cache, None, rows[0], rows[1], 256, rank, b0d)
    torch.cuda.synchronize()
    p.check_segment(1)
