"""Several query rows per kv head: every row count around the edges of a pass (four and eight rows), key shapes that fill a
warp's slabs unevenly, buffers that end inside a 32-token item, flushed segments behind the prompt, per-vector lists."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,hkv,bits,group,s,rank,nb,n,pushed", [
    (2, 1, 2, 64, 2.0, 4, 64, 192, 0),
    (6, 2, 4, 64, 1.0, 8, 64, 64, 64 + 33),          # three rows; a flushed segment, two buffer items
    (4, 1, 2, 128, 2.0, 4, 64, 512, 64 + 17),
    (5, 1, 4, 128, 2.0, 16, 128, 128, 127),
    (7, 1, 2, 32, 4.0, 2, 32, 96, 32 + 1),
    (8, 1, 4, 16, 6.0, 1, 16, 48, 16 + 15),
    (9, 1, 2, 64, 0.0, 0, 64, 128, 5),                # two passes, the second with one row
    (16, 1, 2, 64, 2.0, 4, 64, 16, 3),                # one slab in the prompt
    (8, 2, 4, 0, 2.0, 4, 20, 256, 20 + 7),            # per-vector lists, 20-token blocks
    (17, 1, 2, 0, 2.0, 3, 64, 192, 64 + 40),
])
def test_rows_against_the_oracle(hq, hkv, bits, group, s, rank, nb, n, pushed):
    from paper_2403_05527_b200 import synth
    from tests.gear_harness import Pair, rel_max
    p = Pair(17, 2, hq, hkv, bits, group, s, nb, min(rank, nb), 1024, r_max=rank, keep_fp32=False)

    def check(extra):
        # fp16 storage of A and B alone moves single rows of caches this short by up to 1.1e-3 (measured with the oracle on
        # its own against the stored factors): 2e-3 against its own factors, 1e-3 against the stored ones, and against these
        # the kernel's arithmetic is far nearer: 22-bit operands and fp32 sums, 1e-4 on scores of up to a few dozen
        _, got = p.check_attention(extra=extra, tol=2e-3)
        want = p.with_stored_factors().decode_attn(synth.make_query(17, 2, hq, 128, extra=extra))
        worst = max(rel_max(got[b, h], want[b, h]) for b in range(2) for h in range(hq))
        assert worst <= 1e-4, f"against the oracle on the stored factors: {worst:.2e}"

    try:
        p.compress(n, rank)
        check(0)
        if pushed:
            p.append(pushed)
            check(1)
    finally:
        p.close()


def test_scores_that_keep_growing():
    """Keys ordered so that the running maximum rises in every block, by less and by more than the lag that the fixed point
    allows: the sums are folded or carried on, the result is the same."""
    import torch
    from paper_2403_05527_b200 import binding as G
    from tests.gear_harness import Pair, rel_max
    for hq, step in ((4, 0.4), (8, 1.3), (1, 0.4), (1, 1.3)):
        p = Pair(18, 1, hq, 1, 4, 64, 2.0, 64, 0, 2048, keep_fp32=False)
        try:
            gen = np.random.default_rng(hq)
            n = 1024
            k = gen.standard_normal((1, 1, n, 128)) * 0.05
            k[..., 0] += np.arange(n) // 64 * step * 2.0      # q[0] = 8, scale 1 / sqrt(128): 2 ** about step per block
            k16, v16 = k.astype(np.float16), gen.standard_normal((1, 1, n, 128)).astype(np.float16)
            q = (gen.standard_normal((1, hq, 128)) * 0.1).astype(np.float16)
            q[..., 0] = 8.0
            p.oracle.compress(k16, v16, 0, np.zeros((1, 1, 2, 128, 0), np.float32))
            G.gear_compress(p.cache, None, torch.from_numpy(k16).cuda(), torch.from_numpy(v16).cuda(), n, 0)
            out = torch.empty((1, hq, 128), device="cuda")
            G.gear_decode_attn(p.cache, torch.from_numpy(q).cuda(), out)
            ref = p.oracle.decode_attn(q, None)
            got = out.cpu().numpy().astype(np.float64)
            # 22 bits of p * scale less three bits of lag and exponent, fp32 sums: far below 4e-5
            assert max(rel_max(got[0, h], ref[0, h]) for h in range(hq)) <= 4e-5
        finally:
            p.close()


@pytest.mark.parametrize("batch,hq,hkv,most", [(3, 32, 8, 10), (16, 32, 8, 10), (4, 64, 8, 7), (2, 5, 5, 12)])
def test_every_row_count_up_to_the_cache_s_own(batch, hq, hkv, most):
    """The scratch for partial results does not grow with the row count: seven or eight positions of the first shape need
    more of it than nine or ten.  Every count is taken, and its rows are those of the largest call."""
    import torch
    from paper_2403_05527_b200 import binding as G
    gen = torch.Generator(device="cuda").manual_seed(batch)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda").half()   # noqa: E731
    k, v, q = draw(batch, hkv, 192, 128), draw(batch, hkv, 192, 128), draw(batch, hq, most, 128)
    cache = G.gear_compress(None, G.make_config(batch, hq, hkv, 2, 64, 2.0, 64, 4, 256, seed=1, max_queries=most), k, v, 192, 4)
    try:
        want = torch.empty(q.shape, device="cuda")
        G.gear_decode_attn_multi(cache, q, want, most)
        for rows in range(1, most):
            got = torch.full((batch, hq, rows, 128), float("nan"), device="cuda")
            G.gear_decode_attn_multi(cache, q[:, :, :rows].contiguous(), got, rows)
            # the same arithmetic per row (one row per kv head: another kernel's), split over other ranges of blocks
            err = (got - want[:, :, :rows]).abs().amax(-1) / want[:, :, :rows].abs().amax(-1)
            assert err.max().item() <= 4e-5, rows
        assert G.gear_last_device_status(cache) == 0
    finally:
        G.gear_free(cache)


@pytest.mark.parametrize("bits", [2, 4])
@pytest.mark.parametrize("hq", [1, 4, 8])
def test_small_probabilities_beside_a_large_one(hq, bits):
    """In every block one token holds nearly all of the probability and the others 2^-21 of it, which is one or two units of
    the value fixed point: 22 bits at a probability of one, so an entry of the output is off by at most half a unit per code
    (and fp32 rounding), whatever the maximum may lag by."""
    import torch
    from paper_2403_05527_b200 import binding as G
    from tests.gear_harness import Pair
    p = Pair(18, 1, hq, 1, bits, 64, 0.0, 64, 0, 1024, keep_fp32=False)
    try:
        n, levels = 512, 2 ** bits - 1
        gen = np.random.default_rng(bits)
        k16 = np.zeros((1, 1, n, 128), np.float16)
        k16[0, 0, ::64, 0] = 21.1 / (8.0 / np.sqrt(128.0) * np.log2(np.e))          # the others score 21.1 bits less
        v16 = gen.uniform(0.0, levels, (1, 1, n, 128)).astype(np.float16)
        q = np.zeros((1, hq, 128), np.float16)
        q[..., 0] = 8.0
        p.oracle.compress(k16, v16, 0, np.zeros((1, 1, 2, 128, 0), np.float32))
        tile = p.oracle.segments[0]["V"][0][0]
        assert (0.5 <= tile["scale"]).all() and (tile["scale"] < 1.0).all()        # the exponent that fixes the unit
        G.gear_compress(p.cache, None, torch.from_numpy(k16).cuda(), torch.from_numpy(v16).cuda(), n, 0)
        out = torch.empty((1, hq, 128), device="cuda")
        G.gear_decode_attn(p.cache, torch.from_numpy(q).cuda(), out)
        got, ref = out.cpu().numpy().astype(np.float64)[0], p.oracle.decode_attn(q, None)[0]
        unit = 2.0 ** -22                                # of a scale below one
        bound = tile["codes"].sum(0) * (unit / 2) / (n // 64) + 2.0 ** -20 * np.abs(ref)
        assert (np.abs(got - ref) <= bound).all(), (np.abs(got - ref) / bound).max()
    finally:
        p.close()


@pytest.mark.parametrize("hkv,bits,group,s,rank,n,rows", [
    (32, 2, 64, 2.0, 4, 5888, 16),       # every block shape the kernel is built for, eight rows at a time ...
    (32, 4, 64, 2.0, 8, 4096, 24),
    (24, 2, 128, 2.0, 4, 16384, 15),     # the last pass with seven rows
    (32, 4, 128, 2.0, 4, 8192, 29),      # ... and five
    (32, 4, 0, 2.0, 4, 6144, 16),
    (48, 2, 32, 0.0, 0, 4096, 7),
    (24, 4, 16, 6.0, 2, 4096, 16),
    (32, 2, 64, 2.0, 4, 5888, 12),       # a last pass of four: fours although the cache is long
])
def test_rows_in_eights_against_rows_in_fours(hkv, bits, group, s, rank, n, rows):
    """Long caches take eight rows per pass.  Each row has to be what it is in a call of four rows, before and after the cache
    grows over the line (a prompt of an eighth, the rest behind it)."""
    import torch
    from paper_2403_05527_b200 import binding as G
    gen = torch.Generator(device="cuda").manual_seed(rows)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda").half()   # noqa: E731
    nb = 64 if group != 0 else 20
    cfg = G.make_config(1, hkv, hkv, bits, group, s, nb, min(rank, nb), n + nb, rank_max=max(rank, 0), seed=1, max_queries=rows)
    k, v, q = draw(1, hkv, n, 128), draw(1, hkv, n, 128), draw(1, hkv, rows, 128)
    cache = G.gear_create(cfg)
    try:
        first = n // 8 // 128 * 128
        for lo, hi in ((0, first), (first, n)):
            G.gear_compress(cache, None, k[:, :, lo:hi].contiguous(), v[:, :, lo:hi].contiguous(), hi - lo, rank)
            if hi == n:
                for _ in range(7):
                    G.gear_append_buffer(cache, draw(1, hkv, 128), draw(1, hkv, 128))
            got = torch.full(q.shape, float("nan"), device="cuda")
            G.gear_decode_attn_multi(cache, q, got, rows)
            for r0 in range(0, rows, 4):
                part = q[:, :, r0:r0 + 4].contiguous()
                want = torch.empty(part.shape, device="cuda")
                if part.shape[2] > 1:
                    G.gear_decode_attn_multi(cache, part, want, part.shape[2])
                else:
                    G.gear_decode_attn(cache, part, want)
                err = (got[:, :, r0:r0 + 4] - want).abs().amax(-1) / want.abs().amax(-1)
                assert err.max().item() <= 8e-5          # twice what a kernel's own arithmetic may be off
        assert G.gear_last_device_status(cache) == 0
    finally:
        G.gear_free(cache)


@pytest.mark.parametrize("hkv,group_heads,bits,group,s,rank,n", [
    (32, 1, 2, 64, 2.0, 4, 12032),       # 188 blocks per unit, two passes of one row
    (32, 2, 4, 64, 1.0, 8, 12032),       # two query heads per kv head instead of two positions
    (30, 2, 2, 128, 2.0, 4, 26624),
    (48, 1, 4, 0, 2.0, 4, 8192),         # per-vector lists
    (24, 2, 4, 16, 6.0, 2, 4096),        # groups of 16 keep their kernel
    (64, 1, 2, 32, 0.0, 0, 3072),
])
def test_two_rows_over_long_caches(hkv, group_heads, bits, group, s, rank, n):
    """Two rows per kv head take the kernel of one row twice once the cache is long.  Each has to be what it is alone (a second
    cache with one query head per kv head), before and after the line."""
    import torch
    from paper_2403_05527_b200 import binding as G
    gen = torch.Generator(device="cuda").manual_seed(n)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda").half()   # noqa: E731
    rows = 2 // group_heads
    nb = 64 if group != 0 else 20
    cfg = lambda heads, most: G.make_config(1, hkv * heads, hkv, bits, group, s, nb, min(rank, nb), n + nb,   # noqa: E731
                                            rank_max=rank, seed=1, max_queries=most)
    k, v, q, tail = draw(1, hkv, n, 128), draw(1, hkv, n, 128), draw(1, hkv, 2, 128), draw(7, 2, 1, hkv, 128)
    both, single = G.gear_create(cfg(group_heads, rows)), G.gear_create(cfg(1, 1))
    try:
        first = n // 8 // 128 * 128
        for lo, hi in ((0, first), (first, n)):
            part = k[:, :, lo:hi].contiguous(), v[:, :, lo:hi].contiguous()
            for cache in (both, single):
                G.gear_compress(cache, None, *part, hi - lo, rank)
                for t in tail if hi == n else ():
                    G.gear_append_buffer(cache, t[0], t[1])
            got = torch.full(q.shape, float("nan"), device="cuda")
            for _ in range(2):
                G.gear_decode_attn_multi(both, q, got, rows)
            want = torch.empty((1, hkv, 128), device="cuda")
            for r in range(2):
                G.gear_decode_attn(single, q[:, :, r].contiguous(), want)
                err = (got[:, :, r] - want).abs().amax(-1) / want.abs().amax(-1)
                assert err.max().item() <= 8e-5          # twice what a kernel's own arithmetic may be off
        assert G.gear_last_device_status(both) == 0
    finally:
        G.gear_free(both)
        G.gear_free(single)
