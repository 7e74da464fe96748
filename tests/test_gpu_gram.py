"""Long segments: the loops of Algorithm 2 on R^T R.  Sizes where the work split of the Gram kernel can go wrong (a last
block of 16 rows, fewer blocks than CTAs, ranges that end inside a tile), every factor width, and loop counts."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,n,bits,group,rank,iters", [
    (1, 1, 144, 2, 16, 4, 3),       # three blocks per tile, the last one with 16 rows; one range for both tiles
    (1, 1, 160, 4, 32, 16, 3),      # rank 16, last block of 32 rows
    (1, 3, 1088, 2, 64, 8, 3),      # 17 blocks per tile: ranges end inside tiles
    (2, 5, 576, 2, 64, 5, 1),       # a single loop: B0 itself is orthonormalised
    (1, 2, 2048, 4, 64, 1, 12),     # many loops: the factor is rescaled on the way
    (1, 2, 256, 2, 128, 3, 2),
])
def test_factors_match_the_oracle(B, H, n, bits, group, rank, iters):
    from tests.gear_harness import Pair
    p = Pair(14, B, H, H, bits, group, 2.0, max(group, 16), min(rank, max(group, 16)), n + 128, r_max=rank, iters=iters)
    try:
        p.compress(n, rank)
        # 22 bits of every operand, sums over n rows: 1e-5 is what the shapes above show at most away from close
        # singular values; the oracle's own bound on A B^T is 1e-3
        p.check_segment(0)
        p.check_attention()
    finally:
        p.close()


@pytest.mark.parametrize("group,n", [(32, 2048), (32, 2080), (0, 2048), (0, 2112)])
def test_rows_on_both_sides_of_the_line_between_launches_that_overlap(group, n):
    """A kept residual: up to 16384 rows every launch of the chain may start early, above that the last ones."""
    from tests.gear_harness import Pair
    p = Pair(17, 1, 8, 8, 4, group, 2.0, 64, 4, n + 128)
    try:
        p.compress(n, 4)
        p.check_segment(0)
        p.oracle = p.with_stored_factors()
        p.check_attention(tol=1e-4)
    finally:
        p.close()


def test_residuals_of_zeros_and_of_rank_one():
    """Entries on the quantization grid leave no residual (factors zero); a column off the grid leaves a residual of rank
    one, of which a rank-4 fit must reproduce exactly that and invent nothing."""
    import torch
    from paper_2403_05527_b200 import binding as G
    from tests.gear_harness import Pair
    p = Pair(15, 1, 1, 1, 2, 64, 0.0, 64, 4, 1024)
    try:
        gen = np.random.default_rng(1)
        k16 = gen.permuted(np.tile(np.array([0.0, 1.0, 2.0, 3.0], np.float16), (1, 1, 256, 32)), axis=2)
        k16[0, 0, 2::3, 7] = 1.25
        k16[0, 0, 0::64], k16[0, 0, 1::64] = 0.0, 3.0        # every key group spans the grid exactly
        v16 = np.tile(np.arange(4, dtype=np.float16), (1, 1, 256, 32))
        b0 = gen.standard_normal((1, 1, 2, 128, 4)).astype(np.float32)
        p.oracle.compress(k16, v16, 4, b0)
        G.gear_compress(p.cache, None, torch.from_numpy(k16).cuda(), torch.from_numpy(v16).cuda(), 256, 4,
                        torch.from_numpy(b0).cuda())
        p.check_segment(0)
        ab = {s: G.gear_export(p.cache, 0, s + "_A_FP32", 1, 1)[0, 0] @ G.gear_export(p.cache, 0, s + "_B_FP32", 1, 1)[0, 0].T
              for s in "KV"}
        assert np.array_equal(ab["V"], np.zeros((256, 128)))
        assert np.array_equal(np.delete(ab["K"], 7, axis=1), np.zeros((256, 127)))
        # 22-bit operands and fp32 sums of at most 86 equal terms
        assert np.abs(ab["K"][:, 7] - np.where(k16[0, 0, :, 7] == 1.25, 0.25, 0.0)).max() <= 0.25 * 2.0 ** -20
    finally:
        p.close()


@pytest.mark.parametrize("rank", [2, 8, 16])
def test_tiles_whose_singular_values_span_decades(rank):
    """A few channels 60 times as large as the others: the factor columns differ so much in norm that R^T A0 is taken from
    the residual instead of from R^T R.  Two loops: each one squares the ratio of the directions, and past that the fp32
    iterates of Algorithm 2 hold nothing of the small ones.  (The oracle's bound on A B^T is relative to its largest
    entry; the last assertion looks at the small directions by themselves.)"""
    import torch
    from paper_2403_05527_b200 import binding as G
    from tests.gear_harness import Pair
    p = Pair(16, 1, 1, 1, 4, 64, 2.0, 64, 4, 1024, r_max=16, iters=2)
    try:
        gen = np.random.default_rng(rank)
        x = gen.standard_normal((1, 1, 320, 128))
        x[..., :rank // 2] *= 60.0
        k16, v16 = x.astype(np.float16), gen.standard_normal((1, 1, 320, 128)).astype(np.float16)
        b0 = gen.standard_normal((1, 1, 2, 128, rank)).astype(np.float32)
        p.oracle.compress(k16, v16, rank, b0)
        G.gear_compress(p.cache, None, torch.from_numpy(k16).cuda(), torch.from_numpy(v16).cuda(), 320, rank,
                        torch.from_numpy(b0).cuda())
        p.check_segment(0)
        a, b = (G.gear_export(p.cache, 0, w, 1, 1)[0, 0].astype(np.float64) for w in ("K_A_FP32", "K_B_FP32"))
        assert np.abs(a.T @ a - np.eye(rank)).max() <= 1e-5
        t = p.oracle.segments[0]["K"][0][0]
        got, ref = a @ b.T, t["A"] @ t["B"].T
        small = slice(rank // 2, 128)            # fp32 rounding of the large directions in B: 60^2 * 2^-22, a thousandth
        assert np.abs(got[:, small] - ref[:, small]).max() <= 5e-3 * np.abs(ref[:, small]).max()
    finally:
        p.close()


@pytest.mark.parametrize("batch,hkv,group,nb,rank", [
    (1, 2, 64, 256, 4),
    (2, 32, 64, 256, 4),
    (1, 9, 128, 1024, 16),
    (1, 3, 32, 160, 6),             # 160 tokens: the last 32-row block of a tile is its fifth
])
def test_flush_of_a_long_buffer(batch, hkv, group, nb, rank):
    """Buffers above 128 tokens are compressed like a prompt.  The workspace of that is not the cache's: what it holds does not
    depend on the rank that flushes use, but for the factors themselves."""
    import torch
    from paper_2403_05527_b200 import binding as G, synth
    from tests.gear_harness import Pair
    total = lambda r: alloc(G.make_config(batch, hkv, hkv, 4, group, 2.0, nb, r, 2 * nb, rank_max=16))   # noqa: E731

    def alloc(cfg):
        c = G.gear_create(cfg)
        n = G.gear_cache_bytes(c).alloc_total
        G.gear_free(c)
        return n
    assert total(rank) - total(0) <= batch * hkv * 3 * 2 * 128 * 16 * 2        # B of the flushed segments
    p = Pair(14, batch, hkv, hkv, 4, group, 2.0, nb, rank, 2 * nb)
    try:
        ks, vs = synth.make_appended(14, batch, hkv, 128, nb)
        b0 = synth.make_b0(14, batch, hkv, 128, rank)
        p.oracle.compress(np.stack(list(ks), 2), np.stack(list(vs), 2), rank, b0)
        kd, vd, b0d = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (ks, vs, b0))
        launches = []
        for i in range(nb):
            before = G.gear_kernel_launches()
            flushed = G.gear_append_buffer(p.cache, kd[i], vd[i], b0d)
            assert (flushed == G.GEAR_FLUSHED) == (i == nb - 1)
            launches.append(G.gear_kernel_launches() - before)
        assert set(launches[:-1]) == {1}
        # the push, two of Filter / Quant, three on R^T R, four or five after, the descriptor: not the one-launch path
        assert launches[-1] == (12 if rank > 8 else 11)
        torch.cuda.synchronize()
        p.check_segment(0)
        p.check_attention()
    finally:
        p.close()
