"""Prompts whose residual is not kept: R^T R summed while the blocks are quantized, A0 = R b from the codes.  Residuals that grow past
the range that the sums were scaled for, blocks without a residual, ranges that end inside tiles, chunks that end early.
A CTA's range is one block where there are no more blocks than SMs, so what happens between the blocks of a range takes heads."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _compress(p, k16, v16, rank, seed):
    import torch
    from paper_2403_05527_b200 import binding as G
    B, H, n = k16.shape[:3]
    b0 = np.random.default_rng(seed).standard_normal((B, H, 2, 128, rank)).astype(np.float32)
    p.oracle.compress(k16, v16, rank, b0)
    G.gear_compress(p.cache, None, torch.from_numpy(k16).cuda(), torch.from_numpy(v16).cuda(), n, rank, torch.from_numpy(b0).cuda())
    torch.cuda.synchronize()
    assert G.gear_last_device_status(p.cache) == 0
    p.check_segment(0)


def _blocks_per_range(group, blocks):
    """Of the CTAs that sum `blocks` blocks of a side, at least: a block each up to one per SM, above that two of 64 tokens or one of
    128, and never more CTAs than four (two) per SM."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per = 2 if group == 64 and blocks > sms else 1
    return blocks // min(-(-blocks // per), (4 if group == 64 else 2) * sms)


@pytest.mark.parametrize("bits,group,s_pct,B,H,n,rank", [
    (2, 64, 2.0, 1, 1, 192, 4),     # the shortest: three ranges per side
    (4, 64, 2.0, 1, 3, 704, 8),     # eleven blocks a tile, a range each; the second chunk of rows is short
    (2, 64, 0.0, 2, 2, 576, 16),    # no outliers, sixteen columns
    (4, 64, 0.0, 1, 2, 1024, 1),
    (4, 64, 3.0, 1, 40, 320, 2),
    (2, 128, 2.0, 1, 1, 256, 4),    # two outliers per side: two blocks
    (4, 128, 2.0, 1, 5, 1152, 8),   # nine blocks a tile
    (2, 128, 1.0, 1, 2, 640, 2),    # one outlier
    (4, 128, 1.0, 1, 30, 384, 16),
    (2, 128, 0.0, 1, 3, 384, 5),
    (2, 64, 2.0, 1, 72, 1088, 4),   # 17 blocks a tile and two to three a range: ranges end inside tiles
    (4, 128, 2.0, 1, 72, 1152, 2),  # nine blocks a tile
])
def test_group_shapes(bits, group, s_pct, B, H, n, rank):
    from paper_2403_05527_b200 import synth
    from tests.gear_harness import Pair
    assert H < 72 or _blocks_per_range(group, H * n // group) >= 2
    p = Pair(31, B, H, H, bits, group, s_pct, 64, min(rank, 4), n + 128, r_max=rank)
    try:
        k16, v16 = synth.make_kv(31, B, H, n, 128)
        _compress(p, k16, v16, rank, n)
        # on the factors as stored: fp16 storage moves the attention over short prompts by up to 2e-3, the kernels' arithmetic by less than 1e-4
        p.oracle = p.with_stored_factors()
        p.check_attention(tol=1e-4)
    finally:
        p.close()


@pytest.mark.parametrize("bits,group,s_pct,H", [(2, 64, 2.0, 1), (4, 128, 2.0, 1), (2, 128, 1.0, 1), (4, 64, 0.0, 1),
                                                (4, 64, 2.0, 40), (2, 128, 2.0, 160)])
def test_flat_groups_among_others(bits, group, s_pct, H):
    """Groups whose entries are all equal, equal but for one, two or three, or equal on two levels: the sides of the filter share
    candidates there, and what they clear has to stay out of the sums."""
    from tests.gear_harness import Pair
    assert H == 1 or _blocks_per_range(group, H * 512 // group) >= 2      # flat blocks and others in one range
    p = Pair(33, 1, H, H, bits, group, s_pct, 64, 2, 1024, r_max=2)
    try:
        gen = np.random.default_rng(group + bits)
        x = gen.standard_normal((2, 1, H, 512, 128)).astype(np.float16)
        x[:, 0, :, :group] = 1.25                           # whole blocks of keys, whole groups of values
        x[:, 0, :, group:2 * group] = 0.5
        for at in range(group, 2 * group, 9):               # one to three other entries in a key's and a value's group
            for e in range(1 + at % 3):
                x[:, 0, :, group + (at * 5 + 11 * e) % group, (at * 7) % 128] = gen.standard_normal()
                x[:, 0, :, at, (at * 3 + 17 * e) % 128] = gen.standard_normal()
        x[:, 0, :, 2 * group:2 * group + 64, ::2] = -3.0    # two levels
        x[:, 0, :, 2 * group:2 * group + 64, 1::2] = 3.0
        _compress(p, x[0], x[1], 2, 3)
    finally:
        p.close()


@pytest.mark.parametrize("first", [2.0 ** -10, 0.0])
@pytest.mark.parametrize("bits,group,H,n", [(2, 64, 2, 1088), (4, 64, 2, 1088), (2, 64, 72, 1088), (4, 64, 72, 1088),
                                            (2, 128, 72, 1152), (4, 128, 72, 1152)])
def test_residuals_that_grow(bits, group, H, n, first):
    """Of every four blocks the first, then the second are smaller than the rest by factors that fp16 does not span (with `first` zero:
    without any residual).  Two heads: a range per block, each with a scale of its own.  72 heads: 17 or nine blocks a tile in
    ranges of two or three, several hundred of which grow by 13 or 17 bits behind a block with sums, so that these are scaled
    again (by a warp's 128 columns or by 64), or begin with a block that leaves nothing."""
    from tests.gear_harness import Pair
    assert H == 2 or _blocks_per_range(group, H * n // group) >= 2
    p = Pair(32, 1, H, H, bits, group, 2.0, 64, 4, 2048, r_max=4)
    try:
        gen = np.random.default_rng(bits)
        x = gen.standard_normal((2, 1, H, n, 128)) * np.exp(gen.standard_normal((2, 1, H, 1, 128)))
        for start in range(0, n, 4 * group):                # whatever range a block belongs to: small ones ahead of large ones
            x[..., start:start + group, :] *= first
            x[..., start + group:start + 2 * group, :] *= 2.0 ** -6
            x[..., start + 2 * group:start + 4 * group, :] *= 2.0 ** 7
        k16, v16 = np.clip(x, -6e4, 6e4).astype(np.float16) + np.float16(0)      # no negative zeros: either may be the zero point
        _compress(p, k16, v16, 4, 7)
    finally:
        p.close()


@pytest.mark.parametrize("group,s_pct,H,blocks", [(64, 2.0, 5, 34), (64, 0.0, 5, 34), (128, 2.0, 38, 16), (128, 0.0, 38, 16)])
def test_steps_that_are_subnormal_behind_blocks_of_equal_entries(group, s_pct, H, blocks):
    """A range of 16 to 22 units of 2^-24 has a step of one unit at 4 bits, so that the top entries lie up to seven steps beyond the
    last code; the blocks in front of such blocks have no residual, so that the sums are scaled for the rounding of their zero
    point alone, 2^-35.  fp16 does not span the two."""
    import torch
    from paper_2403_05527_b200 import binding as G
    from tests.gear_harness import Pair, rel_max
    n = group * blocks
    assert _blocks_per_range(group, H * blocks) >= 2
    p = Pair(34, 1, H, H, 4, group, s_pct, 64, 0, n + 128, r_max=4)
    try:
        gen = np.random.default_rng(group)
        top = gen.integers(16, 23, (2, 1, H, blocks // 2, 1, 1))
        x = gen.integers(0, top + 1, (2, 1, H, blocks // 2, group, 128))
        x[0][..., :3, :], x[0][..., 3:6, :] = 0, top[0]                 # three of either end in every group: two leave it at most
        values = x[1].reshape(1, H, blocks // 2, group, 128 // group, group)
        values[..., :3], values[..., 3:6] = 0, top[1][..., None]
        flat = np.zeros_like(x)
        units = 1500 + np.stack([flat, x], 4).reshape(2, 1, H, n, 128)  # all of them below 2^-13: spaced 2^-24
        k16, v16 = (units * 2.0 ** -24).astype(np.float16)
        b0 = gen.standard_normal((1, H, 2, 128, 4)).astype(np.float32)
        p.oracle.compress(k16, v16, 4, b0)
        G.gear_compress(p.cache, None, torch.from_numpy(k16).cuda(), torch.from_numpy(v16).cuda(), n, 4, torch.from_numpy(b0).cuda())
        torch.cuda.synchronize()
        assert G.gear_last_device_status(p.cache) == 0
        p.check_segment(0, tol=1.0)     # codes, scales, outliers; the factors as stored are themselves of a few units of fp16
        for side in "KV":
            a, b = (G.gear_export(p.cache, 0, f"{side}_{w}_FP32", 1, H)[0].astype(np.float64) for w in "AB")
            for h in range(H):
                t = p.oracle.segments[0][side][0][h]
                assert rel_max(a[h] @ b[h].T, t["A"] @ t["B"].T) <= 1e-3
        p.oracle = p.with_stored_factors()
        p.check_attention(tol=1e-4)
    finally:
        p.close()
