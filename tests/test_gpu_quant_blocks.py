"""Quantization of groups of 32, 64 and 128 by CTAs that take one block after the other: more blocks than the device holds
CTAs for, few blocks, and values that lie half way between two codes.  Segments of more than 128 tokens: shorter ones are
compressed by another kernel, in one launch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,group,s_pct,H,n,rank", [
    (2, 64, 2.0, 11, 4096, 1),      # one outlier per side and group; 704 blocks per side
    (4, 64, 2.0, 11, 4096, 0),      # the same without a residual
    (4, 128, 2.0, 6, 16384, 1),     # two outliers; 768 blocks per side
    (2, 128, 2.0, 1, 256, 1),       # few blocks
    (4, 64, 2.0, 1, 192, 1),
    (2, 64, 0.0, 3, 1024, 1),       # no outliers
    (4, 32, 2.0, 13, 4096, 1),      # groups of 32; 1664 blocks per side
    (2, 32, 0.0, 1, 160, 1),
    (2, 128, 1.0, 2, 1024, 1),      # groups of 128 with one outlier
    (4, 128, 0.0, 5, 512, 1),
])
def test_blocks_and_ties(bits, group, s_pct, H, n, rank):
    """A grid of 1.5 under a step of 3: x / 3 is not exact in binary32, and the rounded product is half way between two codes
    where the exact one is not.  Codes, scales and outliers have to be the oracle's bit for bit."""
    import torch
    from paper_2403_05527_b200 import binding as G, synth
    from tests.gear_harness import Pair
    p = Pair(16, 1, H, H, bits, group, s_pct, 64, 1, n + 128, r_max=1, iters=1)
    try:
        top = 3 * (2 ** bits - 1)
        gen = np.random.default_rng(n + bits)
        k16, v16 = ((gen.integers(0, 2 * top // 3 + 1, (1, H, n, 128)) * 1.5).astype(np.float16) for _ in range(2))
        for x in (k16.reshape(1, H, n // group, group, 128).swapaxes(3, 4), v16.reshape(1, H, n, 128 // group, group)):
            x[..., :3], x[..., 3:6] = 0.0, float(top)       # the group spans 0 .. top also without its outliers
        b0 = synth.make_b0(16, 1, H, 128, rank)
        p.oracle.compress(k16, v16, rank, b0)
        before = G.gear_kernel_launches()
        G.gear_compress(p.cache, None, torch.from_numpy(k16).cuda(), torch.from_numpy(v16).cuda(), n, rank,
                        torch.from_numpy(np.ascontiguousarray(b0)).cuda() if rank else None)
        assert G.gear_kernel_launches() - before == (10 if rank else 3)      # a launch per side, seven for the rank, the descriptor
        torch.cuda.synchronize()
        p.check_segment(0)
    finally:
        p.close()


@pytest.mark.parametrize("s_pct", [0.0, 1.0])
@pytest.mark.parametrize("kind", ["equal", "one peak"])
def test_flat_groups(kind, s_pct):
    """Groups whose entries are all equal (the bottom outlier is the next index), or equal but for one on each side."""
    import torch
    from paper_2403_05527_b200 import binding as G
    from tests.gear_harness import Pair
    for group in (32, 64, 128):
        p = Pair(16, 1, 1, 1, 2, group, s_pct, 64, 0, 512)
        try:
            n = 256                                       # more than 128: a launch per side and the descriptor
            x = np.full((1, 1, n, 128), 1.25, np.float16)
            if kind == "one peak":
                x[0, 0, 5::group, :] = 9.0
                x[0, 0, :, 7::group] = -9.0
            p.oracle.compress(x, x, 0, np.zeros((1, 1, 2, 128, 0), np.float32))
            xd = torch.from_numpy(x).cuda()
            before = G.gear_kernel_launches()
            G.gear_compress(p.cache, None, xd, xd, n, 0, None)
            assert G.gear_kernel_launches() - before == 3
            torch.cuda.synchronize()
            p.check_segment(0)
        finally:
            p.close()


@pytest.mark.parametrize("bits,group,s_pct", [(2, 64, 2.0), (4, 64, 0.0), (4, 32, 2.0), (2, 32, 0.0), (2, 128, 2.0), (4, 128, 1.0),
                                              (2, 128, 0.0), (4, 0, 2.0)])
def test_equal_inputs_give_equal_bytes_time_after_time(bits, group, s_pct):
    """A block's bytes in shared memory make room for the next block's while threads still work on what they have loaded: with
    thousands of blocks, and the store pipe full of residuals, every byte of the records is the same each time."""
    import torch
    from paper_2403_05527_b200 import binding as G
    H, n = 256, 1024
    gen = torch.Generator(device="cuda").manual_seed(group)
    k, v = (torch.randn((1, H, n, 128), generator=gen, device="cuda").half() for _ in range(2))
    held = {}

    def alloc(nbytes, _ctx):
        t = torch.zeros(max(int(nbytes), 1), dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    def free(ptr, _ctx):
        del held[ptr]

    a_cb, f_cb = G.ALLOC_FN(alloc), G.FREE_FN(free)
    cfg = G.make_config(1, H, H, bits, group, s_pct, 64 if group else 20, 4, n + 128, seed=1)
    first = None
    G.gear_set_allocator(a_cb, f_cb)
    try:
        for i in range(30):
            cache = G.gear_compress(None, cfg, k, v, n, 4)
            torch.cuda.synchronize()
            arena = max(held.values(), key=lambda t: t.numel())
            if first is None:
                first = arena.clone()
            assert torch.equal(arena, first), i
            del arena
            G.gear_free(cache)
    finally:
        G.gear_set_allocator(None, None)
