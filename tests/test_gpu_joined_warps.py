"""One query row per kv head and one or two blocks per warp: several warps of a unit share a CTA and join in shared memory.
Sizes around the edges of that split: one CTA per unit and several, warps without a block, warps with buffer slabs only,
ranges of two blocks, and the call after one that took the units' tickets."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,bits,group,s,rank,nb,n,pushed", [
    (1, 2, 64, 2.0, 4, 64, 64, 0),            # one block: nothing to join
    (1, 2, 64, 2.0, 4, 64, 64, 1),            # a block and a buffer slab
    (2, 4, 32, 1.0, 4, 64, 256, 63),          # twelve blocks, four of them buffer slabs: no join at this little work
    (3, 2, 64, 2.0, 2, 64, 512, 17),          # ten blocks in one CTA of ten warps
    (1, 2, 64, 2.0, 4, 64, 3072, 64 + 19),    # 51 blocks in seven CTAs of eight warps: five warps have none
    (1, 2, 64, 0.0, 0, 64, 2112, 5),          # 34 blocks in five CTAs of seven warps
    (1, 4, 32, 2.0, 4, 32, 1056, 32 + 7),     # groups of 32
    (1, 2, 0, 2.0, 4, 20, 2176, 20 + 3),      # per-vector lists, a block of 20 tokens
])
def test_against_the_oracle(H, bits, group, s, rank, nb, n, pushed):
    from tests.gear_harness import Pair
    p = Pair(19, 1, H, H, bits, group, s, nb, min(rank, nb), n + 256, r_max=rank, keep_fp32=False)
    try:
        p.compress(n, rank)
        if pushed:
            p.append(pushed)
        first = [p.check_attention(extra=i)[1] for i in range(3)]
        again = [p.check_attention(extra=i)[1] for i in range(3)]
        assert all(np.array_equal(a, b) for a, b in zip(first, again))
    finally:
        p.close()


@pytest.mark.parametrize("batch,H,n,pushed", [
    (1, 32, 2048, 19),      # 34 blocks per unit in six CTAs of six warps
    (2, 32, 768, 19),       # 14 blocks in one CTA
    (8, 32, 512, 19),       # ten blocks, ranges of two, one CTA
    (2, 32, 4096, 19),      # 66 blocks, ranges of two, nine CTAs
    (4, 40, 512, 19),       # more units than SMs
])
def test_many_units_against_the_kernel_of_several_rows(batch, H, n, pushed):
    """The same query twice goes through the kernel of several rows per kv head, which cuts and joins in its own way."""
    import torch
    from paper_2403_05527_b200 import binding as G
    gen = torch.Generator(device="cuda").manual_seed(n)
    draw = lambda *shape: torch.randn(shape, generator=gen, device="cuda").half()   # noqa: E731
    cfg = G.make_config(batch, H, H, 2, 64, 2.0, 64, 4, n + 64, seed=1, max_queries=2)
    cache = G.gear_compress(None, cfg, draw(batch, H, n, 128), draw(batch, H, n, 128), n, 4)
    try:
        for _ in range(pushed):
            G.gear_append_buffer(cache, draw(batch, H, 128), draw(batch, H, 128))
        for _ in range(3):
            q = draw(batch, H, 128)
            got, twice = torch.full(q.shape, float("nan"), device="cuda"), torch.empty((batch, H, 2, 128), device="cuda")
            G.gear_decode_attn(cache, q, got)
            G.gear_decode_attn_multi(cache, q[:, :, None].expand(-1, -1, 2, -1).contiguous(), twice, 2)
            err = (got - twice[:, :, 0]).abs().amax(-1) / twice[:, :, 0].abs().amax(-1)
            assert err.max().item() <= 8e-5          # twice what a kernel's own arithmetic may be off
        assert G.gear_last_device_status(cache) == 0
    finally:
        G.gear_free(cache)
