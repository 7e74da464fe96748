"""Quantization of groups of 64 and 128 by CTAs that take one block after the other: more blocks than the device holds
CTAs for, a single block, and values that lie half way between two codes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,group,H,n,rank", [
    (2, 64, 11, 4096, 1),      # 704 blocks per side
    (4, 64, 11, 4096, 0),      # the same without a residual
    (4, 128, 6, 16384, 1),     # 768 blocks per side
    (2, 128, 1, 128, 1),       # one block
    (4, 64, 1, 64, 1),
])
def test_blocks_and_ties(bits, group, H, n, rank):
    """A grid of 1.5 under a step of 3: x / 3 is not exact in binary32, and the rounded product is half way between two codes
    where the exact one is not.  Codes, scales and outliers have to be the oracle's bit for bit."""
    import torch
    from paper_2403_05527_b200 import binding as G, synth
    from tests.gear_harness import Pair
    p = Pair(16, 1, H, H, bits, group, 2.0, 64, 1, n + 128, r_max=1, iters=1)
    try:
        top = 3 * (2 ** bits - 1)
        gen = np.random.default_rng(n + bits)
        k16, v16 = ((gen.integers(0, 2 * top // 3 + 1, (1, H, n, 128)) * 1.5).astype(np.float16) for _ in range(2))
        for x in (k16.reshape(1, H, n // group, group, 128).swapaxes(3, 4), v16.reshape(1, H, n, 128 // group, group)):
            x[..., :3], x[..., 3:6] = 0.0, float(top)       # the group spans 0 .. top also without its outliers
        b0 = synth.make_b0(16, 1, H, 128, rank)
        p.oracle.compress(k16, v16, rank, b0)
        G.gear_compress(p.cache, None, torch.from_numpy(k16).cuda(), torch.from_numpy(v16).cuda(), n, rank,
                        torch.from_numpy(np.ascontiguousarray(b0)).cuda() if rank else None)
        torch.cuda.synchronize()
        p.check_segment(0)
    finally:
        p.close()
