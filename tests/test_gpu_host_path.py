"""Host-buffer calls: pinned destinations are written by the attention kernel, pageable or unaligned ones through a copy,
and the rows go through a ring of four pinned slots that caches hand on to one another.  The oracle is the same sequence
through device buffers: the kernels are the same, so the results are equal bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _rows(torch, steps, B, H, Hq):
    gen = torch.Generator().manual_seed(3)
    draw = lambda heads: torch.randn((steps, B, heads, 128), generator=gen).half()   # noqa: E731
    return draw(H), draw(H), draw(Hq)


def _cache(torch, G, B, Hq, H, nb):
    gen = torch.Generator().manual_seed(4)
    k, v = (torch.randn((B, H, 128, 128), generator=gen).half().cuda() for _ in range(2))
    cfg = G.make_config(B, Hq, H, 2, 64, 2.0, nb, 4, 512, seed=1)
    return G.gear_compress(None, cfg, k, v, 128, 4)


@pytest.mark.parametrize("where", ["pinned", "pageable", "unaligned"])
@pytest.mark.parametrize("B,Hq,H,nb", [(1, 1, 1, 16), (3, 8, 2, 64), (2, 5, 5, 16)])
def test_steps_queued_beyond_the_ring_match_the_device_calls(where, B, Hq, H, nb):
    import torch
    from paper_2403_05527_b200 import binding as G

    steps = 2 * nb + 5                                   # two flushes; many more calls than slots before the one wait
    k, v, q = _rows(torch, steps, B, H, Hq)
    ref = _cache(torch, G, B, Hq, H, nb)
    want = torch.empty((steps, B, Hq, 128), device="cuda")
    for i in range(steps):
        G.gear_append_buffer(ref, k[i].cuda(), v[i].cuda())
        G.gear_decode_attn(ref, q[i].cuda(), want[i])
    for round_ in range(2):                              # the second cache takes over the first one's pinned rows
        cache = _cache(torch, G, B, Hq, H, nb)
        if where == "unaligned":
            flat = torch.empty(steps * B * Hq * 128 + 1, dtype=torch.float32).pin_memory()
            out = flat[1:].view(steps, B, Hq, 128)
        else:
            out = torch.empty((steps, B, Hq, 128), dtype=torch.float32)
            out = out.pin_memory() if where == "pinned" else out
        scratch_k, scratch_v, scratch_q = (np.empty(t[0].shape, np.float16) for t in (k, v, q))
        for i in range(steps):
            scratch_k[:], scratch_v[:], scratch_q[:] = k[i].numpy(), v[i].numpy(), q[i].numpy()
            if i % 3 == 2:                               # the two calls that a step combines
                G.gear_append_buffer_host(cache, scratch_k, scratch_v)
                G.gear_decode_attn_host(cache, scratch_q, out[i])
            else:
                G.gear_step_host(cache, scratch_k, scratch_v, scratch_q, out[i])
            scratch_k.fill(np.nan), scratch_v.fill(np.nan), scratch_q.fill(np.nan)       # free to be reused on return
        G.gear_cache_wait(cache)
        assert torch.equal(out, want.cpu()), round_
        G.gear_free(cache)
    G.gear_free(ref)
    G.gear_release_workspace()


def test_steps_captured_into_a_graph_match_the_eager_calls():
    """Pushes and attentions of two caches captured token after token: what may be read ahead of the kernel in front is decided
    inside the capture, and the replay gives the bits of the same calls made one by one, flushes among them."""
    import torch
    from paper_2403_05527_b200 import binding as G

    B, Hq, H, nb, steps = 2, 8, 4, 16, 20
    k, v, q = (t.cuda() for t in _rows(torch, steps, B, H, Hq))
    eager, graphed = ([_cache(torch, G, B, Hq, H, nb) for _ in range(2)] for _ in range(2))
    want, got = (torch.full((steps, 2, B, Hq, 128), float("nan"), device="cuda") for _ in range(2))

    def run(caches, out):
        for i in range(steps):
            for j, c in enumerate(caches):
                G.gear_append_buffer(c, k[i], v[i])
                G.gear_decode_attn(c, q[i], out[i, j])
            for j, c in enumerate(caches):               # each behind a call on the other cache
                G.gear_decode_attn(c, q[i], out[i, j])

    run(eager, want)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run(graphed, got)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(got, want)
    # and the caches go on outside the graph
    a, b = torch.empty((B, Hq, 128), device="cuda"), torch.empty((B, Hq, 128), device="cuda")
    for c, out in ((eager[0], a), (graphed[0], b)):
        G.gear_append_buffer(c, k[0], v[0])
        G.gear_decode_attn(c, q[0], out)
    torch.cuda.synchronize()
    assert torch.equal(a, b) and all(G.gear_last_device_status(c) == 0 for c in eager + graphed)
    del graph
    for c in eager + graphed:
        G.gear_free(c)
