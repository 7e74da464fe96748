"""The code path the benchmark times: start vectors of Algorithm 2 drawn by the library from cfg.seed (B0 = NULL),
buffer flushes through the host-buffer entry point, and bitwise reproducibility from run to run.

With a library-drawn start there is no oracle factor pair to compare with (the draw is the library's own), so the
factors are checked against what Algorithm 2 guarantees for ANY start: A has orthonormal columns, B = R^T A, hence
A B^T is the orthogonal projection of R onto range(A) and ||R - A B^T||_F^2 = ||R||_F^2 - ||B||_F^2; the error can
not beat the Eckart-Young bound of a brute-force SVD and, after three loops from a Gaussian start, stays close to
what the oracle reaches from a Gaussian start of its own.  R is the oracle's residual; codes, scales, zero-points
and outliers (which do not depend on the start) are compared bit for bit first, so both sides hold the same R.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _export_all(G, cache, si, B, H):
    return {w: G.gear_export(cache, si, w, B, H) for w in
            ("K_CODES", "V_CODES", "K_SCALE", "V_SCALE", "K_ZERO", "V_ZERO", "K_OUT_IDX", "V_OUT_IDX", "K_OUT_VAL",
             "V_OUT_VAL", "K_A_FP32", "V_A_FP32", "K_B_FP32", "V_B_FP32", "K_A", "V_A", "K_B", "V_B")}


def _build(G, torch, cfg, k16, v16, ks, vs, n, rank):
    dev = torch.device("cuda:0")
    cache = G.gear_compress(None, cfg, torch.from_numpy(k16).to(dev), torch.from_numpy(v16).to(dev), n, rank, None)
    flushed = 0
    for i in range(ks.shape[0]):
        flushed += G.gear_append_buffer(cache, torch.from_numpy(ks[i]).to(dev), torch.from_numpy(vs[i]).to(dev), None) \
            == G.GEAR_FLUSHED
    torch.cuda.synchronize()
    return cache, flushed


@pytest.mark.parametrize("bits,group,rank,n", [(2, 64, 4, 256), (4, 64, 8, 192)])
def test_library_drawn_start_vectors_satisfy_algorithm_2(bits, group, rank, n):
    import torch
    from oracle import gear_oracle as O
    from paper_2403_05527_b200 import binding as G, synth

    B, H, nb = 2, 2, 64
    k16, v16 = synth.make_kv(2, B, H, n, 128, extra=31)
    ks, vs = synth.make_appended(2, B, H, 128, nb + 3)            # one flush, three tokens left in the buffer
    caches, exports = [], []
    try:
        for seed in (11, 11, 12):
            cfg = G.make_config(B, H, H, bits, group, 2.0, nb, rank, n + 4 * nb, rank_max=rank, seed=seed,
                                flags=G.GEAR_FLAG_KEEP_FP32_FACTORS)
            cache, flushed = _build(G, torch, cfg, k16, v16, ks, vs, n, rank)
            caches.append(cache)
            assert flushed == 1
            exports.append([_export_all(G, cache, si, B, H) for si in range(2)])

        # same seed: the same bits everywhere; another seed: other factors, same codes
        for si in range(2):
            for w, arr in exports[0][si].items():
                assert np.array_equal(arr.view(np.uint8), exports[1][si][w].view(np.uint8)), (si, w)
                if w.endswith("_FP32"):
                    assert not np.array_equal(arr, exports[2][si][w]), (si, w, "seed does not reach the start vectors")
                elif "_A" not in w and "_B" not in w:
                    assert np.array_equal(arr.view(np.uint8), exports[2][si][w].view(np.uint8)), (si, w)

        # the oracle on the same inputs: prefill segment (long-segment kernels), then the flushed buffer (tile kernel)
        ref = O.OracleCache(B, H, H, 128, bits, group, 2.0, nb, rank, 3)
        own = np.random.default_rng(5).standard_normal((B, H, 2, 128, rank)).astype(np.float32)
        ref.compress(k16, v16, rank, own)
        for i in range(nb + 3):
            ref.append(ks[i], vs[i], own)
        for si in range(2):
            ex = exports[0][si]
            for side in ("K", "V"):
                for b in range(B):
                    for h in range(H):
                        t = ref.segments[si][side][b][h]
                        assert np.array_equal(ex[f"{side}_CODES"][b, h], t["codes"])
                        assert np.array_equal(ex[f"{side}_SCALE"][b, h].view(np.uint16), t["scale"].view(np.uint16))
                        assert np.array_equal(ex[f"{side}_ZERO"][b, h].view(np.uint16), t["zero"].view(np.uint16))
                        assert np.array_equal(ex[f"{side}_OUT_IDX"][b, h].reshape(t["out_idx"].shape), t["out_idx"])
                        R = t["R"]
                        A = ex[f"{side}_A_FP32"][b, h].astype(np.float64)
                        Bm = ex[f"{side}_B_FP32"][b, h].astype(np.float64)
                        where = f"segment {si} {side} b{b} h{h}"
                        assert np.isfinite(A).all() and np.isfinite(Bm).all(), where
                        assert np.abs(A.T @ A - np.eye(rank)).max() <= 1e-4, where + ": A^T A != I"
                        want_b = R.T @ A
                        assert np.abs(Bm - want_b).max() <= 1e-4 * np.abs(want_b).max(), where + ": B != R^T A"
                        r2 = (R ** 2).sum()
                        err2 = ((R - A @ Bm.T) ** 2).sum()
                        assert abs(err2 - (r2 - (Bm ** 2).sum())) <= 1e-4 * r2, where + ": not a projection of R"
                        sv = np.linalg.svd(R, compute_uv=False)
                        bound2 = (sv[rank:] ** 2).sum()
                        assert err2 >= bound2 * (1 - 1e-6), where + ": beats the Eckart-Young bound"
                        ref_err2 = ((R - t["A"] @ t["B"].T) ** 2).sum()
                        assert err2 <= 1.5 ** 2 * ref_err2, where + f": {err2 ** 0.5:.4g} vs oracle {ref_err2 ** 0.5:.4g}"
                        # the fp16 factors the decode kernel reads are the rounded fp32 ones
                        got16 = ex[f"{side}_A"][b, h].astype(np.float64) @ ex[f"{side}_B"][b, h].astype(np.float64).T
                        den = np.abs(A @ Bm.T).max()
                        assert np.abs(got16 - A @ Bm.T).max() <= 2e-3 * den, where
    finally:
        for c in caches:
            G.gear_free(c)


def test_decode_over_library_drawn_factors_matches_attention_over_the_exported_pieces():
    """Attention over a cache whose low-rank part came from library-drawn start vectors: the float64 reference
    attention is taken over K^ = D^ + A B^T + S assembled from the oracle's D^, S (bit-exact with the library's) and
    the library's own exported fp16 factors."""
    import torch
    from oracle import gear_oracle as O
    from paper_2403_05527_b200 import binding as G, synth

    B, Hq, H, n, nb, rank, bits, group = 1, 4, 2, 192, 64, 4, 2, 64
    k16, v16 = synth.make_kv(2, B, H, n, 128, extra=41)
    ks, vs = synth.make_appended(2, B, H, 128, nb + 9)
    cfg = G.make_config(B, Hq, H, bits, group, 2.0, nb, rank, n + 4 * nb, rank_max=rank, seed=77)
    cache, _ = _build(G, torch, cfg, k16, v16, ks, vs, n, rank)
    try:
        ref = O.OracleCache(B, Hq, H, 128, bits, group, 2.0, nb, 0, 3)      # rank 0: D^ and S only
        ref.compress(k16, v16, 0, None)
        for i in range(nb + 9):
            ref.append(ks[i], vs[i], None)
        q = synth.make_query(2, B, Hq, 128, extra=41)
        dev = torch.device("cuda:0")
        out = torch.full((B, Hq, 128), float("nan"), dtype=torch.float32, device=dev)
        G.gear_decode_attn(cache, torch.from_numpy(q).to(dev), out)
        torch.cuda.synchronize()
        assert G.gear_last_device_status(cache) == 0
        got = out.cpu().numpy().astype(np.float64)
        for b in range(B):
            for hk in range(H):
                ks_, vs_ = [], []
                for si in range(2):
                    for side, dst in (("K", ks_), ("V", vs_)):
                        t = ref.segments[si][side][b][hk]
                        a = G.gear_export(cache, si, f"{side}_A", B, H)[b, hk].astype(np.float64)
                        bm = G.gear_export(cache, si, f"{side}_B", B, H)[b, hk].astype(np.float64)
                        dst.append(t["D"] + t["S"] + a @ bm.T)
                ks_.append(ref.buf_k[b, hk].astype(np.float64))
                vs_.append(ref.buf_v[b, hk].astype(np.float64))
                k_hat, v_hat = np.concatenate(ks_), np.concatenate(vs_)
                for hq in range(hk * 2, hk * 2 + 2):
                    want = O.attention_one(q[b, hq].astype(np.float64), k_hat, v_hat, 1.0 / np.sqrt(128.0))
                    assert np.abs(got[b, hq] - want).max() / np.abs(want).max() <= 1e-3
    finally:
        G.gear_free(cache)


@pytest.mark.parametrize("with_b0", [True, False])
def test_host_buffer_append_through_a_flush(with_b0):
    """gear_append_buffer_host across a full buffer: the flush it triggers (with the start vectors given in host
    memory, or drawn by the library) and the attention after it, against the oracle."""
    import torch
    from oracle import gear_oracle as O
    from paper_2403_05527_b200 import binding as G, synth

    B, H, n, nb, rank = 2, 2, 128, 32, 2
    k16, v16 = synth.make_kv(2, B, H, n, 128, extra=51)
    b0 = synth.make_b0(2, B, H, 128, rank, extra=51)
    ks, vs = synth.make_appended(2, B, H, 128, nb + 5)
    fb0 = synth.make_b0(2, B, H, 128, rank, extra=52)
    cfg = G.make_config(B, H, H, 4, 32, 4.0, nb, rank, 512, rank_max=rank, seed=3)
    dev = torch.device("cuda:0")
    cache = G.gear_compress(None, cfg, torch.from_numpy(k16).to(dev), torch.from_numpy(v16).to(dev), n, rank,
                            torch.from_numpy(b0).to(dev))
    try:
        ref = O.OracleCache(B, H, H, 128, 4, 32, 4.0, nb, rank, 3)
        ref.compress(k16, v16, rank, b0)
        flushed = 0
        for i in range(nb + 5):
            ref.append(ks[i], vs[i], fb0)
            flushed += G.gear_append_buffer_host(cache, ks[i], vs[i], fb0 if with_b0 else None) == G.GEAR_FLUSHED
        assert flushed == 1
        info = G.gear_cache_info(cache)
        assert (info.n_segments, info.buffer_len, info.n_compressed) == (2, 5, n + nb)
        for side in ("K", "V"):
            codes = G.gear_export(cache, 1, f"{side}_CODES", B, H)
            a = G.gear_export(cache, 1, f"{side}_A", B, H).astype(np.float64)
            bm = G.gear_export(cache, 1, f"{side}_B", B, H).astype(np.float64)
            for b in range(B):
                for h in range(H):
                    t = ref.segments[1][side][b][h]
                    assert np.array_equal(codes[b, h], t["codes"])
                    if with_b0:
                        want = t["A"] @ t["B"].T
                        assert np.abs(a[b, h] @ bm[b, h].T - want).max() <= 1e-3 * np.abs(want).max()
        if with_b0:
            q = synth.make_query(2, B, H, 128, extra=51)
            out = np.zeros((B, H, 128), np.float32)
            G.gear_decode_attn_host(cache, q, out)
            want = ref.decode_attn(q)
            for b in range(B):
                for h in range(H):
                    assert np.abs(out[b, h] - want[b, h]).max() / np.abs(want[b, h]).max() <= 1e-3
    finally:
        G.gear_free(cache)


def test_same_inputs_give_the_same_bits_from_run_to_run():
    """Compress + flush + attention twice from scratch on the same inputs: every exported piece and the attention
    output are bit-identical (reductions run in a fixed order; the sparse terms are summed in fixed point)."""
    import torch
    from paper_2403_05527_b200 import binding as G, synth

    B, Hq, H, n, nb, rank = 2, 8, 2, 384, 64, 4
    k16, v16 = synth.make_kv(4, B, H, n, 128, extra=61)
    b0 = synth.make_b0(4, B, H, 128, rank, extra=61)
    ks, vs = synth.make_appended(4, B, H, 128, nb + 21)
    q = synth.make_query(4, B, Hq, 128, extra=61)
    dev = torch.device("cuda:0")
    runs = []
    for _ in range(2):
        cfg = G.make_config(B, Hq, H, 2, 128, 2.0, nb, rank, 1024, rank_max=rank, seed=9)
        cache = G.gear_compress(None, cfg, torch.from_numpy(k16).to(dev), torch.from_numpy(v16).to(dev), n, rank,
                                torch.from_numpy(b0).to(dev))
        try:
            for i in range(nb + 21):
                G.gear_append_buffer(cache, torch.from_numpy(ks[i]).to(dev), torch.from_numpy(vs[i]).to(dev), None)
            outs = []
            for _rep in range(3):
                out = torch.full((B, Hq, 128), float("nan"), dtype=torch.float32, device=dev)
                G.gear_decode_attn(cache, torch.from_numpy(q).to(dev), out)
                torch.cuda.synchronize()
                outs.append(out.cpu().numpy())
            assert G.gear_last_device_status(cache) == 0
            pieces = {(si, w): G.gear_export(cache, si, w, B, H) for si in range(2)
                      for w in ("K_CODES", "V_CODES", "K_A", "V_A", "K_B", "V_B", "K_OUT_VAL", "V_OUT_IDX")}
            runs.append((outs, pieces))
        finally:
            G.gear_free(cache)
    for rep in range(3):
        assert np.array_equal(runs[0][0][0].view(np.uint32), runs[0][0][rep].view(np.uint32)), "repeat calls differ"
        assert np.array_equal(runs[0][0][rep].view(np.uint32), runs[1][0][rep].view(np.uint32)), "runs differ"
    for key, arr in runs[0][1].items():
        assert np.array_equal(arr.view(np.uint8), runs[1][1][key].view(np.uint8)), key


def test_equal_inputs_give_equal_arenas():
    """Every byte of the compressed caches, the block headers among them (largest outlier delta and scale of a block,
    maxima over a CTA's warps in shared memory, which gear_export does not show), is the same from run to run."""
    import torch
    from paper_2403_05527_b200 import binding as G, synth

    dev = torch.device("cuda:0")
    w = synth.WORKLOADS[2]
    gen = torch.Generator(device=dev)
    gen.manual_seed(5)
    k, v = (torch.randn((w.batch, w.n_kv_heads, w.n, 128), generator=gen, device=dev).half() for _ in range(2))
    held = {}

    def alloc(nbytes, _ctx):
        t = torch.zeros(max(int(nbytes), 1), dtype=torch.uint8, device=dev)
        held[t.data_ptr()] = t
        return t.data_ptr()

    def free(ptr, _ctx):
        del held[ptr]

    a_cb, f_cb = G.ALLOC_FN(alloc), G.FREE_FN(free)
    cfg = G.make_config(w.batch, w.n_q_heads, w.n_kv_heads, w.bits, w.group, w.s_pct, w.buffer_cap, 0, w.n + 64)
    arenas = []
    G.gear_set_allocator(a_cb, f_cb)
    try:
        for _ in range(4):
            cache = G.gear_compress(None, cfg, k, v, w.n, 0)
            torch.cuda.synchronize()
            arenas.append(max(held.values(), key=lambda t: t.numel()).clone())
            G.gear_free(cache)
    finally:
        G.gear_set_allocator(None, None)
    assert all(torch.equal(a, arenas[0]) for a in arenas)
