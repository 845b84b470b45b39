"""A plain attention call behind a fused one on the same layer reads the rows that the fused
launch writes: same outputs as the fused call, which takes them from the caller's buffers.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from harness import assert_close  # noqa: E402

pytestmark = pytest.mark.gpu

L, HEADS = 3, 8


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2609_31224_gb300 import build
    build.build()


@pytest.mark.parametrize("n,hist,tokens", [(1, 700, 1), (1, 4100, 1), (6, 900, 1), (40, 2100, 1),
                                           (1, 900, 17), (20, 500, 17)])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("between", [False, True], ids=["next", "after another layer"])
def test_fused_then_plain(n, hist, tokens, dtype, between):
    from paper_2609_31224_gb300 import KVCache
    D, tdtype = (128, torch.bfloat16) if dtype == "bf16" else (64, torch.float32)
    pages = hist // 16 + 8
    rounds = 4
    cache = KVCache(n_sessions=n, layers=L, q_heads=4 * HEADS, kv_heads=HEADS, head_dim=D, budget=-1,
                    window=1, dtype=dtype, n_pages=n * pages, max_pages_per_session=pages,
                    max_positions=hist + rounds * tokens, max_seq_per_call=n,
                    max_tokens_per_call=n * hist)
    g = torch.Generator(device="cuda").manual_seed(n + hist)

    def rand(*shape):
        return torch.randn(shape, generator=g, device="cuda", dtype=tdtype)

    def types(t):
        one = np.zeros(t, np.uint8)
        one[0] = 0x80
        return torch.tensor(np.tile(one, n), device="cuda")

    ids = np.arange(n)
    cache.append_chunk(ids, np.arange(n + 1) * hist, types(hist), rand(L, n * hist, HEADS, D),
                       rand(L, n * hist, HEADS, D))
    st = torch.cuda.current_stream().cuda_stream
    fused, plain = ((cache.attn_decode_kv_raw, cache.attn_decode_raw) if tokens == 1 else
                    (cache.attn_prefill_kv_raw, cache.attn_prefill_raw))
    for _ in range(rounds):
        total = n * tokens
        k, v = rand(L, total, HEADS, D), rand(L, total, HEADS, D)
        q = rand(L, total, 4 * HEADS, D)
        out = torch.full((2, L, total, 4 * HEADS, D), float("nan"), dtype=tdtype, device="cuda")

        def ptr(x, layer):
            return x[layer].data_ptr()

        cache.append_chunk(ids, np.arange(n + 1) * tokens, types(tokens), None, None)
        for layer in range(L):
            fused(layer, ptr(k, layer), ptr(v, layer), ptr(q, layer), ptr(out[0], layer), st)
            if between and layer:
                plain(layer - 1, ptr(q, layer - 1), ptr(out[1], layer - 1), st)
            elif not between:
                plain(layer, ptr(q, layer), ptr(out[1], layer), st)
        if between:
            plain(L - 1, ptr(q, L - 1), ptr(out[1], L - 1), st)
        assert cache.device_status()[1] == 0
        a, b = out[0].float().cpu().numpy(), out[1].float().cpu().numpy()
        assert np.isfinite(a).all()
        # (Two launches of stream-K may merge a pair's parts in another order.)
        assert_close(b, a, dtype, f"{n} sessions")
