"""Calls whose sessions hold other numbers of pages than the host expects when it launches them:
decode and prefill captured with short sessions and replayed on long ones, and sessions of text that a
small budget cannot shorten.  Against the same call launched anew, and on an unbounded cache.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from harness import assert_close  # noqa: E402

pytestmark = pytest.mark.gpu

HEADS, ACOUSTIC, TEXT = 8, 0, 3


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2609_31224_gb300 import build
    build.build()


class Sessions:
    """n sessions of one layer; feed(tokens of each, type) in lockstep from a seeded stream."""

    def __init__(self, n, dtype, budget, most):
        from paper_2609_31224_gb300 import KVCache
        self.n, self.D = n, 128 if dtype == "bf16" else 64
        self.t = torch.bfloat16 if dtype == "bf16" else torch.float32
        pages = 2 * (most // 16 + 4)
        self.cache = KVCache(n_sessions=n, layers=1, q_heads=4 * HEADS, kv_heads=HEADS,
                             head_dim=self.D, budget=budget, window=0, dtype=dtype,
                             n_pages=n * pages, max_pages_per_session=pages, max_positions=most + 1,
                             max_seq_per_call=n, max_tokens_per_call=n * most)
        self.gen = torch.Generator(device="cuda").manual_seed(7)

    def rand(self, *shape):
        return torch.randn(shape, generator=self.gen, device="cuda", dtype=self.t)

    def feed(self, m, kind):
        one = np.full(m, kind, np.uint8)
        if kind == ACOUSTIC:
            one[0] |= 0x80
        self.cache.append_chunk(np.arange(self.n), np.arange(self.n + 1) * m,
                                torch.tensor(np.tile(one, self.n), device="cuda"),
                                self.rand(1, self.n * m, HEADS, self.D),
                                self.rand(1, self.n * m, HEADS, self.D))

    def buffers(self, tokens=1):
        shape = (self.n * tokens, 4 * HEADS, self.D)
        return (self.rand(*shape),
                torch.full(shape, float("nan"), dtype=self.t, device="cuda"))


@pytest.mark.parametrize("n,grown", [(1, 20), (1, 3000), (3, 900), (6, 2100), (20, 700), (40, 600)])
@pytest.mark.parametrize("tokens", [1, 17])
@pytest.mark.parametrize("budget", [-1, 256])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_captured_short_replayed_long(n, grown, tokens, budget, dtype):
    s = Sessions(n, dtype, budget, grown + 2 * tokens)
    attend = s.cache.attn_decode if tokens == 1 else s.cache.attn_prefill_chunk
    q, out = s.buffers(tokens)
    fresh = torch.empty_like(out)
    s.feed(tokens, ACOUSTIC)
    attend(0, q, out)
    torch.cuda.synchronize()
    g, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=stream):
        attend(0, q, out, stream=stream)
    for m in (0, grown):
        if m:
            s.feed(m, TEXT)
            s.cache.evict(np.arange(n))
            s.feed(tokens, TEXT)
        out.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        attend(0, q, fresh)
        assert s.cache.device_status()[1] == 0
        assert_close(out.float().cpu().numpy(), fresh.float().cpu().numpy(), dtype, f"{m} grown")
    del g


@pytest.mark.parametrize("n,text", [(1, 40), (1, 1200), (2, 4000), (6, 1200), (20, 700)])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_text_over_its_budget(n, text, dtype):
    """Nothing of a text is evictable: the same pages, and so the same outputs, at any budget."""
    outs = []
    for budget in (0, -1):
        s = Sessions(n, dtype, budget, text + 1)
        s.feed(text, TEXT)
        s.cache.evict(np.arange(n))
        assert s.cache.resident_size(0) == text
        s.feed(1, TEXT)
        q, out = s.buffers()
        s.cache.attn_decode(0, q, out)
        assert s.cache.device_status()[1] == 0
        outs.append(out.float().cpu().numpy())
    assert np.isfinite(outs[1]).all()
    assert_close(outs[0], outs[1], dtype, f"{n} sessions of {text}")
