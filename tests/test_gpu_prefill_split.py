"""The tcgen05 prefill kernel's two splits against the oracle at the sizes where they can go
wrong: each number of slices per pair, fewer stages than slices, chunks of 1 to 32 tokens
in one call, stream-K pairs over two and over many CTAs, with and without the fused write.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from harness import assert_close  # noqa: E402
from oracle.cache import OracleCache, OracleConfig  # noqa: E402
from synth import gpu as G  # noqa: E402
from synth import values as V  # noqa: E402

pytestmark = pytest.mark.gpu

D, L = 128, 2


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2609_31224_gb300 import build
    build.build()
    G.build()


def _history(n):
    """About n positions: units of 17 acoustic and 3 transcript positions, cut at n."""
    unit = [0x80] + [0] * 16 + [2] * 3
    return np.array((unit * (n // 20 + 1))[:n], np.uint8)


# (tokens of each session's chunk, positions of each session's history, budget).  Pairs are
# 8 per session: 1, 2, 3, 4, 5 and 9 sessions take 8, 6, 5, 4, 3 and 2 slices, 16 sessions
# one, 20 sessions stream-K.
CASES = {
    "8 slices, 32 tokens": ([32], [1500], 1200),
    "8 slices, fewer stages than slices": ([5], [40], -1),
    "8 slices, first chunk of a session": ([17], [0], -1),
    "6 slices, 1 and 17 tokens": ([1, 17], [700, 333], 300),
    "5 slices, 2 to 31 tokens": ([17, 31, 2], [640, 655, 1001], 500),
    "4 slices": ([17] * 4, [500, 64, 65, 1024], 400),
    "3 slices": ([17] * 5, [300, 301, 302, 303, 304], 250),
    "2 slices": ([17, 16, 1, 32, 17, 17, 3, 17, 17], [150 + 37 * i for i in range(9)], 260),
    "1 slice": ([17] * 16, [20 + 11 * i for i in range(16)], 100),
    "stream-K, parts of two CTAs": ([17, 1, 32, 8] * 5, [330 + 16 * i for i in range(20)], 400),
    "stream-K, parts of many CTAs": ([17] * 20, [5000] + [40] * 19, -1),
}


@pytest.mark.parametrize("per_layer", [False, True], ids=["whole", "per_layer"])
@pytest.mark.parametrize("name", list(CASES))
def test_prefill_split(name, per_layer):
    from paper_2609_31224_gb300 import KVCache
    tokens, hist, budget = CASES[name]
    n, heads, seed = len(tokens), 8, 5
    total = sum(h + t for h, t in zip(hist, tokens))
    pages = [2 * ((h + t) // 16 + 3) for h, t in zip(hist, tokens)]
    cache = KVCache(n_sessions=n, layers=L, q_heads=4 * heads, kv_heads=heads, head_dim=D,
                    budget=budget, window=2, dtype="bf16", n_pages=sum(pages),
                    max_pages_per_session=max(pages), max_positions=max(hist) + 64,
                    max_seq_per_call=n, max_tokens_per_call=total)
    orc = OracleCache(OracleConfig(n_sessions=n, layers=L, q_heads=4 * heads, kv_heads=heads,
                                   head_dim=D, page_size=16, budget=budget, window=2,
                                   dtype="bf16", rope_base=10000.0, n_pages=sum(pages)))

    def fill(tag, h, sess, pos):
        x = torch.empty((L, len(pos), h, D), dtype=torch.bfloat16, device="cuda")
        G.fill(x, "bf16", seed, tag, torch.tensor(sess, dtype=torch.int32, device="cuda"),
               torch.tensor(pos, dtype=torch.int32, device="cuda"))
        return x

    def append(who, types, first, with_kv):
        sess = [s for s, t in zip(who, types) for _ in t]
        pos = [f + i for f, t in zip(first, types) for i in range(len(t))]
        k, v = fill(V.TAG_K, heads, sess, pos), fill(V.TAG_V, heads, sess, pos)
        cu = np.concatenate([[0], np.cumsum([len(t) for t in types])])
        cache.append_chunk(who, cu, torch.tensor(np.concatenate(types), device="cuda"),
                           k if with_kv else None, v if with_kv else None)
        orc.append_chunk(list(who), list(types))
        return cu, k, v, fill(V.TAG_Q, 4 * heads, sess, pos)

    who = [s for s in range(n) if hist[s]]
    if who:
        append(who, [_history(hist[s]) for s in who], [0] * len(who), True)
        cache.evict(who)
        orc.evict(who)
    chunk = [np.array([0x80] + [0] * (t - 1), np.uint8) for t in tokens]
    cu, k, v, q = append(list(range(n)), chunk, hist, not per_layer)
    out = torch.full((L, int(cu[-1]), 4 * heads, D), float("nan"), dtype=torch.bfloat16,
                     device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    for _ in range(2):  # the second time overlaps the launches of the first
        for layer in range(L):
            if per_layer:
                cache.attn_prefill_kv_raw(layer, k[layer].data_ptr(), v[layer].data_ptr(),
                                          q[layer].data_ptr(), out[layer].data_ptr(), st)
            else:
                cache.attn_prefill_chunk(layer, q[layer], out[layer])
    assert cache.device_status()[1] == 0

    def kv_source(s, layer, positions):
        return tuple(V.layer_tensor(seed, tag, s, layer, positions, heads, D, "bf16")
                     .astype(np.float64) for tag in (V.TAG_K, V.TAG_V))

    got = out.float().cpu().numpy()
    layer = L - 1
    picked = sorted(set([0, n // 2, n - 1]))
    qs = [V.layer_tensor(seed, V.TAG_Q, s, layer, range(hist[s], hist[s] + tokens[s]), 4 * heads,
                         D, "bf16") for s in picked]
    for s, ref in zip(picked, orc.attend(layer, qs, kv_source, sessions=picked)):
        assert_close(got[layer, cu[s]:cu[s + 1]], ref, "bf16", f"{name}, session {s}")
    assert np.isfinite(got).all()
