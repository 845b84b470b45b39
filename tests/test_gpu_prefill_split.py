"""The prefill kernels against the oracle at the sizes where their splits can go wrong: 1
to 8 (binary32: 16) slices per pair, fewer pages than slices, chunks of 1 to 32 tokens in one
call, the two row-block sizes of binary32, stream-K pairs over two and over many CTAs, with
and without the fused write.
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

L = 2


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2609_31224_gb300 import build
    build.build()
    G.build()


def _history(n):
    """About n positions: units of 17 acoustic and 3 transcript positions, cut at n."""
    unit = [0x80] + [0] * 16 + [2] * 3
    return np.array((unit * (n // 20 + 1))[:n], np.uint8)


# (tokens of each session's chunk, positions of each session's history, budget); 8 KV heads.
CASES = {
    "1 session, 32 tokens": ([32], [1500], 1200),
    "1 session, fewer stages than slices": ([5], [40], -1),
    "first chunk of a session": ([17], [0], -1),
    "1 session, 8 tokens": ([8], [700], 600),
    "2 sessions, 1 and 17 tokens": ([1, 17], [1700, 1333], 1300),
    "2 sessions, one with fewer pages than slices": ([17, 17], [1700, 5], 1300),
    "3 sessions, 2 to 31 tokens": ([17, 31, 2], [1640, 1655, 2001], 1500),
    "4 sessions": ([17] * 4, [1500, 1064, 1065, 1024], 900),
    "5 sessions": ([17] * 5, [1300, 1301, 1302, 1303, 1304], 1250),
    "9 sessions": ([17, 16, 1, 32, 17, 17, 3, 17, 17], [1150 + 37 * i for i in range(9)], 1260),
    "16 sessions, short": ([17] * 16, [20 + 11 * i for i in range(16)], 100),
    "20 sessions": ([17, 1, 32, 8] * 5, [330 + 16 * i for i in range(20)], 400),
    "20 sessions, one much longer": ([17] * 20, [5000] + [40] * 19, -1),
}


@pytest.mark.parametrize("per_layer", [False, True], ids=["whole", "per_layer"])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("name", list(CASES))
def test_prefill_split(name, dtype, per_layer):
    from paper_2609_31224_gb300 import KVCache
    tokens, hist, budget = CASES[name]
    n, heads, seed = len(tokens), 8, 5
    D, tdtype = (128, torch.bfloat16) if dtype == "bf16" else (64, torch.float32)
    total = sum(h + t for h, t in zip(hist, tokens))
    pages = [2 * ((h + t) // 16 + 3) for h, t in zip(hist, tokens)]
    cache = KVCache(n_sessions=n, layers=L, q_heads=4 * heads, kv_heads=heads, head_dim=D,
                    budget=budget, window=2, dtype=dtype, n_pages=sum(pages),
                    max_pages_per_session=max(pages), max_positions=max(hist) + 64,
                    max_seq_per_call=n, max_tokens_per_call=total)
    orc = OracleCache(OracleConfig(n_sessions=n, layers=L, q_heads=4 * heads, kv_heads=heads,
                                   head_dim=D, page_size=16, budget=budget, window=2,
                                   dtype=dtype, rope_base=10000.0, n_pages=sum(pages)))

    def fill(tag, h, sess, pos):
        x = torch.empty((L, len(pos), h, D), dtype=tdtype, device="cuda")
        G.fill(x, dtype, seed, tag, torch.tensor(sess, dtype=torch.int32, device="cuda"),
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
    out = torch.full((L, int(cu[-1]), 4 * heads, D), float("nan"), dtype=tdtype,
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
        return tuple(V.layer_tensor(seed, tag, s, layer, positions, heads, D, dtype)
                     .astype(np.float64) for tag in (V.TAG_K, V.TAG_V))

    got = out.float().cpu().numpy()
    layer = L - 1
    picked = sorted(set([0, n // 2, n - 1]))
    qs = [V.layer_tensor(seed, V.TAG_Q, s, layer, range(hist[s], hist[s] + tokens[s]), 4 * heads,
                         D, dtype) for s in picked]
    for s, ref in zip(picked, orc.attend(layer, qs, kv_source, sessions=picked)):
        assert_close(got[layer, cu[s]:cu[s + 1]], ref, dtype, f"{name}, session {s}")
    assert np.isfinite(got).all()
