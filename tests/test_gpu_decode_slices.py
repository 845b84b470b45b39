"""Decode attention against the oracle over the slice counts that the dispatch picks for
short and long sessions: one page to more pages than warps, one session to more than one
wave holds, sessions much shorter than the call's longest one (empty slices).
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


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2609_31224_gb300 import build
    build.build()
    G.build()


# (KV heads, positions of each session's history, budget)
CASES = {
    "1 pair, first token": (1, [0], -1),
    "1 pair, 1 page": (1, [15], -1),
    "1 pair, 2 pages": (1, [16], -1),
    "1 pair, 33 pages": (1, [700], 512),
    "1 pair, 100 pages": (1, [1700], 1590),
    "4 pairs, 17 pages": (4, [260], -1),
    "8 pairs, 64 pages": (8, [1023], -1),
    "8 pairs, 101 pages": (8, [1610], -1),
    "16 pairs, 7 and 110 pages": (8, [100, 1760], -1),
    "8 pairs, 54 pages": (8, [862], -1),
    "8 pairs, 55 pages": (8, [864], -1),
    "8 pairs, 300 pages": (8, [4800], -1),
    "12 pairs, 190 pages": (4, [3030, 70, 3000], -1),
    "24 pairs, 94 pages": (8, [40, 1490, 16], -1),
    "24 pairs, 96 pages": (8, [40, 1530, 16], -1),
    "24 pairs": (8, [500, 501, 33], 300),
    "48 pairs": (8, [340, 1, 64, 1030, 335, 500], -1),
    "72 pairs": (8, [200 + 16 * i for i in range(9)], 180),
    "128 pairs": (8, [5 + 31 * i for i in range(16)], -1),
    "464 pairs": (8, [20 + i for i in range(58)], -1),
}


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("name", list(CASES))
def test_decode_slices(name, dtype):
    from paper_2609_31224_gb300 import KVCache
    heads, hist, budget = CASES[name]
    n, seed = len(hist), 9
    D, tdtype = (128, torch.bfloat16) if dtype == "bf16" else (64, torch.float32)
    pages = [2 * (h // 16 + 3) for h in hist]
    cfg = dict(n_sessions=n, layers=1, q_heads=4 * heads, kv_heads=heads, head_dim=D,
               budget=budget, window=2, dtype=dtype, n_pages=sum(pages))
    cache = KVCache(**cfg, max_pages_per_session=max(pages), max_positions=max(hist) + 2,
                    max_seq_per_call=n, max_tokens_per_call=sum(hist) + n)
    orc = OracleCache(OracleConfig(**cfg, page_size=16, rope_base=10000.0))

    def append(who, types, first):
        sess = torch.tensor([s for s, t in zip(who, types) for _ in t], dtype=torch.int32, device="cuda")
        pos = torch.tensor([f + i for f, t in zip(first, types) for i in range(len(t))],
                           dtype=torch.int32, device="cuda")

        def fill(tag, h):
            x = torch.empty((1, len(pos), h, D), dtype=tdtype, device="cuda")
            G.fill(x, dtype, seed, tag, sess, pos)
            return x

        cache.append_chunk(who, np.cumsum([0] + [len(t) for t in types]),
                           torch.tensor(np.concatenate(types), device="cuda"),
                           fill(V.TAG_K, heads), fill(V.TAG_V, heads))
        orc.append_chunk(list(who), list(types))
        return fill(V.TAG_Q, 4 * heads)

    unit = [0x80] + [0] * 16 + [2] * 3
    who = [s for s in range(n) if hist[s]]
    if who:
        append(who, [np.array((unit * (hist[s] // 20 + 1))[:hist[s]], np.uint8) for s in who], [0] * len(who))
        cache.evict(who)
        orc.evict(who)
    q = append(list(range(n)), [np.array([2], np.uint8)] * n, hist)
    out = torch.full((2, n, 4 * heads, D), float("nan"), dtype=tdtype, device="cuda")
    for i in range(2):  # the second launch overlaps the first
        cache.attn_decode(0, q[0], out[i])
    assert cache.device_status()[1] == 0
    assert torch.isfinite(out).all()

    def kv_source(s, layer, positions):
        return tuple(V.layer_tensor(seed, tag, s, layer, positions, heads, D, dtype)
                     .astype(np.float64) for tag in (V.TAG_K, V.TAG_V))

    picked = sorted(set([0, n // 2, n - 1]))
    qs = [V.layer_tensor(seed, V.TAG_Q, s, 0, [hist[s]], 4 * heads, D, dtype) for s in picked]
    for s, ref in zip(picked, orc.attend(0, qs, kv_source, sessions=picked)):
        for i in range(2):
            assert_close(out[i, s:s + 1].float().cpu().numpy(), ref, dtype, f"{name}, session {s}")
