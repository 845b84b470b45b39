"""Appends of long chunks (a session's history fed back in one call) against the oracle:
lengths around the ones where the planning changes hands, alone and mixed in one call,
from an empty session and from a partly filled page, with the state after the eviction that
follows; and the stored rows of a long chunk against the same tokens fed in short ones.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from harness import compare_state  # noqa: E402
from oracle.cache import OracleCache, OracleConfig  # noqa: E402

pytestmark = pytest.mark.gpu

HEADS = 2


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2609_31224_gb300 import build
    build.build()


def _types(n, seed):
    rng = np.random.default_rng(seed)
    t = []
    while len(t) < n:
        t += [0x80] + [0] * 16 + [1] + [2] * int(rng.poisson(3)) + [1]
    return np.array(t[:n], np.uint8)


def _cache(n, lens, dtype):
    from paper_2609_31224_gb300 import KVCache
    pages = 2 * sum(m // 16 + 4 for m in lens)
    cfg = dict(n_sessions=n, layers=2, q_heads=4 * HEADS, kv_heads=HEADS,
               head_dim=128 if dtype == "bf16" else 64, budget=200, window=3, dtype=dtype,
               n_pages=pages)
    cache = KVCache(**cfg, max_pages_per_session=2 * (max(lens) // 16 + 4),
                    max_positions=max(lens) + 1, max_seq_per_call=n, max_tokens_per_call=sum(lens))
    return cache, OracleCache(OracleConfig(**cfg, page_size=16, rope_base=10000.0))


@pytest.mark.parametrize("first,then", [
    ([255], [1]), ([256], [257]), ([257], [256]), ([1024], [1025]), ([1], [3000]),
    ([7, 300, 15, 2049], [256, 1, 1100, 513]), ([1] * 40, [258] * 40),
])
def test_long_chunk_state(first, then):
    n = len(first)
    lens = [a + b for a, b in zip(first, then)]
    cache, orc = _cache(n, lens, "bf16")
    streams = [_types(m, i) for i, m in enumerate(lens)]
    for parts in ([s[:a] for s, a in zip(streams, first)], [s[a:] for s, a in zip(streams, first)]):
        total = sum(len(p) for p in parts)
        k = torch.zeros((2, total, HEADS, 128), dtype=torch.bfloat16, device="cuda")
        cache.append_chunk(range(n), np.cumsum([0] + [len(p) for p in parts]),
                           torch.tensor(np.concatenate(parts), device="cuda"), k, k)
        orc.append_chunk(list(range(n)), parts)
        for s in range(n):
            compare_state(cache.export_state(s), orc.state(s), f"session {s}")
    cache.evict(range(n))
    orc.evict(list(range(n)))
    for s in range(n):
        compare_state(cache.export_state(s), orc.state(s), f"session {s}, evicted")


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_long_chunk_rows(dtype):
    lens, d = [5, 700, 301], 128 if dtype == "bf16" else 64
    tdtype = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(3)
    rows = [torch.randn((2, 2, m, HEADS, d), generator=g, device="cuda").to(tdtype) for m in lens]
    whole, _ = _cache(3, lens, dtype)
    short, _ = _cache(3, lens, dtype)
    types = [_types(m, i) for i, m in enumerate(lens)]
    kv = torch.cat(rows, dim=2)
    whole.append_chunk(range(3), np.cumsum([0] + lens), torch.tensor(np.concatenate(types), device="cuda"),
                       kv[0].contiguous(), kv[1].contiguous())
    for s in range(3):
        for a in range(0, lens[s], 64):
            part = rows[s][:, :, a:a + 64]
            m = part.shape[2]
            short.append_chunk([s], [0, m], torch.tensor(types[s][a:a + 64], device="cuda"),
                               part[0].contiguous(), part[1].contiguous())
    for s in range(3):
        for layer in range(2):
            for x, y in zip(whole.export_kv(s, layer), short.export_kv(s, layer)):
                assert np.array_equal(x, y)
