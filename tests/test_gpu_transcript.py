"""Transcript export against the oracle at the edges of its rounds: retained slots around a
thread's share, a round and several rounds, spread over both regions, with short outputs.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle.cache import OracleCache, OracleConfig  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2609_31224_gb300 import build
    build.build()


# (positions of the history, budget of its eviction, positions appended after it)
@pytest.mark.parametrize("heads", [1, 3, 12])  # a part of, one and more batches of a warp
@pytest.mark.parametrize("hist,budget,tail", [(0, -1, 1), (7, -1, 8), (640, 300, 9), (8190, -1, 2),
                                              (8192, -1, 1), (9000, 4000, 4300), (17011, -1, 5)])
def test_export_rounds(hist, budget, tail, heads):
    from paper_2609_31224_gb300 import KVCache
    D, layers = 64, 2
    pages = 2 * ((hist + tail) // 16 + 4)
    cfg = dict(n_sessions=2, layers=layers, q_heads=4 * heads, kv_heads=heads, head_dim=D, budget=budget,
               window=1, dtype="f32", n_pages=2 * pages)
    cache = KVCache(**cfg, max_pages_per_session=pages, max_positions=hist + tail + 1,
                    max_seq_per_call=1, max_tokens_per_call=max(hist, tail))
    orc = OracleCache(OracleConfig(**cfg, page_size=16, rope_base=10000.0))
    rng = np.random.default_rng(hist)
    unit = [0x80] + [0] * 16
    for n in (hist, tail):
        if n == 0:
            continue
        types = np.concatenate([np.array(unit + [2] * int(rng.integers(0, 9)), np.uint8)
                                for _ in range(n // 17 + 1)])[:n] if n > 1 else np.array([2], np.uint8)
        kv = torch.tensor(rng.standard_normal((2, layers, n, heads, D)), dtype=torch.float32, device="cuda")
        cache.append_chunk([1], [0, n], torch.tensor(types, device="cuda"), kv[0], kv[1])
        orc.append_chunk([1], [types])
        if n == hist:
            cache.evict([1])
            orc.evict([1])
    want = orc.transcript_positions(1)
    st = cache.export_state(1)
    where = {p: i for i, p in enumerate(st["pos"])}
    idx = [where[p] for p in want]
    for cap in sorted({st["resident"], len(want), max(0, len(want) - 1), 3}):
        pos, k, v, count = cache.export_transcript(1, cap)
        got = min(cap, len(want))
        assert int(count.item()) == len(want)
        assert pos[:got].cpu().numpy().tolist() == list(want[:got])
        assert not pos[got:].any() and not k[:, got:].any() and not v[:, got:].any()
        for layer in range(layers):
            ks, vs = cache.export_kv(1, layer)
            assert np.array_equal(k[layer, :got].cpu().numpy(), ks[idx[:got]])
            assert np.array_equal(v[layer, :got].cpu().numpy(), vs[idx[:got]])
    assert cache.device_status()[1] == 0
