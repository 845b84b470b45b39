"""Evictions and releases captured in a CUDA graph: the cache goes on afterwards, reads its pages
in use back from eager ones alone, and is destroyed without leaving an error behind.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2609_31224_gb300 import build
    build.build()


def _cache(pages):
    from paper_2609_31224_gb300 import KVCache
    return KVCache(n_sessions=1, layers=1, q_heads=4, kv_heads=1, head_dim=64, budget=16, window=0,
                   dtype="f32", n_pages=pages, max_pages_per_session=pages, max_positions=4096,
                   max_seq_per_call=1, max_tokens_per_call=64)


def _feed(cache, n):
    types = np.zeros(n, np.uint8)
    types[0] = 0x80
    kv = torch.zeros((1, n, 1, 64), device="cuda")
    cache.append_chunk([0], [0, n], torch.tensor(types, device="cuda"), kv, kv)


def _captured(cache, call):
    g, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=stream):
        call(stream)
    return g


@pytest.mark.parametrize("what", ["evict", "release"])
@pytest.mark.parametrize("replays", [0, 3])
def test_destroyed_after_a_captured_call(what, replays):
    cache = _cache(8)
    _feed(cache, 40)
    g = _captured(cache, lambda s: getattr(cache, what)([0], stream=s))
    for _ in range(replays):
        g.replay()
    cache.close()
    assert torch.ones(4, device="cuda").sum().item() == 4  # (raises if an error was left)
    del g


def test_pages_are_read_back_after_a_captured_evict():
    """A pool that the host's bound says is full, after an eager evict and a captured one."""
    cache = _cache(6)
    _feed(cache, 64)
    cache.evict([0])
    g = _captured(cache, lambda s: cache.evict([0], stream=s))
    for _ in range(6):  # 4 pages each, of which an eviction leaves one or none
        _feed(cache, 48)
        g.replay()
        torch.cuda.synchronize()
        cache.evict([0])
    assert cache.device_status()[1] == 0
    assert cache.resident_size(0) <= 16
    del g
