"""Rules of the kernels that a run cannot show to be broken, read off their sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2609_31224_gb300", "csrc")


def code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def statement_before(text, at):
    """The statement that ends before offset `at`."""
    head = text[:at].rstrip().rstrip("{").rstrip()
    return head[max(head[:-1].rfind(";"), head[:-1].rfind("}"), head[:-1].rfind("{")) + 1:].strip()


@pytest.mark.parametrize("name,calls", [
    ("kvc_attn_prefill_f32.cu", [r'asm volatile\("barrier\.cluster\.arrive']),
    ("kvc_attn_prefill_tc.cu", [r"cluster_arrive\(\);", r"cluster_wait\(\);",
                                r'asm volatile\("bar\.sync', r"if \(warp == 2\) tmem_alloc"]),
])
def test_aligned_barriers_follow_a_reconvergence(name, calls):
    """Warp-aligned instructions behind code that lanes run apart (rows of their own, loops of
    different lengths) come right after a __syncwarp() or a barrier of the whole CTA."""
    text = code(name)
    for call in calls:
        found = list(re.finditer(call, text))
        assert found, call
        for m in found:
            assert re.match(r"__sync(warp|threads)\(\);", statement_before(text, m.start())), \
                text[m.start() - 200:m.end()]


def test_launch_state_is_kept_by_the_context():
    """Kernel attributes, grid and cluster limits belong to a CUDA context: nothing of them is kept
    per thread or process, where a context on another device would find the first one's, but in
    tables by the CUDA context's id.  (What else is kept: the driver's entry points, the tensor
    maps of a pool by its address and extent, and the last error's text.)"""
    kept = []
    for name in sorted(os.listdir(CSRC)):
        for line in code(name).splitlines():
            m = re.match(r"\s*(?:static thread_local|thread_local|static(?! constexpr| __device__|_))\s+(.*)", line)
            if m and "(" not in m.group(1):
                kept.append((name, m.group(1).strip().split()[0]))
    assert sorted(set(kept)) == [("kvc_api.cu", "std::string"), ("kvc_attn_prefill.cu", "EncodeTiledFn"),
                                 ("kvc_attn_prefill.cu", "PoolMaps"), ("kvc_noalloc.cu", "PfnCtxGetCurrent"),
                                 ("kvc_noalloc.cu", "PfnCtxGetId"), ("kvc_noalloc.cu", "std::mutex")]
    for name, setter in (("kvc_attn_prefill_f32.cu", "prefill_f32_limits"),
                         ("kvc_attn_prefill_tc.cu", "prefill_tc_limits")):
        assert "cudaFuncSetAttribute" in code(name) and setter in code("kvc_attn_prefill.cu") + \
            code("kvc_decode_dispatch.cu")
    assert "cudaOccupancyMaxActiveClusters" in code("kvc_attn_prefill_f32.cu")
    assert "query_limits(" in code("kvc_api.cu")
    table = code("kvc_decode_dispatch.cu")
    assert "current_context_id(&id)" in table and "g_known[i].ctx_id == id" in table


def test_only_waits_suspend():
    """mbarrier.try_wait may suspend the thread for a while, so it stands in bounded waits alone;
    a look at a phase on the way past it is mbarrier.test_wait."""
    for name in sorted(os.listdir(CSRC)):
        for m in re.finditer(r"(.*)mbar_try_wait\(", code(name)):
            assert re.search(r"if \($|while \(!$|inline bool $", m.group(1)), (name, m.group(0))
