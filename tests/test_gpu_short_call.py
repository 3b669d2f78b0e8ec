"""Short calls of crc_route_and_cache (one token, a few, a small chunk) against
crc_route_scores followed by crc_cache_scan, bit for bit: every access's Top-K
set, misses, proactive loads and caches, and the whole state, over successive
calls of one state and across the sizes at which a call's tile, its clusters or
its kernel changes.
"""
import pytest

import crc_synth as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_04895_gb300 import build
    build.build()
    from paper_2609_04895_gb300 import crc
    crc.load()
    return crc


SHAPES = {
    "n16": S.TINY.with_(L=3),
    "n32": S.GPT_OSS_20B.with_(L=3, d=200),               # a partial K block
    "n64": S.TINY.with_(N=64, K=6, C=12, R=3, L=5, d=520),
    "n128": S.QWEN3_30B.with_(L=3, d=256),
    "n128-r0": S.QWEN3_30B.with_(L=2, d=256, R=0, C=16),
    "n128-one-layer": S.QWEN3_30B.with_(L=1, d=72, R=12, C=8, K=1),
}
# (streams, tokens per call): one tile's edges for T = 1 (128 rows), odd T, the
# longest calls, several stream groups with a ragged last one
SIZES = [(1, 1), (127, 1), (128, 1), (129, 1), (300, 1), (43, 3), (7, 5), (3, 42), (2, 64),
         (5, 64), (1, 65)]


def run_short_calls(C, w, traced, short_kernel):
    """Three successive calls of w.T tokens on one state against the pair's."""
    B, T = w.B, w.T
    p = C.problem_of(w)
    W = C.synth_weights(w.L, w.N, w.d, seed=3)
    ws = torch.empty(C.crc_fused_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    heads = 3 if w.R > 0 else 2
    short, pair = C.State(p), C.State(p)
    carry = None
    for call in range(3):
        h, carry = C.synth_hidden(B, T, w.L, w.d, seed=4, t0=call * T, carry=carry)
        trs = C.Trace.alloc(p, T, caches=True, rank_order=False, topk_set=True)
        trp = C.Trace.alloc(p, T, caches=True, rank_order=False, topk_set=True)
        C.crc_profile_begin()
        C.route_and_cache(p, h, W, short, trs if traced else None, workspace=ws)
        kt = C.crc_profile_end()
        assert kt["fused"]["launches"] == 1 and kt["short"]["launches"] == int(short_kernel)
        scores = torch.zeros((B, T, w.L, 3, w.N), device="cuda")
        C.cache_scan(p, C.route_scores(p, h, W, heads=heads, out=scores), pair, trp)
        if traced:
            for name in ("misses", "proactive", "cache_mid", "cache_after", "topk_set"):
                assert torch.equal(getattr(trs, name), getattr(trp, name)), (call, name)
    a = short.read(want_caches=True, want_retention=True, want_chain_counters=True)
    b = pair.read(want_caches=True, want_retention=True, want_chain_counters=True)
    assert a["error"] == 0 and a["tokens"] == 3 * T
    for name in ("cache_bits", "chain_counters"):
        assert (a[name] == b[name]).all(), name
    assert (a["retention"].view("u4") == b["retention"].view("u4")).all()


# Calls of more clusters than two CTAs an SM hold, where three an SM (of eight
# warps) save a wave, and one on the other side of that line
THREE = {
    "n128-24": S.QWEN3_30B.with_(L=48, B=13, T=24, d=256),
    "n128-24-two": S.QWEN3_30B.with_(L=30, B=13, T=24, d=256),
    "n128-one": S.QWEN3_30B.with_(L=48, B=300, T=1, d=520),
    "n128-r0": S.QWEN3_30B.with_(L=90, B=150, T=1, d=200, R=0, C=16),
    "n64": S.TINY.with_(N=64, K=6, C=12, R=3, L=30, B=400, T=1, d=264),
    "n32": S.GPT_OSS_20B.with_(L=24, B=600, T=1, d=200),
    "n16": S.TINY.with_(L=48, B=300, T=2, d=136),
}


@pytest.mark.parametrize("name", THREE, ids=str)
@pytest.mark.parametrize("traced", [True, False], ids=["traced", "untraced"])
def test_short_calls_of_many_clusters(C, name, traced):
    run_short_calls(C, THREE[name], traced, True)


@pytest.mark.parametrize("w", [S.QWEN3_30B.with_(L=55, B=130, T=2, d=4104),
                               S.QWEN3_30B.with_(L=48, B=200, T=4, d=72)], ids=["two", "four"])
def test_a_small_workspace_keeps_short_calls(C, w):
    """Calls that the persistent kernel takes when its workspace is there run as
    short calls, not as the router's and the scan's launches, when it is not."""
    p = C.problem_of(w)
    W = C.synth_weights(w.L, w.N, w.d, seed=3)
    h, _ = C.synth_hidden(w.B, w.T, w.L, w.d, seed=4)
    got = []
    for nbytes, short in ((C.crc_workspace_bytes(p, 1), 1), (C.crc_fused_workspace_bytes(p), 0)):
        ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        st = C.State(p)
        C.crc_profile_begin()
        C.route_and_cache(p, h, W, st, None, workspace=ws)
        kt = C.crc_profile_end()
        assert kt["fused"]["launches"] == 1 and kt["short"]["launches"] == short
        got.append(st.read(want_caches=True, want_retention=True, want_chain_counters=True))
    for name in ("cache_bits", "chain_counters"):
        assert (got[0][name] == got[1][name]).all(), name
    assert (got[0]["retention"].view("u4") == got[1]["retention"].view("u4")).all()


def test_one_state_over_short_and_persistent_calls(C):
    """A serving loop's mix on one state: single tokens, chunks and long calls in
    turn, traced and not, against one scan of the same scores in the same pieces."""
    w = S.QWEN3_30B.with_(B=6, L=3, d=256)
    p = C.problem_of(w)
    W = C.synth_weights(w.L, w.N, w.d, seed=3)
    ws = torch.empty(C.crc_fused_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    mixed, pair = C.State(p), C.State(p)
    carry, t0 = None, 0
    for i, T in enumerate([1, 150, 1, 24, 2, 200, 64, 1, 66, 3]):
        h, carry = C.synth_hidden(w.B, T, w.L, w.d, seed=4, t0=t0, carry=carry)
        trm = C.Trace.alloc(p, T, caches=True, rank_order=False, topk_set=True)
        trp = C.Trace.alloc(p, T, caches=True, rank_order=False, topk_set=True)
        C.crc_profile_begin()
        C.route_and_cache(p, h, W, mixed, trm if i % 3 else None, workspace=ws)
        assert C.crc_profile_end()["short"]["launches"] == int(T <= 64)
        C.cache_scan(p, C.route_scores(p, h, W), pair, trp)
        if i % 3:
            for name in ("misses", "proactive", "cache_mid", "cache_after", "topk_set"):
                assert torch.equal(getattr(trm, name), getattr(trp, name)), (i, name)
        t0 += T
    a = mixed.read(want_caches=True, want_retention=True, want_chain_counters=True)
    b = pair.read(want_caches=True, want_retention=True, want_chain_counters=True)
    assert a["error"] == 0 and a["tokens"] == t0
    for name in ("cache_bits", "chain_counters"):
        assert (a[name] == b[name]).all(), name
    assert (a["retention"].view("u4") == b["retention"].view("u4")).all()


def test_aborted_short_call_does_not_advance_the_state(C):
    """A call that finds its abort word set (as one of its waits sets it when it
    runs out) leaves the token counter and the carry slot where they were and
    clears the word, so the next call runs."""
    w = SHAPES["n128"].with_(B=4)
    p = C.problem_of(w)
    st = C.State(p)
    W = C.synth_weights(w.L, w.N, w.d, seed=3)
    ws = torch.empty(C.crc_fused_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    h, _ = C.synth_hidden(4, 1, w.L, w.d, seed=4)
    C.route_and_cache(p, h, W, st, None, workspace=ws)
    head = st.buf[:256].view(torch.int32)
    before = head.cpu()
    word = 15                                         # the header's abort word
    head[word] = 1
    C.route_and_cache(p, h, W, st, None, workspace=ws)
    assert torch.equal(head.cpu(), before)            # the word cleared, nothing else moved
    C.route_and_cache(p, h, W, st, None, workspace=ws)
    assert st.read()["tokens"] == 2


@pytest.mark.parametrize("shape", SHAPES, ids=str)
@pytest.mark.parametrize("B,T", SIZES, ids=lambda v: str(v))
@pytest.mark.parametrize("traced", [True, False], ids=["traced", "untraced"])
def test_short_calls_equal_pair(C, shape, B, T, traced):
    w = SHAPES[shape].with_(B=B, T=T)
    # untraced calls of few experts leave the short-call kernel at 32 tokens, others at 64
    run_short_calls(C, w, traced, T <= (64 if traced or w.N > 32 else 32))


def test_short_call_on_another_problems_state(C):
    """A state made for another problem is refused as before, and stays usable."""
    w = SHAPES["n128"].with_(B=4)
    p, other = C.problem_of(w), C.problem_of(w.with_(C=31))
    st = C.State(p)
    W = C.synth_weights(w.L, w.N, w.d, seed=3)
    h, _ = C.synth_hidden(4, 1, w.L, w.d, seed=4)
    ws = torch.empty(C.crc_fused_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    C.crc_route_and_cache(other, h.data_ptr(), W.data_ptr(), 1, st.ptr, st.nbytes, None,
                          ws.data_ptr(), ws.numel())
    with pytest.raises(C.CrcError) as e:
        st.read()
    assert e.value.code == C.CRC_ESTATE
    st.init()
    C.route_and_cache(p, h, W, st, None, workspace=ws)
    assert st.read()["tokens"] == 1
