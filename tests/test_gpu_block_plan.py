"""crc_route_and_cache on the persistent fused kernel with token blocks shorter
than 128 (chosen by the call's size, or all there is of a short call of many
chains) against crc_route_scores followed by crc_cache_scan, bit for bit: every
access and the whole state, over two calls of one state, at batches and lengths
that leave ragged stream groups, ragged blocks and, for N = 128, tiles that do
not pair up.
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


CASES = [
    S.GPT_OSS_20B.with_(L=8, B=128, T=160, d=1024),            # 16-token blocks, all full
    S.GPT_OSS_20B.with_(L=9, B=117, T=135, d=1024),            # ragged groups and block
    S.GPT_OSS_20B.with_(L=9, B=117, T=65, d=1032, R=0),
    S.TINY.with_(N=64, K=6, C=12, R=3, L=9, B=118, T=129, d=1024),
    S.QWEN3_30B.with_(L=8, B=128, T=192, d=1024),              # pairs of 64-token tiles
    S.QWEN3_30B.with_(L=9, B=115, T=90, d=1024),               # 58 groups of 64 tokens
    S.QWEN3_30B.with_(L=9, B=117, T=130, d=1024, R=0, C=16),   # odd at 128 tokens
    S.QWEN3_30B.with_(L=10, B=106, T=100, d=1024, R=8),
    # short calls with more clusters than the GPU holds at once: blocks of 8 tokens
    S.TINY.with_(L=24, B=100, T=8, d=64),
    S.GPT_OSS_20B.with_(L=20, B=117, T=7, d=200),
    S.TINY.with_(N=64, K=6, C=12, R=3, L=24, B=118, T=5, d=72),
    S.QWEN3_30B.with_(L=24, B=128, T=8, d=256),                # pairs: 8 groups of 16 streams
    S.QWEN3_30B.with_(L=32, B=100, T=6, d=256),                # 7 groups, the last of 4
    # of wide rows: blocks of 4
    S.GPT_OSS_20B.with_(L=30, B=128, T=3, d=3080),
    S.QWEN3_30B.with_(L=40, B=128, T=4, d=3080),               # pairs: 4 groups of 32 streams
    S.QWEN3_30B.with_(L=77, B=70, T=3, d=3080),                # 3 groups, the last of 6
    S.QWEN3_30B.with_(L=80, B=128, T=4, d=3080, R=0, C=16),
    # wider still: 2
    S.QWEN3_30B.with_(L=55, B=130, T=2, d=4104),
    # and blocks of 32 and 64
    S.QWEN3_30B.with_(L=20, B=61, T=20, d=128, R=8),
    S.QWEN3_30B.with_(L=20, B=60, T=33, d=128),
]


@pytest.mark.parametrize("w", CASES, ids=lambda w: f"N{w.N}-B{w.B}-T{w.T}-R{w.R}-d{w.d}")
@pytest.mark.parametrize("traced", [True, False], ids=["traced", "untraced"])
def test_block_plans_equal_pair(C, w, traced):
    p = C.problem_of(w)
    W = C.synth_weights(w.L, w.N, w.d, seed=3)
    ws = torch.empty(C.crc_fused_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    fused, pair = C.State(p), C.State(p)
    carry = None
    for call in range(2):
        h, carry = C.synth_hidden(w.B, w.T, w.L, w.d, seed=4, t0=call * w.T, carry=carry)
        trf = C.Trace.alloc(p, w.T, caches=True, rank_order=False, topk_set=True)
        trp = C.Trace.alloc(p, w.T, caches=True, rank_order=False, topk_set=True)
        C.crc_profile_begin()
        C.route_and_cache(p, h, W, fused, trf if traced else None, workspace=ws)
        kt = C.crc_profile_end()
        assert kt["fused"]["launches"] == 1 and kt["short"]["launches"] == 0
        scores = torch.zeros((w.B, w.T, w.L, 3, w.N), device="cuda")
        C.cache_scan(p, C.route_scores(p, h, W, heads=3 if w.R > 0 else 2, out=scores), pair, trp)
        if traced:
            for name in ("misses", "proactive", "cache_mid", "cache_after", "topk_set"):
                assert torch.equal(getattr(trf, name), getattr(trp, name)), (call, name)
    a = fused.read(want_caches=True, want_retention=True, want_chain_counters=True)
    b = pair.read(want_caches=True, want_retention=True, want_chain_counters=True)
    assert a["error"] == 0 and a["tokens"] == 2 * w.T
    for name in ("cache_bits", "chain_counters"):
        assert (a[name] == b[name]).all(), name
    assert (a["retention"].view("u4") == b["retention"].view("u4")).all()
