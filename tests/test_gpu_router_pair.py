"""Router heads of N = 128, on CTA pairs and on one CTA a tile (rows shorter than
2048, or than 4096 in a call of one round, or where pairs would take more
rounds): a layer's tiles pair up whatever their number, so the scores of a call
equal, bit for bit, those of calls on parts of it whose tiles pair up
differently or not at all, and match an fp64 softmax.
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


# (layers, streams, tokens): one tile a layer, two, three (partner idle, one
# round either way), three of more rounds on pairs (single CTAs), nine and more,
# tiles of several streams, ragged lengths
SIZES = [(3, 1, 100), (3, 2, 128), (3, 3, 128), (60, 3, 70), (20, 9, 130), (17, 5, 257),
         (4, 40, 7), (3, 300, 1), (2, 1, 1)]


@pytest.mark.parametrize("L,B,T", SIZES, ids=lambda v: str(v))
@pytest.mark.parametrize("heads", [3, 2])
@pytest.mark.parametrize("d", [328, 2056, 4104])
def test_pairs_equal_parts(C, L, B, T, heads, d):
    w = S.QWEN3_30B.with_(L=L, B=B, T=T, d=d)
    W = C.synth_weights(L, w.N, w.d, seed=3)
    h, _ = C.synth_hidden(B, T, L, w.d, seed=4)
    mark = -7.0
    full = torch.full((B, T, L, 3, w.N), mark, device="cuda")
    C.route_scores(C.problem_of(w), h, W, heads=heads, out=full)
    assert C.crc_device_error() == 0
    if heads == 2:
        assert bool((full[:, :, :, 2] == mark).all())
    cut = max(1, B // 3)
    for b0, b1 in ((0, cut), (cut, B)):
        if b0 == b1:
            continue
        part = torch.full((b1 - b0, T, L, 3, w.N), mark, device="cuda")
        C.route_scores(C.problem_of(w.with_(B=b1 - b0)), h[b0:b1].contiguous(), W, heads=heads,
                       out=part)
        assert torch.equal(part.view(torch.int32), full[b0:b1].view(torch.int32)), (b0, b1)
    for l in {0, L - 1}:
        z = h[:, :, l].double() @ W[l].double().t()
        ref = torch.softmax(z.view(B, T, 3, w.N), dim=-1)[:, :, :heads]
        err = (full[:, :, l, :heads].double() - ref).abs() / ref
        # fp32 sums of d products and the SFU exponential, as for the other router
        # tests (d up to 2880)
        assert float(err.max()) <= 2.5e-4
