"""The means of the coverage losses at the sizes where their summation changes
form (2048 tasks on one CTA, more on a cluster of eight): B L chains of up to 32
tokens are one task each.

Both sides add the same fp32 losses in fp64, n = B (T - 1) L of them in some
order: each sum is within n 2^-53 of the exact one (all terms >= 0), so they
differ by at most 2 n 2^-53 of it, 2.7e-12 for the largest n here.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,top_b", [(64, 9), (16, 3)])
@pytest.mark.parametrize("B,L", [(1, 1), (89, 23), (64, 32), (683, 3), (1365, 3)])
def test_means_at_the_edges(B, L, N, top_b):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_04895_gb300 import build, crc
    build.build()
    T = 4
    pr = crc.problem(L=L, N=N, K=1, d=16, C=1, R=0, B=B, expert_bytes=1)
    g = torch.Generator(device="cuda").manual_seed(7)
    probs = torch.softmax(torch.randn((B, T, L, 3, N), device="cuda", generator=g), -1)
    loss, means, _ = crc.cache_loss(pr, probs, top_b, 0.05)
    torch.cuda.synchronize()
    assert crc.crc_device_error() == 0
    n = B * (T - 1) * L
    want = loss.double().sum((0, 1, 2)) / n
    assert want.min().item() > 0
    for i in range(2):
        assert means[i].item() == pytest.approx(want[i].item(), rel=2 * n * 2.0 ** -53, abs=0)
