"""Failure detection on the GPU without a fault, and checkpoint / resume of
the state.  A bounded wait that runs out (a flag nothing sets; an mbarrier
phase nothing completes) latches CRC_ETIMEOUT in the state, the host reads it
through crc_state_read, the kernel has returned within about the wait limit,
and the context still runs the hot path correctly afterwards.  A state copied
to the host and restored elsewhere continues the streams exactly."""
import ctypes
import time

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


@pytest.mark.parametrize("kind", [0, 1], ids=["flag", "mbarrier"])
def test_expired_wait_reports_timeout_and_context_survives(C, kind):
    lib = C.load()
    w = S.QWEN3_30B.with_(B=2, T=140, L=2, d=128)
    p = C.problem_of(w)
    st = C.State(p)
    torch.cuda.synchronize()
    limit = 50_000_000                                   # 50 ms
    t0 = time.perf_counter()
    assert lib.crc_wait_probe(ctypes.byref(p), st.ptr, st.nbytes, kind, limit,
                              torch.cuda.current_stream().cuda_stream) == C.CRC_OK
    with pytest.raises(C.CrcError) as e:
        st.read()                                        # synchronises, reads the error word
    dt = time.perf_counter() - t0
    assert e.value.code == C.CRC_ETIMEOUT
    assert 0.05 <= dt < 1.5, dt
    assert C.crc_device_error() == C.CRC_OK
    # the context is intact: the fused step on a fresh state equals the two-kernel path
    Wd = C.synth_weights(w.L, w.N, w.d, seed=1)
    hd, _ = C.synth_hidden(w.B, w.T, w.L, w.d, seed=2)
    s1, s2 = C.State(p), C.State(p)
    ws = torch.empty(C.crc_fused_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    C.route_and_cache(p, hd, Wd, s1, workspace=ws)
    C.cache_scan(p, C.route_scores(p, hd, Wd), s2)
    r1 = s1.read(want_caches=True)
    r2 = s2.read(want_caches=True)
    assert r1["error"] == 0 and r1["tokens"] == w.T
    assert (r1["cache_bits"] == r2["cache_bits"]).all() and r1["misses"] == r2["misses"]


def test_checkpoint_to_host_and_resume_elsewhere(C):
    """Checkpoint / resume: the state is position-independent bytes.  Copy it
    to the host after T1 tokens, restore it into a fresh buffer (another
    address), continue with the remaining tokens: the same final caches,
    counters and carried scores as one uninterrupted call."""
    w = S.QWEN3_30B.with_(B=2, T=300, L=3, d=128)
    p = C.problem_of(w)
    Wd = C.synth_weights(w.L, w.N, w.d, seed=7)
    hd, _ = C.synth_hidden(w.B, w.T, w.L, w.d, seed=8)
    ws = torch.empty(C.crc_fused_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    whole = C.State(p)
    C.route_and_cache(p, hd, Wd, whole, workspace=ws)
    ref = whole.read(want_caches=True, want_retention=True, want_chain_counters=True)
    T1 = 170
    first = C.State(p)
    C.route_and_cache(p, hd[:, :T1].contiguous(), Wd, first, workspace=ws)
    saved = first.buf.cpu()                                # checkpoint
    del first
    resumed = C.State(p)
    resumed.buf.copy_(saved)                               # resume into a new buffer
    assert resumed.ptr != saved.data_ptr()
    C.route_and_cache(p, hd[:, T1:].contiguous(), Wd, resumed, workspace=ws)
    got = resumed.read(want_caches=True, want_retention=True, want_chain_counters=True)
    for k, v in ref.items():
        if hasattr(v, "shape"):
            assert (v == got[k]).all(), k
        else:
            assert v == got[k], k


def test_refused_launches_leave_no_error_behind(C):
    """A call whose launch the runtime refuses (its stream's capture has been
    invalidated, a host-side refusal) returns CRC_ECUDA, and the next call on
    an ordinary stream does not report that error as its own."""
    rt = ctypes.CDLL("libcudart.so.13")          # PyTorch's; the library has a runtime of its own
    w = S.QWEN3_30B.with_(B=4, T=100, L=2, d=128)
    p = C.problem_of(w)
    W = C.synth_weights(w.L, w.N, w.d, seed=1)
    h, _ = C.synth_hidden(w.B, w.T, w.L, w.d, seed=2)
    small = S.TINY.with_(B=2, L=2)
    ps = C.problem_of(small)
    Ws = C.synth_weights(small.L, small.N, small.d, seed=1)
    hs, _ = C.synth_hidden(2, 1, small.L, small.d, seed=2)
    st, st1 = C.State(p), C.State(ps)
    out = torch.empty((w.B, w.T, w.L, 3, w.N), device="cuda")
    ws = torch.empty(C.crc_fused_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    ws1 = torch.empty(C.crc_fused_workspace_bytes(ps), dtype=torch.uint8, device="cuda")
    loss = torch.empty((w.B, w.T, w.L, 2), device="cuda")
    means = torch.empty(2, dtype=torch.float64, device="cuda")
    lws = torch.empty(max(256, C.crc_loss_workspace_bytes(p, w.T)), dtype=torch.uint8,
                      device="cuda")
    calls = {
        "pair heads": lambda s: C.route_scores(p, h, W, out=out, stream=s),
        "short": lambda s: C.route_and_cache(ps, hs, Ws, st1, workspace=ws1, stream=s),
        "fused": lambda s: C.route_and_cache(p, h, W, st, workspace=ws, stream=s),
        "scan": lambda s: C.cache_scan(p, out, st, stream=s),
        "policy": lambda s: C.cache_scan_policy(p, out, st, "lru", stream=s),
        "loss": lambda s: C.cache_loss(p, out, 8, 0.05, grad=False, loss=loss, means=means,
                                       workspace=lws, stream=s),
        "state": lambda s: C.crc_state_init(p, st.ptr, st.nbytes, s),
    }
    for call in calls.values():                  # one-time setup is done outside any capture
        st.init()
        call(None)
    torch.cuda.synchronize()
    for name, call in calls.items():
        s = ctypes.c_void_p()
        assert rt.cudaStreamCreateWithFlags(ctypes.byref(s), 1) == 0      # non-blocking
        assert rt.cudaStreamBeginCapture(s, 2) == 0
        assert rt.cudaStreamSynchronize(s) != 0          # not permitted: ends the capture's validity
        with pytest.raises(C.CrcError) as e:
            call(s.value)
        assert e.value.code == C.CRC_ECUDA, name
        graph = ctypes.c_void_p()
        assert rt.cudaStreamEndCapture(s, ctypes.byref(graph)) != 0
        rt.cudaGetLastError()
        st.init()                                        # raises if it finds the old error
        assert rt.cudaStreamDestroy(s) == 0
    # a size that the generator refuses after asking the runtime for its shared memory
    with pytest.raises(C.CrcError) as e:
        C.crc_synth_hidden(1, 1, 4096, 64, 0, 0, 0.5, 0.5, None, h.data_ptr(), out.data_ptr())
    assert e.value.code == C.CRC_EUNSUPPORTED
    st.init()
    C.route_and_cache(p, h, W, st, workspace=ws)
    assert st.read()["tokens"] == w.T
