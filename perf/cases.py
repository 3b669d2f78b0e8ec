"""The measured work of this framework: what a program that uses it has it do.

A serving loop calls the fused step once per decoded token (or once per short
chunk of tokens) for all of its streams, continuing one cache state, and reads
the access trace to know which experts to move; an offline evaluation replays
whole recorded sequences from a cold cache, or compares the caching policies
over one set of router probabilities; a training step runs the router heads
and the coverage losses with their gradient.  Sizes are the repository's
configurations (`crc_synth.WORKLOADS`) and ragged ones of the same kind.

Inputs are what the benchmark uses: hidden states from the seeded AR(1)
generator (unit variance, correlated over tokens and layers), router weights
N(0, 1/d).  Calls that continue a state walk a window of successive inputs, so
that successive passes see successive tokens and the caches keep changing.
"""
import math

import torch

import paper_2609_04895_gb300 as P

BF16, F32 = 2, 4

# Backbone shapes of the repository's workloads (layers, experts, Top-K,
# hidden size, cache slots, refinement budget, token correlation), and a
# generic one with 64 experts.
SHAPES = {
    "tiny": dict(L=4, N=16, K=2, d=256, C=4, R=1, rho=0.9),
    "gptoss": dict(L=24, N=32, K=4, d=2880, C=8, R=2, rho=0.85),
    "n64": dict(L=26, N=64, K=6, d=2048, C=16, R=2, rho=0.9),
    "qwen3": dict(L=48, N=128, K=8, d=2048, C=32, R=4, rho=0.9),
    "large": dict(L=94, N=128, K=8, d=4096, C=32, R=8, rho=0.9),
}
POLICIES = ("lru", "lfu", "lrfu", "spatio_lru")
WARM = 8            # tokens a continued state has seen before the measured calls


def _case(name, kind, shape, B, T, **over):
    c = dict(name=name, kind=kind, **SHAPES[shape], B=B, T=T)
    c.update(over)
    return c


def listed():
    return [
        # one decoded token of a few streams of the smallest configuration:
        # nothing but latency and launches
        _case("decode-tiny", "step", "tiny", 4, 1, window=64),
        # one decoded token of a full serving batch
        _case("decode-qwen3", "step", "qwen3", 64, 1, window=32),
        # the same for the 32-expert backbone with a batch that is not a power of two
        _case("decode-gptoss", "step", "gptoss", 37, 1, window=32),
        # a short chunk per call (chunked prefill, several draft tokens), odd batch and length
        _case("chunk-qwen3", "step", "qwen3", 13, 24, window=8),
        # one chunk of the largest configuration, streamed chunk by chunk: d = 4096, R = 8
        _case("chunk-large", "step", "large", 64, 128, window=2),
        # one recorded sequence replayed on its own, as in the paper's batch-1 evaluation
        _case("stream-qwen3", "replay", "qwen3", 1, 1000),
        # the benchmark's workload: 64 sequences of 1024 tokens from a cold cache
        _case("replay-qwen3", "replay", "qwen3", 64, 1024),
        # 32 experts, d = 2880, a length that fills no whole number of tiles
        _case("replay-gptoss", "replay", "gptoss", 64, 1000),
        # the update-only capacity sweep: two heads, no refinement, ragged length
        _case("replay-update-only", "replay", "qwen3", 48, 777, C=64, R=0),
        # the router heads alone (a trainer's forward pass)
        _case("scores-qwen3", "scores", "qwen3", 24, 500),
        # the method and the four comparison policies over the same probabilities
        _case("compare-policies", "compare", "qwen3", 40, 600),
        # the coverage losses and their gradient, the paper's B = 20 and tau = 0.03
        _case("loss-qwen3", "loss", "qwen3", 64, 512, top_b=20, tau=0.03),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "replay", "replay", "scores", "compare", "loss"])
    shape = rng.choice(["tiny", "gptoss", "n64", "qwen3", "qwen3", "large"])
    s = dict(SHAPES[shape])
    s["K"] = rng.randint(1, s["K"])
    s["C"] = rng.randint(s["K"], max(s["K"], s["N"] // 2))
    s["R"] = rng.choice([0, 1, 2, 4, 8]) if s["N"] > 16 else rng.choice([0, 1, 2])
    # tokens x streams so that a pass costs no more than a fraction of the largest case
    units = {"step": 4.0e5, "replay": 8.0e5, "scores": 4.0e5, "compare": 6.0e5, "loss": 8.0e5}[kind]
    most = max(4, int(units / s["L"] * min(1.0, 2048.0 / s["d"])))
    if kind == "step":
        B = _log_int(rng, 1, 128)
        T = rng.choice([1, 1, _log_int(rng, 1, max(1, min(128, most // B)))])
    else:
        B = _log_int(rng, 1, 64)
        T = _log_int(rng, min(16, most // B), max(16, min(1500, most // B)))
    c = dict(kind=kind, **s, B=B, T=T)
    if kind == "step":
        c["window"] = 4
    if kind == "loss":
        c["top_b"] = rng.randint(1, s["N"] // 4)
        c["tau"] = rng.choice([0.01, 0.03, 0.1])
    return c


def _problem(c):
    return P.crc.problem(c["L"], c["N"], c["K"], c["d"], c["C"], c["R"], c["B"],
                         3 * c["d"] * 768 * BF16)


def _hidden(c, seed, T, t0=0, carry=None):
    return P.synth_hidden(c["B"], T, c["L"], c["d"], seed=seed, rho_t=c["rho"], t0=t0,
                          carry=carry)


def _weights(c, seed):
    return P.synth_weights(c["L"], c["N"], c["d"], seed=seed + 1)


def _probs(c, seed):
    """Router probabilities [B][T][L][3][N]: the softmax of unit-variance
    logits correlated over tokens, the law that random router weights give."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    z = torch.randn((c["B"], c["T"], c["L"], 3, c["N"]), device="cuda", generator=g)
    r, s = c["rho"], math.sqrt(1.0 - c["rho"] ** 2)
    for t in range(1, c["T"]):
        z[:, t].mul_(s).add_(z[:, t - 1], alpha=r)
    return torch.softmax(z, dim=-1, out=z) if z.numel() else z


def prepare(case, seed):
    c = case
    p = _problem(c)
    s = {"case": c, "p": p}
    if c["kind"] in ("step", "replay"):
        s["W"] = _weights(c, seed)
        s["state"] = P.State(p)
        s["ws"] = torch.empty(P.crc.crc_fused_workspace_bytes(p), dtype=torch.uint8, device="cuda")
    if c["kind"] == "step":
        h, carry = _hidden(c, seed, WARM)
        P.route_and_cache(p, h, s["W"], s["state"], None, workspace=s["ws"])
        s["inputs"] = []
        for i in range(c["window"]):
            h, carry = _hidden(c, seed, c["T"], t0=WARM + i * c["T"], carry=carry)
            s["inputs"].append(h)
        s["next"] = 0
        s["trace"] = P.Trace.alloc(p, c["T"], caches=True, rank_order=False, topk_set=True)
    elif c["kind"] == "replay":
        s["h"], _ = _hidden(c, seed, c["T"])
    elif c["kind"] == "scores":
        s["W"] = _weights(c, seed)
        s["h"], _ = _hidden(c, seed, c["T"])
        s["out"] = torch.empty((c["B"], c["T"], c["L"], 3, c["N"]), device="cuda")
    elif c["kind"] == "compare":
        s["probs"] = _probs(c, seed)
        s["states"] = {n: P.State(p) for n in ("method",) + POLICIES}
    elif c["kind"] == "loss":
        s["probs"] = _probs(c, seed)
        s["loss"] = torch.empty((c["B"], c["T"], c["L"], 2), device="cuda")
        s["means"] = torch.empty(2, dtype=torch.float64, device="cuda")
        s["grad"] = torch.empty_like(s["probs"])
        s["ws"] = torch.empty(max(256, P.crc.crc_loss_workspace_bytes(p, c["T"])),
                              dtype=torch.uint8, device="cuda")
    return s


def _state_views(c, state):
    """The state buffer's parts: per chain the cache bitmask and the counters,
    the retention scores, the carried Spatio predictions."""
    B, L, N = c["B"], c["L"], c["N"]
    r0 = 256 + 64 * B * L
    c0 = r0 + F32 * B * L * N
    f = state.buf.view(torch.float32)
    return {"chains": state.buf[256:r0].view(torch.int32).view(B, L, 16),
            "retention": f[r0 // 4:c0 // 4].view(B, L, N),
            "carry": f[c0 // 4:c0 // 4 + 2 * B * N].view(2, B, N)}


def run(state):
    s = state
    c, p = s["case"], s["p"]
    kind = c["kind"]
    if kind == "step":
        h = s["inputs"][s["next"]]
        s["next"] = (s["next"] + 1) % len(s["inputs"])
        tr = s["trace"]
        P.route_and_cache(p, h, s["W"], s["state"], tr, workspace=s["ws"])
        return dict(_state_views(c, s["state"]), misses=tr.misses, proactive=tr.proactive,
                    cache_mid=tr.cache_mid, cache_after=tr.cache_after, topk=tr.topk_set)
    if kind == "replay":
        s["state"].init()
        P.route_and_cache(p, s["h"], s["W"], s["state"], None, workspace=s["ws"])
        return _state_views(c, s["state"])
    if kind == "scores":
        return P.route_scores(p, s["h"], s["W"], heads=3, out=s["out"])
    if kind == "compare":
        out = {}
        for name, st in s["states"].items():
            st.init()
            if name == "method":
                P.cache_scan(p, s["probs"], st)
            else:
                P.crc.cache_scan_policy(p, s["probs"], st, name)
            v = _state_views(c, st)
            out[name] = {"chains": v["chains"], "retention": v["retention"]}
        return out
    if kind == "loss":
        return P.cache_loss(p, s["probs"], c["top_b"], c["tau"], loss=s["loss"], means=s["means"],
                            grad_out=s["grad"], workspace=s["ws"])
    raise ValueError(kind)


def work(case):
    """What a pass has to read, write and multiply, each array once."""
    c = case
    B, T, L, N, d = c["B"], c["T"], c["L"], c["N"], c["d"]
    units = B * T * L
    heads = 3 if c["R"] > 0 else 2
    chain_state = B * L * (64 + F32 * N)
    words = (N + 31) // 32
    if c["kind"] in ("step", "replay"):
        b = units * d * BF16 + L * heads * N * d * BF16
        if c["kind"] == "step":
            b += 2 * chain_state + units * (2 + 3 * words * 4)
        else:
            b += chain_state
        return {"bytes": b, "flops": 2.0 * units * heads * N * d}
    if c["kind"] == "scores":
        return {"bytes": units * (d * BF16 + 3 * N * F32) + L * 3 * N * d * BF16,
                "flops": 2.0 * units * 3 * N * d}
    if c["kind"] == "compare":
        return {"bytes": units * 3 * N * F32 + 5 * chain_state, "flops": 0.0}
    return {"bytes": units * (6 * N * F32 + 8), "flops": 0.0}


def tolerance(case):
    c = case
    if c["kind"] == "compare":
        # comparisons, sums of two and products of two fp32 values in a stated order
        return "exact"
    if c["kind"] == "loss":
        # fp32 terms and sums of N products with approximate exponentials and reciprocals
        return {"rel": 1e-6, "max": 1e-4}
    if c["kind"] == "scores":
        # bf16 products summed in fp32 over d, softmax with an approximate exponential
        return {"rel": 2e-5, "max": 2e-4}
    # the same for s^T and p^S; a rounding may turn a decision between two
    # nearly equal scores, which moves a few cache words and counters
    return {"rel": 2e-5, "max": 2e-4, "differ": 2e-3}


# --------------------------------------------------------------------------- #
# 64-bit values, without this repository's kernels
# --------------------------------------------------------------------------- #
def _probs64(h, W, N):
    """softmax in 64 bits of hidden [M][L][d] against W [L][3N][d]: [M][L][3][N]."""
    M, L = h.shape[:2]
    out = torch.empty((M, L, 3, N), dtype=torch.float64, device=h.device)
    for l in range(L):
        z = h[:, l].double() @ W[l].double().t()
        out[:, l] = torch.softmax(z.view(M, 3, N), dim=-1)
    return out


def _loss64(c, probs):
    B, T, L, N = c["B"], c["T"], c["L"], c["N"]
    tau, top_b = c["tau"], c["top_b"]
    n = B * (T - 1) * L
    loss = torch.zeros((B, T, L, 2), dtype=torch.float64, device=probs.device)
    grad = torch.zeros((B, T, L, 3, N), dtype=torch.float64, device=probs.device)

    def term(s32, s, q):
        # theta is the top_b-th entry of the fp32 priorities, score descending, index ascending
        e = torch.sort(s32, dim=-1, descending=True, stable=True)[1][..., top_b - 1:top_b]
        m = torch.sigmoid((s - s.gather(-1, e)) / tau)
        return (q * (1.0 - m)).sum(-1)

    for b in range(B):
        x = probs[b]
        p = x.double().requires_grad_(True)
        # p^S of the causal predecessor of (t, l), t >= 1
        def rho(y):
            return torch.cat([y[:-1, -1:, 2], y[1:, :-1, 2]], dim=1)
        sT32 = x[:-1, :, 0] + x[:-1, :, 1]
        sT = p[:-1, :, 0] + p[:-1, :, 1]
        lT = term(sT32, sT, p[1:, :, 0])
        lST = term(sT32 + rho(x), sT + rho(p), p[1:, :, 0])
        ((lT.sum() + lST.sum()) / n).backward()
        loss[b, :-1, :, 0] = lT.detach()
        loss[b, 1:, :, 1] = lST.detach()
        g, pd = p.grad, p.detach()
        grad[b] = pd * (g - (pd * g).sum(-1, keepdim=True))
    return loss, loss.sum(dim=(0, 1, 2)) / max(n, 1), grad


def exact(case, seed):
    c = case
    B, T, L, N = c["B"], c["T"], c["L"], c["N"]
    if c["kind"] in ("step", "replay"):
        W = _weights(c, seed)
        if c["kind"] == "step":
            h0, k = _hidden(c, seed, WARM)
            h, _ = _hidden(c, seed, T, t0=WARM, carry=k)
        else:
            h0, (h, _) = None, _hidden(c, seed, T)
        last = _probs64(h[:, -1], W, N)
        carry = None
        if c["R"] > 0:
            # the two carry slots alternate from call to call, slot 1 first
            other = torch.zeros((B, N), dtype=torch.float64, device="cuda")
            if h0 is None:
                carry = torch.stack([other, last[:, -1, 2]])
            else:
                carry = torch.stack([last[:, -1, 2], _probs64(h0[:, -1], W, N)[:, -1, 2]])
        out = {"chains": None, "retention": last[:, :, 0] + last[:, :, 1], "carry": carry}
        if c["kind"] == "step":
            out.update(misses=None, proactive=None, cache_mid=None, cache_after=None, topk=None)
        return out
    if c["kind"] == "scores":
        W = _weights(c, seed)
        h, _ = _hidden(c, seed, T)
        return _probs64(h.view(B * T, L, c["d"]), W, N).view(B, T, L, 3, N)
    if c["kind"] == "compare":
        pr = _probs(c, seed)[:, -1].double()
        out = {n: {"chains": None, "retention": None} for n in ("method",) + POLICIES}
        out["method"]["retention"] = pr[:, :, 0] + pr[:, :, 1]
        out["spatio_lru"]["retention"] = pr[:, :, 0]
        return out
    if T < 2:
        return None
    return _loss64(c, _probs(c, seed))
