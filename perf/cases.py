"""The work this library is timed on, through its public calls.

Three kinds of case, over the sizes of the five synthetic layers in paper_2310_15929_b200/inputs.py:

  product    esp_spgemm / esp_spgemm_grouped: the forward product of pruned linears, from one decode token to a prefill of
             8192 tokens; token-major and channel-major activations, fp16 and fp32 output, bias and ReLU
  prune      esp_metric_prune: statistics, score, both shuffles run to their end, selection, compression, packing
  calibrate  esp_calib_*: the channel statistics accumulated over chunks of calibration activations
"""
import math

import torch

from paper_2310_15929_b200 import binding as b

DEV = "cuda"


# ---------------------------------------------------------------------------------------------------------- the cases
def _product(name, M, K, Ns, layout="token", out="f16", bias_relu=False, calls=None):
    """Ns: output features of the linears of one pass as "N+N,N": a comma separates calls, a plus joins a grouped call; a
    linear whose input differs from K is written N:K."""
    c = {"kind": "product", "M": M, "K": K, "linears": Ns, "layout": layout, "out": out, "bias_relu": bias_relu}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one decode step of a LLaMA-7B-shaped layer as an engine runs it: q,k,v and gate,up grouped, one sequence
        _product("decode7b_m1", 1, 4096, "4096+4096+4096,4096,11008+11008,4096:11008"),
        # a small batch of decode sequences through one attention projection of a LLaMA-13B-shaped layer
        _product("decode13b_q_m16", 16, 5120, "5120"),
        # batched decode through the largest weight of the OPT-66B-shaped layer, with OPT's bias and ReLU
        _product("opt66b_fc1_m32", 32, 9216, "36864", layout="channel", bias_relu=True),
        # the smallest layer: launch and latency bound
        _product("single512_m128", 128, 512, "512"),
        # a mid-sized ragged batch (chunked prefill, speculative decoding) through a down projection
        _product("down7b_m200", 200, 11008, "4096"),
        # a short prefill of the OPT-66B-shaped layer's attention projection
        _product("opt66b_q_m512", 512, 9216, "9216", layout="channel"),
        # prefill of an odd number of tokens through a gate projection, fp32 output kept for a later sum
        _product("gate7b_m2001_f32", 2001, 4096, "11008", out="f32"),
        # the largest prefill: 8192 tokens through a gate projection of the LLaMA-65B-shaped layer
        _product("gate65b_m8192", 8192, 8192, "22016", layout="channel"),
        # pruning the smallest layer: few rows, few tokens
        {"name": "prune512", "kind": "prune", "No": 512, "C": 512, "T": 128, "heavy": False, "outlier": 20.0},
        # pruning one attention projection of a LLaMA-7B-shaped layer on 16 x 2048 calibration tokens
        {"name": "prune7b_q", "kind": "prune", "No": 4096, "C": 4096, "T": 32768, "heavy": True, "outlier": 30.0},
        # pruning a gate projection of the LLaMA-13B-shaped layer on a shorter calibration set
        {"name": "prune13b_gate", "kind": "prune", "No": 13824, "C": 5120, "T": 8192, "heavy": True, "outlier": 30.0},
        # streaming calibration of a LLaMA-65B-shaped layer's input, eight sequences of 2048 tokens, each its own chunk
        {"name": "calib65b", "kind": "calibrate", "C": 8192, "T": 2048, "chunks": 8, "outlier": 30.0},
    ]


def _log_int(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choice(("decode", "decode", "middle", "prefill", "prefill", "prune", "prune", "calibrate"))
    if kind == "prune":
        return {"kind": "prune", "No": _log_int(rng, 512, 8192, 2 if rng.random() < 0.5 else 128),
                "C": _log_int(rng, 512, 5120, 8 if rng.random() < 0.5 else 256), "T": _log_int(rng, 128, 32768),
                "heavy": rng.random() < 0.7, "outlier": rng.choice((20.0, 30.0, 60.0))}
    if kind == "calibrate":
        return {"kind": "calibrate", "C": _log_int(rng, 512, 9216, 8), "T": _log_int(rng, 500, 2048),
                "chunks": rng.randint(1, 8), "outlier": rng.choice((20.0, 30.0, 60.0))}
    layout = rng.choice(("token", "channel"))
    out = "f32" if rng.random() < 0.2 else "f16"
    bias_relu = rng.random() < 0.25
    if kind == "decode":
        M, K, N = _log_int(rng, 1, 64), _log_int(rng, 512, 22016, 8), _log_int(rng, 512, 22016, 2)
        if rng.random() < 0.3:                              # same-input linears in one call (no bias there)
            return _product(None, M, K, "+".join([str(N)] * rng.randint(2, 3)), layout, out, False)
    elif kind == "middle":
        M, K, N = _log_int(rng, 65, 1024), _log_int(rng, 512, 11008, 8), _log_int(rng, 512, 11008, 2)
    else:
        M, K, N = _log_int(rng, 1024, 8192), _log_int(rng, 2048, 9216, 8), _log_int(rng, 2048, 16384, 8)
    return _product(None, M, K, str(N), layout, out, bias_relu)


def _linears(case):
    """[[(N, K), ...] per call]"""
    return [[(int(s.split(":")[0]), int(s.split(":")[1]) if ":" in s else case["K"]) for s in call.split("+")]
            for call in case["linears"].split(",")]


# ------------------------------------------------------------------------------------------------------------- inputs
def _weight(g, No, C, heavy):
    """N(0, 0.02^2) rows; heavy: each row scaled so that the marginals are Student-t with four degrees of freedom."""
    scale = torch.full((No, 1), 0.02, device=DEV)
    if heavy:
        chi2 = torch.randn(No, 4, generator=g, device=DEV).square().sum(1, keepdim=True)
        scale = scale * torch.sqrt(4.0 / chi2)
    W = torch.empty(No, C, dtype=torch.float16, device=DEV)
    for r in range(0, No, 8192):
        n = min(8192, No - r)
        W[r:r + n] = torch.randn(n, C, generator=g, device=DEV).mul_(scale[r:r + n]).half()
    return W


def _activations(g, T, C, outlier):
    """N(0, 1) with one channel in a hundred scaled up: the outlier channels of a trained model."""
    scale = torch.where(torch.rand(C, generator=g, device=DEV) < 0.01, outlier, 1.0)
    X = torch.empty(T, C, dtype=torch.float16, device=DEV)
    for r in range(0, T, 8192):
        n = min(8192, T - r)
        X[r:r + n] = torch.randn(n, C, generator=g, device=DEV).mul_(scale).half()
    return X


def _compressed(g, N, K):
    """(packed weight, permutation) of a pruned linear: global shuffle and 2:4 selection under a score like the metric's."""
    W = _weight(g, N, K, True)
    score = torch.rand(K, generator=g, device=DEV, dtype=torch.float64) + 3.5
    score[torch.rand(K, generator=g, device=DEV) < 0.01] += 30.0
    o = b.esp_prune_opts_default()
    o.use_lbs = 0
    o.score_override = score.data_ptr()
    ws = torch.empty(b.esp_metric_prune_workspace_bytes(N, K, 0, o), dtype=torch.uint8, device=DEV)
    vals = torch.empty(N, K // 2, dtype=torch.float16, device=DEV)
    meta = torch.empty(N, K // 8, dtype=torch.uint8, device=DEV)
    perm = torch.empty(K, dtype=torch.int32, device=DEV)
    packed = torch.empty(b.esp_packed_bytes(N, K), dtype=torch.uint8, device=DEV)
    b.esp_metric_prune(W, None, o, vals, meta, perm, packed, workspace=ws)
    torch.cuda.current_stream().synchronize()               # W, the score and the scratch end here
    return packed, perm


def _prepare_product(case, g):
    M = case["M"]
    o = b.esp_gemm_opts_default()
    o.x_layout = b.ESP_X_CHANNEL_MAJOR if case["layout"] == "channel" else b.ESP_X_TOKEN_MAJOR
    o.out_dtype = b.ESP_OUT_F32 if case["out"] == "f32" else b.ESP_OUT_F16
    o.static_weights = 1                                    # inference: nothing on the stream writes weights
    o.activation = b.ESP_ACT_RELU if case["bias_relu"] else b.ESP_ACT_NONE
    out_t = torch.float32 if case["out"] == "f32" else torch.float16
    calls, ws_bytes, keep = [], 16, []
    for call in _linears(case):
        K = call[0][1]
        X = _activations(g, M, K, 30.0)
        if case["layout"] == "channel":
            Xt = torch.zeros(K, (M + 7) // 8 * 8, dtype=torch.float16, device=DEV)
            Xt[:, :M] = X.t()
            X = Xt[:, :M]
        weights = [_compressed(g, N, K) for N, _ in call]
        Ys = [torch.zeros(M, N, dtype=out_t, device=DEV) for N, _ in call]
        ws_bytes = max(ws_bytes, len(call) * b.esp_spgemm_workspace_bytes(M, max(N for N, _ in call), K, o))
        if case["bias_relu"]:
            keep.append((0.1 * torch.randn(call[0][0], generator=g, device=DEV)).half())
            o.bias = keep[-1].data_ptr()
        calls.append((X, [w[0] for w in weights], [w[1] for w in weights], Ys))
    return {"opts": o, "calls": calls, "ws": torch.empty(ws_bytes, dtype=torch.uint8, device=DEV), "keep": keep}


def _prepare_prune(case, g):
    No, C, T = case["No"], case["C"], case["T"]
    o = b.esp_prune_opts_default()
    o.alpha = 1.0 / math.sqrt(T)
    return {"opts": o, "W": _weight(g, No, C, case["heavy"]), "X": _activations(g, T, C, case["outlier"]),
            "vals": torch.empty(No, C // 2, dtype=torch.float16, device=DEV),
            "meta": torch.empty(No, C // 8, dtype=torch.uint8, device=DEV),
            "perm": torch.empty(C, dtype=torch.int32, device=DEV),
            "packed": torch.empty(b.esp_packed_bytes(No, C), dtype=torch.uint8, device=DEV),
            "score": torch.empty(C, dtype=torch.float64, device=DEV),
            "ws": torch.empty(b.esp_metric_prune_workspace_bytes(No, C, T, o), dtype=torch.uint8, device=DEV)}


def _prepare_calibrate(case, g):
    C = case["C"]
    o = b.esp_prune_opts_default()
    T = case["T"] * case["chunks"]
    o.alpha = 1.0 / math.sqrt(T)
    X = _activations(g, T, C, case["outlier"])
    f64 = lambda: torch.empty(C, dtype=torch.float64, device=DEV)
    return {"opts": o, "C": C, "T": T, "chunks": list(X.split(case["T"])), "norm": f64(), "entropy": f64(), "score": f64(),
            "state": torch.empty(b.esp_calib_state_bytes(C, o.bins), dtype=torch.uint8, device=DEV)}


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    make = {"product": _prepare_product, "prune": _prepare_prune, "calibrate": _prepare_calibrate}[case["kind"]]
    return dict(make(case, g), kind=case["kind"])


# ------------------------------------------------------------------------------------------------------------ one pass
def run(state):
    s, o = state, state["opts"]
    if s["kind"] == "product":
        for X, packed, perm, Y in s["calls"]:
            if len(Y) == 1:
                b.esp_spgemm(X, packed[0], perm[0], Y[0], o, s["ws"])
            else:
                b.esp_spgemm_grouped([X] * len(Y), packed, perm, Y, o, s["ws"])
        return [y for call in s["calls"] for y in call[3]]
    if s["kind"] == "prune":
        stats = b.esp_prune_stats()
        b.esp_metric_prune(s["W"], s["X"], o, s["vals"], s["meta"], s["perm"], s["packed"], chan_score=s["score"], stats=stats,
                           workspace=s["ws"])
        return [s["vals"], s["meta"], s["perm"], s["packed"], s["score"], int(stats.lbs_swaps_total), int(stats.near_tie_groups),
                int(stats.near_tie_sort), int(stats.near_tie_swaps), float(stats.obj_identity), float(stats.obj_after_gns),
                float(stats.obj_after_lbs)]
    b.esp_calib_reset(s["state"], s["C"], o.bins)
    for x in s["chunks"]:
        b.esp_calib_range(s["state"], x, o.bins)
    for x in s["chunks"]:
        b.esp_calib_histogram(s["state"], x, o.bins)
    b.esp_calib_finish(s["state"], s["C"], s["T"], o, s["norm"], s["entropy"], s["score"])
    return [s["norm"], s["entropy"], s["score"]]


def work(case):
    if case["kind"] == "product":
        M, item = case["M"], 4 if case["out"] == "f32" else 2
        nbytes = flops = 0.0
        for call in _linears(case):
            K = call[0][1]
            nbytes += 2.0 * M * K
            for N, _ in call:
                nbytes += 1.125 * N * K + float(item) * M * N + 4.0 * K
                flops += 1.0 * M * N * K                    # two operations for every kept weight: half of the dense product's
        return {"bytes": nbytes, "flops": flops}
    if case["kind"] == "prune":
        No, C, T = case["No"], case["C"], case["T"]
        # read W and the activations, write the compressed and the packed weight; the block shuffle's first table compares
        # every channel of a block with every slot of the block, in every row
        return {"bytes": 2.0 * No * C + 2.0 * T * C + 2 * 1.125 * No * C + 12.0 * C, "flops": 2.0 * 256 * No * C}
    return {"bytes": 2.0 * case["T"] * case["chunks"] * case["C"] + 24.0 * case["C"],
            "flops": 4.0 * case["T"] * case["chunks"] * case["C"]}


def tolerance(case):
    # Four times the distance of this path from the same product in fp64: fp16 output 2.1e-4 (max 5.0e-4: the rounding of the
    # result), fp32 output 2.3e-6 (max 4.4e-5: fp32 accumulation).
    if case["kind"] == "product":
        return {"rel": 1e-5, "max": 2e-4} if case["out"] == "f32" else {"rel": 8e-4, "max": 2e-3}
    # Statistics are fp64 sums (2e-16 from the same additions in another order, the entropy a few ulps of its logarithms);
    # everything discrete follows from them and stays the same.
    return {"rel": 1e-14, "max": 1e-12}
