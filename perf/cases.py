"""The work that users of this library have it do, as cases with inputs, one pass, necessary work and tolerance.

A case is a plain dict.  Its "kind" says which public entry points a pass goes through:

  linear    one elutq_lut_gemm call on one layer
  block     the four merged linears of a transformer block (qkv, o, gate_up, down) as separate elutq_lut_gemm calls
  step      a decode step (M = 1): the four linears once per bit-width of "qs", planned once and run as one chain
  host      one elutq_lut_gemm_host call: activations and outputs in pinned host memory
  quantise  the offline step: elutq_hlq_fit on dense fp16 weights, then elutq_pack

Sizes are those of the benchmark configurations (LLaMA-3.1 8B and 70B linears with q/k/v and gate/up merged) and
generic ones; values follow the benchmark's recipe: activations N(0,1), on request with 1 % of the channels times 20,
bit-planes Bernoulli(1/2), scales |N(0,0.02)|, offsets N(0,0.01).
"""

import torch

import paper_2510_19482_b200 as elutq

# A transformer block: width of the merged q/k/v output, hidden width, inner width of the feed-forward part
LLAMA_8B = {"qkv": 6144, "hidden": 4096, "ffn": 14336}
LLAMA_70B = {"qkv": 10240, "hidden": 8192, "ffn": 28672}


def listed():
    return [
        # the smallest call: one token through one attention-output layer (launches and latency)
        {"name": "decode_one_call", "kind": "linear", "M": 1, "N": 4096, "K": 4096, "q": 2, "G": 128, "outliers": False},
        # one token through a block without a plan, as a framework calls layer by layer
        {"name": "decode_block_q4", "kind": "block", **LLAMA_8B, "M": 1, "q": 4, "G": 128, "outliers": False},
        # the headline decode step: twelve planned linears, 2-, 3- and 4-bit
        {"name": "decode_step_8b", "kind": "step", **LLAMA_8B, "qs": "234", "G": 128},
        # the large model's decode step
        {"name": "decode_step_70b", "kind": "step", **LLAMA_70B, "qs": "23", "G": 128},
        # activations come from and go to a host program: a few requests at once
        {"name": "host_call_m2", "kind": "host", "M": 2, "N": 6144, "K": 4096, "q": 3, "G": 128, "outliers": False},
        # small-batch serving, 3-bit, activations with outlier channels
        {"name": "batch4_block_q3", "kind": "block", **LLAMA_8B, "M": 4, "q": 3, "G": 128, "outliers": True},
        # batched decoding, 2-bit
        {"name": "batch16_block_q2", "kind": "block", **LLAMA_8B, "M": 16, "q": 2, "G": 128, "outliers": True},
        # finer quantisation groups on odd sizes, a batch that fills no tile
        {"name": "batch27_ragged_g64", "kind": "linear", "M": 27, "N": 5003, "K": 2880, "q": 3, "G": 64, "outliers": True},
        # a large layer at a large decoding batch, 4-bit
        {"name": "batch64_gate_up_70b_q4", "kind": "linear", "M": 64, "N": 57344, "K": 8192, "q": 4, "G": 128, "outliers": False},
        # a short prompt
        {"name": "prefill384_block_q2", "kind": "block", **LLAMA_8B, "M": 384, "q": 2, "G": 128, "outliers": False},
        # a long prompt: the largest work
        {"name": "prefill2048_block_q2", "kind": "block", **LLAMA_8B, "M": 2048, "q": 2, "G": 128, "outliers": False},
        # quantising a layer: Algorithm 1 with the paper's ten rounds, then packing
        {"name": "quantise_4096_q2", "kind": "quantise", "N": 4096, "K": 4096, "q": 2, "G": 128, "rounds": 10},
    ]


def _log(rng, lo, hi):
    """A whole number, its logarithm uniform over [lo, hi]."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def _draw_block(rng):
    hidden = 128 * _log(rng, 8, 64)
    return {"qkv": hidden + 256 * rng.randint(1, hidden // 256), "hidden": hidden, "ffn": 128 * int(hidden * rng.uniform(2.5, 3.6) / 128)}


def draw(rng):
    kind = rng.choice(["linear", "linear", "linear", "block", "block", "step", "host", "quantise"])
    q = rng.choice([2, 3, 4])
    outliers = rng.random() < 0.5
    if kind == "linear":
        G = rng.choice([128, 128, 128, 64])
        N, K = _log(rng, 1000, 57344), G * _log(rng, 1024 // G, 16384 // G)
        # bounded by the multiply-adds (prefill is done at G = 128; finer groups: decoding and small batches)
        top = min(2048, int(2.5e11 / (N * K))) if G == 128 else min(32, int(6e9 / (N * K)))
        return {"kind": kind, "M": _log(rng, 1, max(1, top)), "N": N, "K": K, "q": q, "G": G, "outliers": outliers}
    if kind == "block":
        case = {"kind": kind, **_draw_block(rng), "M": 1, "q": q, "G": 128, "outliers": outliers}
        case["M"] = _log(rng, 1, min(2048, int(2.5e11 / sum(n * k for _, n, k in _shapes(case)))))
        return case
    if kind == "step":
        return {"kind": kind, **_draw_block(rng), "qs": rng.choice(["2", "3", "4", "23", "34", "234"]), "G": 128}
    G = rng.choice([128, 128, 64, 32])
    if kind == "host":
        return {"kind": kind, "M": _log(rng, 1, 64), "N": _log(rng, 1000, 28672), "K": G * _log(rng, 1024 // G, 8192 // G),
                "q": q, "G": G, "outliers": outliers}
    return {"kind": kind, "N": _log(rng, 256, 2048), "K": G * _log(rng, 1024 // G, 4096 // G), "q": q, "G": G,
            "rounds": rng.choice([5, 10])}


def _shapes(case):
    """(q, N, K) of every call of a pass."""
    if case["kind"] in ("block", "step"):
        hidden, ffn = case["hidden"], case["ffn"]
        linears = ((case["qkv"], hidden), (hidden, hidden), (2 * ffn, hidden), (hidden, ffn))     # in model order
        return [(int(c), n, k) for c in str(case.get("qs", case.get("q"))) for n, k in linears]
    return [(case["q"], case["N"], case["K"])]


def _activations(gen, M, K, outliers):
    x = torch.randn((M, K), generator=gen, device="cuda", dtype=torch.float32)
    if outliers:
        x[:, torch.randperm(K, generator=gen, device="cuda")[: (K + 99) // 100]] *= 20.0
    return x.half()


def _layer(gen, q, G, N, K):
    planes = torch.randint(0, 2, (q, N, K), generator=gen, device="cuda", dtype=torch.uint8)
    scales = (torch.randn((N, K // G, q), generator=gen, device="cuda", dtype=torch.float32) * 0.02).abs().half()
    offsets = (torch.randn((N, K // G), generator=gen, device="cuda", dtype=torch.float32) * 0.01).half()
    return elutq.elutq_pack(planes, scales, offsets, q, G, N, K)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    if kind == "quantise":
        # dense weights as trained layers have them: a narrow bell with a few large entries
        W = torch.randn((case["N"], case["K"]), generator=gen, device="cuda", dtype=torch.float32) * 0.02
        W = torch.where(torch.rand(W.shape, generator=gen, device="cuda") < 0.002, W * 6.0, W).half()
        return {"case": case, "W": W}
    M = case.get("M", 1)
    calls = []
    for q, N, K in _shapes(case):
        x = _activations(gen, M, K, case.get("outliers", False))
        y = torch.empty((M, N), dtype=torch.float16, device="cuda")
        calls.append((x, _layer(gen, q, case["G"], N, K), y, N, K))
    state = {"case": case, "M": M, "calls": calls}
    if kind == "step":
        state["plan"] = elutq.elutq_chain_plan(calls)
    if kind == "host":
        x, packed, y, N, K = calls[0]
        state["x_host"] = x.cpu().pin_memory()
        state["y_host"] = torch.empty((M, N), dtype=torch.float16, pin_memory=True)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "quantise":
        planes, scales, offsets = elutq.elutq_hlq_fit(state["W"], case["q"], case["G"], case["rounds"])
        packed = elutq.elutq_pack(planes, scales, offsets, case["q"], case["G"], case["N"], case["K"])
        return planes, scales, offsets, packed
    calls = state["calls"]
    if kind == "step":
        elutq.elutq_chain_run(state["plan"], len(calls))
        return [c[2] for c in calls]
    if kind == "host":
        _, packed, _, N, K = calls[0]
        elutq.elutq_lut_gemm_host(state["x_host"], packed, state["y_host"], state["M"], N, K)
        return state["y_host"]
    for x, packed, y, N, K in calls:
        elutq.elutq_lut_gemm(x, packed, y, state["M"], N, K)
    return [c[2] for c in calls]


def work(case):
    if case["kind"] == "quantise":
        n, g = case["N"] * case["K"], case["G"]
        q = case["q"]
        params = 2 * (q + 1) * (n // g)
        # dense weights in; one byte per bit-plane entry and the parameters out; these in again for the packing; blob out.
        # Every round needs at least one subtraction and one comparison per weight and bit, and one addition per bit set.
        return {"bytes": 2 * n + 2 * (q * n + params) + q * n // 8 + params, "flops": 3 * q * n * case["rounds"]}
    M = case.get("M", 1)
    G = case["G"]
    nbytes = flops = 0
    for q, N, K in _shapes(case):
        nbytes += q * N * K // 8 + 2 * (q + 1) * N * (K // G) + 2 * M * K + 2 * M * N
        flops += 2 * M * N * K
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Quantising is exact by design (fp64 in a fixed order, integer packing).
    if case["kind"] == "quantise":
        return "exact"
    # Measured against the product in 64 bits, and about four times that.  fp16 outputs from fp32 sums carry one rounding:
    # 2.1e-4 in norm, at most 2^-11 of a value.  Batches of more than a few rows may rebuild the weights in fp16: up to
    # 4.8e-4 in norm, 2.8e-3 of the mean magnitude in one element.
    if case.get("M", 1) <= 4 or case["G"] != 128:
        return {"rel": 8e-4, "max": 2e-3}
    return {"rel": 2e-3, "max": 1.2e-2}
