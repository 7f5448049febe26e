"""The work whose speed this library is judged by: linear layers evaluated through the public entry points.

A case is one of five kinds of calls:

  linear    `sq_linear` over one or more layers, as an inference step makes them: rotation + INT4
            quantisation of the tokens, then the W4A4 product (decode and prefill)
  wo        `sq_linear_wo` in the same way: fp16 activations, 4- or 3-bit weights (W4A16 / W3A16)
  grouped   `sq_linear_grouped`: the experts of one mixture-of-experts layer, tokens sorted by expert
  pack      `sq_pack_weight` / `sq_pack_weight_wo`: loading time, a layer's fp16 weights are rotated,
            quantised and packed

Activations carry the two kinds of outliers that the method is about (channels scaled x20 on every
token, four channels at +-1000 on the first one), weights are N(0, 0.02): the recipe of
`paper_2511_22316_b200.workloads`, drawn on the GPU.  A state holds what a serving program keeps: the
rotation handles, the packed weights, one workspace and the output buffers.

Decode cases run several layers with weights of their own, as a decoding step does, so that weights
come from HBM as they do in use and not from the L2 cache that a single layer would fit.
"""
import math

import torch

from paper_2511_22316_b200 import binding as sq

# (K, N) of the layers of the benchmark configurations, with the factor pair n1 x n2 = K they name.
_ATTN = (4096, 4096)
_UP, _DOWN = (4096, 14336), (14336, 4096)
_N2 = {512: 32, 1024: 32, 2048: 32, 3072: 64, 4096: 64, 5120: 64, 8192: 128, 11008: 64, 14336: 128, 28672: 128}


def _case(name, kind, rows, layers, n2=0, bits=4, experts=0):
    """`layers`: "KxN" of each layer, separated by blanks.  `n2`: the power-of-two factor (0: the
    configured one)."""
    case = {"kind": kind, "rows": rows, "layers": " ".join("%dx%d" % kn for kn in layers), "n2": n2, "bits": bits,
            "experts": experts}
    return dict(case, name=name) if name else case


def listed():
    return [
        # The smallest call: one layer of a tiny network, where launches and latency are all there is.
        _case("tiny_64x512x512", "linear", 64, [(512, 512)]),
        # One user decoding: the MLP of a block (gate, up, down), one token.
        _case("decode_m1", "linear", 1, [_UP, _UP, _DOWN]),
        # A batch of sixteen users decoding the same three layers.
        _case("decode_m16", "linear", 16, [_UP, _UP, _DOWN]),
        # A large, ragged decode batch.
        _case("decode_m50", "linear", 50, [_UP, _UP, _DOWN]),
        # A short prompt of odd length through the four attention projections.
        _case("prefill_m333_attn", "linear", 333, [_ATTN] * 4),
        # The headline layer: a 2048-token prompt through an attention projection.
        _case("prefill_m2048_attn", "linear", 2048, [_ATTN]),
        # The wide-input MLP projection of the same prompt (factor pair 172 x 64).
        _case("prefill_m2048_down", "linear", 2048, [(11008, 4096)]),
        # The largest call: 4096 tokens through the gate/up projection of a 70B-sized block.
        _case("prefill_m4096_70b", "linear", 4096, [(8192, 28672)]),
        # Weight-only deployment, decoding: W4A16 over the three MLP layers.
        _case("wo_decode_m16", "wo", 16, [_UP, _UP, _DOWN]),
        # Weight-only deployment, a prompt of odd length: W3A16.
        _case("wo_prefill_m777", "wo", 777, [(4096, 11008)], bits=3),
        # A mixture-of-experts layer decoding 16 tokens, two experts each.
        _case("grouped_decode_m32", "grouped", 32, [_UP], experts=8),
        # Loading a layer: offline rotation, quantisation and packing of its weights.
        _case("pack_11008x4096", "pack", 0, [(4096, 11008)]),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the same ranges: any batch size from one token to a long prompt, the layer
    shapes of the configurations and generic ones beside them, both usable factor pairs."""
    small = [(512, 512), (512, 2048), (1024, 1024), (1024, 4096), (2048, 2048), (2048, 5632), (2048, 8192)]
    large = [_ATTN, _UP, _DOWN, (4096, 11008), (11008, 4096), (3072, 3072), (3072, 8192), (5120, 5120), (5120, 1280),
             (8192, 1024), (8192, 8192), (4096, 32000), (8192, 28672), (28672, 8192)]

    def pair(K):
        return rng.choice([64, 128]) if K >= 3072 and K % 128 == 0 and K // 64 <= 256 else 0

    kind = rng.choice(["tiny", "decode", "decode", "prefill", "prefill", "wo_decode", "wo_prefill", "grouped", "pack"])
    if kind == "tiny":
        K, N = rng.choice(small)
        return _case(None, "linear", _log_int(rng, 1, 512), [(K, N)])
    if kind in ("decode", "wo_decode"):
        K, N = rng.choice(large)
        count = max(1, min(6, int(1.2e8 / (K * N / 2))))            # layers enough to exceed the L2 cache
        return _case(None, "wo" if kind == "wo_decode" else "linear", _log_int(rng, 1, 128), [(K, N)] * count, pair(K),
                     rng.choice([4, 4, 3]) if kind == "wo_decode" else 4)
    if kind in ("prefill", "wo_prefill"):
        K, N = rng.choice(large)
        most = min(4096, int(1.4e12 / (2.0 * K * N)) if kind == "prefill" else int(4e11 / (2.0 * K * N)))
        return _case(None, "wo" if kind == "wo_prefill" else "linear", _log_int(rng, 129, max(400, most)), [(K, N)], pair(K),
                     rng.choice([4, 4, 3]) if kind == "wo_prefill" else 4)
    if kind == "grouped":
        K, N = rng.choice([_UP, _DOWN, (4096, 11008), (2048, 5632), (5120, 1280)])
        return _case(None, "grouped", _log_int(rng, 8, 2048), [(K, N)], experts=rng.choice([4, 8, 16]))
    K, N = rng.choice([kn for kn in small + large if kn[0] * kn[1] <= 6e7])
    return _case(None, "pack", rng.choice([0, 0, 1]), [(K, N)], pair(K), rng.choice([4, 4, 3]))


def _layers(case):
    return [tuple(int(v) for v in layer.split("x")) for layer in case["layers"].split()]


def _activations(gen, M, K):
    X = torch.randn(M, K, generator=gen, device="cuda")
    channels = torch.randperm(K, generator=gen, device="cuda")
    X[:, channels[:max(4, K // 128)]] *= 20.0
    X[0, channels[-4:]] = torch.tensor([1000.0, -1000.0, 1000.0, -1000.0], device="cuda")
    return X.half()


def _weights(gen, N, K):
    return torch.randn(N, K, generator=gen, device="cuda").mul_(0.02).half()


def _rotation(X, K, n2, seed):
    n2 = n2 or _N2[K]
    return sq.sq_build_rotation(X[:8].float().cpu().numpy(), K // n2, n2, seed=seed & 0x7FFFFFFF)


def _empty_bytes(n):
    return torch.empty(n, dtype=torch.uint8, device="cuda")


def _packed(case, rot, W, N, K):
    Wq, sw = _empty_bytes(N * K // 2).view(N, K // 2), torch.empty(N, dtype=torch.float16, device="cuda")
    if case["kind"] == "wo":
        sq.sq_pack_weight_wo(rot, W, N, K, case["bits"], Wq, sw)
    else:
        sq.sq_pack_weight(rot, W, N, K, Wq, sw)
    return Wq, sw


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind, M, layers = case["kind"], case["rows"], _layers(case)
    state = {"kind": kind, "M": M, "bits": case["bits"], "layers": []}
    if kind == "pack":
        # `rows` = 1: the weight-only storage order, else the W4A4 one
        (K, N), = layers
        rot = _rotation(_activations(gen, 8, K), K, case["n2"], seed)
        state.update(rot=rot, N=N, K=K, W=_weights(gen, N, K), Wq=_empty_bytes(N * K // 2).view(N, K // 2),
                     sw=torch.empty(N, dtype=torch.float16, device="cuda"), wo=bool(M) or case["bits"] != 4)
        return state
    if kind == "grouped":
        (K, N), = layers
        E = case["experts"]
        owner = torch.randint(0, E, (M,), generator=gen, device="cuda").sort().values
        offsets = [0] + torch.bincount(owner, minlength=E).cumsum(0).tolist()
        X = _activations(gen, M, K)
        rot = _rotation(X, K, case["n2"], seed)
        packed = [_packed(case, rot, _weights(gen, N, K), N, K) for _ in range(E)]
        ws = sq.sq_linear_workspace_bytes(M, K)
        state.update(rots=[rot] * E, offsets=offsets, X=X, Wq=[p[0] for p in packed], sw=[p[1] for p in packed], N=N, K=K,
                     ws=_empty_bytes(ws), ws_bytes=ws, Y=torch.empty(M, N, dtype=torch.float16, device="cuda"))
        return state
    inputs = {}                                       # layers of one input width read the same tokens (gate and up, q, k and v)
    ws = 0
    for K, N in layers:
        if K not in inputs:
            X = _activations(gen, M, K)
            inputs[K] = (X, _rotation(X, K, case["n2"], seed))
        X, rot = inputs[K]
        Wq, sw = _packed(case, rot, _weights(gen, N, K), N, K)
        ws = max(ws, (sq.sq_linear_wo_workspace_bytes if kind == "wo" else sq.sq_linear_workspace_bytes)(M, K))
        state["layers"].append((rot, X, Wq, sw, N, K, torch.empty(M, N, dtype=torch.float16, device="cuda")))
    state.update(ws=_empty_bytes(ws), ws_bytes=ws)
    return state


def run(state):
    kind, M = state["kind"], state["M"]
    if kind == "pack":
        rot, W, N, K, Wq, sw = (state[k] for k in ("rot", "W", "N", "K", "Wq", "sw"))
        if state["wo"]:
            sq.sq_pack_weight_wo(rot, W, N, K, state["bits"], Wq, sw)
        else:
            sq.sq_pack_weight(rot, W, N, K, Wq, sw)
        return Wq, sw
    if kind == "grouped":
        sq.sq_linear_grouped(state["rots"], state["offsets"], state["X"], state["Wq"], state["sw"], state["N"], state["K"],
                             state["ws"], state["ws_bytes"], state["Y"])
        return state["Y"]
    call = sq.sq_linear_wo if kind == "wo" else sq.sq_linear
    for rot, X, Wq, sw, N, K, Y in state["layers"]:
        call(rot, X, M, Wq, sw, N, K, state["ws"], state["ws_bytes"], Y)
    return [layer[-1] for layer in state["layers"]]


def work(case):
    """Bytes: fp16 tokens and the two factors once, packed weights and steps once, outputs once.  Flops: the rotation
    (2 n1 + 2 n2 per element) and the product."""
    M, nbytes, flops = case["rows"], 0, 0
    read = set()
    for K, N in _layers(case):
        n2 = case["n2"] or _N2[K]
        n1 = K // n2
        factors, turn = 4 * (n1 * n1 + n2 * n2), 2 * (n1 + n2)
        if case["kind"] == "pack":
            return {"bytes": N * K * 2.5 + 2 * N + factors, "flops": N * K * turn}
        count = case["experts"] or 1
        if K not in read:
            nbytes += 2 * M * K + factors
            read.add(K)
        # an expert without tokens is not read: the expected number of experts that have some
        used = count * (1 - (1 - 1 / count) ** M) if count > 1 else 1
        nbytes += used * (N * K / 2 + 2 * N) + 2 * M * N
        flops += M * K * turn + 2 * M * N * K
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Measured against the same arithmetic with the rotation in float64.  The integer product is exact, so W4A4 outputs
    differ only where a rotated value lies within fp32 rounding of a boundary between two codes: a share of 1e-6 to
    2e-6 of the codes.  Over many rows that is up to 1.2e-3 of the result; one such code in the outlier token of a small
    batch was 4.4e-3 of it, and up to 0.08 of the rms in single entries."""
    if case["kind"] == "pack":          # bytes of two codes: 3e-6 to 5e-6 differ; steps: one fp16 ulp now and then
        return {"rel": 1.2e-4, "max": 4e-3, "differ": 3e-5}
    if case["kind"] == "wo":            # one fp16 rounding of tokens and outputs: 7e-5 to 1.2e-4, single entries one ulp
        return {"rel": 5e-4, "max": 4e-3}
    return {"rel": 2e-2 if case["rows"] < 64 else 5e-3, "max": 0.35}
