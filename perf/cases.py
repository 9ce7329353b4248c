"""What a user of the library has it do, as timed cases: decoder linears with 2-bit weights at the
token counts of decoding and of prefill, through the entry points of ``binding``.

A case is a plain dict:
  work     "linear": one matrix (K -> N), called eagerly;
           "layer": the seven linears of one decoder layer (q|k|v, o, gate|up, down)
  entry    "linear" (bf16 in: quantiser and GEMM), "h16" (a8_quantize, then binary16 scales and a
           bf16 result), "a16" (bf16 activations, no quantiser), "host" (activations and results in
           page-locked host memory)
  model    "8b" or "70b" for a layer; K and N for a linear
  M        tokens;  group: values of k per weight scale, 0 = one scale per channel
  ternary  codes {1,2,3} instead of {0..3};  outliers: 1 % of the activations at +-20
  graph    the calls of a pass are captured once and replayed, as a decode loop does; else each
           call is made from Python, as a prefill does
"""
import math

import torch

from paper_2508_06753_b200 import binding as b
from paper_2508_06753_b200 import synth

_LAYERS = {"8b": synth.LLAMA3_8B_LAYER, "70b": synth.LLAMA3_70B_LAYER}
_SHARED = [("q", "k", "v"), ("o",), ("gate", "up"), ("down",)]      # linears that share their activations


def _layer(name, model, M, group=64, entry="linear", ternary=False, outliers=False, graph=True):
    return dict(name=name, work="layer", entry=entry, model=model, M=M, group=group, ternary=ternary,
                outliers=outliers, graph=graph)


def _linear(name, K, N, M, group=64, entry="linear", ternary=False, outliers=False):
    return dict(name=name, work="linear", entry=entry, K=K, N=N, M=M, group=group, ternary=ternary,
                outliers=outliers, graph=False)


def listed():
    return [
        # one call on one small matrix: latency of a single GEMV outside any graph
        _linear("gemv_2048_m1", 2048, 2048, 1),
        # single-stream decoding, the headline use
        _layer("decode_8b_m1", "8b", 1),
        # batched decoding
        _layer("decode_8b_m16", "8b", 16),
        # a ternary model with one scale per channel, a small batch
        _layer("decode_8b_ternary_m8", "8b", 8, group=0, ternary=True),
        # the larger model with outliers in its activations, a large decode batch
        _layer("decode_70b_m32", "70b", 32, group=128, outliers=True),
        # the 16-bit storage recipe: groups of 128, binary16 scales, bf16 results
        _layer("decode_8b_h16_m4", "8b", 4, group=128, entry="h16"),
        # activations left at 16 bits (an accuracy option), a ragged small batch
        _layer("decode_8b_a16_m3", "8b", 3, entry="a16"),
        # activations and results in host memory: the end-to-end path of the benchmark
        _layer("host_8b_m4", "8b", 4, entry="host"),
        # a short prompt or a verification batch with a ragged number of tokens
        _layer("chunk_8b_m100", "8b", 100, graph=False),
        # prefill of an ordinary prompt through the matrix with few output channels
        _linear("prefill_down_m512", 14336, 4096, 512),
        # prefill of a ternary model
        _linear("prefill_gate_ternary_m2048", 4096, 14336, 2048, group=0, ternary=True),
        # the largest prefill of the benchmark
        _linear("prefill_gate_m8192", 4096, 14336, 8192),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# (K, N) of single linears: the paper's small GEMV shapes and the linears of the layers
_SMALL = [(1600, 1600), (2048, 2048), (2560, 2560), (2560, 3840), (3200, 3200)]
_LARGE = [(4096, 4096), (4096, 1024), (4096, 14336), (14336, 4096), (8192, 8192)]


def draw(rng):
    kind = rng.choice(["small", "decode", "decode", "decode", "chunk", "prefill", "prefill"])
    ternary = rng.random() < 0.25
    outliers = rng.random() < 0.25
    if kind == "small":
        K, N = rng.choice(_SMALL)
        c = _linear("", K, N, _log_int(rng, 1, 32), rng.choice([64, 0] if K % 128 else [64, 128, 0]),
                    rng.choice(["linear", "linear", "h16", "a16"]), ternary, outliers)
    elif kind == "prefill":
        K, N = rng.choice(_LARGE)
        most = min(8192, 8192 * 4096 * 14336 // (K * N))
        c = _linear("", K, N, _log_int(rng, 256, most), rng.choice([64, 64, 128, 0]),
                    rng.choice(["linear", "linear", "linear", "h16", "a16"]), ternary, outliers)
    else:
        M = _log_int(rng, 1, 32) if kind == "decode" else _log_int(rng, 33, 256)
        entry = rng.choice(["linear", "linear", "linear", "h16", "a16", "host"] if kind == "decode" else ["linear"])
        c = _layer("", rng.choice(["8b", "8b", "70b"]), M, rng.choice([64, 128, 0]), entry, ternary, outliers,
                   graph=kind == "decode")
    del c["name"]
    return c


def _linears(case):
    """[(name, K, N)], [indices that share their activations]"""
    if case["work"] == "linear":
        return [("linear", case["K"], case["N"])], [[0]]
    lins = _LAYERS[case["model"]]
    index = {name: i for i, (name, _, _) in enumerate(lins)}
    return lins, [[index[n] for n in names] for names in _SHARED]


def _group(case, K):
    return case["group"] or K


def _activations(g, M, K, outliers):
    x = torch.randn((M, K), generator=g, device="cuda")
    if outliers:
        pos = torch.rand((M, K), generator=g, device="cuda").topk(K // 100, dim=1).indices
        sign = torch.randint(0, 2, pos.shape, generator=g, device="cuda") * 2 - 1
        x.scatter_(1, pos, 20.0 * sign)
    return x.to(torch.bfloat16)


class _State:
    pass


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    M, entry = case["M"], case["entry"]
    lins, groups = _linears(case)
    s = _State()
    s.case, s.groups = case, groups
    packed, scale = [], []
    for _, K, N in lins:
        codes = torch.randint(1 if case["ternary"] else 0, 4, (N, K), generator=g, device="cuda", dtype=torch.uint8)
        packed.append(b.w2_pack(codes))
        sc = 0.02 * torch.exp(0.5 * torch.randn((N, K // _group(case, K)), generator=g, device="cuda"))
        scale.append(sc.to(torch.float16) if entry == "h16" else sc)
        del codes
    s.packed, s.scale = packed, scale
    # one set of buffers per set of linears that share their activations
    s.x, s.a, s.a_scale, s.y, s.grp, s.ws, s.g = [], [], [], [], [], [], []
    for ids in groups:
        K, Ns = lins[ids[0]][1], [lins[i][2] for i in ids]
        gr = _group(case, K)
        x = _activations(g, M, K, case["outliers"])
        out = dict(dtype=torch.bfloat16 if entry == "h16" else torch.float32)
        if entry == "host":
            x = x.cpu().pin_memory()
            ws = b.w2a8_linear_grouped_host_workspace_bytes(Ns, M, K, gr)
            out["pin_memory"] = True
        else:
            ws = b.w2a8_grouped_workspace_bytes(Ns, M, K, gr)
            out["device"] = "cuda"
        y = [torch.zeros((M, n), **out) for n in Ns]
        s.x.append(x)
        s.a.append(torch.zeros((M, K), dtype=torch.int8, device="cuda"))
        s.a_scale.append(torch.zeros((M,), dtype=torch.float32, device="cuda"))
        s.y.append(y)
        s.grp.append(b.Group([packed[i] for i in ids], [scale[i] for i in ids], None if entry == "host" else y))
        s.ws.append(b.new_workspace(ws))
        s.g.append(gr)
    s.graph = None
    if case["graph"]:
        _calls(s)                                   # first use outside the capture
        torch.cuda.synchronize()
        s.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s.graph):
            _calls(s)
    return s


def _calls(s):
    entry = s.case["entry"]
    single = s.case["work"] == "linear"
    for i, ids in enumerate(s.groups):
        x, a, a_scale, y, gr, ws = s.x[i], s.a[i], s.a_scale[i], s.y[i], s.g[i], s.ws[i]
        if entry == "host":
            b.w2a8_linear_grouped_host(x, s.grp[i], gr, y, ws)
        elif entry == "h16":
            b.a8_quantize(x, a, a_scale)
            for j, w in enumerate(ids):
                b.w2a8_gemm_h16(a, a_scale, s.packed[w], s.scale[w], gr, ws, y=y[j])
        elif entry == "a16":
            for j, w in enumerate(ids):
                b.w2a16_gemm(x, s.packed[w], s.scale[w], gr, ws, y=y[j])
        elif single:
            b.w2a8_linear(x, s.packed[0], s.scale[0], gr, ws, a=a, a_scale=a_scale, y=y[0])
        else:
            b.w2a8_linear_grouped(x, s.grp[i], gr, ws, a=a, a_scale=a_scale)


def run(s):
    if s.graph is not None:
        s.graph.replay()
    else:
        _calls(s)
    out = {"y": [t for y in s.y for t in y]}
    if s.case["entry"] in ("linear", "h16"):
        out["a"], out["a_scale"] = s.a, s.a_scale
    return out


def work(case):
    M, entry = case["M"], case["entry"]
    lins, groups = _linears(case)
    nbytes = flops = 0
    for _, K, N in lins:
        G = K // _group(case, K)
        nbytes += K * N // 4 + N * G * (2 if entry == "h16" else 4) + M * N * (2 if entry == "h16" else 4)
        flops += 2 * M * N * K
    for ids in groups:
        K = lins[ids[0]][1]
        nbytes += 2 * M * K
        if entry in ("linear", "h16"):
            nbytes += M * K + 4 * M                 # the int8 rows and their scales are results too
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # int8 rows are exact.  fp32 results: exact integer group sums (int8) or exact products (bf16),
    # then fp32 sums in another order (against sums in 64 bits: rel 3e-7, max 2e-6 on the int8 path).
    # bf16 results: the same, where the two fp32 values fall on either side of a rounding boundary
    # one bf16 step apart (up to one value in a thousand).
    if case["entry"] == "h16":
        return {"rel": 2e-4, "max": 8e-3}
    return {"rel": 2e-6, "max": 2e-5}
