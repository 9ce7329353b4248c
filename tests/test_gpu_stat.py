"""GPU parity of the streaming kernel with stationary activations against the CPU
reference: edges of token slabs, half channel pairs, every scale group form, K shares with unequal
block counts, cells cut between warps, several rounds of pairs, grouped matrices, both scale types."""
import numpy as np
import pytest

from conftest import Guarded
from paper_2508_06753_b200 import synth

pytestmark = pytest.mark.gpu
TOL = 1e-4


@pytest.fixture(scope="module")
def gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_06753_b200 import binding, build
    build.build()
    binding.lib()
    return torch, binding


def _dev(torch, arr):
    return torch.from_numpy(np.ascontiguousarray(arr)).cuda()


CASES = [
    # M, K, [N], group (0 = K), forced K shares (0 = the plan's)
    (9, 256, [16], 64, 0),                    # one cell, half a pair
    (16, 512, [48, 16], 128, 0),              # half pairs at the end of both matrices
    (17, 1280, [64], 64, 2),                  # shares of 2 and 3 blocks
    (24, 1792, [160, 32], 256, 3),
    (25, 2048, [4096], 0, 2),                 # one scale per channel
    (32, 4096, [4096, 1024, 1024], 64, 4),
    (32, 14336, [272], 64, 0),                # long rows: eight shares
    (31, 512, [20480], 128, 1),               # no cluster, several rounds of pairs
    (1, 1024, [96], 64, 0),                   # forced below its range: a single token
    (8, 4352, [80], 64, 2),
    (40, 1024, [2048], 64, 0),                # five slabs
    (47, 768, [96, 48], 256, 2),              # six
    (64, 4096, [1024], 128, 0),               # eight: a full group
    (100, 2048, [272], 64, 2),                # two groups of seven slabs, the second not full
    (130, 512, [1024], 0, 0),                 # three groups
    (3, 8192, [12304], 128, 0),               # large: the 16 bytes around the scales of a block
    (2, 8192, [12288], 64, 0),
]


@pytest.mark.parametrize("h16", [False, True])
@pytest.mark.parametrize("M,K,Ns,group,shares", CASES)
def test_stat_against_reference(gpu, oracle, monkeypatch, M, K, Ns, group, shares, h16):
    torch, b = gpu
    monkeypatch.setenv("W2A8_STAT", "2")
    if shares:
        monkeypatch.setenv("W2A8_STAT_C", str(shares))
    g = K if group == 0 else group
    mats = [synth.make_linear(5 * M + K + i, K, N, g) for i, N in enumerate(Ns)]
    if h16:
        mats = [(c, s.astype(np.float16)) for c, s in mats]
    bits = synth.activations_bf16(M + K, M, K, 0.01)
    a, s_a = b.a8_quantize(_dev(torch, bits.view(np.int16)).view(torch.bfloat16))
    packed, scales = [b.w2_pack(_dev(torch, c)) for c, _ in mats], [_dev(torch, s) for _, s in mats]
    ws = b.new_workspace(b.w2a8_grouped_workspace_bytes(Ns, M, K, g))
    ys = []
    for _ in range(2):
        guards = [Guarded(torch, (M, N), torch.float32, float("nan")) for N in Ns]
        if h16:
            for pk, sc, gd in zip(packed, scales, guards):
                b.w2a8_gemm_h16(a, s_a, pk, sc, g, ws, y=gd.view)
        else:
            b.w2a8_gemm_grouped(a, s_a, b.Group(packed, scales), g, ws, y=[gd.view for gd in guards])
        torch.cuda.synchronize()
        for gd in guards:
            gd.check("y")
        ys.append([gd.view.clone() for gd in guards])
    a_ref, s_ref = oracle.quantize(bits)
    for (codes, s_w), y, again in zip(mats, *ys):
        assert torch.equal(y, again)
        ref = oracle.gemm(a_ref, s_ref, codes, s_w.astype(np.float32), g)
        err = np.abs(y.cpu().numpy().astype(np.float64) - ref).max(axis=1)
        assert (err <= TOL * np.abs(ref).max(axis=1)).all(), float(err.max())


@pytest.mark.parametrize("M,K,Ns,group", [
    (2, 8192, [28672, 28672], 128),         # few tokens: each matrix alone is large enough for the kernel too
    (32, 4096, [14336, 14336], 64),
    (12, 8192, [8192, 1024, 1024], 0),      # and two that alone go to the persistent kernel
])
def test_grouped_against_single_calls(gpu, M, K, Ns, group):
    """By default, i.e. by the dispatch rule: the fp32 additions may come in another order than alone (at most
    K / 64 of them per output, so a few times 2^-24 of the largest output of a row), equal bits on repeats."""
    torch, b = gpu
    g = K if group == 0 else group
    gen = torch.Generator(device="cuda").manual_seed(M + K)
    rand = lambda *shape: torch.rand(shape, generator=gen, device="cuda")
    packed = [b.w2_pack((4 * rand(N, K)).to(torch.uint8).clamp_(max=3)) for N in Ns]
    scales = [0.01 + 0.02 * rand(N, K // g) for N in Ns]
    a, s_a = b.a8_quantize((rand(M, K) - 0.5).to(torch.bfloat16))
    ws = b.new_workspace(b.w2a8_grouped_workspace_bytes(Ns, M, K, g))
    ys = [y.clone() for y in b.w2a8_gemm_grouped(a, s_a, b.Group(packed, scales), g, ws)]
    again = b.w2a8_gemm_grouped(a, s_a, b.Group(packed, scales), g, ws)
    for pk, sc, y, y2 in zip(packed, scales, ys, again):
        assert torch.equal(y, y2)
        alone = b.w2a8_gemm(a, s_a, pk, sc, g, ws)
        assert torch.equal(alone, b.w2a8_gemm(a, s_a, pk, sc, g, ws))
        err = (y.double() - alone.double()).abs().amax(dim=1)
        assert bool((err <= 1e-5 * alone.double().abs().amax(dim=1)).all()), float(err.max())


@pytest.mark.parametrize("M,K,Ns,shares", [
    (64, 14336, [256], 1),               # eight slabs of 56 blocks do not fit one CTA
    (32, 28672, [64, 32], 2),            # a group: to the persistent kernel
    (40, 28672, [64, 32], 2),            # more tokens than that one takes
])
def test_shapes_without_a_plan_take_another_kernel(gpu, oracle, monkeypatch, M, K, Ns, shares):
    torch, b = gpu
    monkeypatch.setenv("W2A8_STAT", "2")
    monkeypatch.setenv("W2A8_STAT_C", str(shares))
    mats = [synth.make_linear(K + i, K, N, 64) for i, N in enumerate(Ns)]
    bits = synth.activations_bf16(M, M, K)
    a, s_a = b.a8_quantize(_dev(torch, bits.view(np.int16)).view(torch.bfloat16))
    grp = b.Group([b.w2_pack(_dev(torch, c)) for c, _ in mats], [_dev(torch, s) for _, s in mats])
    ws = b.new_workspace(b.w2a8_grouped_workspace_bytes(Ns, M, K, 64))
    ys = b.w2a8_gemm_grouped(a, s_a, grp, 64, ws)
    a_ref, s_ref = oracle.quantize(bits)
    for (codes, s_w), y in zip(mats, ys):
        ref = oracle.gemm(a_ref, s_ref, codes, s_w, 64)
        err = np.abs(y.cpu().numpy().astype(np.float64) - ref).max(axis=1)
        assert (err <= TOL * np.abs(ref).max(axis=1)).all(), float(err.max())
