"""GPU parity of the streaming kernel on the tensor cores (weights unpacked into tensor memory) against the CPU
reference: edges of the token tiles, ragged last channel tiles, every scale group form, unequal shares of K, groups cut
between shares, several tiles per cluster, grouped matrices, both scale types and result types."""
import numpy as np
import pytest

from conftest import Guarded
from paper_2508_06753_b200 import synth

pytestmark = pytest.mark.gpu
# y is a sum of K / group <= 512 fp32 terms from exact integer sums, 1e-6 of its row's largest value; the other kernels are
# held to the same 1e-4, and test_error_does_not_grow_with_the_row holds the sums to their bound
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
    # M, K, [N], group (0 = K), forced shares of K (0 = the plan's)
    (1, 256, [16], 64, 0),                     # one block, an eighth of a tile
    (8, 512, [128], 128, 2),
    (9, 1280, [144], 64, 2),                   # shares of 3 and 2 blocks; a second tile of 16 channels
    (16, 4096, [272, 16], 256, 4),
    (16, 2048, [128 * 9], 0, 8),               # one scale per channel, a block per CTA
    (17, 1792, [640, 32], 64, 4),              # shares of 2 and 1 blocks
    (32, 1536, [384], 512, 4),                 # groups of two blocks cut between shares of 2, 2, 1, 1
    (31, 768, [128 * 150], 64, 1),             # more tiles than SMs
    (20, 2048, [256], 128, 8),                 # parts of four of 24 columns: two ranks have none
    (24, 1024, [128 * 170], 128, 2),           # two tiles for some clusters: both exchange buffers
    (12, 512, [128 * 310], 64, 1),             # a second round
    (33, 2048, [1024], 64, 8),
    (48, 4096, [256, 128], 0, 0),
    (64, 7168, [512], 64, 4),                  # the ring of stages comes round
    (64, 512, [128 * 160], 128, 2),
    (50, 3072, [144], 1024, 8),
    (5, 14336, [256], 64, 8),
    (48, 2048, [384, 16], 128, 2),
    (24, 1024, [272], 0, 4),
    (23, 3072, [256, 144], 1024, 2),
    (32, 2048, [256], 128, 4),
]


@pytest.mark.parametrize("h16", [False, True])
@pytest.mark.parametrize("M,K,Ns,group,shares", CASES)
def test_against_reference(gpu, oracle, monkeypatch, M, K, Ns, group, shares, h16):
    torch, b = gpu
    monkeypatch.setenv("W2A8_TSTREAM", "2")
    if shares:
        monkeypatch.setenv("W2A8_TSTREAM_C", str(shares))
    g = K if group == 0 else group
    mats = [synth.make_linear(7 * M + K + i, K, N, g) for i, N in enumerate(Ns)]
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
        assert b.w2a8_workspace_status(ws) == 0
        for gd in guards:
            gd.check("y")
        ys.append([gd.view.clone() for gd in guards])
    a_ref, s_ref = oracle.quantize(bits)
    for i, ((codes, s_w), y, again) in enumerate(zip(mats, *ys)):
        assert torch.equal(y, again)
        N = codes.shape[0]
        sel = np.unique(np.concatenate([np.arange(min(N, 160)), np.arange(max(0, N - 160), N), np.arange(0, N, 37)]))
        ref = oracle.gemm(a_ref, s_ref, codes[sel], s_w[sel].astype(np.float32), g)
        err = np.abs(y.cpu().numpy()[:, sel].astype(np.float64) - ref).max(axis=1)
        assert (err <= TOL * np.abs(ref).max(axis=1)).all(), float(err.max())
        if h16:
            y16 = b.w2a8_gemm_h16(a, s_a, packed[i], scales[i], g, ws,
                                  y=torch.full((M, N), float("nan"), dtype=torch.bfloat16, device="cuda"))
            assert torch.equal(y16, y.to(torch.bfloat16))


@pytest.mark.parametrize("group", [64, 2048])
def test_largest_sums_and_scales(gpu, oracle, monkeypatch, group):
    """Every product at its extreme (code 0 = -2 times +-127) and scales from 2^-100 to 2^95 (the running sums carry
    64 times sums of up to 2^19, so that larger ones leave fp32)."""
    torch, b = gpu
    monkeypatch.setenv("W2A8_TSTREAM", "2")
    M, N, K = 16, 128, 2048
    codes = np.zeros((N, K), np.uint8)
    codes[1::2] = 3
    s_w = np.exp2(np.linspace(-100, 95, N * (K // group))).reshape(N, K // group).astype(np.float32)
    a = np.where(np.arange(M)[:, None] % 2 == 0, 127, -127).astype(np.int8).repeat(K, axis=1)
    s_a = np.full(M, 0.5, np.float32)
    ws = b.new_workspace(b.w2a8_workspace_bytes(M, N, K, group))
    y = b.w2a8_gemm(_dev(torch, a), _dev(torch, s_a), b.w2_pack(_dev(torch, codes)), _dev(torch, s_w), group, ws)
    ref = oracle.gemm(a, s_a, codes, s_w, group)
    err = np.abs(y.cpu().numpy().astype(np.float64) - ref)
    assert (err <= 1e-5 * np.abs(ref)).all()          # all terms of an output have one sign: relative to each output


@pytest.mark.parametrize("M,K,N", [(32, 8192, 8192), (64, 4096, 4096)])
def test_default_dispatch_in_a_replayed_graph(gpu, monkeypatch, M, K, N):
    """By the rule, captured and replayed on changed activations: the bits of a plain call."""
    torch, b = gpu
    gen = torch.Generator(device="cuda").manual_seed(M)
    codes = torch.randint(0, 4, (N, K), generator=gen, device="cuda", dtype=torch.uint8)
    packed, scale = b.w2_pack(codes), torch.rand((N, K // 128), generator=gen, device="cuda") + 0.01
    x = torch.randn((M, K), generator=gen, device="cuda").to(torch.bfloat16)
    a, s = b.a8_quantize(x)
    ws = b.new_workspace(b.w2a8_workspace_bytes(M, N, K, 128))
    y = torch.empty((M, N), device="cuda")
    b.w2a8_gemm(a, s, packed, scale, 128, ws, y=y)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        b.a8_quantize(x, a, s)
        b.w2a8_gemm(a, s, packed, scale, 128, ws, y=y)
    x.copy_(torch.randn((M, K), generator=gen, device="cuda").to(torch.bfloat16))
    graph.replay()
    got = y.clone()
    a2, s2 = b.a8_quantize(x)
    plain = b.w2a8_gemm(a2, s2, packed, scale, 128, ws)
    assert torch.equal(got, plain)
    import ctypes
    assert b.lib().w2a8_grouped_plan(1, (ctypes.c_int * 1)(N), M, K, 128, b.FUSE_OFF) & 4
    monkeypatch.setenv("W2A8_TSTREAM", "0")
    other = b.w2a8_gemm(a2, s2, packed, scale, 128, b.new_workspace(b.w2a8_workspace_bytes(M, N, K, 128)))
    assert (other - plain).abs().max() <= 1e-5 * plain.abs().max()


def test_behind_a_long_kernel(gpu, monkeypatch):
    """The bounded waits do not count the time of the kernel before (eight quantiser launches of 0.26 s)."""
    torch, b = gpu
    monkeypatch.setenv("W2A8_TSTREAM", "2")
    M, N, K = 20, 512, 8192                            # four shares of eight blocks: the ring comes round
    monkeypatch.setenv("W2A8_TSTREAM_C", "4")
    gen = torch.Generator(device="cuda").manual_seed(1)
    packed = b.w2_pack(torch.randint(0, 4, (N, K), generator=gen, device="cuda", dtype=torch.uint8))
    scale = torch.rand((N, K // 64), generator=gen, device="cuda")
    a, s = b.a8_quantize(torch.randn((M, K), generator=gen, device="cuda").to(torch.bfloat16))
    ws = b.new_workspace(b.w2a8_workspace_bytes(M, N, K, 64))
    alone = b.w2a8_gemm(a, s, packed, scale, 64, ws)
    x = torch.randn((1, 1 << 30), dtype=torch.bfloat16, device="cuda")
    row, row_scale = torch.empty((1, 1 << 30), dtype=torch.int8, device="cuda"), torch.empty(1, device="cuda")
    y = torch.full_like(alone, float("nan"))
    torch.cuda.synchronize()
    for _ in range(8):
        b.a8_quantize(x, row, row_scale)
    b.w2a8_gemm(a, s, packed, scale, 64, ws, y=y)
    torch.cuda.synchronize()
    assert b.w2a8_workspace_status(ws) == 0
    assert torch.equal(y, alone)


# One running total over the groups of these rows was up to 2.2 times as far from 64-bit sums as the kernels that had
# such launches before.
@pytest.mark.parametrize("M,K,N,group,shares", [
    (16, 10240, 512, 64, 1), (24, 10240, 512, 128, 1), (32, 8192, 512, 64, 1), (32, 28672, 256, 128, 1),
    (48, 10240, 512, 64, 1), (64, 10240, 512, 64, 1), (64, 28672, 256, 64, 2), (60, 16384, 256, 256, 1),
])
def test_error_does_not_grow_with_the_row(gpu, monkeypatch, M, K, N, group, shares):
    """Distance from sums in 64 bits.  Chains of eight groups add 4.5 roundings of a relative size of 2.6e-8 (rms) at
    most, a share's last addition, the sum of the shares and the token scale one each: sqrt(7.5) * 2.6e-8 = 7.1e-8 for
    terms of equal size (7.3e-8 in numpy); a running total over the groups of these rows is at 1.0e-7 and more."""
    torch, b = gpu
    monkeypatch.setenv("W2A8_TSTREAM", "2")
    monkeypatch.setenv("W2A8_TSTREAM_C", str(shares))
    gen = torch.Generator(device="cuda").manual_seed(K + M)
    codes = torch.randint(0, 4, (N, K), generator=gen, device="cuda", dtype=torch.uint8)
    scale = 0.02 * torch.exp(0.5 * torch.randn((N, K // group), generator=gen, device="cuda"))
    a = torch.randint(-127, 128, (M, K), generator=gen, device="cuda", dtype=torch.int8)
    a_scale = torch.rand(M, generator=gen, device="cuda") + 0.5
    ws = b.new_workspace(b.w2a8_workspace_bytes(M, N, K, group))
    y = b.w2a8_gemm(a, a_scale, b.w2_pack(codes), scale, group, ws).double()
    sums = torch.einsum("mgk,ngk->mng", a.double().view(M, -1, group), codes.double().view(N, -1, group) - 2)
    exact = torch.einsum("mng,ng->mn", sums, scale.double()) * a_scale.double()[:, None]
    assert b.w2a8_workspace_status(ws) == 0
    assert ((y - exact).norm() / exact.norm()).item() <= 8e-8


@pytest.mark.parametrize("group", [64, 128, 256, 4096])
@pytest.mark.parametrize("M,shares", [(16, 1), (16, 8), (24, 4), (32, 1), (48, 2), (64, 4)])
def test_infinities_and_nan(gpu, monkeypatch, M, shares, group):
    """Infinite and NaN scales, and products that leave fp32: what a plain sum of the scaled group sums gives."""
    torch, b = gpu
    monkeypatch.setenv("W2A8_TSTREAM", "2")
    monkeypatch.setenv("W2A8_TSTREAM_C", str(shares))
    N, K = 160, 4096
    G = K // group
    gen = torch.Generator(device="cuda").manual_seed(M + group)
    codes = torch.randint(0, 4, (N, K), generator=gen, device="cuda", dtype=torch.uint8)
    a = torch.randint(-127, 128, (M, K), generator=gen, device="cuda", dtype=torch.int8)
    scale = torch.rand((N, G), generator=gen, device="cuda") + 0.01
    for ch in range(0, 64, 2):                        # one, then two infinite scales, somewhere in the row
        scale[ch, (5 * ch) % G] = float("inf")
        scale[ch, (11 * ch + 3) % G] = -float("inf") if ch % 4 else float("inf")
    scale[64:80, G // 2] = float("nan")
    scale[80:96, (G - 1) // 2] = 3.0e38               # finite, its products are not
    ones = torch.ones(M, device="cuda")
    ws = b.new_workspace(b.w2a8_workspace_bytes(M, N, K, group))
    y = b.w2a8_gemm(a, ones, b.w2_pack(codes), scale, group, ws)
    sums = 64 * torch.einsum("mgk,ngk->mng", a.double().view(M, G, group), codes.double().view(N, G, group) - 2)
    ref = (sums * scale.double()).float().sum(dim=2) / 64        # (terms in fp32: infinite where theirs are)
    assert b.w2a8_workspace_status(ws) == 0
    assert torch.equal(y.isnan(), ref.isnan()) and torch.equal(y.isinf(), ref.isinf())
    assert torch.equal(y.sign()[y.isinf()], ref.sign()[ref.isinf()])
    fin = ref.isfinite()
    assert int(fin.sum()) > M * 60
    assert (y - ref)[fin].abs().max() <= 1e-5 * ref[fin].abs().max()


@pytest.mark.parametrize("N,K", [(1024, 8192), (1152, 2560)])
@pytest.mark.parametrize("shares", [1, 2, 4, 8])
def test_one_scale_per_channel_is_exact_up_to_the_scales(gpu, monkeypatch, N, K, shares):
    """Integer sums, then the two scales: the bits of the int8 tensor-core kernel, whatever the shares of K."""
    torch, b = gpu
    M = 64
    gen = torch.Generator(device="cuda").manual_seed(K)
    packed = b.w2_pack(torch.randint(0, 4, (N, K), generator=gen, device="cuda", dtype=torch.uint8))
    scale = torch.rand((N, 1), generator=gen, device="cuda") + 0.01
    a, s = b.a8_quantize(torch.randn((M, K), generator=gen, device="cuda").to(torch.bfloat16))
    monkeypatch.setenv("W2A8_PREFILL", "2")
    monkeypatch.setenv("W2A8_PF_KSPLIT", "1")
    monkeypatch.setenv("W2A8_TSTREAM_C", str(shares))
    ws = b.new_workspace(b.w2a8_workspace_bytes(M, N, K, K))
    ys = {}
    for mode in ("0", "2"):
        monkeypatch.setenv("W2A8_TSTREAM", mode)
        ys[mode] = b.w2a8_gemm(a, s, packed, scale, K, ws)
        assert b.w2a8_workspace_status(ws) == 0
    assert torch.equal(ys["0"], ys["2"])


@pytest.mark.parametrize("M", [16, 32, 64])
@pytest.mark.parametrize("shares", [1, 2, 8])
@pytest.mark.parametrize("group", [64, 1024])
def test_a_wait_that_gives_up(gpu, monkeypatch, M, shares, group):
    """With no polls allowed the waits give up: the call ends, the status word says so, and the next call is whole."""
    torch, b = gpu
    monkeypatch.setenv("W2A8_TSTREAM", "2")
    monkeypatch.setenv("W2A8_TSTREAM_C", str(shares))
    N, K = 1024, 32768
    gen = torch.Generator(device="cuda").manual_seed(M)
    packed = b.w2_pack(torch.randint(0, 4, (N, K), generator=gen, device="cuda", dtype=torch.uint8))
    scale = torch.rand((N, K // group), generator=gen, device="cuda") + 0.01
    a, s = b.a8_quantize(torch.randn((M, K), generator=gen, device="cuda").to(torch.bfloat16))
    ws = b.new_workspace(b.w2a8_workspace_bytes(M, N, K, group))
    whole = b.w2a8_gemm(a, s, packed, scale, group, ws)
    assert b.w2a8_workspace_status(ws) == 0
    monkeypatch.setenv("W2A8_TSTREAM_POLLS", "0")
    b.w2a8_gemm(a, s, packed, scale, group, ws)
    assert b.w2a8_workspace_status(ws) == -7                  # W2A8_ERR_TIMEOUT
    monkeypatch.delenv("W2A8_TSTREAM_POLLS")
    ws.zero_()
    assert torch.equal(b.w2a8_gemm(a, s, packed, scale, group, ws), whole)
    assert b.w2a8_workspace_status(ws) == 0


@pytest.mark.parametrize("M,K,Ns,group,h16", [
    (12, 2560, [3840], 64, False),                 # short rows, 9 to 16 tokens
    (16, 3072, [1984], 3072, False),
    (32, 8192, [8192], 128, True),                 # binary16 scales
    (24, 8192, [8192], 8192, True),
    (48, 4096, [4096, 1024, 1024], 64, False),     # matrices that share their activations
    (32, 8192, [8192, 1024, 1024], 8192, False),
    (63, 14336, [4096], 1024, False),
])
def test_by_the_rule(gpu, monkeypatch, M, K, Ns, group, h16):
    """Launches that come here by the rule: the bits of the forced kernel, which plans alike."""
    torch, b = gpu
    gen = torch.Generator(device="cuda").manual_seed(K + M)
    packed = [b.w2_pack(torch.randint(0, 4, (N, K), generator=gen, device="cuda", dtype=torch.uint8)) for N in Ns]
    scales = [torch.rand((N, K // group), generator=gen, device="cuda") + 0.01 for N in Ns]
    if h16:
        scales = [s.half() for s in scales]
    a, s_a = b.a8_quantize(torch.randn((M, K), generator=gen, device="cuda").to(torch.bfloat16))
    ws = b.new_workspace(b.w2a8_grouped_workspace_bytes(Ns, M, K, group))
    run = lambda: ([b.w2a8_gemm_h16(a, s_a, packed[0], scales[0], group, ws)] if h16 else
                   [y.clone() for y in b.w2a8_gemm_grouped(a, s_a, b.Group(packed, scales), group, ws)])
    ys = {}
    for mode in (None, "2", "0"):
        if mode is None:
            monkeypatch.delenv("W2A8_TSTREAM", raising=False)
        else:
            monkeypatch.setenv("W2A8_TSTREAM", mode)
        ys[mode] = run()
        assert b.w2a8_workspace_status(ws) == 0
    for rule, forced, other in zip(ys[None], ys["2"], ys["0"]):
        assert torch.equal(rule, forced)
        assert (rule - other).abs().max() <= 1e-5 * other.abs().max()
