"""One workspace for a sequence of shapes: what one call leaves in it (partial outputs of a K split) must not be
taken for the arrival counters of the next (rows of more than 32768 values, whose K chunks do not fit a cluster)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_06753_b200 import binding, build
    build.build()
    binding.lib()
    return torch, binding


def _problem(torch, b, M, N, K, entry):
    gen = torch.Generator(device="cuda").manual_seed(M + N)
    packed = b.w2_pack(torch.randint(0, 4, (N, K), generator=gen, device="cuda", dtype=torch.uint8))
    scale = torch.rand((N, K // 64), generator=gen, device="cuda") + 0.01
    x = torch.randn((M, K), generator=gen, device="cuda").to(torch.bfloat16)
    a, s = b.a8_quantize(x)
    y = torch.empty((M, N), device="cuda")

    def run(ws):
        y.fill_(float("nan"))
        if entry == "a16":
            b.w2a16_gemm(x, packed, scale, 64, ws, y=y)
        elif entry == "h16":
            b.w2a8_gemm_h16(a, s, packed, scale.to(torch.float16), 64, ws, y=y)
        else:
            b.w2a8_gemm(a, s, packed, scale, 64, ws, y=y)
        return y.clone()
    return run, b.w2a8_workspace_bytes(M, N, K, 64)


@pytest.mark.parametrize("entry", ["h16", "a16"])
@pytest.mark.parametrize("first", [(4, 16, 65536, None), (128, 256, 4096, "gemm")])
def test_sequence_on_one_workspace(gpu, monkeypatch, first, entry):
    torch, b = gpu
    M, N, K, kind = first
    if kind == "gemm":                   # a K split of the tensor-core kernel
        monkeypatch.setenv("W2A8_PREFILL", "2")
        monkeypatch.setenv("W2A8_PF_KSPLIT", "4")
    run1, bytes1 = _problem(torch, b, M, N, K, kind or entry)
    run2, bytes2 = _problem(torch, b, 4, 2048, 65536, entry)
    fresh = run2(b.new_workspace(max(bytes1, bytes2)))
    ws = b.new_workspace(max(bytes1, bytes2))
    run1(ws)
    assert torch.equal(run2(ws), fresh)
    assert torch.equal(run2(ws), fresh)
    assert not torch.isnan(fresh).any()
