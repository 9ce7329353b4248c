"""The tensor-core kernels start while the previous kernel of the stream still runs (programmatic dependent
launch).  Their bounded waits must not count the time of that kernel: a correct call behind a long one gives
the outputs it gives on an idle device, and no wait gives up."""
import numpy as np
import pytest

from paper_2508_06753_b200 import synth

pytestmark = pytest.mark.gpu

# One row of 2^30 values keeps a single CTA of the quantiser busy for 0.26 s, from a launch that lets its
# successor start at once and leaves 147 SMs to it.  A wait gives up after 2^20 polls of 1.48 us (measured on a
# barrier that nothing completes), i.e. 1.55 s: eight such launches in a row take 2.1 s.
LONG_ROW = 1 << 30
LAUNCHES = 8


@pytest.fixture(scope="module")
def gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_06753_b200 import binding, build
    build.build()
    binding.lib()
    return torch, binding


@pytest.mark.parametrize("switches,group,tile", [
    ({"W2A8_TC_KIND": "8"}, 64, 128),
    ({"W2A8_TC_KIND": "8"}, 256, 128),
    ({"W2A8_TC_KIND": "16"}, 64, 128),
    ({"W2A8_PF_WIDE": "2"}, 2048, 256),
])
def test_behind_a_long_kernel(gpu, monkeypatch, switches, group, tile):
    torch, b = gpu
    M, N, K = 200, 256, 2048                      # a ring of three or four stages is used more than twice
    monkeypatch.setenv("W2A8_PREFILL", "2")
    for k, v in switches.items():
        monkeypatch.setenv(k, v)
    assert b.w2a8_tensor_core_tile_tokens(M, N, K, group) == tile
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()
    codes, s_w = synth.make_linear(group, K, N, group)
    bits = synth.activations_bf16(group + 1, M, K)
    a, s_a = b.a8_quantize(dev(bits.view(np.int16)).view(torch.bfloat16))
    packed, scales = b.w2_pack(dev(codes)), dev(s_w)
    ws = b.new_workspace(b.w2a8_workspace_bytes(M, N, K, group))
    alone = b.w2a8_gemm(a, s_a, packed, scales, group, ws)
    torch.cuda.synchronize()
    assert b.w2a8_workspace_status(ws) == 0
    x = torch.randn((1, LONG_ROW), dtype=torch.bfloat16, device="cuda")
    row, scale = torch.empty((1, LONG_ROW), dtype=torch.int8, device="cuda"), torch.empty(1, device="cuda")
    y = torch.full_like(alone, float("nan"))
    torch.cuda.synchronize()
    for _ in range(LAUNCHES):
        b.a8_quantize(x, row, scale)
    b.w2a8_gemm(a, s_a, packed, scales, group, ws, y=y)
    torch.cuda.synchronize()
    assert b.w2a8_workspace_status(ws) == 0
    assert torch.equal(y, alone)
