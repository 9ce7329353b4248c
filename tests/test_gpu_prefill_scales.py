"""Scales at the ends of the fp32 range on the int8 tensor-core kernel: its drain multiplies a scale by 2^23 on
the way, which must not take a scale out of range that the product with the token scale brings back."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 1e-5        # at most 16 fp32 additions of exact group sums, three roundings each: below 3e-6


@pytest.fixture(scope="module")
def gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_06753_b200 import binding, build
    build.build()
    binding.lib()
    return torch, binding


@pytest.mark.parametrize("split", ["1", "2"])
@pytest.mark.parametrize("group", [64, 128])
@pytest.mark.parametrize("s_max,s_tok", [(1e30, 1e-30), (4.1e31, 1e-30), (1e33, 1e-33), (5e32, 1e-32),
                                         (1e-36, 1e30)])
def test_scales_at_the_ends_of_the_range(gpu, oracle, monkeypatch, s_max, s_tok, group, split):
    """Rows whose scales all lie near s_max, and rows where only one group does, at every place of a turn of the
    drain loop (four groups); the running sums before it then hold ordinary scales."""
    torch, b = gpu
    monkeypatch.setenv("W2A8_PREFILL", "2")
    monkeypatch.setenv("W2A8_PF_KSPLIT", split)
    M, N, K = 130, 256, 1024
    rng = np.random.default_rng(group)
    codes = rng.integers(0, 4, (N, K)).astype(np.uint8)
    a = rng.integers(-127, 128, (M, K)).astype(np.int8)
    s_w = (0.01 * s_max * rng.uniform(0.5, 1.0, (N, K // group))).astype(np.float32)
    for n in range(N):
        if n % 3 == 0:
            s_w[n, n % (K // group)] = s_max
    s_a = (s_tok * rng.uniform(0.5, 1.0, M)).astype(np.float32)
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()
    ws = b.new_workspace(b.w2a8_workspace_bytes(M, N, K, group))
    y = b.w2a8_gemm(dev(a), dev(s_a), b.w2_pack(dev(codes)), dev(s_w), group, ws)
    torch.cuda.synchronize()
    assert b.w2a8_workspace_status(ws) == 0
    ref = oracle.gemm(a, s_a, codes, s_w, group)
    assert np.isfinite(ref).all()
    err = np.abs(y.cpu().numpy().astype(np.float64) - ref)
    assert (err <= TOL * np.abs(ref).max(axis=1, keepdims=True)).all(), float(err.max())
