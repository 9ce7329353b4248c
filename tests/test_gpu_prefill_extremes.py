"""The int8 tensor-core kernel at the ends of its accumulator range: groups of 64 and 128 start from a
constant that every sum of a group has to stay above, and their scales are fetched four at a time where a
row holds a multiple of four."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 1e-5        # at most 12 fp32 additions of exact group sums, two roundings each: below 2e-6


@pytest.fixture(scope="module")
def gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2508_06753_b200 import binding, build
    build.build()
    binding.lib()
    return torch, binding


@pytest.mark.parametrize("value", [127, -128])
@pytest.mark.parametrize("code", [0, 3])
@pytest.mark.parametrize("K,group", [(256, 64), (256, 128), (768, 128)])     # the last: six scales per row
def test_extreme_sums(gpu, oracle, monkeypatch, K, group, code, value):
    torch, b = gpu
    monkeypatch.setenv("W2A8_PREFILL", "2")
    M, N = 65, 128
    codes = np.full((N, K), code, np.uint8)
    a = np.full((M, K), value, np.int8)
    a[1::2, ::3] = 1
    rng = np.random.default_rng(K + group + code)
    s_w = (0.02 * np.exp(0.5 * rng.standard_normal((N, K // group)))).astype(np.float32)
    s_a = rng.uniform(0.001, 0.1, M).astype(np.float32)
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()
    packed, ta, tsa = b.w2_pack(dev(codes)), dev(a), dev(s_a)
    ws = b.new_workspace(b.w2a8_workspace_bytes(M, N, K, group))
    y = b.w2a8_gemm(ta, tsa, packed, dev(s_w), group, ws)
    ref = oracle.gemm(a, s_a, codes, s_w, group)
    err = np.abs(y.cpu().numpy().astype(np.float64) - ref)
    assert (err <= TOL * np.abs(ref).max(axis=1, keepdims=True)).all(), float(err.max())
