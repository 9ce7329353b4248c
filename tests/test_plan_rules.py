"""Dispatch rules on the host (no GPU needed): the automatic fuse rule at the edges of its range, and the switches
that force the tensor-core kernel."""
import pytest

from paper_2508_06753_b200 import binding as b


@pytest.fixture(autouse=True)
def library(monkeypatch):
    from paper_2508_06753_b200 import build
    build.build()
    for name in ("W2A8_FUSE_MAX_ELEMS", "W2A8_GEMV", "W2A8_STAT", "W2A8_GEMV_WARPS", "W2A8_GEMV_BCACHE",
                 "W2A8_PREFILL", "W2A8_PF_KSPLIT", "W2A8_PF_WIDE", "W2A8_TC_KIND"):
        monkeypatch.delenv(name, raising=False)


@pytest.mark.parametrize("Ns,M,K,fused", [
    ([2048], 1, 2048, True),
    ([16], 1, 1024, True),                # one tile
    ([4736], 1, 4096, True),              # one tile per CTA, the last such size
    ([4752], 1, 4096, True),
    ([4096, 1024, 1024], 1, 4096, True),
    ([14192], 1, 4096, True),
    ([14336, 14336], 1, 4096, True),
    ([2048], 1, 3072, False),             # no instance with these rows in registers
    ([2048], 1, 8192, False),
    ([2048], 2, 2048, False),             # more than one token
    ([4096], 1, 14336, False),            # activations do not stay in registers
])
def test_automatic_fuse_rule(Ns, M, K, fused):
    assert b.w2a8_grouped_plan(Ns, M, K, 64)["fused"] is fused


def test_limit_replaces_the_rule(monkeypatch):
    monkeypatch.setenv("W2A8_FUSE_MAX_ELEMS", "0")
    assert b.w2a8_grouped_plan([2048], 1, 2048, 64)["fused"] is False
    monkeypatch.setenv("W2A8_FUSE_MAX_ELEMS", "4096")
    assert b.w2a8_grouped_plan([2048], 2, 2048, 64)["fused"] is True


@pytest.mark.parametrize("M", [64, 65, 128, 256])
@pytest.mark.parametrize("N,K", [(4096, 4096), (14336, 4096), (4096, 14336), (128, 256)])
def test_tensor_core_kernel_when_forced(monkeypatch, M, N, K):
    for more in ({}, {"W2A8_PF_KSPLIT": "2"}, {"W2A8_PF_WIDE": "2"}, {"W2A8_TC_KIND": "16"}):
        monkeypatch.setenv("W2A8_PREFILL", "2")
        for name, value in more.items():
            monkeypatch.setenv(name, value)
        assert b.w2a8_kernel_for(M, N, K, 64) == "tensor_core", more
        assert b.w2a8_kernel_for(M, N, K, K) == "tensor_core", more
        for name in more:
            monkeypatch.delenv(name)
    monkeypatch.setenv("W2A8_PREFILL", "0")
    assert b.w2a8_kernel_for(M, N, K, 64) == "streaming"


def test_workspace_covers_the_channel_remainder_of_bf16_activations(monkeypatch):
    """w2a16_gemm has a tensor-core rule of its own and may split channels where w2a8_gemm does not; one query
    sizes the workspace of both."""
    found = 0
    for M in (65, 100, 136, 140, 180, 200, 256, 300, 512, 700):
        for N in (4096, 8192, 14336, 19456, 28672):
            for K in (1024, 2048, 4096, 8192):
                for group in (64, 128, K):
                    monkeypatch.setenv("W2A8_TC_KIND", "16")         # the rule for 16-bit operands
                    takes = b.w2a8_kernel_for(M, N, K, group) == "tensor_core"
                    channels = b.w2a8_tensor_core_channels(M, N, K, group)
                    monkeypatch.delenv("W2A8_TC_KIND")
                    if not takes or channels == N:
                        continue
                    found += 1
                    size = b.w2a8_workspace_bytes(M, N, K, group)
                    monkeypatch.setenv("W2A8_PREFILL", "0")          # the remainder runs on a streaming kernel
                    rest = b.w2a8_workspace_bytes(M, N - channels, K, group)
                    monkeypatch.delenv("W2A8_PREFILL")
                    assert size >= rest, (M, N, K, group)
    assert found > 10


@pytest.mark.parametrize("N,K,group,kernel", [
    (28672, 8192, 8192, "tensor_core"),
    (28672, 8192, 128, "tensor_core"),
    (14336, 4096, 4096, "tensor_core"),
    (4096, 14336, 128, "tensor_core"),
    (4096, 14336, 64, "streaming"),
    (4096, 4096, 64, "streaming"),
    (8192, 8192, 64, "streaming"),
    (5120, 14336, 128, "streaming"),
])
def test_64_tokens(monkeypatch, N, K, group, kernel):
    """The fewest tokens of the tensor-core kernel, which is ahead there with large groups only (of the kernels other
    than the streaming one on the tensor cores), and not by a K split whose scratch w2a8_gemm_static does not have."""
    monkeypatch.setenv("W2A8_TSTREAM", "0")
    assert b.w2a8_kernel_for(64, N, K, group) == kernel
    if (N, K) == (5120, 14336):
        assert b.w2a8_workspace_bytes(64, N, K, group) <= 8 << 20


@pytest.mark.parametrize("M,taken", [(8, False), (32, True), (33, True), (64, True), (65, False)])
def test_streaming_tensor_core_kernel(monkeypatch, M, taken):
    import ctypes
    monkeypatch.delenv("W2A8_TSTREAM", raising=False)
    plan = lambda: bool(b.lib().w2a8_grouped_plan(2, (ctypes.c_int * 2)(28672, 28672), M, 8192, 128, b.FUSE_OFF) & 4)
    assert plan() is taken
    for name in ("W2A8_GEMV", "W2A8_STAT"):           # another kernel forced, or kept out
        monkeypatch.setenv(name, "2")
        assert plan() is False
        monkeypatch.setenv(name, "0")
        assert plan() is taken
        monkeypatch.delenv(name)
    monkeypatch.setenv("W2A8_TSTREAM", "0")
    assert plan() is False


@pytest.mark.parametrize("Ns,M,K,group,taken", [
    ([14336, 14336], 8, 4096, 128, False),
    ([3840], 9, 2560, 64, True),                  # short rows that the persistent kernel does not hold
    ([3840], 16, 2560, 2560, True),
    ([3840], 17, 2560, 64, False),
    ([4096], 16, 2048, 64, False),                # rows that it holds
    ([16384], 12, 1280, 64, False),               # too short for the sums
    ([57344], 64, 1280, 128, False),
    ([57344], 64, 1280, 1280, True),
    ([4096], 32, 4096, 128, False),               # 512 blocks
    ([4096], 64, 4096, 128, True),
    ([28672], 64, 4096, 1024, False),             # four groups at 64 tokens
    ([28672], 63, 4096, 1024, True),
    ([28672, 28672], 64, 8192, 64, True),
])
def test_where_the_streaming_tensor_core_kernel_is_taken(monkeypatch, Ns, M, K, group, taken):
    import ctypes
    monkeypatch.delenv("W2A8_TSTREAM", raising=False)
    plan = b.lib().w2a8_grouped_plan(len(Ns), (ctypes.c_int * len(Ns))(*Ns), M, K, group, b.FUSE_OFF)
    assert bool(plan & 4) is taken


@pytest.mark.parametrize("M", [32, 48, 64])
def test_reports_say_what_runs(monkeypatch, M):
    """Two matrices that the streaming kernel on the tensor cores takes: one launch, and no tensor-core kernel with its
    splits and tiles; without it a launch per matrix above 32 tokens, on the tensor-core kernel at 64."""
    plan = lambda: b.w2a8_grouped_plan([28672, 28672], M, 8192, 8192, b.FUSE_OFF)
    reports = lambda: (b.w2a8_kernel_for(M, 28672, 8192, 8192), b.w2a8_tensor_core_kind(M, 28672, 8192, 8192),
                       b.w2a8_tensor_core_channels(M, 28672, 8192, 8192) > 0, b.w2a8_tensor_core_ksplit(M, 28672, 8192, 8192) > 0,
                       b.w2a8_tensor_core_tile_tokens(M, 28672, 8192, 8192) > 0)
    monkeypatch.delenv("W2A8_TSTREAM", raising=False)
    assert plan() == {"one_launch": True, "fused": False}
    assert reports() == ("streaming", 0, False, False, False)
    monkeypatch.setenv("W2A8_TSTREAM", "0")
    assert plan()["one_launch"] is (M == 32)
    assert reports() == (("tensor_core", 8, True, True, True) if M == 64 else ("streaming", 0, False, False, False))

