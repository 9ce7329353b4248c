"""The W2A8_* switches are looked up anew whenever the environment changes, however it changes (host only)."""
import ctypes

import pytest

from paper_2508_06753_b200 import binding as b

SHAPE = (96, 4096, 4096, 64)        # M, N, K, group: streaming kernel by default, tensor cores without W2A8_STAT


@pytest.fixture(autouse=True)
def library(monkeypatch):
    from paper_2508_06753_b200 import build
    build.build()
    monkeypatch.delenv("W2A8_STAT", raising=False)


def test_set_and_unset(monkeypatch):
    assert b.w2a8_kernel_for(*SHAPE) == "streaming"
    monkeypatch.setenv("W2A8_STAT", "0")
    assert b.w2a8_kernel_for(*SHAPE) == "tensor_core"
    monkeypatch.delenv("W2A8_STAT")
    assert b.w2a8_kernel_for(*SHAPE) == "streaming"


def test_string_edited_in_place():
    """putenv makes the caller's own string part of the environment: an edit of it is a new value."""
    libc = ctypes.CDLL(None)
    text = ctypes.create_string_buffer(b"W2A8_STAT=1")
    assert libc.putenv(text) == 0
    try:
        assert b.w2a8_kernel_for(*SHAPE) == "streaming"
        text[len("W2A8_STAT=")] = b"0"
        assert b.w2a8_kernel_for(*SHAPE) == "tensor_core"
    finally:
        libc.unsetenv(b"W2A8_STAT")
