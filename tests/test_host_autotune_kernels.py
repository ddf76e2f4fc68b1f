"""A stored choice belongs to the kernels it was timed on."""
import pytest

pytest.importorskip("torch")

from paper_2601_17354_gb300 import autotune as A


def test_key_changes_with_the_kernels(monkeypatch):
    key = lambda: A.workload_key("single-T16", ["640x480"], 1000, 3)
    now = key()
    assert key() == now
    monkeypatch.setattr(A, "_kernels", lambda: "other")
    other = key()
    assert other != now and other.split("|")[1:] == now.split("|")[1:]
