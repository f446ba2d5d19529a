"""The autotuner's cache file: one per GPU and per state of the sources, so that
mappings chosen on other kernels are not installed again."""
import torch

from paper_2104_07638_gb300 import batch


def test_cache_file_changes_with_the_sources(monkeypatch, tmp_path):
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda: "NVIDIA GB300")
    src = tmp_path / "kernel.cu"
    src.write_text("a")
    monkeypatch.setattr(batch._build, "_deps", lambda: [str(src)])
    first = batch._cache_path()
    assert batch._cache_path() == first
    src.write_text("b")
    assert batch._cache_path() != first
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda: "another GPU")
    assert "another_GPU" in batch._cache_path()
