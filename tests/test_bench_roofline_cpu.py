"""The benchmark's roofline names the SpMM kernel that runs, and its traffic
figure follows that kernel's source."""
import os
import re
import shutil

import pytest

pytest.importorskip("torch")
import bench  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_roofline_kernels_exist():
    text = open(os.path.join(ROOT, "bench.py")).read()
    names = set(re.findall(r"\bk_[a-z0-9_]+", " ".join(
        re.findall(r'"kernels?":\s*((?:"[^"]*"\s*)+)', text))))
    assert {"k_spmm_fix", "k_fft_rows", "k_fft_cols", "k_fft_back"} <= names
    src = "".join(open(os.path.join(bench.CSRC, f)).read() for f in os.listdir(bench.CSRC)
                  if f.endswith((".cu", ".cuh")))
    for name in names:
        assert re.search(r"\b%s\(" % name, src), name


def test_traffic_digest_follows_the_sweep(tmp_path, monkeypatch):
    dst = tmp_path / "csrc"
    shutil.copytree(bench.CSRC, dst)
    monkeypatch.setattr(bench, "CSRC", str(dst))
    before = bench.fix_kernel_digest()
    for name in ("fix.cu", "tma.cuh"):
        with open(dst / name, "a") as f:
            f.write("\n// edited\n")
        after = bench.fix_kernel_digest()
        assert after != before
        before = after
        assert bench.traffic_ratio_from_profile() is None
