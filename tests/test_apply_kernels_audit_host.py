"""Host audit of the index arithmetic of the kernels that a plan chooses by estimated time: the two-CTA
pencil-load kernel and the two-exchange 16^3 kernels (tests/native/apply_kernels_audit.cu, no GPU);
test_index_audit_host.py covers the other layouts.
"""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_two_cta_and_two_exchange_indices(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "audit")
    src = os.path.join(HERE, "native", "apply_kernels_audit.cu")
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-diag-suppress", "177,1886", "-x", "cu", src, "-o", exe], check=True, capture_output=True, text=True)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    print(res.stdout)
    assert res.returncode == 0, res.stdout
    for n in (8, 10, 12, 18, 20):
        assert f"n={n} two CTAs:" in res.stdout
    assert res.stdout.strip().endswith("audit ok")
