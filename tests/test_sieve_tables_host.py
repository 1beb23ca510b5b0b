"""The sieve form's tables, compiled for the host from the kernels' own source: contexts created by
several threads at once upload the same bytes as one thread does."""
import os
import subprocess

import pytest

from test_sigma_search_host import ROOT, _nvcc


def test_tables_uploaded_by_several_threads_are_whole(tmp_path):
    nvcc = _nvcc()
    if not nvcc:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "sieve_tables_host")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-diag-suppress", "550",
                    "-I", os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "host", "sieve_tables_host.cu"),
                    "-o", exe, "-lpthread"], check=True, capture_output=True)
    uploads, wrong = subprocess.run([exe], capture_output=True, text=True, check=True, timeout=120).stdout.split()
    assert int(uploads) == 2 * (8 * 100 + 1)
    assert int(wrong) == 0
