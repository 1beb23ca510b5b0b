"""The form a DNA solve takes, from the runtime's own estimate compiled for the host: the cases listed
for each of the sieve's kernels (test_gpu_sieve.py) take it, so that none goes untested unnoticed."""
import os
import subprocess

import pytest

from test_gpu_sieve import FORMS
from test_sigma_search_host import ROOT, _nvcc

# (n, m, l, d, q, alone): quorums whose sieve would wait for the warp of one block; the tree took half as long
TREE = [(20, 1500, 9, 0, 19, 1), (8, 1392, 10, 0, 7, 1), (5, 3000, 11, 0, 4, 1), (8, 1392, 12, 1, 7, 1), (40, 600, 10, 2, 38, 1)]
# every kernel that launch_sieve holds: middle letters, counter planes, warps per block (0: a sequence a warp)
KERNELS = {(3, 0, 0), (3, 0, 1), (4, 0, 0), (4, 0, 1), (5, 0, 1), (5, 0, 8), (6, 0, 8), (3, 7, 1), (4, 5, 1), (5, 5, 8)}


def test_listed_cases_take_their_form(tmp_path):
    nvcc = _nvcc()
    if not nvcc:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "sieve_forms_host")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-diag-suppress", "550",
                    "-I", os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "host", "sieve_forms_host.cu"),
                    "-o", exe, "-Xlinker", "--unresolved-symbols=ignore-all"],   # the kernels: none is launched
                   check=True, capture_output=True)
    assert set(FORMS) == KERNELS
    cases = [(f, c) for f in FORMS for c in FORMS[f]] + [((0, 0, 0), c) for c in TREE]
    lines = "\n".join(" ".join(map(str, (152,) + c)) for _, c in cases)
    out = subprocess.run([exe], input=lines, capture_output=True, text=True, check=True, timeout=120).stdout.split("\n")
    got = [tuple(int(v) for v in line.split()) for line in out if line]
    assert len(got) == len(cases)
    for (form, case), g in zip(cases, got):
        assert g == form, case
