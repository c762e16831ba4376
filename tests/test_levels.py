"""The float64 path's single launch per anti-diagonal (leaf blocks of 16, the
next anti-diagonal's early sums beside the leaves): how a launch's work is cut
(on the CPU), and results against the oracle where the blocks can go wrong."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1607_06303_gb300.inputs import make_T

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_level_split(tmp_path):
    exe = str(tmp_path / "level_split_check")
    csrc = os.path.join(ROOT, "paper_1607_06303_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-I", csrc,
                    os.path.join(ROOT, "tests", "level_split_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    assert out.stdout.startswith("ok ")


# one block and a ragged one (17, 31), the first anti-diagonals whose near
# blocks coincide or touch the diagonal (33 .. 65), an odd ordinary order, and
# more leaves than SMs (2449: two CTAs on an SM)
@pytest.mark.gpu
@pytest.mark.parametrize("n", [17, 31, 33, 47, 48, 49, 65, 333, 2449])
@pytest.mark.parametrize("n_neg", [1, None])
def test_levels_vs_oracle(gpu_lib, oracle_mod, n, n_neg):
    import torch
    T = make_T(n, 0.5, seed=3 * n, n_neg=n_neg)
    U = gpu_lib.to_numpy(gpu_lib.sign(gpu_lib.to_device(T), gpu_lib.Variant.PH_FP64_EFFICIENT))
    torch.cuda.synchronize()
    ref = oracle_mod.sign_tri(T, schedule="antidiag")
    # each entry is a sum of at most n products, each rounding at most eps / 2
    # of the sum's size: n eps covers both sides
    assert np.linalg.norm(U - ref) <= n * np.finfo(float).eps * np.linalg.norm(ref)
    assert np.array_equal(np.diag(U), np.sign(np.diag(T))) and np.all(np.tril(U, -1) == 0)
