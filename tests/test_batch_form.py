"""The rule that chooses between the batch kernel's two forms (csrc/spmspv_batch_form.h), compiled for the host."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def one_by_one(tmp_path_factory):
    out = tmp_path_factory.mktemp("form") / "libplan_shim.so"
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2607_21985_b200", "csrc"),
                    "-o", str(out), os.path.join(ROOT, "tests", "plan_shim.cpp")], check=True)
    f = ctypes.CDLL(str(out)).shim_batch_loads_one_by_one
    f.argtypes = [ctypes.c_longlong] * 3
    return lambda nnz, M, K: bool(f(nnz, M, K))


@pytest.mark.parametrize("M", [1, 16, 255, 256, 257, 300, 512, 520, 700, 4096, 28672])
@pytest.mark.parametrize("K", [16, 1000, 8192])
def test_the_form_follows_the_density_and_not_the_rows_of_the_last_tile(one_by_one, M, K):
    """80 values of a full tile of 256 rows, whatever share of the last row tile the matrix has."""
    line = 80 * M * K // 256
    assert one_by_one(line, M, K) and not one_by_one(line + 1, M, K)
    assert one_by_one(0, M, K) and not one_by_one(M * K, M, K)
    assert not one_by_one(M * K // 2, M, K) and one_by_one(M * K * 3 // 10, M, K)
