"""The rule that chooses between the batch kernel's two forms (csrc/spmspv_batch_form.h), compiled for the host."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def compile_rule(folder):
    """one_by_one(counts, M): does a layer whose column tiles hold counts[row tile, column] values take 16-bit loads?"""
    out = os.path.join(str(folder), "libplan_shim.so")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2607_21985_b200", "csrc"),
                    "-o", out, os.path.join(ROOT, "tests", "plan_shim.cpp")], check=True)
    f = ctypes.CDLL(out).shim_batch_loads_one_by_one
    f.argtypes = [ctypes.c_longlong] * 4

    def one_by_one(counts, M):
        counts = np.asarray(counts, np.int64)
        K = counts.shape[1]
        diff = counts[:, 0:K // 2 * 2:2] - counts[:, 1:K // 2 * 2:2]
        return bool(f(int(counts.sum()), int(2 * (diff * diff).sum()), M, K))
    return one_by_one


@pytest.fixture(scope="module")
def one_by_one(tmp_path_factory):
    return compile_rule(tmp_path_factory.mktemp("form"))


def rows_of(M):
    return np.array([min(256, M - r) for r in range(0, M, 256)])


def binomial(rng, M, densities):
    return rng.binomial(rows_of(M)[:, None], np.asarray(densities)[None, :])


@pytest.mark.parametrize("M", [250, 256, 300, 512, 520, 700, 1100, 4096])
def test_partial_row_tiles_count_like_whole_ones(one_by_one, M):
    """The form follows the density, whatever share of the last row tile the matrix has: 300 rows at 50 % are 128 values of a full
    tile and not 75."""
    rng = np.random.Generator(np.random.PCG64(M))
    for sparsity, loads in ((0.3, False), (0.5, False), (0.6, False), (0.66, False), (0.76, True), (0.8, True), (0.9, True), (1.0, True)):
        assert one_by_one(binomial(rng, M, np.full(4096, 1.0 - sparsity)), M) == loads, sparsity


@pytest.mark.parametrize("M,K", [(4096, 4096), (28672, 8192)])
def test_columns_of_different_density_take_words(one_by_one, M, K):
    """Both forms measured at these points: 28672x8192 at 70 % with columns up to 12 % apart takes 6.5 % longer with loads than before
    there were any."""
    rng = np.random.Generator(np.random.PCG64(K))
    large = M * K // 256 >= 200000
    measured = {(0.66, 0.0): False, (0.74, 0.0): not large, (0.82, 0.0): True, (0.9, 0.0): True, (0.7, 0.12): False, (0.74, 0.06): False,
                (0.74, 0.12): False, (0.78, 0.12): False, (0.74, 0.2): False, (0.9, 0.04): True, (0.82, 0.04): True}
    for (sparsity, spread), loads in measured.items():
        assert one_by_one(binomial(rng, M, 1.0 - sparsity + spread * rng.uniform(-1, 1, K)), M) == loads, (sparsity, spread)


def test_smallest_layers(one_by_one):
    assert one_by_one([[0]], 1) and not one_by_one([[1]], 1) and one_by_one([[0, 0, 0]], 5) and one_by_one([[256] + [0] * 999], 256)
