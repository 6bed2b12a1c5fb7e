"""The folded layout of a skew tensor (csrc/k1t.cuh) without a GPU: its values
give the dense contraction, and the kernel's row ranges and copies cover the
stored tensor (folded_plan.cpp)."""
import os
import subprocess

import numpy as np
import pytest

import oracle
import synth
import paper_2311_03694_gb300 as grom
from test_plan_invariants import _cuda_include

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def folded_contraction(C, u):
    """c from the stored values: group m, rows q <= m, positions p < m."""
    c = np.zeros(len(u))
    for m in range(1, len(u)):
        F = C[:m, : m + 1, m].copy()                      # C_pqm
        F[:, :m] += C[:m, m, :m]                          # + C_pmq, q < m
        F[np.arange(m), np.arange(m)] = C[np.arange(m), np.arange(m), m]  # C_pmp is zero in a skew tensor
        D = F @ u[: m + 1]
        c[:m] += D * u[m]
        c[m] -= D @ u[:m]
    return c


@pytest.mark.parametrize("n", [1, 2, 3, 4, 7, 16, 33])
def test_folded_values_give_the_dense_contraction(n):
    C = synth.skew_normal_tensor(n, 40 + n)
    u = synth.initial_condition(n, 50 + n)[0]
    ref = oracle.nonlinear_full(C, u)
    # n^2 terms of three roundings each, on the scale of their absolute sum
    bound = 8 * 2.0 ** -53 * np.max(oracle.nonlinear_full(np.abs(C), np.abs(u)), initial=0.0) * max(n, 4)
    c = folded_contraction(C, u)
    assert np.max(np.abs(c - ref)) <= bound
    assert abs(u @ c) <= bound * np.sum(np.abs(u))


def test_folded_plan(tmp_path):
    lib = grom.build()
    inc = _cuda_include()
    if inc is None:
        pytest.skip("CUDA headers not found")
    exe = str(tmp_path / "folded_plan")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I" + inc, "-I" + os.path.join(ROOT, "paper_2311_03694_gb300", "csrc"),
                    os.path.join(HERE, "folded_plan.cpp"), lib, "-Wl,-rpath," + os.path.dirname(lib), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and ", 0 failed" in r.stdout, r.stdout[-2000:]
