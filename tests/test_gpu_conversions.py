"""The integer-pipe conversions, bit for bit over their whole range
(conversions.cu), and K2's sums at the edges of theirs: partial sums whose total
leaves the FP32 range are summed in FP64, and a non-finite trajectory stays alone."""
import importlib
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2311_03694_gb300 as grom  # noqa: E402

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
grom_build = importlib.import_module("paper_2311_03694_gb300.build")


def test_conversions_equal_the_instructions(tmp_path):
    exe = str(tmp_path / "conversions")
    subprocess.run([grom_build._nvcc()] + grom_build.ARCH + ["-O2", "-std=c++17", "-I" + grom_build.CSRC,
                   os.path.join(HERE, "conversions.cu"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


def test_k2_sums_beyond_the_fp32_range():
    grom.build()
    n, batch, value = 64, 16, 2.0 ** 117
    C = np.full((n, n, n), value)
    rom = grom.Rom(n, "full", "bf16", tensor=C, stiffness=np.ones(n), max_batch=batch)
    rom.set_kernel("tensor")
    u = torch.ones(batch, n, dtype=torch.float64, device="cuda")
    u[3, 5] = float("inf")
    c = torch.empty_like(u)
    rom.nonlinear(u, c)
    c = c.cpu().numpy()
    # powers of two throughout: n^2 terms sum exactly, beyond the largest float
    assert value * n * n > float(np.finfo(np.float32).max)
    for b in range(batch):
        if b == 3:
            assert not np.isfinite(c[b]).any()
        else:
            np.testing.assert_array_equal(c[b], np.full(n, value * n * n))
    rom.close()
