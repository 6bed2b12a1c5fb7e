"""grom_als_stats counts every solve in full: a factorisation beside an MTTKRP
costs what one alone costs.  With residuals, the first update of every later
iteration has its MTTKRP already and factorises alone (8 of 27 updates here);
without them all 27 run beside one.  The same 27 solves, so the sums agree up to
what sharing the device costs (the ones beside an MTTKRP are the slower); a sum
that left out the hidden factorisations would lack more than half of theirs."""
import ctypes

import pytest

import synth

torch = pytest.importorskip("torch")
import paper_2311_03694_gb300 as grom  # noqa: E402

pytestmark = pytest.mark.gpu


def test_solves_beside_an_mttkrp_count_in_full():
    grom.build()
    n, r, iters = 512, 32, 9
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    als = grom.Als(torch.randn(n, n, n, generator=g, dtype=torch.float64, device="cuda"))
    F0 = [synth.normal(7, 30 + q, 0, n * r).reshape(n, r) / n ** 0.5 for q in range(3)]

    def solve_ms(residual):
        F = [f.copy() for f in F0]
        res = (ctypes.c_double * iters)()
        als.stats()
        assert grom.load().grom_als_fit(als._h, r, 0, iters, 0.5, 1, 1e-5, *(f.ctypes.data for f in F),
                                        res if residual else None) == 0
        return als.stats()[2]

    solve_ms(True)  # warm-up
    alone, beside = (min(solve_ms(residual) for _ in range(3)) for residual in (True, False))
    als.close()
    assert alone <= 1.15 * beside, (alone, beside)
