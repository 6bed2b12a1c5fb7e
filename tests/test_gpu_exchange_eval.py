"""One-launch evaluations of FP64 CP forms (one to four trajectories): against
the oracle within the FP64 tolerance (1e-12) and against the two-kernel path, at
the edges of its columns and rows (CTAs without a column or without a row,
several columns a CTA), in place, between steps that share its published words,
and replayed from a captured graph."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
import paper_2311_03694_gb300 as grom  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    grom.build()


def _factors(form, n, r):
    if form == "cp_skew":
        U, V, W, _, _ = synth.cp_workload(n, r, 1)
        return (U, V, W), lambda u: oracle.nonlinear_cp_skew(U, V, W, u)
    rng = np.random.default_rng(n + r)
    A, B, C = (rng.standard_normal((n, r)) / np.sqrt(r) for _ in range(3))
    return (A, B, C), lambda u: oracle.nonlinear_cp(A, B, C, u)


@pytest.mark.parametrize("form", ["cp_skew", "cp"])
@pytest.mark.parametrize("n,r,batch", [(1, 1, 1), (5, 300, 2), (9, 3, 4), (257, 150, 1), (300, 153, 2), (600, 257, 3),
                                       (640, 700, 1), (2048, 9, 4)])
def test_evaluation_matches_the_oracle(form, n, r, batch):
    fac, ref = _factors(form, n, r)
    U = synth.initial_condition(n, 3 + n, 0, batch)
    rom = grom.Rom(n, form, "f64", factors=fac, stiffness=synth.diag_stiffness(n), max_batch=batch)
    u = torch.from_numpy(U).cuda()
    got = {}
    for kernel in ("stream", "auto"):
        rom.set_kernel(kernel)
        c = torch.full_like(u, float("nan"))
        rom.nonlinear(u, c)
        torch.cuda.synchronize()
        got[kernel] = c.cpu().numpy()
    tr = grom.Trajectories(rom, U)
    tr.step(6)  # its words follow the evaluation's
    v = u.clone()
    rom.nonlinear(v, v)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(v.cpu().numpy(), got["auto"])
    assert tr.status()[0] == 0
    tr.close()
    rom.close()
    for b in range(batch):
        want = ref(U[b])
        # below one rounding of each product and sum where the terms cancel (n = 1: c = 0)
        floor = 1e-12 * np.linalg.norm(want) + (1e-15 if n == 1 else 0.0)
        for c in got.values():
            assert np.linalg.norm(c[b] - want) <= floor, b


def test_evaluation_replays_from_a_graph():
    n, r = 200, 100
    fac, ref = _factors("cp_skew", n, r)
    s = torch.cuda.Stream()
    rom = grom.Rom(n, "cp_skew", "f64", factors=fac, stiffness=synth.diag_stiffness(n), max_batch=1, stream=s)
    u = torch.zeros((1, n), dtype=torch.float64, device="cuda")
    c = torch.empty_like(u)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        rom.nonlinear(u, c)
    for k in range(3):
        U = synth.initial_condition(n, 40 + k, 0, 1)
        u.copy_(torch.from_numpy(U))
        g.replay()
        torch.cuda.synchronize()
        want = ref(U[0])
        assert np.linalg.norm(c.cpu().numpy()[0] - want) <= 1e-12 * np.linalg.norm(want), k
    rom.close()
