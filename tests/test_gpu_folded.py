"""The folded skew-packed kernels (F64, F32X2) against the FP64 oracle where
their tiles change: one and two vectors a thread and row, four, two and one
row groups a warp, passes of one to four trajectories, CTAs with no row, one
group or many.  Tolerances: 1e-12 an evaluation (the FP64-class storages), 1e-11
for the states after a few steps, as in the other tests of the layout."""
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


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("storage", ["f64", "f32x2"])
@pytest.mark.parametrize("n", [5, 33, 130, 258, 515])
def test_evaluations_and_steps(storage, n):
    batch, steps = 7, 4  # passes of four and three, or of fewer
    C = synth.skew_normal_tensor(n, 900 + n)
    a = synth.diag_stiffness(n)
    U = synth.initial_condition(n, 901 + n, 0, batch)
    rom = grom.Rom(n, "full", storage, tensor=C, stiffness=a, max_batch=batch, layout="skew_packed")
    u = torch.from_numpy(U).cuda()
    c = torch.full_like(u, float("nan"))
    rom.nonlinear(u, c)
    torch.cuda.synchronize()
    for b in range(batch):
        assert _rel(c[b].cpu().numpy(), oracle.nonlinear_full(C, U[b])) <= 1e-12, b
    ref = oracle.Rom("full", n, a, 1e-2, 1e-3, C=C)
    for count in (1, 2, 3, 4, 7):  # the last takes the per-step kernels
        tr = grom.Trajectories(rom, U[:count])
        tr.step(steps)
        H = tr.get_state()
        tr.close()
        for b in (0, count - 1):
            h = ref.initial_history(U[b])
            ref.step(h, steps)
            assert _rel(H[b][:n], h[:n]) <= 1e-11, (count, b)
    rom.close()


@pytest.mark.parametrize("storage,n", [("f64", 1030), ("f64", 2052), ("f32x2", 2052)])
def test_rows_of_several_vectors_a_thread(storage, n):
    # two and four vectors a thread and row; a CP-structured tensor, uploaded
    # in slabs made on the device, whose contraction has a closed form
    batch, rank = 4, 3
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    U, V, W = (torch.randn(n, rank, generator=g, dtype=torch.float64, device="cuda") / n ** 0.5 for _ in range(3))
    rom = grom.Rom(n, "full", storage, stiffness=synth.diag_stiffness(n), max_batch=batch, layout="skew_packed",
                   defer_tensor=True)
    for i0 in range(0, n, 60):
        i1 = min(n, i0 + 60)
        X = ((U[i0:i1, None, :] * V[None]).reshape(-1, rank) @ W.T - (W[i0:i1, None, :] * V[None]).reshape(-1, rank) @ U.T)
        rom.upload_slab(i0, X.reshape(i1 - i0, n, n).contiguous())
    u = torch.randn(batch, n, generator=g, dtype=torch.float64, device="cuda") / torch.arange(1, n + 1, device="cuda")
    c = torch.full_like(u, float("nan"))
    rom.nonlinear(u, c)
    p, q, s = u @ V, u @ W, u @ U
    want = (p * q) @ U.T - (p * s) @ W.T
    torch.cuda.synchronize()
    for b in range(batch):
        assert float(torch.linalg.norm(c[b] - want[b]) / torch.linalg.norm(want[b])) <= 1e-12, b
    tr = grom.Trajectories(rom, u[:1])
    tr.step(2)
    assert tr.status()[0] == 0
    tr.close()
    rom.close()
