"""The folded stepper with several vectors a thread and row (F64 above n = 1024
and 2048, F32X2 above 2048): states, energy and invariant of a few steps, for one
trajectory and for the most a launch takes, against the same steps in torch FP64
on a CP-structured tensor, whose contraction has a closed form.  Tolerances: 1e-11
for states and energy, as in the other tests of the layout; the invariant u . c is
zero, so it is compared on the scale |u| |c| of its terms."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import paper_2311_03694_gb300 as grom  # noqa: E402

pytestmark = pytest.mark.gpu
NU, DT = 1e-2, 1e-3
BETA = ((1.0, -1.0), (1.5, -2.0, 0.5), (11.0 / 6.0, -3.0, 1.5, -1.0 / 3.0))
ALPHA = ((1.0,), (2.0, -1.0), (3.0, -3.0, 1.0))


@pytest.mark.parametrize("storage,n,batch", [("f64", 1030, 1), ("f64", 1030, 4), ("f64", 2052, 1), ("f64", 2052, 2),
                                             ("f32x2", 2052, 1), ("f32x2", 2052, 2)])
def test_states_energy_and_invariant(storage, n, batch):
    grom.build()
    steps, rank = 4, 3
    g = torch.Generator(device="cuda")
    g.manual_seed(n + batch)
    U, V, W = (torch.randn(n, rank, generator=g, dtype=torch.float64, device="cuda") / n ** 0.5 for _ in range(3))
    a = synth.diag_stiffness(n)
    rom = grom.Rom(n, "full", storage, stiffness=a, nu=NU, dt=DT, max_batch=batch, layout="skew_packed",
                   defer_tensor=True)
    for i0 in range(0, n, 60):
        i1 = min(n, i0 + 60)
        X = ((U[i0:i1, None, :] * V[None]).reshape(-1, rank) @ W.T - (W[i0:i1, None, :] * V[None]).reshape(-1, rank) @ U.T)
        rom.upload_slab(i0, X.reshape(i1 - i0, n, n).contiguous())
    u = torch.randn(batch, n, generator=g, dtype=torch.float64, device="cuda") / torch.arange(1, n + 1, device="cuda")
    tr = grom.Trajectories(rom, u)
    energy = torch.full((steps, batch), float("nan"), dtype=torch.float64, device="cuda")
    invariant = torch.full_like(energy, float("nan"))
    tr.step(steps, energy, invariant)
    H = tr.get_state()
    code, _ = tr.status()
    assert code == 0
    A = torch.from_numpy(np.asarray(a)).cuda()
    us, cs = [u], []
    for s in range(steps):
        k = min(s + 1, 3)
        p = us[0] @ V
        cs = [(p * (us[0] @ W)) @ U.T - (p * (us[0] @ U)) @ W.T] + cs[:2]
        scale = torch.linalg.norm(us[0], dim=1) * torch.linalg.norm(cs[0], dim=1)
        assert bool((invariant[s].abs() <= 1e-11 * scale).all()), s
        rhs = sum(ALPHA[k - 1][q] * cs[q] for q in range(k)) + sum(BETA[k - 1][q + 1] / DT * us[q] for q in range(k))
        us = [-rhs / (BETA[k - 1][0] / DT + NU * A)] + us[:2]
        torch.testing.assert_close(energy[s], 0.5 * (us[0] ** 2).sum(1), rtol=1e-11, atol=0)
    for b in range(batch):
        want = us[0][b].cpu().numpy()
        assert np.linalg.norm(H[b][:n] - want) <= 1e-11 * np.linalg.norm(want), b
    tr.close()
    rom.close()
