"""The exchange stepper of the CP forms (one to four trajectories, factors in
shared memory by columns and by rows) against the oracle's stepper on the same
rounded factors and against the per-step kernels: sizes around its tiles (one
CTA, columns or rows without a CTA of their own, ragged vectors), both forms, all
operators, energies and invariants.  FP64: 1e-11 after 12 steps; FP32 sums:
2e-6 (each advection term to ~1e-6, its effect on a state scaled by dt)."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
import paper_2311_03694_gb300 as grom  # noqa: E402

pytestmark = pytest.mark.gpu
TOL = {"f64": 1e-11, "f32": 2e-6, "bf16": 2e-6}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    grom.build()


def _stored(x, storage):
    t = torch.from_numpy(x)
    return {"f64": t, "f32": t.float(), "bf16": t.float().bfloat16()}[storage].double().numpy()


@pytest.mark.parametrize("storage,batch", [("f64", 1), ("f64", 2), ("f32", 3), ("bf16", 1), ("bf16", 4)])
@pytest.mark.parametrize("form", ["cp_skew", "cp"])
@pytest.mark.parametrize("n,r", [(5, 3), (70, 9), (9, 130), (257, 100), (300, 300)])
def test_steps_match_the_oracle(storage, batch, form, n, r):
    steps, dt, nu = 12, 1e-3, 1e-2
    U, V, W, _, seed = synth.cp_workload(n, r, 1)
    F = [_stored(f, storage) for f in (U, V * 20.0, W)]
    a, rng = synth.diag_stiffness(n), np.random.default_rng(n)
    extra = dict(mass=1.0 + 0.1 * rng.random(n), linear=0.1 * rng.random(n), forcing=0.01 * rng.random(n)) if n == 70 else {}
    U0 = synth.initial_condition(n, seed, 0, batch)
    rom = grom.Rom(n, form, storage, factors=F, stiffness=a, nu=nu, dt=dt, max_batch=batch, **extra)
    ref = oracle.Rom(form, n, a, nu, dt, factors=F, B=np.diag(extra["mass"]) if extra else None,
                     L=np.diag(extra["linear"]) if extra else None, f=extra.get("forcing"))
    tr = grom.Trajectories(rom, U0)
    E = torch.empty((steps, batch), dtype=torch.float64, device="cuda")
    inv = torch.empty_like(E)
    tr.step(5, E[:5], inv[:5])
    tr.step(7, E[5:], inv[5:])
    assert tr.status()[0] == 0
    plain = grom.Trajectories(rom, U0)
    plain.step(steps)  # one call, no sums: the same bits
    H = tr.get_state()
    np.testing.assert_array_equal(plain.get_state(), H)
    for b in range(batch):
        h = ref.initial_history(U0[b])
        e_ref, i_ref = ref.step(h, steps, want_energy=True, want_invariant=True)
        assert np.linalg.norm(H[b][:n] - h[:n]) <= TOL[storage] * np.linalg.norm(h[:n]), b
        np.testing.assert_allclose(E.cpu().numpy()[:, b], e_ref, rtol=4 * TOL[storage])
        assert H[b][6 * n] == steps
    tr.close()
    plain.close()
    rom.close()
