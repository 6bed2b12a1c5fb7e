"""The plain diagonal step of large batches (no energy or invariant asked for)
against the general step kernel, which runs when they are: the same element
arithmetic, so the same bits, at the edges of its tiles (256, 512 and 1024
elements a block, one block or several a trajectory) and at all three orders."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import paper_2311_03694_gb300 as grom  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    grom.build()


def _both(rom, U, steps):
    t1, t2 = grom.Trajectories(rom, U), grom.Trajectories(rom, U)
    E = torch.empty((1, U.shape[0]), dtype=torch.float64, device="cuda")
    for _ in range(steps):
        t1.step(1)
        t2.step(1, E, torch.empty_like(E))
    a, b = t1.get_state(), t2.get_state()
    t1.close()
    t2.close()
    return a, b


@pytest.mark.parametrize("n,batch", [(65, 256), (256, 257), (257, 300), (512, 256), (513, 260), (1024, 256), (1025, 130)])
def test_cp_batches_step_to_the_same_bits(n, batch):
    U, V, W, _, seed = synth.cp_workload(n, 24, 1)
    rom = grom.Rom(n, "cp_skew", "bf16", factors=(U, V * 50.0, W), stiffness=synth.diag_stiffness(n), max_batch=batch)
    a, b = _both(rom, synth.initial_condition(n, seed, 0, batch), 4)
    np.testing.assert_array_equal(a, b)
    assert np.all(a[:, 6 * n] == 4)
    rom.close()


def test_full_batch_steps_to_the_same_bits():
    n, batch = 70, 300
    C = synth.skew_normal_tensor(n, 5)
    rom = grom.Rom(n, "full", "bf16", tensor=C, stiffness=synth.diag_stiffness(n), max_batch=batch)
    a, b = _both(rom, synth.initial_condition(n, 6, 0, batch), 4)
    np.testing.assert_array_equal(a, b)
    rom.close()
