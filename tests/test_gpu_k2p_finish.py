"""K2P's finish kernel on both sides of its rule (a warp per test index below
two blocks an SM, eight warps a block above), against the FP64 oracle on the
stored BF16 values: exact up to the 2^-17 hi/lo split of the states and FP32
sums, so 2^-14 of A_i = sum_jk |C_ijk| |u_j| |u_k| bounds each entry."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
import paper_2311_03694_gb300 as grom  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch", [(49, 94), (161, 96), (161, 1000)])
def test_finish_matches_oracle(n, batch):
    grom.build()
    C = synth.skew_normal_tensor(n, 77 + n)
    Cr = torch.from_numpy(C).to(torch.bfloat16).to(torch.float64).numpy()
    U = synth.initial_condition(n, 78 + n, 0, batch)
    rom = grom.Rom(n, "full", "bf16", tensor=C, stiffness=synth.diag_stiffness(n), max_batch=batch,
                   layout="skew_packed")
    rom.set_kernel("tensor")
    u = torch.from_numpy(U).cuda()
    c = torch.full_like(u, float("nan"))
    rom.nonlinear(u, c)
    torch.cuda.synchronize()
    c = c.cpu().numpy()
    assert np.all(np.isfinite(c))
    for b in (0, 31, 32, batch // 2, batch - 1):
        A = np.einsum("ijk,j,k->i", np.abs(Cr), np.abs(U[b]), np.abs(U[b]))
        assert np.all(np.abs(c[b] - oracle.nonlinear_full(Cr, U[b])) <= 2.0 ** -14 * A), (n, batch, b)
    rom.close()
