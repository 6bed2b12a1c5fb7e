"""K3O's level-by-level slice products (k3_tri.cu) at the edges of their column
tiles and summed ranges, and the one-product-per-pair form that N > 1024 keeps,
against the FP64 oracle within the FP64 tolerance (1e-12)."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
import paper_2311_03694_gb300 as grom  # noqa: E402

pytestmark = pytest.mark.gpu


def _factors(form, n, r, seed):
    if form == "cp_skew":
        U, V, W, _, _ = synth.cp_workload(n, r, 1)
        return (U, V, W), lambda u: oracle.nonlinear_cp_skew(U, V, W, u)
    rng = np.random.default_rng(seed)
    A, B, C = (rng.standard_normal((n, r)) / np.sqrt(r) for _ in range(3))
    return (A, B, C), lambda u: oracle.nonlinear_cp(A, B, C, u)


@pytest.mark.parametrize("form", ["cp_skew", "cp"])
@pytest.mark.parametrize("n,r,batch", [(64, 130, 64), (129, 64, 65), (400, 449, 16), (1024, 40, 33), (100, 1500, 16), (1030, 40, 16)])
def test_k3o_level_products_at_tile_edges(form, n, r, batch):
    # one and several column tiles, summed ranges of one to six steps a CTA,
    # with a shorter last one and over many CTAs (rank 1500: 47 steps, skew)
    grom.build()
    fac, ref = _factors(form, n, r, 900 + n)
    rom = grom.Rom(n, form, "f64", factors=fac, stiffness=synth.diag_stiffness(n), max_batch=batch)
    rom.set_kernel("tensor")
    U = synth.initial_condition(n, 31 + n, 0, batch)
    u = torch.from_numpy(U).cuda()
    c = torch.full_like(u, float("nan"))
    rom.nonlinear(u, c)
    torch.cuda.synchronize()
    got = c.cpu().numpy()
    for b in (0, batch // 2, batch - 1):
        want = ref(U[b])
        assert np.linalg.norm(got[b] - want) <= 1e-12 * np.linalg.norm(want), (n, r, b)
    rom.close()


@pytest.mark.parametrize("form,n,r,batch,tensor", [
    ("cp_skew", 1024, 512, 16, True), ("cp", 1024, 512, 16, True),     # N R = 2^19 from 2^23 on
    ("cp_skew", 1024, 448, 16, False), ("cp", 1024, 448, 16, False),   # below it: double-single
    ("cp_skew", 128, 128, 768, True), ("cp", 128, 128, 768, False),    # 3 2^22
])
def test_k3o_rule_takes_the_path_it_states(form, n, r, batch, tensor):
    # the default choice gives the bits of the path that its rule names, at FP64 tolerance
    grom.build()
    fac, ref = _factors(form, n, r, 77)
    U = synth.initial_condition(n, 5, 0, batch)
    rom = grom.Rom(n, form, "f64", factors=fac, stiffness=synth.diag_stiffness(n), max_batch=batch)
    u = torch.from_numpy(U).cuda()
    got = []
    for kernel in ("auto", "tensor"):
        rom.set_kernel(kernel)
        c = torch.empty_like(u)
        rom.nonlinear(u, c)
        torch.cuda.synchronize()
        got.append(c.cpu().numpy())
    rom.close()
    assert np.array_equal(got[0], got[1]) == tensor
    for b in (0, batch - 1):
        want = ref(U[b])
        for c in got:
            assert np.linalg.norm(c[b] - want) <= 1e-12 * np.linalg.norm(want), b
