"""K3O's error where a tile's contracted index is split most: the sums over the
splits must not add to what a double-single value rounds off by itself, 2^-48,
which bounds the median error of an evaluation (against long double, the oracle's
64 bits being too short to judge it)."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
import paper_2311_03694_gb300 as grom  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form,n,r,batch", [("cp_skew", 1024, 512, 64), ("cp_skew", 512, 256, 200), ("cp", 1000, 900, 40)])
def test_median_error_of_an_evaluation(form, n, r, batch):
    grom.build()
    d = 1.0 / (np.arange(1, r + 1) * r ** 0.5)
    F = [synth.normal(40 + n, 30 + q, 0, n * r).reshape(n, r) * d for q in range(3)]
    U = synth.initial_condition(n, 41 + n, 0, batch)
    rom = grom.Rom(n, form, "f64", factors=F, stiffness=synth.diag_stiffness(n), max_batch=batch)
    rom.set_kernel("tensor")
    u = torch.from_numpy(U).cuda()
    c = torch.empty_like(u)
    rom.nonlinear(u, c)
    c = c.cpu().numpy().astype(np.longdouble)
    rom.close()
    A, B, C = (f.astype(np.longdouble) for f in F)
    v = U[:32].astype(np.longdouble)
    mm = lambda x, y: np.einsum("ij,jk->ik", x, y)  # noqa: E731 (no BLAS for long double)
    p = mm(v, B)
    want = mm(p * mm(v, C), A.T)
    if form == "cp_skew":
        want = want - mm(p * mm(v, A), C.T)
    err = np.sqrt(np.sum((c[:32] - want) ** 2, axis=1)) / np.sqrt(np.sum(want ** 2, axis=1))
    assert np.median(err) <= 2.0 ** -48, float(np.median(err))
