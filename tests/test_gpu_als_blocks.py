"""CP fitting's FP64 solves at the edges of their 32-wide blocks and 16-wide
Gram tiles, against the oracle (1e-4, the MTTKRP's precision on BF16-exact
tensors), and under scaling of the factors by powers of two, which every step
of the solves carries exactly (even exponents in H)."""
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


def _problem(n, r):
    # multiples of 1/64 of at most 8 significant bits: exact in BF16
    z = synth.normal(500 + r, 13, 0, n ** 3).reshape(n, n, n)
    X = np.clip(np.round(z * 64.0), -255, 255) / 64.0
    return X, [synth.normal(600 + r, 20 + q, 0, n * r).reshape(n, r) for q in range(3)]


@pytest.mark.parametrize("n,r", [(20, 1), (33, 15), (21, 31), (30, 33), (47, 64), (40, 97), (26, 161)])
def test_one_iteration_at_block_edges(n, r):
    X, F0 = _problem(n, r)
    als = grom.Als(X)
    F, res = als.fit(F0, 1)
    Fo, reso = oracle.cp_als(X, F0, 1)
    als.close()
    for q in range(3):
        assert np.linalg.norm(F[q] - Fo[q]) <= 1e-4 * np.linalg.norm(Fo[q]), (n, r, q)
    assert res[0] == pytest.approx(reso[0], rel=1e-4)


def test_powers_of_two_pass_through_the_solves():
    n, r = 30, 70
    X, F0 = _problem(n, r)
    als = grom.Als(X)
    F, _ = als.fit(F0, 1)
    G, _ = als.fit([F0[0], F0[1] * 2.0 ** 20, F0[2] * 2.0 ** 20], 1)
    als.close()
    for q, e in enumerate((-40, 20, 20)):
        np.testing.assert_array_equal(G[q], F[q] * 2.0 ** e)
