"""Kept-determinant sigma (forte_set_gas_route 1) where its class lists can go wrong: a
single space (one class: everything allowed), one orbital per space (a class per string,
up to 20 classes of one string), limits that leave rows without an unmoved or without
a moved source, an empty spin, classes of more strings than a tile, FP32 vectors through
a mixed solve.

Tolerances as in the other restricted-sigma tests: 1e-12 of the largest element; energies
1e-9 Eh against the dense restricted problem."""
import numpy as np
import pytest

import oracle
import synth_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2405_10197_gb300 as fg  # noqa: E402

SETS = [
    (5, 2, 2, (5,), (0,), (10,)),
    (6, 3, 3, (1, 1, 1, 1, 1, 1), (0,) * 6, (2, 2, 2, 1, 1, 1)),
    (7, 2, 4, (2, 5), (1, 0), (3, 9)),
    (7, 3, 0, (3, 4), (1, 0), (2, 8)),
    (8, 3, 5, (2, 4, 2), (3, 0, 0), (4, 8, 1)),
    (11, 5, 4, (2, 7, 2), (3, 0, 0), (4, 14, 1)),
]


@pytest.mark.parametrize("n,na,nb,spaces,gmin,gmax", SETS)
def test_kept_sigma_matches_oracle(n, na, nb, spaces, gmin, gmax):
    h, eri = si.integrals(n, 2 * n, seed=17 + n)
    prob = fg.CASProblem(n, na, nb, h, eri)
    try:
        prob.set_gas(spaces, gmin, gmax)
        fg.forte_set_gas_route(prob.ctx, 1)
        C = si.random_vectors(2, prob.na, prob.nb, seed=n)
        S = prob.sigma(torch.tensor(C, device="cuda")).cpu().numpy()
        ref = oracle.sigma_gas(n, na, nb, h, eri, C, spaces, gmin, gmax)
        assert np.abs(S - ref).max() < 1e-12 * np.abs(ref).max()
    finally:
        prob.close()


def test_fp32_route_of_a_mixed_solve():
    n, na, nb, spaces, gmin, gmax = 8, 4, 4, (3, 2, 3), (5, 0, 0), (6, 4, 1)
    h, eri = si.integrals(n, 2 * n, seed=2)
    prob = fg.CASProblem(n, na, nb, h, eri, precision=fg.FORTE_BF16X2)
    try:
        prob.set_gas(spaces, gmin, gmax)
        fg.forte_set_gas_route(prob.ctx, 1)
        E, _, rn, _ = prob.davidson(nroots=1, tol=1e-9)
        w, _ = oracle.solve_dense_gas(n, na, nb, h, eri, spaces, gmin, gmax, nroots=1)
        assert rn[0] < 1e-9 and abs(E[0] - w[0]) < 1e-9
    finally:
        prob.close()
