"""Davidson solves whose vectors take the short-vector kernels (up to 77,824 elements, any
count and alignment) against dense or stored energies: odd vector lengths, lengths
below, at and above one block's 128 elements, bases above the 16 columns that are
reduced at a time (several roots), FP64 and FP32 vectors.

Tolerance: the solver's own contract, 1e-10 Eh at a residual of 1e-10, and the residual
of the returned vectors recomputed in numpy from the dense Hamiltonian."""
import numpy as np
import pytest

import oracle
import synth_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2405_10197_gb300 as fg  # noqa: E402


@pytest.mark.parametrize("mode", [fg.FORTE_FP64, fg.FORTE_BF16X2])
@pytest.mark.parametrize("n,na,nb,nroots", [(5, 1, 1, 1), (5, 2, 1, 2), (7, 3, 1, 1), (7, 2, 2, 3), (6, 3, 3, 5), (7, 3, 3, 2)])
def test_solve_matches_dense(n, na, nb, nroots, mode):
    h, eri = si.integrals(n, 2 * n, seed=91 + n + na)
    w, V = oracle.solve_dense(n, na, nb, h, eri, nroots=nroots)
    prob = fg.CASProblem(n, na, nb, h, eri, precision=mode)
    try:
        fg.forte_set_davidson_params(prob.ctx, 12, 2, 1000, 1e-8)
        E, C, rn, it = prob.davidson(nroots=nroots, tol=1e-10)
        assert np.abs(E - w).max() < 1e-10
        X = C.cpu().numpy().reshape(nroots, -1)
        S = oracle.sigma(n, na, nb, h, eri, X)
        assert np.linalg.norm(S - E[:, None] * X, axis=1).max() < 1.1e-10
        assert np.abs(X @ X.T - np.eye(nroots)).max() < 1e-11
    finally:
        prob.close()
