"""Mixed-precision solves whose reduced-precision inner operator cannot resolve the
corrections: one integral of 1e5 Eh beside the ordinary ones makes its error as large as the
gaps, so that the residuals stop halving and the inner solves have to take the FP64-class
sigma.  The solve has to converge all the same.

Tolerances: the residual asked for; energies 1e-8 Eh, some 1e2 roundings of the largest
diagonal elements (a few 1e5 Eh, 2^-53 each)."""
import numpy as np
import pytest

import oracle
import synth_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2405_10197_gb300 as fg  # noqa: E402


def _integrals(n, seed, size=1e5):
    h, eri = si.integrals(n, 2 * n, seed=3 + seed)
    rng = np.random.default_rng(seed)
    v = np.zeros((n, n))
    v[0, 0], v[1, 1] = 1.0, rng.uniform(0.2, 1.0)
    v[0, 1] = v[1, 0] = rng.uniform(0.0, 0.8)
    return h, eri + size * np.einsum("pq,rs->pqrs", v, v)


TF, BF = fg.FORTE_TF32, fg.FORTE_BF16X2
CASES = [(TF, 0, 6, 3, 3, 3), (BF, 0, 6, 3, 3, 3), (TF, 1, 6, 3, 3, 3), (BF, 1, 7, 3, 4, 2), (BF, 1, 8, 4, 4, 3),
         (TF, 4, 6, 3, 3, 3)]


@pytest.mark.parametrize("mode,seed,n,na,nb,nroots", CASES)
def test_solve_converges_with_the_outer_operator(mode, seed, n, na, nb, nroots):
    h, eri = _integrals(n, seed)
    w, _ = oracle.solve_dense(n, na, nb, h, eri, nroots=nroots)
    prob = fg.CASProblem(n, na, nb, h, eri, precision=mode)
    try:
        fg.forte_set_davidson_params(prob.ctx, 12, 2, 400, 1e-8)
        E, _, rn, _ = prob.davidson(nroots=nroots, tol=1e-9)
        assert np.all(rn < 1e-9)
        assert np.abs(E - w).max() < 1e-8
        # outer steps alone take at most 33 FP64-class sigmas a root
        assert fg.forte_get_counters(prob.ctx)[0] > 33 * nroots
    finally:
        prob.close()
