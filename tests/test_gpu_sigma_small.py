"""FP64 and double-FP32 sigma on both sides of the line between the gathered small-space
kernels and the tiled ones, against the oracle: empty and full spins (no moving
replacement, or none of the other kind), one beta string, columns that do not fill a
block, up to five vectors, and the largest number of orbitals with few strings of one
spin (all 136 integral pairs, alpha rows that do and do not fit in shared memory).

Tolerance as for the other FP64-class sigma tests: 1e-12 of the largest element
(FP64: ~1000 terms of 2^-53; double-FP32: ~2^-46 a term)."""
import numpy as np
import pytest

import oracle
import synth_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2405_10197_gb300 as fg  # noqa: E402

CASES = [(1, 1, 1, 1), (3, 0, 2, 2), (3, 3, 1, 1), (5, 5, 5, 1), (6, 2, 0, 5), (8, 7, 1, 3), (9, 4, 4, 2), (10, 5, 5, 1),
         (10, 3, 6, 2), (11, 5, 4, 1), (11, 2, 9, 3), (12, 3, 4, 1), (16, 1, 2, 2), (16, 3, 1, 1), (16, 2, 15, 1)]


@pytest.mark.parametrize("mode", [fg.FORTE_FP64, fg.FORTE_DF32])
@pytest.mark.parametrize("n,na,nb,nvec", CASES)
def test_sigma_matches_oracle(n, na, nb, nvec, mode):
    h, eri = si.integrals(n, 2 * n, seed=11 * n + na)
    prob = fg.CASProblem(n, na, nb, h, eri, precision=mode)
    try:
        C = si.random_vectors(nvec, prob.na, prob.nb, seed=2)
        S = prob.sigma(torch.tensor(C, device="cuda")).cpu().numpy().reshape(nvec, -1)
        rng = np.random.default_rng(n)
        rows = np.unique(np.concatenate([[0, prob.ndet - 1], rng.integers(0, prob.ndet, size=4000)]))
        ref = oracle.sigma(n, na, nb, h, eri, C.reshape(nvec, -1), rows=rows)
        for v in range(nvec):
            assert np.abs(S[v, rows] - ref[v]).max() <= 1e-12 * np.abs(S[v]).max()
    finally:
        prob.close()
