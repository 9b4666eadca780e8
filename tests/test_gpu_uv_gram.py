"""FP64 2- and 3-RDM from the Grams of the symmetric and antisymmetric one-body images
against the oracle, at the sizes where the tiling can go wrong: one orbital (no
antisymmetric pair), pair counts around multiples of the 3 x 3 tile, fewer
determinants than a 32-determinant slab, the last slab partly filled, several tile
groups per slab (n = 10 and up), the largest number of orbitals, an empty spin.

Tolerance: an image element is a sum of two entries of C, so the products of an RDM
element add up to at most 4 |C|^2 = 4 in magnitude (2-RDM; 8 for the 3-RDM, whose ket
is an image of an image) and a sum of N_det of them in any order is off by at most
N_det 2^-53 times that; the lower-rank terms add a few 2^-53 of numbers below N^2.
With N_det <= 1600 the worst case is 1e-12; rounding errors do not all add up."""
import numpy as np
import pytest

import oracle
import synth_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2405_10197_gb300 as fg  # noqa: E402

TOL = 1e-12


def _state(n, na, nb, seed):
    h, eri = si.integrals(n, 2 * n, seed=seed)
    prob = fg.CASProblem(n, na, nb, h, eri)
    C = si.random_vectors(1, prob.na, prob.nb, seed=seed)[0]
    return prob, C


@pytest.mark.parametrize("n,na,nb", [(1, 1, 0), (1, 1, 1), (2, 1, 1), (3, 1, 2), (4, 2, 2), (5, 3, 2), (6, 6, 1), (7, 0, 3),
                                     (8, 2, 3), (10, 1, 2), (13, 1, 1), (16, 1, 1), (16, 2, 0)])
def test_rdm12_small_and_ragged(n, na, nb):
    prob, C = _state(n, na, nb, 3 * n + na)
    try:
        r1, r2 = oracle.rdm12(n, na, nb, C.reshape(-1))
        g1, g2 = prob.rdms(torch.tensor(C, device="cuda"))
        assert np.abs(g1.cpu().numpy() - r1).max() < TOL
        assert np.abs(g2.cpu().numpy() - r2).max() < TOL
    finally:
        prob.close()


@pytest.mark.parametrize("n,na,nb", [(1, 1, 1), (2, 2, 1), (3, 2, 1), (4, 2, 2), (5, 1, 3), (6, 2, 2), (7, 2, 1), (10, 1, 1)])
def test_rdm3_small_and_ragged(n, na, nb):
    prob, C = _state(n, na, nb, 5 * n + nb)
    try:
        g3 = prob.rdm3(torch.tensor(C, device="cuda")).cpu().numpy()
        assert np.abs(g3 - oracle.rdm3(n, na, nb, C.reshape(-1))).max() < TOL
    finally:
        prob.close()


def test_tdm1_of_two_states_is_not_symmetrised():
    prob, C = _state(6, 3, 2, 4)
    D = si.random_vectors(1, prob.na, prob.nb, seed=9)[0]
    try:
        t = prob.tdm1(torch.tensor(C, device="cuda"), torch.tensor(D, device="cuda")).cpu().numpy()
        assert np.abs(t - oracle.rdm12(6, 3, 2, C.reshape(-1), D.reshape(-1), two=False)[0]).max() < TOL
    finally:
        prob.close()
