"""List sigma at the edges of its screen and queues against the oracle: list lengths
around a plane word (32), a warp's load (4096 determinants) and a block's rows (8);
every spin orbital position of a 64-bit word; words listed twice; lists that mix
electron counts down to the empty determinant (where the screen passes pairs that the
element rules refuse); complete small spaces, where a third of the pairs is connected;
one to six vectors.

Tolerance: a row sums at most ~2000 elements in another order than the oracle and both
are FP64: 2000 2^-53 of the sum of magnitudes in the worst case, held to 1e-12 of the
largest row as in the other list tests."""
import numpy as np
import pytest

import oracle
import synth_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2405_10197_gb300 as fg  # noqa: E402


def _check(n, words, nvec, seed):
    words = np.asarray(words, dtype=np.uint64)
    h, eri = si.integrals(n, 2 * n, seed=seed)
    C = np.random.default_rng(seed).normal(size=(nvec, len(words)))
    sci = fg.forte_sci_create(n, h, eri)
    try:
        Ct = torch.tensor(C, device="cuda")
        S = torch.full_like(Ct, np.nan)
        d = torch.tensor(words.view(np.int64), device="cuda")
        fg.forte_sci_sigma(sci, d, Ct, S, nvec)
        again = torch.empty_like(S)
        fg.forte_sci_sigma(sci, d, Ct, again, nvec)
        assert torch.equal(S, again)  # the order of the sums is fixed
        S = S.cpu().numpy()
    finally:
        fg.forte_sci_destroy(sci)
    ref = oracle.sci_sigma(n, words, h, eri, C)
    assert np.abs(S - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("count,nvec", [(1, 1), (7, 2), (8, 3), (31, 4), (32, 1), (33, 5), (129, 6), (4095, 1),
                                        (4096, 1), (4097, 2)])
def test_list_lengths(count, nvec):
    exc = si.excitation_list(16, 6, 5)
    rng = np.random.default_rng(count)
    _check(16, rng.choice(exc, size=count, replace=False), nvec, seed=count)


@pytest.mark.parametrize("n,na,nb", [(1, 1, 1), (2, 1, 1), (4, 2, 2), (5, 3, 2), (6, 3, 3)])
def test_complete_spaces(n, na, nb):
    A, B = oracle.strings(n, na), oracle.strings(n, nb)
    _check(n, oracle.det_words(n, np.repeat(A, len(B)), np.tile(B, len(A))), 2, seed=n)


def test_all_64_positions_and_full_words():
    # 32 orbitals; 31 + 31 and 32 + 32 electrons reach every bit of the word
    n = 32
    full = (1 << 64) - 1
    words = [full] + [full ^ (1 << p) ^ (1 << (n + q)) for p in range(0, 32) for q in (0, 1, 13, 31)]
    _check(n, words, 1, seed=5)


def test_mixed_electron_counts_and_repeated_words():
    n = 6
    rng = np.random.default_rng(3)
    words = np.concatenate([[0, 0, 1, 64, 65, 4095], rng.integers(0, 1 << 12, size=700), [65, 1]])
    _check(n, words, 3, seed=6)
