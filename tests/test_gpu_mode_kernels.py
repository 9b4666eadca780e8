"""The double-FP32 and digit-slice kernels on small spaces, where the modes take the FP64
kernels unless forte_set_small_route asks for their own: tile edges, padded rows, ragged
chunks, empty and full spins, the smallest and the largest number of integral pairs.  Every
test names the kernels that have to run and reads the trace to see that they did, so that
another size rule cannot leave these kernels untested.

Tolerances, those of the other tests of the same arithmetic: sigma 1e-12 of the largest
element (about 2^-45 a term), 2-RDM elements 1e-11 of a normalised vector (fixed point
2^-46 of a row's largest element), energies 1e-10 Eh at a residual of 1e-10."""
import numpy as np
import pytest

import oracle
import synth_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2405_10197_gb300 as fg  # noqa: E402

OZ_GRAM = {"gram_oz_u", "gram_oz_v", "oz_rowmax"}
FP64_KERNELS = {"ab_fp64", "ss_spmm", "gram"}


def _problem(n, na, nb, seed, mode):
    h, eri = si.integrals(n, 2 * n, seed=seed)
    prob = fg.CASProblem(n, na, nb, h, eri, precision=mode)
    fg.forte_set_small_route(prob.ctx, 0)
    return prob, h, eri


class _trace:
    """with _trace(prob, kernels): those kernels run and no FP64 one does."""

    def __init__(self, prob, kernels):
        self.ctx, self.kernels = prob.ctx, set(kernels)

    def __enter__(self):
        fg.forte_profile_enable(self.ctx, 1)

    def __exit__(self, kind, *_):
        names = set(fg.profile_table(self.ctx))
        fg.forte_profile_enable(self.ctx, 0)
        if kind is None:
            assert self.kernels <= names and not names & FP64_KERNELS, names


def _sigma_kernels(mode, n, na, nb):
    if na == 0 or nb == 0:
        return {"ss_spmm_df"}
    return {"ss_spmm_df", "ab_oz" if mode == fg.FORTE_OZ64 and n <= 15 else "ab_df"}


# n_kl from 0 to 39, one row or one column, 64-string tiles with ragged tails
SIGMA = [(1, 1, 1, 1), (2, 1, 1, 2), (3, 3, 1, 1), (4, 2, 2, 2), (5, 2, 3, 2), (5, 5, 5, 1), (5, 0, 2, 2), (6, 3, 3, 3),
         (6, 3, 0, 2), (6, 2, 6, 1), (7, 3, 2, 2), (8, 4, 4, 2), (8, 7, 1, 3), (9, 2, 5, 2), (15, 1, 2, 1), (16, 1, 1, 2),
         (16, 3, 1, 1), (16, 2, 15, 1)]


@pytest.mark.parametrize("mode", [fg.FORTE_DF32, fg.FORTE_OZ64])
@pytest.mark.parametrize("n,na,nb,nvec", SIGMA)
def test_sigma_matches_oracle(n, na, nb, nvec, mode):
    prob, h, eri = _problem(n, na, nb, 13 * n + na + 2 * nb, mode)
    try:
        C = si.random_vectors(nvec, prob.na, prob.nb, seed=4)
        with _trace(prob, _sigma_kernels(mode, n, na, nb)):
            S = prob.sigma(torch.tensor(C, device="cuda")).cpu().numpy()
        ref = oracle.sigma(n, na, nb, h, eri, C)
        for v in range(nvec):
            assert np.abs(S[v] - ref[v]).max() < 1e-12 * np.abs(ref[v]).max()
    finally:
        prob.close()


def _wide_range(na, nb, seed):
    rng = np.random.default_rng(seed)
    x = np.exp(rng.uniform(np.log(1e-14), 0.0, size=na * nb)) * rng.choice([-1.0, 1.0], size=na * nb)
    return torch.tensor((x / np.linalg.norm(x)).reshape(1, na, nb), device="cuda")


@pytest.mark.parametrize("mode", [fg.FORTE_DF32, fg.FORTE_OZ64])
def test_sigma_wide_dynamic_range_and_scaling(mode):
    """Entries from 1e-14 to 1, the vector scaled by 1e-7 and the zero vector."""
    prob, h, eri = _problem(8, 4, 4, 21, mode)
    try:
        C = _wide_range(prob.na, prob.nb, 4)
        ref = oracle.sigma(8, 4, 4, h, eri, C.cpu().numpy())
        with _trace(prob, _sigma_kernels(mode, 8, 4, 4)):
            S, Ss, Z = (prob.sigma(x).cpu().numpy() for x in (C, C * 1e-7, torch.zeros_like(C)))
        assert np.abs(S - ref).max() < 1e-12 * np.abs(ref).max()
        assert np.abs(Ss * 1e7 - ref).max() < 1e-12 * np.abs(ref).max()
        assert np.abs(Z).max() == 0.0
    finally:
        prob.close()


@pytest.mark.parametrize("mode", [fg.FORTE_DF32, fg.FORTE_OZ64])
def test_davidson_matches_dense(mode):
    cfg = si.CAS88
    h, eri = si.integrals(8, cfg["n_l"], cfg["seed"])
    w, _ = oracle.solve_dense(8, 4, 4, h, eri, nroots=3)
    prob = fg.CASProblem(8, 4, 4, h, eri, precision=mode)
    try:
        fg.forte_set_small_route(prob.ctx, 0)
        with _trace(prob, _sigma_kernels(mode, 8, 4, 4)):
            E, _, rn, _ = prob.davidson(nroots=3, tol=1e-10)
        assert np.all(rn < 1e-10)
        assert np.abs(E - w).max() < 1e-10
    finally:
        prob.close()


# every padded row count of the Gram kernel: 16 .. 112 symmetric, 16 .. 96 antisymmetric rows
RDMS = [(2, 1, 1), (3, 1, 2), (4, 2, 2), (5, 2, 3), (6, 3, 3), (6, 3, 0), (6, 0, 2), (7, 3, 2), (8, 4, 4), (9, 2, 5),
        (10, 3, 3), (11, 3, 3), (12, 2, 3), (13, 2, 2), (14, 2, 3), (15, 1, 2)]


@pytest.mark.parametrize("mode", [fg.FORTE_BF16X2, fg.FORTE_TF32, fg.FORTE_OZ64, fg.FORTE_DF32])
@pytest.mark.parametrize("n,na,nb", RDMS)
def test_rdms_match_oracle(n, na, nb, mode):
    prob, _, _ = _problem(n, na, nb, 60 + n, mode)
    try:
        c = si.random_vectors(1, prob.na, prob.nb, seed=n)[0]
        c /= np.linalg.norm(c)
        with _trace(prob, OZ_GRAM):
            g1, g2 = prob.rdms(torch.tensor(c, device="cuda"))
        r1, r2 = oracle.rdm12(n, na, nb, c.reshape(-1))
        assert np.abs(g1.cpu().numpy() - r1).max() < 1e-12
        assert np.abs(g2.cpu().numpy() - r2).max() < 1e-11
    finally:
        prob.close()


@pytest.mark.parametrize("n,na,nb", [(6, 3, 3), (8, 3, 4)])
def test_rdms_wide_dynamic_range_and_scaling(n, na, nb):
    prob, _, _ = _problem(n, na, nb, 7, fg.FORTE_BF16X2)
    try:
        C = _wide_range(prob.na, prob.nb, n)[0]
        _, r2 = oracle.rdm12(n, na, nb, C.cpu().numpy().reshape(-1))
        with _trace(prob, OZ_GRAM):
            g2, g2s, g2z = (prob.rdms(x)[1].cpu().numpy() for x in (C, C * 1e-7, torch.zeros_like(C)))
        assert np.abs(g2 - r2).max() < 1e-11
        assert np.abs(g2s * 1e14 - g2).max() < 1e-11
        assert np.abs(g2z).max() == 0.0
    finally:
        prob.close()


def test_state_averaged_gradient_takes_the_tensor_core_gram():
    n, na, nb = 8, 4, 4
    prob, h, eri = _problem(n, na, nb, 12, fg.FORTE_BF16X2)
    try:
        _, V = oracle.solve_dense(n, na, nb, h, eri, nroots=2)
        C = torch.tensor(V.reshape(2, prob.na, prob.nb), device="cuda")
        dh = torch.zeros(n, n, dtype=torch.float64, device="cuda")
        de = torch.zeros((n,) * 4, dtype=torch.float64, device="cuda")
        with _trace(prob, OZ_GRAM):
            fg.forte_sa_gradient(prob.ctx, 2, np.array([0.5, 0.5]), C, 1.0, dh, de, n)
        r = [oracle.rdm12(n, na, nb, V[k].reshape(-1)) for k in range(2)]
        assert np.abs(dh.cpu().numpy() - 0.5 * (r[0][0] + r[1][0])).max() < 1e-12
        assert np.abs(de.cpu().numpy() - 0.25 * (r[0][1] + r[1][1])).max() < 1e-11
    finally:
        prob.close()


@pytest.mark.parametrize("mode,call", [(fg.FORTE_OZ64, "sigma"), (fg.FORTE_BF16X2, "rdms")])
def test_context_computes_again_after_expired_waits(mode, call):
    """A budget of a few cycles makes the waits expire; with the default one the same
    kernels of the same context give the right result."""
    n, na, nb = 8, 4, 4
    prob, h, eri = _problem(n, na, nb, 31, mode)
    try:
        c = si.random_vectors(1, prob.na, prob.nb, seed=8)
        c /= np.linalg.norm(c)
        C = torch.tensor(c, device="cuda")
        fg.forte_set_wait_budget(prob.ctx, 4)
        if call == "sigma":
            prob.sigma(C)
            assert fg.forte_get_status(prob.ctx, allow=(fg.FORTE_ERR_TIMEOUT,)) == fg.FORTE_ERR_TIMEOUT
        else:
            with pytest.raises(fg.ForteError) as ex:
                prob.rdms(C[0])
            assert ex.value.code == fg.FORTE_ERR_TIMEOUT
        fg.forte_set_wait_budget(prob.ctx, 0)
        if call == "sigma":
            with _trace(prob, {"ab_oz"}):
                out = prob.sigma(C).cpu().numpy()
            ref = oracle.sigma(n, na, nb, h, eri, c)
            tol = 1e-12 * np.abs(ref).max()
        else:
            with _trace(prob, OZ_GRAM):
                out = prob.rdms(C[0])[1].cpu().numpy()
            ref, tol = oracle.rdm12(n, na, nb, c.reshape(-1))[1], 1e-11
        assert fg.forte_get_status(prob.ctx) == fg.FORTE_OK
        assert np.abs(out - ref).max() < tol
    finally:
        prob.close()


@pytest.mark.parametrize("route,budget,own", [(-1, 0, False), (0, 0, True), (1, 0, False), (1, 4000000000, False)])
def test_route_selects_the_kernels(route, budget, own):
    prob, _, _ = _problem(8, 4, 4, 3, fg.FORTE_OZ64)
    try:
        fg.forte_set_small_route(prob.ctx, route)
        fg.forte_set_wait_budget(prob.ctx, budget)
        C = torch.tensor(si.random_vectors(1, prob.na, prob.nb, seed=1), device="cuda")
        fg.forte_profile_enable(prob.ctx, 1)
        prob.sigma(C)
        prob.rdms(C[0])
        names = set(fg.profile_table(prob.ctx))
        assert ("ab_oz" in names) == own and ("gram_oz_u" in names) == own
        assert ("ab_fp64" in names) != own and ("gram" in names) != own
        with pytest.raises(fg.ForteError):
            fg.forte_set_small_route(prob.ctx, 2)
    finally:
        prob.close()
