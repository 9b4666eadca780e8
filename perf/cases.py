"""Performance cases of the CASCI engine: what a user's program has it do, timed call by call.

Every case is one kind of call through the public entry points, at a size this repository's
configurations and benchmark name (CAS(8,8), CAS(12,12), CAS(14,14), the RAS(2h,2p) restriction,
determinant lists of 30 orbitals, batches of small half-filled spaces) or one between them:

  sigma     sigma = H C for given CI vectors (the inner call of a user's own eigensolver)
  gas       the same under an occupation restriction (RAS)
  list      sigma over a list of determinants (selected CI)
  solve     Davidson solve to the default residual 1e-10 of an existing problem, and the RDMs of its
            lowest root where the program asks for them
  rdms      1- and 2-RDM of a given CI vector
  rdm3      3-RDM of a given CI vector
  grad      state-averaged energy and its gradient with respect to the integrals (forward and backward),
            from the integrals on
  batch     many independent small problems, from the integrals on

Integrals: h diagonal -1 + 0.25 p, off-diagonal N(0, 0.05^2); (pq|rs) = sum_L B^L_pq B^L_rs with
2 n symmetric factors of N(0, 0.15^2).  CI vectors: N(0,1) amplitudes divided by 1 + (H_II - min H_II),
the decay a first-order wave function has, normalised.
"""
import math

import numpy as np
import torch

import paper_2405_10197_gb300 as fg

MODES = {"fp64": fg.FORTE_FP64, "tf32": fg.FORTE_TF32, "bf16x2": fg.FORTE_BF16X2, "df32": fg.FORTE_DF32,
         "oz64": fg.FORTE_OZ64}


def _cas(kind, mode, n, na, nb, **more):
    return dict(kind=kind, mode=mode, norb=n, nalpha=na, nbeta=nb, **more)


def listed():
    return [
        # The smallest call: one vector of a small space in the default precision; launches and latency.
        dict(name="sigma_fp64_cas8", **_cas("sigma", "fp64", 8, 4, 4, nvec=1)),
        # An ordinary call: a block of four vectors of CAS(12,12) in the default precision.
        dict(name="sigma_fp64_cas12", **_cas("sigma", "fp64", 12, 6, 6, nvec=4)),
        # The largest space in the FP64-class arithmetic for GPUs with little FP64.
        dict(name="sigma_oz64_cas14", **_cas("sigma", "oz64", 14, 7, 7, nvec=1)),
        # An open shell with unequal, odd string counts (1716 x 1287) in double-FP32.
        dict(name="sigma_df32_cas13", **_cas("sigma", "df32", 13, 7, 5, nvec=1)),
        # RAS with up to two holes and two particles in CAS(14,14): 3 % of the determinants.
        dict(name="gas_fp64_cas14", **_cas("gas", "fp64", 14, 7, 7, nvec=1, ras1=4, ras3=4, holes=2, particles=2)),
        # A selected-CI list of the size adaptive CI ends with, beyond what a CAS grid holds.
        dict(name="list_30o", kind="list", norb=30, nalpha=10, nbeta=10, ndet=50001, nvec=1),
        # Solving a small space: some 150 short iterations.
        dict(name="solve_fp64_cas8", **_cas("solve", "fp64", 8, 4, 4, nroots=1, rdms=False)),
        # The flagship: ground state of CAS(14,14) in mixed precision, then its 1- and 2-RDM.
        dict(name="solve_bf16x2_cas14", **_cas("solve", "bf16x2", 14, 7, 7, nroots=1, rdms=True)),
        # RDMs of an open-shell state in the default precision.
        dict(name="rdms_fp64_cas12", **_cas("rdms", "fp64", 12, 7, 5)),
        # The 3-RDM a perturbative treatment on top of a CASCI asks for.
        dict(name="rdm3_fp64_cas9", **_cas("rdm3", "fp64", 9, 5, 4)),
        # State-averaged energy of three roots and its gradient: one step of an orbital optimisation.
        dict(name="grad_bf16x2_cas12", **_cas("grad", "bf16x2", 12, 6, 6, nroots=3)),
        # A batch of uneven small problems in the default precision.
        dict(name="batch_fp64", kind="batch", mode="fp64", count=24, norb=6, norb_max=8),
    ]


def _draw_occ(rng, n):
    """Electron counts around half filling, the spins not always alike."""
    lo, hi = max(1, n // 2 - 1), min(n - 1, n // 2 + 1)
    return rng.randint(lo, hi), rng.randint(lo, hi)


def draw(rng):
    kind = rng.choice(["sigma", "sigma", "gas", "list", "solve", "solve", "rdms", "rdm3", "grad", "batch"])
    if kind == "list":
        n = rng.randint(16, 32)
        e = rng.randint(4, 10)
        return dict(kind=kind, norb=n, nalpha=e, nbeta=max(3, e - rng.randint(0, 2)),
                    ndet=int(round(math.exp(rng.uniform(math.log(300), math.log(50000))))), nvec=rng.randint(1, 4))
    if kind == "batch":
        mode, hi = rng.choice(["fp64", "bf16x2"]), rng.randint(5, 7)
        return dict(kind=kind, mode=mode, count=rng.randint(6, 32), norb=hi if mode == "bf16x2" else rng.randint(4, hi - 1),
                    norb_max=hi)
    mode = {"sigma": ["fp64", "df32", "oz64"], "gas": ["fp64", "oz64"], "solve": ["fp64", "oz64", "bf16x2", "tf32"],
            "rdms": ["fp64", "bf16x2", "oz64"], "rdm3": ["fp64"], "grad": ["bf16x2", "tf32"]}[kind]
    mode = rng.choice(mode)
    top = {"sigma": {"fp64": 13, "df32": 14, "oz64": 14}, "gas": {"fp64": 14, "oz64": 14},
           "solve": {"fp64": 10, "oz64": 10, "bf16x2": 13, "tf32": 13},
           "rdms": {"fp64": 12, "bf16x2": 14, "oz64": 14}, "rdm3": {"fp64": 9}, "grad": {"bf16x2": 11, "tf32": 11}}
    low = {"sigma": 4, "gas": 10, "solve": 5, "rdms": 4, "rdm3": 4, "grad": 5}[kind]
    n = rng.randint(low, top[kind][mode])
    na, nb = _draw_occ(rng, n)
    case = _cas(kind, mode, n, na, nb)
    if kind in ("sigma", "gas"):
        case["nvec"] = rng.randint(1, 5 if math.comb(n, na) * math.comb(n, nb) < 500000 else 2)
    if kind == "gas":
        case.update(ras1=n // 3 - rng.randint(0, 1), ras3=n // 3 - rng.randint(0, 1), holes=rng.randint(1, 2),
                    particles=rng.randint(1, 2))
    if kind == "solve":
        case.update(nroots=1, rdms=rng.random() < 0.5)
    if kind == "grad":
        case["nroots"] = rng.randint(1, 3)
    return case


# ------------------------------------------------------------------------------------------ inputs

def _integrals(n, rng):
    h = np.zeros((n, n))
    iu = np.triu_indices(n, 1)
    h[iu] = rng.normal(0.0, 0.05, len(iu[0]))
    h = h + h.T + np.diag(-1.0 + 0.25 * np.arange(n))
    B = rng.normal(0.0, 0.15, (2 * n, n, n))
    B = np.triu(B) + np.triu(B, 1).transpose(0, 2, 1)
    B = B.reshape(2 * n, n * n)
    eri = (B.T @ B).reshape(n, n, n, n)
    # every permutation of an integral the same number, as integral files have it
    pair = np.arange(n * n).reshape(n, n)
    pair = np.minimum(pair, pair.T).reshape(-1)
    eri = eri.reshape(n * n, n * n)[pair][:, pair]
    eri = np.triu(eri) + np.triu(eri, 1).T
    return np.ascontiguousarray(h), np.ascontiguousarray(eri.reshape(n, n, n, n))


def _problem(case, rng):
    h, eri = _integrals(case["norb"], rng)
    prob = fg.CASProblem(case["norb"], case["nalpha"], case["nbeta"], h, eri, precision=MODES[case["mode"]])
    return prob, h, eri


def _vectors(hdiag, nvec, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    fin = torch.isfinite(hdiag)
    low = hdiag[fin].min()
    wt = torch.where(fin, 1.0 / (1.0 + hdiag - low), torch.zeros_like(hdiag))
    C = torch.randn((nvec,) + tuple(hdiag.shape), generator=g, device="cuda", dtype=torch.float64) * wt
    return C / C.reshape(nvec, -1).norm(dim=1).reshape(nvec, 1, 1)


def _ras(case):
    """Spaces and electron limits of a RAS restriction: the holes and particles counted from the aufbau filling."""
    n, e = case["norb"], case["nalpha"] + case["nbeta"]
    sizes = [case["ras1"], n - case["ras1"] - case["ras3"], case["ras3"]]
    most = min(e, 2 * sizes[0])
    return sizes, [max(0, most - case["holes"]), 0, 0], [2 * sizes[0], 2 * sizes[1], case["particles"]]


def _excite(words, n, rng, spin):
    """One random replacement within a spin for every word."""
    bits = ((words[:, None] >> (np.arange(n, dtype=np.uint64) + np.uint64(spin * n))[None, :]) & np.uint64(1)).astype(bool)
    r = rng.random(bits.shape)
    hole = np.argmax(np.where(bits, r, -1.0), axis=1).astype(np.uint64) + np.uint64(spin * n)
    part = np.argmax(np.where(bits, -1.0, r), axis=1).astype(np.uint64) + np.uint64(spin * n)
    return (words & ~(np.uint64(1) << hole)) | (np.uint64(1) << part)


def _det_list(n, na, nb, count, rng):
    """Distinct determinants of one to four replacements from the aufbau determinant, ascending: doubles of the
    reference and, from those, what a few more rounds of selection add."""
    ref = ((1 << na) - 1) | (((1 << nb) - 1) << n)
    have = np.array([ref], dtype=np.uint64)
    while True:
        base = rng.choice(have[: max(1, len(have) // 2)], size=2 * count) if len(have) < count // 2 else rng.choice(have, size=count)
        base[: len(base) // 2] = ref
        one = _excite(base, n, rng, 0)
        two = np.where(rng.random(len(base)) < 0.5, _excite(one, n, rng, 1), _excite(one, n, rng, 0))
        flip = rng.random(len(base)) < 0.25
        two = np.where(flip, np.where(rng.random(len(base)) < 0.5, _excite(base, n, rng, 1), _excite(_excite(base, n, rng, 1), n, rng, 1)), two)
        have = np.unique(np.concatenate([have, two]))
        if len(have) >= count:
            keep = rng.choice(len(have), size=count, replace=False)
            return np.sort(have[keep])


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    st = {"case": case}
    if kind == "batch":
        st["problems"] = []
        for i in range(case["count"]):
            n = case["norb"] + i % (case["norb_max"] + 1 - case["norb"])
            h, eri = _integrals(n, rng)
            st["problems"].append(dict(norb=n, nalpha=(n + 1) // 2, nbeta=n // 2, nroots=1 + i % 2, h=h, eri=eri))
        return st
    if kind == "list":
        n = case["norb"]
        h, eri = _integrals(n, rng)
        st["sci"] = _List(n, h, eri)
        st["dets"] = torch.from_numpy(_det_list(n, case["nalpha"], case["nbeta"], case["ndet"], rng).view(np.int64)).cuda()
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        C = torch.randn(case["nvec"], case["ndet"], generator=g, device="cuda", dtype=torch.float64)
        st["C"] = C / C.norm(dim=1, keepdim=True)
        st["h"], st["eri"] = h, eri
        return st
    if kind == "grad":
        h, eri = _integrals(case["norb"], rng)
        st["h"] = torch.from_numpy(h).cuda().requires_grad_(True)
        st["eri"] = torch.from_numpy(eri).cuda().requires_grad_(True)
        return st
    prob, st["h"], st["eri"] = _problem(case, rng)
    st["prob"] = prob
    if kind == "gas":
        prob.set_gas(*_ras(case))
    if kind == "solve":
        fg.forte_set_davidson_params(prob.ctx, 12, 2, 1000, 1e-8)
    else:
        st["C"] = _vectors(prob.hdiag(), case.get("nvec", 1), seed)
    return st


class _List:
    """A determinant-list handle that is given back with its last user."""

    def __init__(self, n, h, eri):
        self.sci = fg.forte_sci_create(n, h, eri)

    def __del__(self):
        fg.forte_sci_destroy(self.sci)


# ------------------------------------------------------------------------------------------ the calls

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("sigma", "gas"):
        return state["prob"].sigma(state["C"])
    if kind == "list":
        S = torch.empty_like(state["C"])
        fg.forte_sci_sigma(state["sci"].sci, state["dets"], state["C"], S, case["nvec"])
        return S
    if kind == "rdms":
        return list(state["prob"].rdms(state["C"][0]))
    if kind == "rdm3":
        return state["prob"].rdm3(state["C"][0])
    if kind == "solve":
        E, C, _, _ = state["prob"].davidson(case["nroots"])
        return [E, C] + (list(state["prob"].rdms(C[0])) if case["rdms"] else [])
    if kind == "grad":
        state["h"].grad = state["eri"].grad = None
        E = fg.sa_energy(state["h"], state["eri"], case["norb"], case["nalpha"], case["nbeta"],
                         [1.0 / case["nroots"]] * case["nroots"], precision=MODES[case["mode"]])
        E.backward()
        return [E.detach(), state["h"].grad, state["eri"].grad]
    return fg.forte_batch_solve(state["problems"], precision=MODES[case["mode"]])[0]


# ------------------------------------------------------------------------------------------ the least work

def _counts(n, na, nb):
    A, B = math.comb(n, na), math.comb(n, nb)
    ka, kb = na * (n - na) + 1, nb * (n - nb) + 1  # replacements of a string, its own occupation once
    two = lambda e: math.comb(e, 2) * math.comb(n - e, 2)  # noqa: E731
    return A * B, ka, kb, ka + two(na), kb + two(nb)


def _sigma_work(n, na, nb, nvec):
    N, ka, kb, sa, sb = _counts(n, na, nb)
    return dict(bytes=16.0 * N * nvec, flops=2.0 * N * nvec * (ka * kb + sa + sb))


def work(case):
    kind, n = case["kind"], case["norb"]
    if kind == "batch":
        by, fl = 0.0, 0.0
        for m in range(case["norb"], case["norb_max"] + 1):  # two roots each, some 20 sigma vectors a root
            w = _sigma_work(m, (m + 1) // 2, m // 2, 40)
            share = case["count"] / (case["norb_max"] + 1 - case["norb"])
            by, fl = by + share * 8.0 * m ** 4, fl + share * w["flops"]
        return dict(bytes=by, flops=fl)
    na, nb = case["nalpha"], case["nbeta"]
    if kind == "list":
        # one element for every pair of the list that could be connected: of the order of the singles and doubles
        # of a determinant, at most the list
        near = min(case["ndet"], na * (n - na) + nb * (n - nb) + math.comb(na, 2) * math.comb(n - na, 2)
                   + math.comb(nb, 2) * math.comb(n - nb, 2) + na * (n - na) * nb * (n - nb))
        return dict(bytes=8.0 * case["ndet"] * (1 + 2 * case["nvec"]), flops=2.0 * case["ndet"] * near * case["nvec"] / 8)
    N, ka, kb, sa, sb = _counts(n, na, nb)
    if kind == "sigma":
        return _sigma_work(n, na, nb, case["nvec"])
    if kind == "gas":
        kept = _kept_count(case)
        return dict(bytes=16.0 * N * case["nvec"], flops=2.0 * kept * case["nvec"] * (ka * kb + sa + sb) * kept / N)
    pairs = n * (n + 1) // 2
    rdm = dict(bytes=8.0 * (N + n ** 4 + n * n), flops=2.0 * N * (pairs * (pairs + 1) // 2 + pairs * (pairs - 1) // 2))
    if kind == "rdms":
        return rdm
    if kind == "rdm3":
        m = n * n  # the pairs commute, and bra and ket can be exchanged
        return dict(bytes=8.0 * (N + n ** 6), flops=2.0 * N * m * (m + 1) * (m + 2) / 12)
    w = _sigma_work(n, na, nb, 20 * case["nroots"])  # some 20 sigma vectors a root
    if kind == "solve":
        by, fl = 8.0 * N * case["nroots"], w["flops"]
        return dict(bytes=by + (rdm["bytes"] if case["rdms"] else 0), flops=fl + (rdm["flops"] if case["rdms"] else 0))
    return dict(bytes=16.0 * (n ** 4 + n * n), flops=w["flops"] + case["nroots"] * rdm["flops"])


# ------------------------------------------------------------------------------------------ 64-bit values

def _strings(n, e):
    return [m for m in range(1 << n) if bin(m).count("1") == e]


def _table(n, e):
    """J[r, s, I], sgn[r, s, I] of a+_r a_s |I> (sgn 0 where it vanishes)."""
    S = _strings(n, e)
    at = {m: i for i, m in enumerate(S)}
    J = np.zeros((n, n, len(S)), dtype=np.int64)
    g = np.zeros((n, n, len(S)))
    for i, m in enumerate(S):
        for s in range(n):
            if not (m >> s) & 1:
                continue
            m1 = m & ~(1 << s)
            for r in range(n):
                if (m1 >> r) & 1:
                    continue
                lo, hi = min(r, s), max(r, s)
                between = bin(m1 & (((1 << hi) - 1) & ~((1 << (lo + 1)) - 1))).count("1")
                J[r, s, i] = at[m1 | (1 << r)]
                g[r, s, i] = -1.0 if between & 1 else 1.0
    return torch.from_numpy(J).cuda(), torch.from_numpy(g).cuda()


class _Exact:
    """E_pq in the determinant basis with plain torch."""

    def __init__(self, n, na, nb):
        self.n = n
        self.Ja, self.ga = _table(n, na)
        self.Jb, self.gb = (self.Ja, self.ga) if na == nb else _table(n, nb)

    def E(self, r, s, X):
        """E_rs X: row I takes the string that E_sr I names."""
        more = (1,) * (X.dim() - 2)
        return (X[self.Ja[s, r]] * self.ga[s, r].reshape(-1, 1, *more)
                + X[:, self.Jb[s, r]] * self.gb[s, r].reshape(1, -1, *more))

    def images(self, C):
        return torch.stack([self.E(r, s, C) for r in range(self.n) for s in range(self.n)])

    def sigma(self, h, eri, C):
        n = self.n
        h, eri = torch.from_numpy(h).cuda(), torch.from_numpy(eri).cuda()
        k = h - 0.5 * torch.einsum("prrq->pq", eri)
        D = self.images(C).reshape(n * n, -1)
        F = (0.5 * eri.reshape(n * n, n * n)) @ D
        S = (k.reshape(-1) @ D).reshape(C.shape)
        del D
        F = F.reshape((n, n) + tuple(C.shape))
        for p in range(n):
            for q in range(n):
                S += self.E(p, q, F[p, q])
        return S

    def rdms(self, C):
        n = self.n
        D = self.images(C).reshape(n * n, -1)
        g1 = (D @ C.reshape(-1)).reshape(n, n)
        G = (D @ D.T).reshape(n, n, n, n)  # <E_ab C | E_rs C> = <E_ba E_rs>
        g2 = G.permute(1, 0, 2, 3).clone()
        for q in range(n):
            g2[:, q, q, :] -= g1
        return g1, g2

    def rdm3(self, C):
        n = self.n
        D = self.images(C)
        g1, g2 = self.rdms(C)
        g3 = torch.empty((n,) * 6, dtype=torch.float64, device="cuda")
        Dt = D.reshape(n, n, -1).transpose(0, 1).reshape(n * n, -1)  # row pq: E_qp C
        for t in range(n):
            for u in range(n):
                g3[:, :, :, :, t, u] = (Dt @ self.images(D[t * n + u]).reshape(n * n, -1).T).reshape((n,) * 4)
        for i in range(n):
            g3[:, i, :, :, i, :] -= g2.permute(0, 2, 3, 1)  # q = t: Gamma_purs at [p, r, s, u]
            g3[:, :, :, i, i, :] -= g2.permute(0, 1, 2, 3)  # s = t: Gamma_pqru
            g3[:, i, i, :, :, :] -= g2.permute(0, 1, 2, 3)  # q = r: Gamma_pstu
            for j in range(n):
                g3[:, i, i, j, j, :] -= g1  # q = r and s = t
        return g3


def _kept(case):
    """Which determinants a RAS restriction keeps."""
    sizes, lo, hi = _ras(case)
    at, occ = 0, []
    for g in sizes:
        mask = ((1 << g) - 1) << at
        occ.append(tuple(np.array([bin(m & mask).count("1") for m in _strings(case["norb"], e)])
                         for e in (case["nalpha"], case["nbeta"])))
        at += g
    keep = True
    for (a, b), l, u in zip(occ, lo, hi):
        both = a[:, None] + b[None, :]
        keep = keep & (both >= l) & (both <= u)
    return keep


def _kept_count(case):
    return int(_kept(case).sum())


def _lowest(h, eri, n, na, nb, k):
    """Lowest k eigenpairs by dense diagonalisation."""
    X = _Exact(n, na, nb)
    A, B = math.comb(n, na), math.comb(n, nb)
    h, eri = torch.from_numpy(h).cuda(), torch.from_numpy(eri).cuda()
    ops = X.images(torch.eye(A * B, dtype=torch.float64, device="cuda").reshape(A, B, A * B)).reshape(n * n, A * B, A * B)
    F = ((0.5 * eri.reshape(n * n, n * n)) @ ops.reshape(n * n, -1)).reshape(ops.shape)
    F += (h - 0.5 * torch.einsum("prrq->pq", eri)).reshape(-1, 1, 1) * torch.eye(A * B, dtype=torch.float64, device="cuda")
    H = torch.bmm(ops, F).sum(0)
    w, V = torch.linalg.eigh(0.5 * (H + H.T))
    V = V[:, :k].T.reshape(k, A, B).contiguous()
    for v in V:
        if v.reshape(-1)[v.abs().argmax()] < 0:
            v.neg_()
    return w[:k], V


def _popcount(x):
    x = x - ((x >> 1) & 0x5555555555555555)
    x = (x & 0x3333333333333333) + ((x >> 2) & 0x3333333333333333)
    x = (x + (x >> 4)) & 0x0F0F0F0F0F0F0F0F
    return (x + (x >> 8) + (x >> 16) + (x >> 24) + (x >> 32) + (x >> 40) + (x >> 48) + (x >> 56)) & 0x7F


def _low_bit(x):
    b = x & -x
    return b, torch.log2(b.double().abs()).round().long()


def _between(word, i, j):
    lo, hi = torch.minimum(i, j), torch.maximum(i, j)
    return word & ((torch.ones_like(word) << hi) - 1) & ~((torch.ones_like(word) << (lo + 1)) - 1)


def _odd(word):
    return 1.0 - 2.0 * (_popcount(word) & 1).double()


def _list_sigma(n, h, eri, dets, C):
    """Slater-Condon elements of every pair of the list, row block by row block."""
    h, eri = torch.from_numpy(h).cuda(), torch.from_numpy(eri).cuda()
    J = torch.einsum("ppqq->pq", eri)
    K = torch.einsum("pqqp->pq", eri)
    occ = ((dets[:, None] >> torch.arange(2 * n, device="cuda")[None, :]) & 1).double()
    a, b = occ[:, :n], occ[:, n:]
    t = a + b
    diag = t @ h.diagonal() + 0.5 * ((t @ J) * t).sum(1) - 0.5 * ((a @ K) * a).sum(1) - 0.5 * ((b @ K) * b).sum(1)
    S = C * diag[None, :]
    sector = _popcount(dets & ((1 << n) - 1))
    step = max(1, (1 << 26) // len(dets))
    for i0 in range(0, len(dets), step):
        Di = dets[i0:i0 + step]
        d = _popcount(Di[:, None] ^ dets[None, :])
        near = (d <= 4) & (d > 0) & (sector[i0:i0 + step, None] == sector[None, :])
        d = d[near]
        ii, jj = near.nonzero(as_tuple=True)
        bra, ket = Di[ii], dets[jj]
        val = torch.zeros(len(ii), dtype=torch.float64, device="cuda")
        one = d == 2
        B, Kt = bra[one], ket[one]
        _, p = _low_bit(B & ~Kt)
        _, q = _low_bit(Kt & ~B)
        sg = _odd(_between(Kt, p, q))
        sp, po, qo = p // n, p % n, q % n
        v = h[po, qo].clone()
        common = occ[jj[one]]
        for r in range(n):
            v += (common[:, r] + common[:, n + r]) * eri[po, qo, r, r]
            same = torch.where(sp == 0, common[:, r], common[:, n + r])
            v -= same * eri[po, r, r, qo]
        # (the hole itself is in `common` too: its Coulomb and exchange parts cancel)
        val[one] = sg * v
        two = d == 4
        B, Kt = bra[two], ket[two]
        b1, p1 = _low_bit(B & ~Kt)
        _, p2 = _low_bit((B & ~Kt) ^ b1)
        k1, q1 = _low_bit(Kt & ~B)
        k2, q2 = _low_bit((Kt & ~B) ^ k1)
        sg = _odd(_between(Kt, p1, q1)) * _odd(_between((Kt ^ k1) | b1, p2, q2))
        s = lambda x: x // n  # noqa: E731
        o = lambda x: x % n  # noqa: E731
        v = torch.where((s(p1) == s(q1)) & (s(p2) == s(q2)), eri[o(p1), o(q1), o(p2), o(q2)], 0.0)
        v = v - torch.where((s(p1) == s(q2)) & (s(p2) == s(q1)), eri[o(p1), o(q2), o(p2), o(q1)], 0.0)
        val[two] = sg * v
        for k in range(C.shape[0]):
            S[k].index_add_(0, ii + i0, val * C[k][jj])
    return S


def exact(case, seed):
    kind = case["kind"]
    if kind == "grad":
        return None
    if kind == "solve" and case["norb"] > 7:
        return None
    if kind == "batch":
        out = []
        for p in prepare(case, seed)["problems"]:
            small = math.comb(p["norb"], p["nalpha"]) * math.comb(p["norb"], p["nbeta"]) <= 400
            out.append(_lowest(p["h"], p["eri"], p["norb"], p["nalpha"], p["nbeta"], p["nroots"])[0] if small else None)
        return out if any(x is not None for x in out) else None
    st = prepare(case, seed)
    n = case["norb"]
    if kind == "list":
        return _list_sigma(n, st["h"], st["eri"], st["dets"], st["C"])
    if kind == "solve":
        E, C = _lowest(st["h"], st["eri"], n, case["nalpha"], case["nbeta"], case["nroots"])
        return [E, C] + (list(_Exact(n, case["nalpha"], case["nbeta"]).rdms(C[0])) if case["rdms"] else [])
    X = _Exact(n, case["nalpha"], case["nbeta"])
    C = st["C"]
    if kind == "rdms":
        return list(X.rdms(C[0]))
    if kind == "rdm3":
        return X.rdm3(C[0])
    keep = torch.from_numpy(_kept(case)).cuda().double() if kind == "gas" else 1.0
    return torch.stack([X.sigma(st["h"], st["eri"], c * keep) * keep for c in C])
