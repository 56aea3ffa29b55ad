"""The GPU eigen-decomposition of the Tanner-graph Laplacian on graphs where it can go wrong: the smallest
ones, disconnected ones (a split tridiagonal matrix), clusters of equal eigenvalues of every size class
(one CTA, Cholesky QR, past its node limit), dependent nodes, the largest token count; and the attention's
fixed-point rows against the double-precision rows that wide scores take."""
import numpy as np
import pytest

from paper_2410_05911_gb300 import aecct as A
from paper_2410_05911_gb300 import inputs as I
from paper_2410_05911_gb300 import spe

pytest.importorskip("torch")

EPS = np.finfo(np.float64).eps


def _random(n, m, p, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    H = (rng.random((m, n)) < p).astype(np.uint8)
    H[rng.integers(0, m, n), np.arange(n)] = 1
    H[np.arange(m), rng.integers(0, n, m)] = 1
    return H


GRAPHS = {
    "one edge pair": np.ones((1, 2), np.uint8),
    "star": np.ones((1, 40), np.uint8),                                              # one eigenvalue 39 times
    "complete": np.ones((5, 37), np.uint8),
    "ten copies": np.kron(np.eye(10, dtype=np.uint8), np.ones((2, 5), np.uint8)),    # disconnected
    "five hamming": np.kron(np.eye(5, dtype=np.uint8), I.make_code("hamming7_4").H),
    "random 80": _random(60, 20, 0.1, 0),
    "random 300": _random(200, 100, 0.02, 1),
    "ldpc 450": I.ldpc_regular_code(300, 150, 3, 6, seed=1).H,                       # 150 times, dependent nodes
    "ldpc 690": I.ldpc_regular_code(460, 230, 3, 6, seed=2).H,                       # 230 times
    "wide star": np.kron(np.eye(2, dtype=np.uint8), np.ones((1, 400), np.uint8)),    # 798 times
    "ldpc 1020": I.ldpc_regular_code(680, 340, 3, 6, seed=3).H,
}


@pytest.mark.gpu
@pytest.mark.parametrize("name", GRAPHS)
def test_eigenpairs_of_graph(name):
    H = GRAPHS[name]
    T = sum(H.shape)
    p = I.spe_params(H, 8, seed=1)
    tab, t64, lam, U = A.spe_table(H, p, want_eigen=True)
    ref_lam, ref_U = spe.eigenpairs(H)
    top = ref_lam[-1]
    L = spe.tanner_laplacian(H)
    assert np.abs(lam - ref_lam).max() <= 4 * EPS * top * T
    # residuals and orthogonality: backward errors of T-step reductions, divided by the smallest gap
    # between clusters for the vectors themselves
    gaps = np.diff(ref_lam)
    gap = gaps[gaps > 1e-8 * max(1.0, top)].min(initial=top)
    assert np.abs(L @ U - U * lam).max() <= 32 * EPS * top * T
    assert np.abs(U.T @ U - np.eye(T)).max() <= 32 * EPS * T * max(1.0, top / gap)
    assert np.abs(U - ref_U).max() <= 128 * EPS * T * max(1.0, top / gap)
    if T <= 100:
        ref = spe.spe_from_eigenpairs(ref_lam, ref_U, p)
        assert np.abs(t64 - ref).max() <= 1e-9 * (1 + np.abs(ref).max())
        assert np.abs(tab - ref).max() <= 1e-6 * (1 + np.abs(ref).max())


# eigenvalues that lie close without being equal (5e-6 apart for Polar(64,32)): their vectors are orthogonal to
# rounding, a few T eps, whatever the gap
CLOSE = dict(GRAPHS, **{"polar": I.make_code("polar64_32").H, "bch63": I.make_code("bch63_36").H,
                        "ldpc 192": I.make_code("ldpc128_64").H,
                        "ninety hamming": np.kron(np.eye(90, dtype=np.uint8), I.make_code("hamming7_4").H)})


@pytest.mark.gpu
@pytest.mark.parametrize("name", CLOSE)
def test_eigenvectors_are_orthonormal(name):
    H = CLOSE[name]
    T = sum(H.shape)
    _, _, lam, U = A.spe_table(H, I.spe_params(H, 8, seed=1), want_eigen=True)
    assert np.abs(U.T @ U - np.eye(T)).max() <= 2 * EPS * T
    L = spe.tanner_laplacian(H)
    assert np.abs(L @ U - U * lam).max() <= 32 * EPS * lam[-1] * T


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [1e-3, 1.0, 4.0, 8.0, 20.0, 40.0, 1e3])
def test_table_over_score_ranges(scale):
    # scores from about 1e-6 over both fixed-point ranges (1024 and 16384 in base 2) to where rows take doubles; the
    # error of a row's probabilities is that of its scores, 2^-52 of their size or more
    H = I.make_code("bch31_16").H
    p = I.spe_params(H, 16, seed=3)
    p.wq = p.wq * scale
    p.wk = p.wk * scale
    lam, U = spe.eigenpairs(H)
    ref = spe.spe_from_eigenpairs(lam, U, p)
    _, t64, lam_g, U_g = A.spe_table(H, p, want_eigen=True)
    # the same attention on the GPU's own eigenpairs, so that only the softmax is compared
    own = spe.spe_from_eigenpairs(lam_g, U_g, p)
    size = 1 + np.abs(ref).max()
    assert np.abs(t64 - own).max() <= 64 * EPS * size * max(1.0, 16.0 * scale * scale)


def _attention(lam, U, p, nodes):
    """SPE rows of `nodes` by the definition, and the largest score."""
    heads, d_e = p.wq.shape[0], p.wq.shape[2]
    rows, top = [], 0.0
    for j in nodes:
        X = np.stack([lam, U[j]], 1) @ p.w_pe
        parts = []
        for e in range(heads):
            S = (X @ p.wq[e]) @ (X @ p.wk[e]).T / np.sqrt(d_e)
            top = max(top, np.abs(S).max())
            P = np.exp(S - S.max(1, keepdims=True))
            parts.append((P / P.sum(1, keepdims=True) @ (X @ p.wv[e])).mean(0))
        rows.append(np.concatenate(parts) @ p.wo)
    return np.array(rows), top


# past 576 nodes a thread takes several rows; the larger scales reach the wide fixed-point rows and the double ones
@pytest.mark.gpu
@pytest.mark.parametrize("name", ["random 300", "ldpc 450", "ldpc 690", "wide star", "ldpc 1020"])
@pytest.mark.parametrize("scale", [1.0, 8.0, 40.0])
def test_table_of_long_codes_on_sampled_nodes(name, scale):
    H = GRAPHS[name]
    T = sum(H.shape)
    p = I.spe_params(H, 8, seed=4)
    p.wq, p.wk = p.wq * scale, p.wk * scale
    tab, t64, lam, U = A.spe_table(H, p, want_eigen=True)
    nodes = [0, 1, T // 3, T // 2, T - 2, T - 1]
    ref, top = _attention(lam, U, p, nodes)
    # the error of a probability is that of its score, 2^-52 of the largest score or more
    bound = 64 * EPS * (1 + np.abs(ref).max()) * max(1.0, top)
    assert np.abs(t64[nodes] - ref).max() <= bound
    assert np.abs(tab - t64).max() <= 1e-7 * (1 + np.abs(t64).max())
