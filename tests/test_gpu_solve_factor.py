"""What the factorisation's rounding leaves in eps of an ill-conditioned solve: no more than fp64 numbers' own."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2607_00712_gb300 import abi  # noqa: E402
from paper_2607_00712_gb300.device import LS  # noqa: E402

pytestmark = pytest.mark.gpu
WIDE = np.longdouble   # 64 bits of mantissa or more


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00712_gb300.build import build_library
    build_library()
    abi.lib()


def _activations(kind, g, T, D):
    a = g.standard_normal((T, D))
    if kind == "pairs":        # every other feature nearly its neighbour's copy
        a[:, 1::2] = a[:, 0::2] + 1e-4 * a[:, 1::2]
    else:                      # singular values falling to 1e-4, in no feature's direction
        u, v = (np.linalg.qr(g.standard_normal((D, D)))[0] for _ in range(2))
        a = (a @ (u * np.logspace(0, -4, D))) @ v
    return a


def _cholesky(M):
    L = np.zeros_like(M)
    for j in range(len(M)):
        c = M[j:, j] - L[j:, :j] @ L[j, :j]
        L[j:, j] = c / np.sqrt(c[0])
    return L


def _forward(L, B):
    Y = B.copy()
    for i in range(len(B)):
        Y[i] = (B[i] - L[i, :i] @ Y[:i]) / L[i, i]
    return Y


def _backward(L, Y):
    Z = Y.copy()
    for i in range(len(Y) - 1, -1, -1):
        Z[i] = (Y[i] - L[i + 1:, i] @ Z[i + 1:]) / L[i, i]
    return Z


def _sym(m):
    return np.triu(m) + np.triu(m, 1).T


@pytest.mark.parametrize("seed", [0, 1, 2])
@pytest.mark.parametrize("kind", ["pairs", "decay"])
def test_eps_of_an_ill_conditioned_system(kind, seed):
    # A factor of M + E (M scaled to a diagonal near 1) changes eps by sum_ij K_ij E_ij to first order, with
    # K = Z Z^T + V Z^T + Z V^T, M Z = X W and M V = lambda Z.  An E of independent elements of 2^-56, the rounding of
    # an fp64 number in [1/4, 1), gives 2^-56 |K| (Frobenius) for a standard deviation; elements that all lean the same
    # way add up to more.  The products and sums outside the factor are off by a few 2^-53 of eps's terms.
    D, n, lam = 256, 32, 1e-3
    g = np.random.default_rng(seed)
    a = _activations(kind, g, 3 * D, D)
    d = 0.5 * g.standard_normal(a.shape) + 0.2 * a
    W = (g.standard_normal((D, n)) / np.sqrt(D)).astype(np.float32)
    G, X, S = ((p.T @ q).astype(np.float32) for p, q in ((a, a), (a, d), (d, d)))
    M = (_sym(G.astype(np.float64)) + lam * np.eye(D)).astype(WIDE)
    s = WIDE(2) ** -((np.frexp(np.diag(M).astype(np.float64))[1] + 1) >> 1)
    Ww, Sw = W.astype(WIDE), _sym(S).astype(WIDE)
    L = _cholesky(M * s[:, None] * s[None, :])
    Y = _forward(L, (X.astype(WIDE) @ Ww) * s[:, None])
    Z = _backward(L, Y)
    term = np.sum(Ww * (Sw @ Ww))
    exact = term - np.sum(Y * Y) - WIDE(lam) * np.sum((Z * s[:, None]) ** 2)
    L64, Z64 = L.astype(np.float64), Z.astype(np.float64)
    V = _backward(L64, _forward(L64, lam * Z64 * s.astype(np.float64)[:, None] ** 2))
    K = Z64 @ Z64.T + V @ Z64.T + Z64 @ V.T

    st = LS(D)
    gram = np.zeros((2 * D, 2 * D), np.float32)
    gram[:D, :D], gram[:D, D:], gram[D:, D:] = np.triu(G), X, np.triu(S)
    st.gram.copy_(torch.from_numpy(gram.reshape(-1)))
    wsb = abi.ispa_ls_solve_workspace_size(D, n)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    out = torch.empty(D, n, dtype=torch.float32, device="cuda")
    eps = abi.ispa_ls_solve(st.c, torch.from_numpy(W).cuda(), n, lam, out, ws, wsb)
    err = abs(float(eps - exact))
    assert err <= 2.0 ** -56 * np.linalg.norm(K) + 8 * 2.0 ** -53 * float(term), err / np.linalg.norm(K) * 2.0 ** 56
