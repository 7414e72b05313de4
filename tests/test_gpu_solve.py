"""The absorption solve at the edges of its blocks: panels of 64 columns, blocks of 128 rows,
products in tiles of 128 x 64 and chunks of 32, and its fixed-point factorisation's range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ls as ols  # noqa: E402
from paper_2607_00712_gb300 import abi  # noqa: E402
from paper_2607_00712_gb300.device import LS, to_f32  # noqa: E402

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00712_gb300.build import build_library
    build_library()
    abi.lib()


def _sums(seed, D, T, spread=0.0):
    """fp32 G, X, S of T tokens; features scaled by exp(spread * N(0, 1))."""
    g = np.random.default_rng(seed)
    f = np.exp(spread * g.standard_normal(D))
    a = g.standard_normal((T, D)) * f
    d = 0.5 * g.standard_normal((T, D)) * f + 0.2 * a
    return (a.T @ a).astype(np.float32), (a.T @ d).astype(np.float32), (d.T @ d).astype(np.float32)


def _sym(m):
    m = m.astype(np.float64)
    return np.triu(m) + np.triu(m, 1).T


def _gpu(G, X, S, W, lam):
    D, n = W.shape
    st = LS(D)
    gram = np.zeros((2 * D, 2 * D), np.float32)
    gram[:D, :D], gram[:D, D:], gram[D:, D:] = np.triu(G), X, np.triu(S)   # what the state maintains for any D
    st.gram.copy_(torch.from_numpy(gram.reshape(-1)))
    wsb = abi.ispa_ls_solve_workspace_size(D, n)
    ws = torch.full((wsb,), 0xA5, dtype=torch.uint8, device="cuda")     # no entry may count on zeros
    dW = torch.empty(D, n, dtype=torch.float32, device="cuda")
    eps = abi.ispa_ls_solve(st.c, torch.from_numpy(W).cuda(), n, lam, dW, ws, wsb)
    assert abi.ispa_last_device_error()[0] == abi.ISPA_OK
    return to_f32(dW).astype(np.float64), eps


@pytest.mark.parametrize("D,n,spread", [(1, 1, 0.0), (5, 3, 0.0), (63, 64, 0.0), (64, 65, 0.0), (65, 31, 2.0), (127, 128, 0.0),
                                        (129, 33, 2.0), (192, 200, 0.0), (320, 63, 1.0), (384, 384, 0.0), (520, 129, 2.0)])
def test_solve_matches_the_oracle(D, n, spread):
    # Both sides solve the same fp32 sums.  dW: fp32 rounding (2^-24) plus what 64-bit arithmetic may
    # lose, D 2^-53 times the condition number of the scaled matrix (diagonal scaling does not
    # enter the error of a Cholesky solve), row by row of the scaled solution.  eps: a difference of three terms.
    G, X, S = _sums(D + n, D, 3 * D + 40, spread)
    W = (np.random.default_rng(n).standard_normal((D, n)) / np.sqrt(D)).astype(np.float32)
    lam = 1e-3
    dW, eps = _gpu(G, X, S, W, lam)
    Gs, Ss = _sym(G), _sym(S)
    ref, eps_ref = ols.ls_solve(Gs, X.astype(np.float64), Ss, W, lam, factor=np.linalg.cholesky)
    M = Gs + lam * np.eye(D)
    s = 1 / np.sqrt(np.diag(M))
    cond = np.linalg.cond(M * s[:, None] * s[None, :])
    err = np.linalg.norm((dW - ref) / s[:, None])
    assert err <= (2.0 ** -24 + 8 * D * cond * U64) * np.linalg.norm(ref / s[:, None]), err
    terms = abs(np.sum(ref * (Gs @ ref))) + 2 * abs(np.sum(ref * (X.astype(np.float64) @ W))) + abs(np.sum(W * (Ss @ W)))
    assert abs(eps - eps_ref) <= 8 * D * cond * U64 * terms


@pytest.mark.parametrize("D,bad", [(200, "late pivot"), (200, "off-diagonal"), (200, "nan"), (200, "inf"), (130, "zero row")])
def test_not_positive_definite(D, bad):
    G, X, S = _sums(7, D, 3 * D)
    if bad == "late pivot":       # the last Schur complement turns negative
        L = np.linalg.cholesky(_sym(G))
        G[-1, -1] -= np.float32(1.01 * L[-1, -1] ** 2)
    elif bad == "off-diagonal":
        G[20, 170] = 2 * np.sqrt(G[20, 20] * G[170, 170])
    elif bad == "zero row":
        G[:, 100] = G[100, :] = 0
    else:
        G[3, 150] = np.float32(bad)
    W = np.eye(D, 40, dtype=np.float32)
    with pytest.raises(abi.IspaError) as e:
        _gpu(G, X, S, W, 0.0)
    assert e.value.status == abi.ISPA_ERR_NOT_SPD


def test_a_nan_weight_stays_in_its_column():
    D, n = 150, 70
    G, X, S = _sums(9, D, 500)
    W = (np.random.default_rng(1).standard_normal((D, n)) / 12).astype(np.float32)
    clean, _ = _gpu(G, X, S, W, 1e-3)
    W[17, 5] = np.nan
    dW, eps = _gpu(G, X, S, W, 1e-3)
    assert np.isnan(dW[:, 5]).all() and np.isnan(eps)
    keep = np.arange(n) != 5
    assert np.array_equal(dW[:, keep], clean[:, keep])


@pytest.mark.parametrize("D,n,spread", [(520, 16384, 0.0), (700, 10900, 1.0), (1030, 6600, 0.0)])
def test_solve_in_windows(D, n, spread):
    # many columns: the substitutions go by windows of 512 rows, the last of which is partial
    test_solve_matches_the_oracle(D, n, spread)
