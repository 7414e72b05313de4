"""The absorption solve where the weights undo large differences between the features' sizes: X W is formed from
numbers of 56 bits under a row's or a column's largest, so the features have to meet in it at one size."""
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


def _problem(kind, D, n):
    """fp32 G, X, S of 3 D + 40 tokens and a W whose row j goes with 1 / (the size of Delta's feature j)."""
    g = np.random.default_rng(D + n)
    T = 3 * D + 40
    fa, fd = np.ones(D), np.ones(D)
    if kind == "two groups":
        fa = fd = np.where(np.arange(D) % 2, 2.0 ** 20, 2.0 ** -20)
    elif kind == "log-normal":
        fa = fd = np.exp(6 * g.standard_normal(D))
    elif kind == "few large":
        fd = np.where(np.arange(D) % 50 == 0, 2.0 ** 40, 1.0)
    a = g.standard_normal((T, D)) * fa
    d = (0.5 * g.standard_normal((T, D)) + 0.2 * a / fa) * fd
    W = g.standard_normal((D, n)) / np.sqrt(D) / fd[:, None]
    if kind == "no difference":   # features whose Delta is zero, with by far the largest weights
        d[:, ::2] = 0
        W[::2] *= 2.0 ** 40
    return tuple(m.astype(np.float32) for m in (a.T @ a, a.T @ d, d.T @ d, W))


def _sym(m):
    m = m.astype(np.float64)
    return np.triu(m) + np.triu(m, 1).T


@pytest.mark.parametrize("D,n", [(65, 31), (256, 64), (520, 33)])
@pytest.mark.parametrize("kind", ["two groups", "log-normal", "few large", "no difference"])
def test_weights_against_the_features(kind, D, n):
    # The bounds of the solve's other tests: fp32 rounding of dW plus D 2^-53 times the scaled matrix's condition
    # number, row by row of the scaled solution; eps against the size of its terms.
    G, X, S, W = _problem(kind, D, n)
    lam = 0.0 if kind in ("two groups", "log-normal") else 1e-3   # the small features' own sums are far below 1e-3
    st = LS(D)
    gram = np.zeros((2 * D, 2 * D), np.float32)
    gram[:D, :D], gram[:D, D:], gram[D:, D:] = np.triu(G), X, np.triu(S)
    st.gram.copy_(torch.from_numpy(gram.reshape(-1)))
    wsb = abi.ispa_ls_solve_workspace_size(D, n)
    ws = torch.full((wsb,), 0xA5, dtype=torch.uint8, device="cuda")
    out = torch.empty(D, n, dtype=torch.float32, device="cuda")
    eps = abi.ispa_ls_solve(st.c, torch.from_numpy(W).cuda(), n, lam, out, ws, wsb)
    assert abi.ispa_last_device_error()[0] == abi.ISPA_OK
    dW = to_f32(out).astype(np.float64)
    Gs, Ss, Xd, Wd = _sym(G), _sym(S), X.astype(np.float64), W.astype(np.float64)
    ref, eps_ref = ols.ls_solve(Gs, Xd, Ss, W, lam, factor=np.linalg.cholesky)
    M = Gs + lam * np.eye(D)
    s = 1 / np.sqrt(np.diag(M))
    cond = np.linalg.cond(M * s[:, None] * s[None, :])
    err = np.linalg.norm((dW - ref) / s[:, None]) / np.linalg.norm(ref / s[:, None])
    assert err <= 2.0 ** -24 + 8 * D * cond * U64, err
    terms = abs(np.sum(ref * (Gs @ ref))) + 2 * abs(np.sum(ref * (Xd @ Wd))) + abs(np.sum(Wd * (Ss @ Wd)))
    assert abs(eps - eps_ref) <= 8 * D * cond * U64 * terms
