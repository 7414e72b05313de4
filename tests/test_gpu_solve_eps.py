"""eps of the absorption solve against whole-number arithmetic, where its first term is all there is."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2607_00712_gb300 import abi  # noqa: E402
from paper_2607_00712_gb300.device import LS, to_f32  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00712_gb300.build import build_library
    build_library()
    abi.lib()


def test_the_sum_over_the_features_is_rounded_a_few_times():
    # X = 0 and G = I: dW = 0 and eps = sum_ij S_ij (W W^T)_ij.  S below 2^23 and W below 2^6 are whole and positive,
    # so is every term, below 2^41, and a CTA's share of them (2^51) is exact; what rounds is the addition of shares to
    # one sum of 2^54.2.  Added up in random order (200 trials), 12 shares, the tiles of 128 x 64, leave 0.6 units in
    # its last place (root mean square), 48, a plain kernel's blocks of 256 numbers, 1.2, and 192, one a warp, 2.0.
    D, n, draws = 384, 32, 40
    st = LS(D)
    wsb = abi.ispa_ls_solve_workspace_size(D, n)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    out = torch.empty(D, n, dtype=torch.float32, device="cuda")
    units = []
    for seed in range(draws):
        g = np.random.default_rng(seed)
        S = np.triu(g.integers(1, 1 << 23, (D, D)))
        S = S + np.triu(S, 1).T
        W = g.integers(1, 1 << 6, (D, n))
        exact = int(np.sum(S * (W @ W.T)))   # exact in 64-bit whole numbers
        gram = np.zeros((2 * D, 2 * D), np.float32)
        gram[:D, :D], gram[D:, D:] = np.eye(D), np.triu(S)
        st.gram.copy_(torch.from_numpy(gram.reshape(-1)))
        eps = abi.ispa_ls_solve(st.c, torch.from_numpy(W.astype(np.float32)).cuda(), n, 0.0, out, ws, wsb)
        assert not to_f32(out).any()
        units.append((int(eps) - exact) / float(np.spacing(float(exact))))
    assert np.sqrt(np.mean(np.square(units))) <= 1.2, units
