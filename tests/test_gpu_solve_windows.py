"""The absorption solve where its substitutions go by three windows of 512 rows and more: windows that are both updated
by others and update them, and slices of L at an offset in the operand."""
import pytest

torch = pytest.importorskip("torch")

import test_gpu_solve as base  # noqa: E402
from paper_2607_00712_gb300 import abi  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00712_gb300.build import build_library
    build_library()
    abi.lib()


@pytest.mark.parametrize("D,n,windows", [(1030, 8250, 3),    # 512, 512 and 128 rows
                                         (1600, 5500, 4)])   # 3 x 512 and 128, features spread
def test_three_windows_and_more(D, n, windows):
    rows = -(-D // 128) * 128
    assert rows // 256 * -(-n // 64) >= 512 and -(-rows // 512) == windows   # the solve's own rule for windows
    base.test_solve_matches_the_oracle(D, n, 1.0 if windows == 4 else 0.0)
