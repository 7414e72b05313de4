"""Normal-equation sums of few tokens on the grids that cut fewer tiles than one CTA per SM does: whole passes a CTA,
full waves of one kind of tile and a tail, and the first token count past them.  Small integers, whose sums fp32
holds exactly, so the sums have to be exact whatever the grid."""
import pytest

torch = pytest.importorskip("torch")

import test_gpu_ls_partition as base  # noqa: E402
from paper_2607_00712_gb300 import abi  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00712_gb300.build import build_library
    build_library()
    abi.lib()


@pytest.mark.parametrize("exact", [False, True])
@pytest.mark.parametrize("D,T", [(1792, 500), (2048, 84), (2560, 1), (2560, 500), (3072, 200), (3328, 300), (3840, 60),
                                 (3840, 84), (4096, 84), (4608, 136), (2048, 1024), (2048, 1025)])
def test_sums_are_exact_on_fewer_ctas(D, T, exact):
    base.test_sums_are_exact(D, T, exact)
