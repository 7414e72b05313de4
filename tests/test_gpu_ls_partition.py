"""Normal-equation sums at the sizes where the split of the work over CTAs changes: one token, one step
of 64 tokens, tiles cut into several parts, a part of a step, one CTA per SM.  The inputs are small integers, whose
sums fp32 holds exactly, so the sums have to be exact whatever the split."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2607_00712_gb300 import abi  # noqa: E402
from paper_2607_00712_gb300.device import LS  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00712_gb300.build import build_library
    build_library()
    abi.lib()


@pytest.mark.parametrize("exact", [False, True])
@pytest.mark.parametrize("D,T", [(128, 1), (128, 65), (256, 1), (256, 64), (256, 4680), (384, 60), (384, 1000), (384, 4680),
                                 (512, 300), (512, 1000), (640, 1000), (768, 129), (896, 1000), (1024, 60), (1024, 1000),
                                 (1280, 4680), (1536, 300), (2048, 60), (2560, 64)])
def test_sums_are_exact(D, T, exact):
    g = torch.Generator(device="cuda").manual_seed(D + T)
    a = torch.randint(-2, 3, (T, D), device="cuda", generator=g).float()
    d = torch.randint(-2, 3, (T, D), device="cuda", generator=g).float()
    a[0, 0], d[0, 0] = 2, 2
    n = abi.ispa_ls_accumulate_workspace_size(D, T)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    st = LS(D)
    for _ in range(2):
        abi.ispa_ls_accumulate_ex(st.c, a.bfloat16(), (a + d).bfloat16(), T, abi.ISPA_LS_EXACT_DELTA if exact else 0, ws, n)
    torch.cuda.synchronize()
    assert abi.ispa_last_device_error()[0] == abi.ISPA_OK
    gram = st.gram.view(2 * D, 2 * D).double()
    a, d = a.double(), d.double()
    upper = torch.ones(D, D, device="cuda").triu() > 0      # G and S keep the upper triangle's tiles
    assert torch.equal(gram[:D, :D][upper], 2 * (a.t() @ a)[upper])
    assert torch.equal(gram[:D, D:], 2 * (a.t() @ d))
    assert torch.equal(gram[D:, D:][upper], 2 * (d.t() @ d)[upper])
