"""Launches that start while the one before them finishes: back-to-back calls whose inputs the call
before has just written (or whose ring the call before still reads) equal the same calls one at a time."""
import pytest

torch = pytest.importorskip("torch")

from paper_2607_00712_gb300 import abi  # noqa: E402
from paper_2607_00712_gb300.device import Ring  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00712_gb300.build import build_library
    build_library()
    abi.lib()


def _chain(H, P, frames, sync):
    """Attention -> projection -> the next step's q, k, v -> append -> attention, eight times."""
    g = torch.Generator(device="cuda")
    g.manual_seed(H * P)
    d, n = 128, P
    D = H * d
    ring = Ring(H, d, P, frames, 1)
    x = torch.randn(n, H, d, generator=g, device="cuda").bfloat16()
    W = (torch.randn(D, D, generator=g, device="cuda") / D ** 0.5).contiguous()
    w8, ws = torch.empty(D, D, dtype=torch.uint8, device="cuda"), torch.empty(D, device="cuda")
    abi.ispa_quantize_weight_e4m3(W, None, D, D, w8, ws)
    out, lse = torch.empty(n, D, dtype=torch.bfloat16, device="cuda"), torch.empty(H, n, device="cuda")
    a8, sa = torch.empty(n, D, dtype=torch.uint8, device="cuda"), torch.empty(n, device="cuda")
    y = torch.empty_like(out)
    seen = []
    for _ in range(8):
        for call in (lambda: abi.ispa_attn_full(ring.c, x, x, x, n, 0.0, out, lse),
                     lambda: abi.ispa_quantize_rows_e4m3(out, n, D, a8, sa),
                     lambda: abi.ispa_linear_w8a8(a8, sa, w8, ws, n, D, D, y),
                     lambda: abi.ispa_kv_append(ring.c, x, x, 1),
                     lambda: x.copy_((x.view(n, D) * 0.5 + y).view_as(x))):
            call()
            if sync:
                torch.cuda.synchronize()
        seen += [out.clone(), lse.clone(), y.clone()]
    torch.cuda.synchronize()
    assert abi.ispa_last_device_error()[0] == abi.ISPA_OK
    return seen


@pytest.mark.parametrize("H,P,frames", [(2, 100, 3),     # everything small
                                        (2, 640, 5),     # split items alone
                                        (12, 1664, 3)])  # 156 items: whole ones, then split ones
def test_back_to_back_calls_equal_synchronised_ones(H, P, frames):
    want = _chain(H, P, frames, True)
    for _ in range(3):
        for a, b in zip(want, _chain(H, P, frames, False)):
            assert torch.equal(a, b)
