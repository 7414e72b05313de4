"""The 8-bit chain back to back: quantisers, attention and append are launched while the kernel before them finishes,
and each reads what that kernel writes or writes what it reads.  The same calls one at a time give the same bits."""
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


def _chain(fmt, H, P, frames, sync):
    """Codes of q, k (and v) -> attention -> append -> attention over the new ring, six times."""
    g = torch.Generator(device="cuda")
    g.manual_seed(H * P)
    d, n, kv8 = 128, P, fmt == "kv8"
    D, ld = H * d, (P + 15) // 16 * 16
    ring = Ring(H, d, P, frames, 1, k_e4m3=not kv8, kv_e4m3=kv8)
    x = torch.randn(n, H, d, generator=g, device="cuda").bfloat16()
    scale = torch.full((H,), 4 / 448, device="cuda")
    q8, k8 = (torch.empty(n, H, d, dtype=torch.uint8, device="cuda") for _ in range(2))
    qs = torch.empty(H, (n + 127) // 128, device="cuda")
    v8 = torch.zeros(H, d, ld, dtype=torch.uint8, device="cuda")
    out, again = (torch.empty(n, D, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    lse = torch.empty(H, n, device="cuda")

    def attend(o):
        if kv8:
            abi.ispa_attn_full_kv8(ring.c, scale, scale, q8, qs, k8, scale, v8, ld, n, 0.0, o, lse)
        else:
            abi.ispa_attn_full_qk8(ring.c, scale, q8, qs, k8, scale, x, n, 0.0, o, lse)

    def append():
        if kv8:
            abi.ispa_kv_append_kv8(ring.c, x, x, 1, scale, scale)
        else:
            abi.ispa_kv_append_qk8(ring.c, x, x, 1, scale)

    seen = []
    for _ in range(6):
        for call in (lambda: abi.ispa_quantize_q_e4m3(x, n, H, d, q8, qs),
                     lambda: abi.ispa_quantize_k_e4m3(x, n, H, d, scale, k8),
                     lambda: abi.ispa_quantize_vt_e4m3(x, n, H, d, scale, v8, ld),
                     lambda: attend(out), append, lambda: attend(again),
                     lambda: x.copy_((out.view_as(x) * 3 + again.view_as(x) + x * 0.5))):
            call()
            if sync:
                torch.cuda.synchronize()
        seen += [q8.clone(), k8.clone(), v8.clone(), out.clone(), again.clone(), lse.clone()]
    seen += [ring.k.clone(), ring.v.clone()]
    torch.cuda.synchronize()
    assert abi.ispa_last_device_error()[0] == abi.ISPA_OK
    return seen


@pytest.mark.parametrize("fmt", ["qk8", "kv8"])
@pytest.mark.parametrize("H,P,frames", [(2, 100, 3), (2, 640, 5), (12, 1664, 3)])
def test_back_to_back_8bit_calls_equal_synchronised_ones(fmt, H, P, frames):
    want = _chain(fmt, H, P, frames, True)
    for _ in range(3):
        for a, b in zip(want, _chain(fmt, H, P, frames, False)):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
