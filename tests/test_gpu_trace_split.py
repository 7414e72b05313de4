"""The tile trace (ispa_debug_set_trace) of calls whose items are split over clusters: after whole items the events are
those of the first whole item alone; where all items are split, those of the first CTA's share."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_helpers import Step  # noqa: E402
from paper_2607_00712_gb300 import abi  # noqa: E402

pytestmark = pytest.mark.gpu
SLOTS, TILE = 32, 192


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00712_gb300.build import build_library
    build_library()
    abi.lib()


@pytest.mark.parametrize("H,P,whole", [(12, 1560, True),    # 156 items: 152 and 4
                                       (3, 400, False)])    # 12 items
def test_one_item_is_traced(H, P, whole):
    past = 4
    st = Step(H, P=P, H=H, d=128, n_past=past, n_chunk_frames=1, capacity=past)
    n, keys = st.n_q, past * P
    out = torch.empty(n, H * 128, dtype=torch.bfloat16, device="cuda")
    abi.ispa_attn_full(st.ring.c, st.q, st.kc, st.vc, n, 0.0, out)
    plain = out.clone()
    buf = torch.zeros(128 * SLOTS, dtype=torch.int64, device="cuda")
    abi.ispa_debug_set_trace(buf, 128)
    try:
        abi.ispa_attn_full(st.ring.c, st.q, st.kc, st.vc, n, 0.0, out)
        torch.cuda.synchronize()
    finally:
        abi.ispa_debug_set_trace(None, 0)
    assert torch.equal(out, plain)
    t = buf.view(-1, SLOTS).cpu().numpy()
    tiles = int((t[:, 0] != 0).sum())
    all_tiles = -(-keys // TILE) + -(-P // TILE)
    assert tiles == all_tiles if whole else 2 <= tiles < all_tiles
    # softmax warp 0, one after the other: kernel entry, every tile's scores seen and P arrived, the epilogue
    order = np.concatenate([t[0, 12:13], t[:tiles, [0, 2]].reshape(-1), t[0, 15:16]])
    assert np.all(np.diff(order) > 0)
