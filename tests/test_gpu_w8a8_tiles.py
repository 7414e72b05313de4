"""W8A8 projection where it runs on pairs of CTAs, and its stores at ragged row tiles: nothing past the
last row is written."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import quant as qt  # noqa: E402
from paper_2607_00712_gb300 import abi, synth  # noqa: E402
from paper_2607_00712_gb300.device import to_f32  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00712_gb300.build import build_library
    build_library()
    abi.lib()


# pairs: the last 256-row tile has 228, 66 and 256 rows; one CTA: 1, 31, 33, 127 and 129 rows, each tile width
@pytest.mark.parametrize("T,D,Do", [(3300, 1024, 7680), (4930, 1024, 5120), (3328, 1024, 7680),
                                    (1, 128, 256), (31, 128, 384), (33, 256, 128), (127, 384, 512), (129, 256, 384),
                                    (2300, 256, 1536), (4800, 128, 768)])
def test_rows_and_edges(T, D, Do):
    # fp32 accumulation of exact e4m3 products in one chain of D terms, two fp32 scale multiplies, bf16 rounding
    g = np.random.default_rng(T + D)
    aq, sa = qt.quantize_rows(synth.bf16_round(g.standard_normal((T, D), dtype=np.float32)))
    wq, sw = qt.quantize_weight((g.standard_normal((D, Do)) / np.sqrt(D)).astype(np.float32), None)
    out = torch.full((T + 256, Do), 7.0, dtype=torch.bfloat16, device="cuda")
    abi.ispa_linear_w8a8(torch.from_numpy(aq).cuda(), torch.from_numpy(sa).cuda(), torch.from_numpy(wq).cuda(),
                         torch.from_numpy(sw).cuda(), T, D, Do, out)
    torch.cuda.synchronize()
    assert abi.ispa_last_device_error()[0] == abi.ISPA_OK
    assert bool((out[T:] == 7.0).all())
    last = np.arange(max(0, T - 260), T)
    rows = np.unique(np.concatenate([[0, T // 2], last, g.integers(0, T, 40)]))
    y = to_f32(out)[rows].astype(np.float64)
    ref = qt.linear_w8a8(aq[rows], sa[rows], wq, sw)
    mag = (np.abs(qt.decode(aq[rows])) @ np.abs(qt.decode(wq)).T) * sa[rows][:, None].astype(np.float64) * sw.astype(np.float64)
    assert np.all(np.abs(y - ref) <= 2.0 ** -8 * np.abs(ref) + (D + 6) * 2.0 ** -24 * mag)


@pytest.mark.parametrize("T,D", [(9, 16), (50, 1024), (33, 1040), (50, 1536), (21, 1552), (50, 2048), (17, 2064), (8, 3072),
                                 (7, 3088), (3, 8960)])
def test_quantised_rows_at_the_register_limits(T, D):
    # rows that fill 4, 6, 8 and 12 words a lane exactly, or need a little more: codes and scales bit for bit
    x = synth.bf16_round(np.random.default_rng(D).standard_normal((T, D), dtype=np.float32))
    x[T // 2, D - 1] = 1e4
    q = torch.empty(T, D, dtype=torch.uint8, device="cuda")
    s = torch.empty(T, dtype=torch.float32, device="cuda")
    abi.ispa_quantize_rows_e4m3(torch.from_numpy(x).to(torch.bfloat16).cuda(), T, D, q, s)
    torch.cuda.synchronize()
    rq, rs = qt.quantize_rows(synth.bf16_round(x))
    assert np.array_equal(q.cpu().numpy(), rq) and np.array_equal(s.cpu().numpy(), rs)


# few tiles: 8, 4 and 2 CTAs share a tile's k-blocks, evenly or not; the last row tile is ragged
@pytest.mark.parametrize("T,D,Do", [(40, 1536, 1536), (1, 5120, 128), (129, 4736, 256), (52, 4224, 2048), (300, 2688, 768),
                                    (128, 5120, 5120), (200, 3200, 4096)])
def test_split_contractions(T, D, Do):
    test_rows_and_edges(T, D, Do)
