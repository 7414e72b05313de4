"""Attention launches whose items leave SMs idle: their key tiles are split over a cluster and merged.

The shapes put the cut everywhere: two tiles a CTA, ranges that start inside a segment or at its end, a
ragged last tile, CTAs whose keys a frame-causal row never sees, a full wave of whole items before
the split ones.  Tolerances are the unsplit kernel's (the merge is fp32)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_helpers import Step, assert_close_attn  # noqa: E402
from oracle import attention as at  # noqa: E402
from paper_2607_00712_gb300 import abi  # noqa: E402
from paper_2607_00712_gb300.device import Window, to_f32  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00712_gb300.build import build_library
    build_library()
    abi.lib()


def _check(st, win=None, causal=False, rows=None):
    n = st.n_q
    out = torch.full((n, st.H * st.d), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((st.H, n), float("nan"), dtype=torch.float32, device="cuda")
    flags = abi.ISPA_ATTN_FRAME_CAUSAL if causal else 0
    if win is None:
        abi.ispa_attn_full_ex(st.ring.c, st.q, st.kc, st.vc, n, 0.0, flags, out, lse)
        ro, rl = at.attn_full(*st.oracle_args(), rows=rows, frame_causal=causal)
    else:
        abi.ispa_attn_local_ex(st.ring.c, Window(*win), st.q, st.kc, st.vc, n, 0.0, flags, out, lse)
        ro, rl = at.attn_local(*st.oracle_args(), *win, rows=rows, frame_causal=causal)
    torch.cuda.synchronize()
    assert abi.ispa_last_device_error()[0] == abi.ISPA_OK
    sel = slice(None) if rows is None else rows
    assert_close_attn(to_f32(out).reshape(n, st.H, st.d)[sel], ro)
    assert np.abs(to_f32(lse)[:, sel] - rl).max() < 2e-3


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("H,P,past,chunk", [(1, 192, 3, 1),     # 4 tiles, none ragged
                                            (2, 100, 9, 1),     # one query tile, ragged segments
                                            (3, 190, 14, 2),    # 380 queries
                                            (1, 1, 600, 1),     # one query, frames of one token
                                            (5, 250, 20, 3)])
def test_small_launches(d, H, P, past, chunk):
    st = Step(100 * H + P, P=P, H=H, d=d, n_past=past, n_chunk_frames=chunk, capacity=past, n_sink_pinned=0)
    _check(st)


@pytest.mark.parametrize("cap,pinned,win", [(8, 1, (1, 3)), (8, 0, (0, 5)), (6, 2, (2, 2)), (9, 1, (0, 8))])
def test_windows_over_a_wrapped_ring(cap, pinned, win):
    # up to three ring segments and the chunk
    st = Step(7 + cap, P=230, H=2, d=128, n_past=17, n_chunk_frames=2, capacity=cap, n_sink_pinned=pinned)
    _check(st, win)


@pytest.mark.parametrize("past", [0, 1, 6])
def test_frame_causal_ranges_that_a_row_never_sees(past):
    # the chunk is most of the keys: the last CTAs' ranges lie wholly past the first frames' own keys
    st = Step(60 + past, P=260, H=2, d=128, n_past=past, n_chunk_frames=6, capacity=6)
    _check(st, causal=True)


@pytest.mark.parametrize("H,P,chunk", [(12, 1560, 1),    # 156 items: 152 and 4
                                       (11, 1920, 1),    # 165: 152 and 13
                                       (4, 1600, 3)])    # 152: no item left over
def test_a_wave_of_whole_items_first(H, P, chunk):
    st = Step(H, P=P, H=H, d=128, n_past=3, n_chunk_frames=chunk, capacity=3)
    n = st.n_q
    rows = np.unique(np.concatenate([[0, 127, 128, n - 1], np.random.default_rng(H).choice(n, 40, False)]))
    _check(st, rows=rows)
