"""The 8-bit quantisers and appends at the edges of their blocks (128 tokens of d-major values, four
words a thread, frames inside a block), codes bit for bit against the oracle's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import keysets as ks  # noqa: E402
from oracle import quant as qt  # noqa: E402
from paper_2607_00712_gb300 import abi, synth  # noqa: E402
from paper_2607_00712_gb300.device import Ring, bf16_tensor  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00712_gb300.build import build_library
    build_library()
    abi.lib()


def _x(seed, n, H, d):
    g = np.random.default_rng(seed)
    return synth.bf16_round((g.standard_normal((n, H, d)) * np.exp(g.standard_normal((1, H, 1)))).astype(np.float32))


@pytest.mark.parametrize("n,H", [(1, 1), (3, 2), (4, 1), (5, 3), (127, 2), (128, 1), (129, 3), (1563, 2)])
def test_values_d_major(n, H):
    x = _x(n, n, H, 128)
    sc = (qt.head_scales(x) * np.float32(0.9)).astype(np.float32)
    ld = (n + 15) // 16 * 16 + 16
    out = torch.full((H, 128, ld), 0xCD, dtype=torch.uint8, device="cuda")
    abi.ispa_quantize_vt_e4m3(bf16_tensor(x), n, H, 128, torch.from_numpy(sc).cuda(), out, ld)
    got = out.cpu().numpy()
    assert np.array_equal(got[:, :, :n], qt.quantize_heads_with_scale(x, sc).transpose(1, 2, 0))
    assert (got[:, :, n:] == 0xCD).all()


@pytest.mark.parametrize("n,H,d", [(1, 1, 16), (7, 3, 48), (128, 1, 64), (65, 5, 128), (129, 2, 256)])
def test_queries_and_keys(n, H, d):
    x = _x(n + d, n, H, d)
    sc = (qt.head_scales(x) * np.float32(0.9)).astype(np.float32)
    guard = 64
    k8 = torch.full((n * H * d + guard,), 0xCD, dtype=torch.uint8, device="cuda")
    abi.ispa_quantize_k_e4m3(bf16_tensor(x), n, H, d, torch.from_numpy(sc).cuda(), k8)
    got = k8.cpu().numpy()
    assert np.array_equal(got[:-guard].reshape(n, H, d), qt.quantize_heads_with_scale(x, sc))
    q8 = torch.full((n * H * d + guard,), 0xCD, dtype=torch.uint8, device="cuda")
    qs = torch.empty(H, (n + 127) // 128, dtype=torch.float32, device="cuda")
    abi.ispa_quantize_q_e4m3(bf16_tensor(x), n, H, d, q8, qs)
    want, want_s = qt.quantize_query_blocks(x)
    got_q = q8.cpu().numpy()
    assert np.array_equal(got_q[:-guard].reshape(n, H, d), want) and np.array_equal(qs.cpu().numpy(), want_s)
    assert (got[-guard:] == 0xCD).all() and (got_q[-guard:] == 0xCD).all()


@pytest.mark.parametrize("P,H,n_frames,cap,written", [(4, 1, 3, 5, 4), (12, 3, 16, 17, 9), (128, 2, 1, 3, 5), (132, 2, 3, 4, 1)])
def test_append_into_wrapped_slots(P, H, n_frames, cap, written):
    # the d-major values of several frames share one block when P < 128, and slots wrap inside it
    k, v = _x(P, n_frames * P, H, 128), _x(P + 1, n_frames * P, H, 128)
    ksc, vsc = (qt.head_scales(t).astype(np.float32) for t in (k, v))
    dev = [torch.from_numpy(t).cuda() for t in (ksc, vsc)]
    for kv8 in (True, False):
        ring = Ring(H, 128, P, cap, 1, k_e4m3=not kv8, kv_e4m3=kv8)
        ring.c.frames_written = written
        if kv8:
            abi.ispa_kv_append_kv8(ring.c, bf16_tensor(k), bf16_tensor(v), n_frames, *dev)
        else:
            abi.ispa_kv_append_qk8(ring.c, bf16_tensor(k), bf16_tensor(v), n_frames, dev[0])
        kr, vr = ring.k.cpu().numpy(), ring.v.float().cpu().numpy() if not kv8 else ring.v.cpu().numpy()
        want_k, want_v = qt.quantize_heads_with_scale(k, ksc), qt.quantize_heads_with_scale(v, vsc)
        for i in range(n_frames):
            sl = ks.ring_slot(written + i, cap, 1)
            rows, src = slice(sl * P, (sl + 1) * P), slice(i * P, (i + 1) * P)
            assert np.array_equal(kr[:, rows], want_k[src].transpose(1, 0, 2))
            if kv8:
                assert np.array_equal(vr[:, :, rows], want_v[src].transpose(1, 2, 0))
            else:
                assert np.array_equal(vr[:, rows], v[src].transpose(1, 0, 2))
        untouched = [s for s in range(cap) if s not in {ks.ring_slot(written + i, cap, 1) for i in range(n_frames)}]
        for s in untouched:
            assert (kr[:, s * P:(s + 1) * P] == 0).all()
            assert (vr[:, :, s * P:(s + 1) * P] == 0).all() if kv8 else (vr[:, s * P:(s + 1) * P] == 0).all()
