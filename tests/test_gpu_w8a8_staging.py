"""The two shared blocks that a read-back warp of the W8A8 GEMM stores through: a block is written again only
once the store that reads it is done.  A tile of 192 columns has three stores a warp, so the blocks have
to alternate on from one tile of a CTA to the next."""
import pytest

torch = pytest.importorskip("torch")


def _clashes(columns, tiles, carry):
    """Stores of a warp that may find the store before them still reading their block: the warp waits until one
    is pending at most.  `carry`: a tile goes on with the block after the last tile's."""
    order, first = [], 0
    for _ in range(tiles):
        order += [(first + c) & 1 for c in range(columns // 64)]
        first ^= (columns // 64) & 1 if carry else 0
    return [i for i in range(1, len(order)) if order[i] == order[i - 1]]


@pytest.mark.parametrize("columns", [128, 192, 256])
def test_a_pending_store_is_never_on_the_block_written_next(columns):
    assert not _clashes(columns, 5, carry=True)


def test_the_model_sees_a_tile_that_starts_again_on_the_first_block():
    assert _clashes(192, 3, carry=False) == [3, 6]


@pytest.mark.gpu
@pytest.mark.parametrize("T,D,Do", [(9400, 128, 1152), (9400, 256, 1152), (6000, 128, 1920)])
def test_several_tiles_of_192_columns_a_cta(T, D, Do):
    # 192 divides D_out and 256 doesn't: three tiles and more a CTA, one or two k-blocks each.  One chain of D
    # terms in fp32 (exact products), two fp32 multiplies, bf16 rounding; every call the same bits.
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00712_gb300 import abi
    from paper_2607_00712_gb300.build import build_library
    build_library()
    g = torch.Generator(device="cuda")
    g.manual_seed(T + D)
    a, w = (torch.randn(n, D, generator=g, device="cuda").to(torch.float8_e4m3fn) for n in (T, Do))
    sa, sw = (torch.rand(n, generator=g, device="cuda") + 0.5 for n in (T, Do))
    exact = (a.double() @ w.double().t()) * sa.double()[:, None] * sw.double()
    mag = (a.double().abs() @ w.double().abs().t()) * sa.double()[:, None] * sw.double()
    first = None
    for _ in range(40):
        out = torch.full((T, Do), float("nan"), dtype=torch.bfloat16, device="cuda")
        abi.ispa_linear_w8a8(a.view(torch.uint8), sa, w.view(torch.uint8), sw, T, D, Do, out)
        if first is None:
            first = out
            err = (out.double() - exact).abs() - (2.0 ** -8 * exact.abs() + (D + 6) * 2.0 ** -24 * mag)
            assert not bool(err.isnan().any()) and float(err.max()) <= 0
        assert torch.equal(out, first)
    assert abi.ispa_last_device_error()[0] == abi.ISPA_OK
