"""The split of a complex64 matrix into BF16 planes (bip_debug_split), bit for
bit against the same roundings in PyTorch: remainders of its 32-row, 64-column
blocks, both source layouts, unaligned rows and destinations, conjugation; what
lies outside the written columns stays."""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00756_gb300 import build
    build.build()
    from paper_2607_00756_gb300 import capi
    from paper_2607_00756_gb300.context import BipContext
    ctx = BipContext(synth.config1(), prec="mixed")
    yield capi, ctx.ctx
    ctx.close()


@pytest.mark.parametrize("rows,cols", [(1, 1), (1, 64), (32, 2), (31, 63), (33, 65), (32, 64), (100, 257), (5, 1000)])
@pytest.mark.parametrize("layout", ["k", "r"])
@pytest.mark.parametrize("pad,dcol0,dpad,skip,conj", [(0, 0, 0, 0, 0), (2, 2, 2, 0, 1), (1, 1, 0, 1, 0), (0, 3, 2, 1, 1)])
def test_planes(env, rows, cols, layout, pad, dcol0, dpad, skip, conj):
    capi, ctx = env
    rng = torch.Generator("cuda").manual_seed(rows * 1000 + cols)
    shape = (rows, cols + pad) if layout == "k" else (cols, rows + pad)
    flat = torch.randn(shape[0] * shape[1] + skip, dtype=torch.complex64, device="cuda", generator=rng)
    flat *= torch.exp(4 * torch.randn(flat.shape, device="cuda", generator=rng))
    src = flat[skip:]
    x = src.view(shape)
    x = x[:, :cols] if layout == "k" else x[:, :rows].T
    x = torch.conj_physical(x) if conj else x
    d_cols = dcol0 + cols + dpad
    dst = torch.full((4, rows, d_cols), 7.0, dtype=torch.bfloat16, device="cuda")
    s = (cols + pad, 1) if layout == "k" else (1, rows + pad)
    capi.bip_debug_split(ctx, rows, cols, src, *s, d_cols, dcol0, conj, dst)
    want = torch.full_like(dst, 7.0)
    for p, part in enumerate((x.real, x.imag)):
        hi = part.to(torch.bfloat16)
        want[2 * p, :, dcol0:dcol0 + cols] = hi
        want[2 * p + 1, :, dcol0:dcol0 + cols] = (part - hi.float()).to(torch.bfloat16)
    assert torch.equal(dst.view(torch.int16), want.view(torch.int16))
