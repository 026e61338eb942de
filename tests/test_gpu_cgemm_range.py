"""The FP32 complex contraction (bip_debug_cgemm) at the ends of the FP32
range, the largest finite elements and infinite ones, and the triangle of a
product that is not square."""
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
    ctx = BipContext(synth.config1(), prec="fp32")
    yield capi, ctx.ctx
    ctx.close()


def operands(layout, M, N, K):
    """[M, K] and [N, K] with parts of magnitude 0.5 to 1, and the strides
    of their storage, k or row contiguous."""
    rng = torch.Generator("cuda").manual_seed(5)
    out = []
    for rows, lay in ((M, layout[0]), (N, layout[1])):
        x = torch.rand(rows, K, 2, device="cuda", generator=rng) * 0.5 + 0.5
        x *= torch.where(torch.rand(x.shape, device="cuda", generator=rng) < 0.5, -1.0, 1.0)
        t = torch.view_as_complex(x)
        out.append((t, (K, 1, 0, 0)) if lay == "k" else (t.T.contiguous(), (1, rows, 0, 0)))
    return out


def call(env, A, sA, B, sB, M, N, K):
    capi, ctx = env
    C = torch.full((M, N), float("nan"), dtype=torch.complex64, device="cuda")
    capi.bip_debug_cgemm(ctx, M, N, K, 1, 1, A, sA, B, sB, 0, None, C)
    return C


@pytest.mark.parametrize("layout", ["kk", "rr", "kr"])
@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("big", [torch.finfo(torch.float32).max, torch.finfo(torch.float32).min, 3.3965e38, 3.39e38])
def test_largest_finite_elements(env, layout, side, big):
    """Elements up to the largest finite one, whose nearest BF16 is infinite,
    with partners small enough for a finite product: as any other element
    ((K / 16 + 40) 2^-24 of sum |a||b| per entry)."""
    M, N, K = 130, 40, 50
    (A, sA), (B, sB) = operands(layout, M, N, K)
    ts = [A, B]
    ts[1 - side].mul_(2.0 ** -12)
    rows = (M, N)[side]
    t = ts[side] if layout[side] == "k" else ts[side].T
    t[3, 7] = big
    t[rows - 1, K - 1] = complex(0.25, big)
    a, b = (x if lay == "k" else x.T for x, lay in zip(ts, layout))
    C = call(env, A, sA, B, sB, M, N, K)
    a, b = a.to(torch.complex128), b.to(torch.complex128)
    assert torch.all((C - a @ b.T).abs() <= (K / 16 + 40) * 2.0 ** -24 * (a.abs() @ b.abs().T))


@pytest.mark.parametrize("layout", ["kk", "rr", "kr"])
@pytest.mark.parametrize("side", [0, 1])
def test_infinite_elements(env, layout, side):
    """An infinite real or imaginary part gives what its products give, an
    infinity of their sign in both parts of C."""
    M, N, K = 130, 40, 50
    (A, sA), (B, sB) = operands(layout, M, N, K)
    ts = [A, B]
    rows = (M, N)[side]
    t = ts[side] if layout[side] == "k" else ts[side].T
    inf = float("inf")
    t[3, 7] = complex(inf, 0.5)
    t[rows - 1, K - 1] = complex(-0.5, -inf)
    a, b = (torch.view_as_real(x if lay == "k" else x.T).double() for x, lay in zip(ts, layout))
    # the real products one by one (a complex one in PyTorch makes NaN of inf)
    re = (a[:, None, :, 0] * b[None, :, :, 0]).sum(-1) - (a[:, None, :, 1] * b[None, :, :, 1]).sum(-1)
    im = (a[:, None, :, 0] * b[None, :, :, 1]).sum(-1) + (a[:, None, :, 1] * b[None, :, :, 0]).sum(-1)
    C = torch.view_as_real(call(env, A, sA, B, sB, M, N, K)).double()
    for got, want in ((C[..., 0], re), (C[..., 1], im)):
        assert torch.isinf(want).sum() == 2 * (N if side == 0 else M)
        assert torch.equal(torch.isinf(got), torch.isinf(want)) and not torch.isnan(got).any()
        assert torch.equal(got[torch.isinf(want)], want[torch.isinf(want)])


@pytest.mark.parametrize("M,N", [(512, 256), (300, 129), (1000, 40), (129, 500)])
def test_upper_triangle_of_a_rectangle(env, M, N):
    """Flag 4 with more rows than columns, and with fewer: every entry on or
    above the diagonal is written."""
    capi, ctx = env
    K = 48
    (A, sA), (B, sB) = operands("kk", M, N, K)
    C = torch.full((M, N), float("nan"), dtype=torch.complex64, device="cuda")
    capi.bip_debug_cgemm(ctx, M, N, K, 1, 1, A, sA, B, sB, 4, None, C)
    a, b = A.to(torch.complex128), B.to(torch.complex128)
    up = torch.ones(M, N, dtype=torch.bool, device="cuda").triu()
    assert torch.all((C - a @ b.T).abs()[up] <= ((K / 16 + 40) * 2.0 ** -24 * (a.abs() @ b.abs().T))[up])
