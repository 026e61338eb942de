"""The FP32 complex contraction (bip_debug_cgemm) against complex128 at the
edges of its tiles: single elements, remainders of the 128-row, nt-column and
16-k tiles, split and unsplit k ranges, both operand layouts, unaligned
strides, weights, conjugation, k in blocks, the upper triangle."""
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


def bound(K):
    """Per element, of sum |a||b|: one rounding per chunk of 16 k, and per
    chunk the two full-magnitude tensor-core additions with their alignment
    (16 terms), the dropped products and the elements' 24 bits."""
    return (K / 16 + 40) * 2.0 ** -24


CASES = [
    # M, N, K, blocks, batch, layout of A and B (k or row contiguous), pad of the row length
    (1, 1, 1, 1, 1, "kk", 0), (1, 1, 1, 1, 1, "rr", 0), (128, 128, 16, 1, 1, "kk", 0), (129, 127, 17, 1, 2, "kk", 0),
    (129, 131, 33, 1, 2, "kr", 1), (45, 45, 1000, 1, 3, "rk", 1), (257, 9, 40, 1, 1, "rr", 3), (193, 257, 193, 1, 8, "kr", 0),
    (45, 137, 4096, 1, 4, "kk", 0), (300, 515, 640, 1, 5, "kk", 2), (200, 1032, 45, 3, 2, "rr", 0), (70, 90, 129, 2, 1, "kk", 1),
    (1305, 1515, 64, 1, 1, "kk", 0),
]


def operand(rng, rows, K, blocks, batch, layout, pad):
    """A tensor with [batch][blocks] sheets stored k- or row-contiguous, its
    strides, and its [batch, rows, blocks K] values in complex128."""
    shape = (batch, blocks, rows, K + pad) if layout == "k" else (batch, blocks, K, rows + pad)
    t = torch.randn(*shape, dtype=torch.complex64, device="cuda", generator=rng)
    t *= torch.exp(2 * torch.randn(*shape, device="cuda", generator=rng))
    sheet = shape[2] * shape[3]
    if layout == "k":
        val, s = t[..., :K], (K + pad, 1)
    else:
        val, s = t[..., :rows].transpose(2, 3), (1, rows + pad)
    return t, (*s, blocks * sheet, sheet), val.to(torch.complex128).transpose(1, 2).reshape(batch, rows, blocks * K)


@pytest.mark.parametrize("M,N,K,blocks,batch,layout,pad", CASES)
@pytest.mark.parametrize("flags", [0, 1, 2])
def test_against_complex128(env, M, N, K, blocks, batch, layout, pad, flags):
    capi, ctx = env
    rng = torch.Generator("cuda").manual_seed(M * 7 + N * 3 + K)
    A, sA, a = operand(rng, M, K, blocks, batch, layout[0], pad)
    B, sB, b = operand(rng, N, K, blocks, batch, layout[1], pad)
    w = torch.rand(K, device="cuda", generator=rng) if blocks == 1 and flags == 2 else None
    C = torch.full((batch, M, N), float("nan"), dtype=torch.complex64, device="cuda")
    capi.bip_debug_cgemm(ctx, M, N, K, blocks, batch, A, sA, B, sB, flags, w, C)
    a = a.conj().resolve_conj() if flags & 1 else a
    b = b.conj().resolve_conj() if flags & 2 else b
    if w is not None:
        a = a * w.double()
    want, size = a @ b.transpose(1, 2), a.abs() @ b.abs().transpose(1, 2)
    assert torch.all((C - want).abs() <= bound(blocks * K) * size)


@pytest.mark.parametrize("M,N,K,blocks,batch,layout,pad", CASES[3:9])
def test_transposed_output(env, M, N, K, blocks, batch, layout, pad):
    capi, ctx = env
    rng = torch.Generator("cuda").manual_seed(M + N + K)
    A, sA, _ = operand(rng, M, K, blocks, batch, layout[0], pad)
    B, sB, _ = operand(rng, N, K, blocks, batch, layout[1], pad)
    C = torch.full((batch, M, N), float("nan"), dtype=torch.complex64, device="cuda")
    T = torch.full((batch, N, M), float("nan"), dtype=torch.complex64, device="cuda")
    capi.bip_debug_cgemm(ctx, M, N, K, blocks, batch, A, sA, B, sB, 0, None, C)
    capi.bip_debug_cgemm(ctx, M, N, K, blocks, batch, A, sA, B, sB, 8, None, T)
    assert torch.equal(torch.view_as_real(C), torch.view_as_real(T.transpose(1, 2).contiguous()))


@pytest.mark.parametrize("M", [64, 128, 256, 384, 513])
def test_upper_triangle(env, M):
    """Hermitian products: every column tile that reaches the diagonal or
    lies right of it is written; entries above the diagonal are right."""
    capi, ctx = env
    rng = torch.Generator("cuda").manual_seed(M)
    K, batch = 480, 3
    A, sA, a = operand(rng, M, K, 1, batch, "k", 0)
    C = torch.full((batch, M, M), float("nan"), dtype=torch.complex64, device="cuda")
    capi.bip_debug_cgemm(ctx, M, M, K, 1, batch, A, sA, A, sA, 5, None, C)
    want, size = a.conj() @ a.transpose(1, 2), a.abs() @ a.abs().transpose(1, 2)
    up = torch.ones(M, M, dtype=torch.bool, device="cuda").triu()
    assert torch.all((C - want).abs()[:, up] <= bound(K) * size[:, up])


def test_repeats_bit_for_bit_and_keeps_nonfinite_rows_apart(env):
    """A split k range repeats bit for bit; a NaN or infinite element makes
    its own row non-finite and no other."""
    capi, ctx = env
    rng = torch.Generator("cuda").manual_seed(3)
    M, N, K = 130, 140, 2048
    A, sA, _ = operand(rng, M, K, 1, 1, "k", 0)
    B, sB, _ = operand(rng, N, K, 1, 1, "k", 0)
    C = [torch.empty(1, M, N, dtype=torch.complex64, device="cuda") for _ in range(2)]
    for c in C:
        capi.bip_debug_cgemm(ctx, M, N, K, 1, 1, A, sA, B, sB, 0, None, c)
    assert torch.equal(torch.view_as_real(C[0]), torch.view_as_real(C[1]))
    A[0, 0, 5, 77] = float("nan")
    A[0, 0, 129, 3] = float("inf")
    bad = torch.empty_like(C[0])
    capi.bip_debug_cgemm(ctx, M, N, K, 1, 1, A, sA, B, sB, 0, None, bad)
    fine = torch.isfinite(torch.view_as_real(bad)).all(-1)[0]
    rows = torch.ones(M, dtype=torch.bool, device="cuda")
    rows[[5, 129]] = False
    assert torch.all(fine[rows]) and not torch.any(fine[~rows])
    assert torch.equal(torch.view_as_real(bad[0][rows]), torch.view_as_real(C[0][0][rows]))


@pytest.mark.parametrize("layout", ["k", "r"])
def test_operands_of_more_than_31_bits(env, layout):
    """Rows (or k) 2^24 elements apart: the last lies past 2^31 elements."""
    capi, ctx = env
    rng = torch.Generator("cuda").manual_seed(8)
    far, n, near = 1 << 24, 131, 17
    M, K = (n, near) if layout == "k" else (near, n)
    a = torch.randn(M, K, dtype=torch.complex64, device="cuda", generator=rng)
    t = torch.empty((n - 1) * far + near, dtype=torch.complex64, device="cuda")
    torch.as_strided(t, (n, near), (far, 1)).copy_(a if layout == "k" else a.T)
    s = (far, 1, 0, 0) if layout == "k" else (1, far, 0, 0)
    B, sB, b = operand(rng, 40, K, 1, 1, "k", 0)
    for flags in (0, 8):
        C = torch.full((M, 40) if flags == 0 else (40, M), float("nan"), dtype=torch.complex64, device="cuda")
        capi.bip_debug_cgemm(ctx, M, 40, K, 1, 1, t, s, B, sB, flags, None, C)
        got = C if flags == 0 else C.T
        a2, b2 = a.to(torch.complex128), b[0]
        assert torch.all((got - a2 @ b2.T).abs() <= bound(K) * (a2.abs() @ b2.abs().T))
    C = torch.full((40, M), float("nan"), dtype=torch.complex64, device="cuda")
    capi.bip_debug_cgemm(ctx, 40, M, K, 1, 1, B, sB, t, s, 0, None, C)
    assert torch.all((C - b2 @ a2.T).abs() <= bound(K) * (b2.abs() @ a2.abs().T))
