"""The exact cube's beams through their sweeps in chunks: the memory the cube
may take decides how many beams a chunk has, and no value depends on it."""
import numpy as np
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
    from paper_2607_00756_gb300.context import BipContext
    return BipContext


@pytest.mark.parametrize("prec", ["fp32", "split_bf16", "mixed"])
@pytest.mark.parametrize("n", [128, 256, 512])
def test_bits_do_not_depend_on_the_chunk(env, n, prec):
    """208 beams in one chunk, in chunks of 160 and 48, of 64 and of 32, on
    rows of 128, 256 and 512 points; the sums over the window split or not."""
    L = 10.0 * n / 128
    cells = int(L / 2.5)
    cfg = synth.config1().replace(ny=n, nx=n, ly=L, lx=L, cells_y=cells, cells_x=cells, ion_cells=(cells // 2 - 1, cells // 2 + 1),
                                  fy=n // 64, fx=n // 64, cube_ky=16, cube_kx=13, scan_y=(n / 2 - 8, 3.0, 6),
                                  scan_x=(n / 2 - 8, 3.5, 5))
    sp = synth.make_specimen(cfg)
    V = torch.tensor(sp.V, dtype=torch.float32, device="cuda")
    H = torch.tensor(sp.H, dtype=torch.complex64, device="cuda")
    ctx = env(cfg, prec=prec)
    try:
        ctx.build(V, sp.atoms, sp.nch)
        per_beam = (ctx.n_sites * cfg.win ** 2 + n * n) * 8
        got = []
        for beams in (0, 160, 64, 32):
            ctx.set_cube_memory(beams * per_beam + (beams > 0))
            got.append(ctx.cube(V, H, sp.scans).cpu().numpy())
    finally:
        ctx.close()
    assert got[0].shape[1] == 208 and got[0].max() > 0
    for g in got[1:]:
        assert np.array_equal(g, got[0])


@pytest.mark.parametrize("first,then", [(0, 32), (32, 0), (160, 64)])
def test_nothing_is_left_of_a_cube_with_nan(env, first, then):
    """A cube of transition potentials with a NaN, then one of good ones in
    chunks of another size, on scans that are no raster: only the good one's."""
    cfg = synth.config1().replace(cube_ky=16, cube_kx=13)
    sp = synth.make_specimen(cfg)
    V = torch.tensor(sp.V, dtype=torch.float32, device="cuda")
    H = torch.tensor(sp.H, dtype=torch.complex64, device="cuda")
    scans = sp.scans[:9] + np.random.default_rng(1).random((9, 2))
    ctx = env(cfg, prec="fp32")
    try:
        ctx.build(V, sp.atoms, sp.nch)
        per_beam = (ctx.n_sites * cfg.win ** 2 + cfg.ny * cfg.nx) * 8
        memory = {b: b * per_beam + (b > 0) for b in (first, then)}
        ctx.set_cube_memory(memory[then])
        want = ctx.cube(V, H, scans).cpu().numpy()
        bad = H.clone()
        bad[:, 5, 7] = float("nan")
        ctx.set_cube_memory(memory[first])
        assert not np.isfinite(ctx.cube(V, bad, scans).cpu().numpy()).all()
        ctx.set_cube_memory(memory[then])
        assert np.array_equal(ctx.cube(V, H, scans).cpu().numpy(), want)
    finally:
        ctx.close()
