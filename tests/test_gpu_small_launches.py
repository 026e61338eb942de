"""Few sites, few scans: the launch shapes that fill the chip there (split
contractions, small reconstruction units, narrow raster blocks) against the
general ones."""
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
    cfg = synth.config1()
    sp = synth.make_specimen(cfg)
    V = torch.tensor(sp.V, dtype=torch.float32, device="cuda")
    H = torch.tensor(sp.H, dtype=torch.complex64, device="cuda")
    return BipContext, cfg, sp, V, H


def raster(my, mx, step):
    y, x = 20.0 + step * np.arange(my), 11.5 + step * np.arange(mx)
    return np.stack(np.meshgrid(y, x, indexing="ij"), -1).reshape(-1, 2)


@pytest.mark.parametrize("my,mx,step", [(1, 1, 1.0), (1, 130, 0.75), (16, 16, 4.0), (70, 65, 1.25), (3, 200, 0.5), (129, 64, 0.5),
                                        (5, 20000, 0.005)])
def test_raster_blocks(env, my, mx, step):
    """Rasters of every block shape: as Horner's rule per scan to 1e-5, and
    bit for bit as the same raster off by 1e-10 px past its first row and
    column (the per-scan crop test), away from the crop's edge."""
    BipContext, cfg, sp, V, H = env
    scans = raster(my, mx, step)
    off = scans.copy()
    if my > 1 and mx > 1:
        off.reshape(my, mx, 2)[1:, 1:] += 1e-10
    ctx = BipContext(cfg, prec="mixed")
    try:
        ctx.build(V, sp.atoms, sp.nch)
        a, b = ctx.sites(H, scans).cpu().numpy(), ctx.sites(H, off).cpu().numpy()
        ctx.set_raster_eval(False)
        h = ctx.sites(H, scans).cpu().numpy()
    finally:
        ctx.close()
    assert np.array_equal(a == 0, h == 0)
    assert np.linalg.norm(a - h) <= 1e-5 * np.linalg.norm(h)
    same = (a == 0) == (b == 0)
    assert np.array_equal(a[same], b[same]) and same.mean() > 0.99


@pytest.mark.parametrize("prec", ["mixed", "split_bf16", "fp8", "fp32"])
def test_one_site_as_among_many(env, prec):
    """A site by itself (contractions split over K) against the same site
    among seventy-two copies of four sites (whole K per tile)."""
    BipContext, cfg, sp, V, H = env
    ion = np.nonzero(sp.nch > 0)[0]
    reps = 18
    atoms = np.concatenate([sp.atoms[ion]] * reps)
    nch = np.full(len(atoms), 3, dtype=np.int32)
    ctx = BipContext(cfg, prec=prec)
    try:
        ctx.build(V, atoms, nch)
        many = ctx.sites(H.repeat(reps, 1, 1), sp.scans).cpu().numpy()
        ctx.build(V, sp.atoms[ion[:1]], sp.nch[ion[:1]])
        one = ctx.sites(H[:3].contiguous(), sp.scans).cpu().numpy()
    finally:
        ctx.close()
    # FP32 sums in another order; BF16 roundings of M that flip move single
    # entries by 2^-9 of them, 1e-5 of a map of 3 x 193 x 45
    assert np.linalg.norm(one[0] - many[0]) <= 2e-5 * np.linalg.norm(many[0])
    for k in range(4):                                # the first batch and the short last one
        assert np.array_equal(many[k], many[k + 4 * (reps - 1)])


@pytest.mark.parametrize("prec", ["mixed", "split_bf16", "fp8", "fp32"])
def test_batches_do_not_matter(env, prec):
    """Five sites in batches of one to five: the same bits."""
    BipContext, cfg, sp, V, H = env
    ion = np.nonzero(sp.nch > 0)[0][[0, 1, 2, 3, 0]]
    H5 = H[torch.tensor(np.concatenate([[3 * k, 3 * k + 1, 3 * k + 2] for k in (0, 1, 2, 3, 0)]), device="cuda")]
    ctx = BipContext(cfg, prec=prec)
    try:
        ctx.build(V, sp.atoms[ion], sp.nch[ion])
        got = []
        for sb in (0, 1, 2, 3, 5):
            ctx.set_launch(sites_per_batch=sb)
            got.append(ctx.sites(H5.contiguous(), sp.scans).cpu().numpy())
    finally:
        ctx.close()
    for g in got[1:]:
        assert np.array_equal(g, got[0])
