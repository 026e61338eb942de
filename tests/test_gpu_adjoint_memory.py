"""dL/dV on a device with little memory left: one adjoint sweep after the
other in one set of workspaces where two sets do not fit, with the bits of
the two side by side."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MB = 1 << 20


def run(planes, nrad1, leave):
    """dL/dV of two sites' map (one site each in the given slices) with
    leave bytes of the device free beside what the context holds already
    (None: all)."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00756_gb300.context import BipContext
    cfg = synth.config1().replace(name="tight", ny=512, nx=512, ly=40.0, lx=40.0, nz=26, cells_y=16, cells_x=16, fy=4, fx=4,
                                  nrad1=nrad1, win=32, ion_slices=planes, ion_cells=(8, 9), channels=(0,),
                                  scan_y=(250.0, 4.0, 4), scan_x=(250.0, 4.0, 4))
    sp = synth.make_specimen(cfg)
    V = torch.tensor(sp.V, dtype=torch.float32, device="cuda")
    H = torch.tensor(sp.H, dtype=torch.complex64, device="cuda")
    g = torch.linspace(-1.0, 1.0, len(sp.scans), dtype=torch.float64, device="cuda")
    ctx = BipContext(cfg, prec="fp32")
    hold = None
    try:
        ctx.build(V, sp.atoms, sp.nch)
        ctx.grad(H, sp.scans, g, occ=False, aberr=False)
        out = torch.empty_like(V)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        if leave is not None:
            hold = torch.empty(torch.cuda.mem_get_info()[0] - leave - out.nbytes, dtype=torch.uint8, device="cuda")
        out.copy_(ctx.grad(H, sp.scans, g, occ=False, h=False, aberr=False, V=V)["V"])
        return out.cpu().numpy()
    finally:
        ctx.close()
        del hold
        torch.cuda.empty_cache()


def test_memory_for_one_set_only():
    """Sites near the exit surface and more columns on the probe side: S2's
    second set is small and would fit by itself, but not beside S1's."""
    want = run((24, 25), 4, None)
    state = 61 * 512 * 512 * 8
    s1 = (1 + 5 + 5) * state + state // 2             # adjoint, checkpoints, segment, partial sums of 24 slices
    got = run((24, 25), 4, s1 + 64 * MB)              # (S2's set: 200 MB)
    assert np.linalg.norm(got) > 0
    assert np.linalg.norm(got - want) <= 1e-6 * np.linalg.norm(want)


def test_one_after_the_other_gives_the_bits_of_both_at_once():
    """Sites in slices 2 and 22: both sweeps reach the slices between."""
    want = run((2, 23, 20), 2, None)
    state = 19 * 512 * 512 * 8
    one = (1 + 5 + 5) * state + state // 2
    assert np.array_equal(run((2, 23, 20), 2, one + 64 * MB), want)
