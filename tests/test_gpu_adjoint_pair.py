"""The two adjoint sweeps of dL/dV run side by side on two streams when both
are there, and S2's alone when every site lies in the first slice.  Against
the oracle's reverse pass (the bound of tests/test_gpu_grad.py, 1e-4), and,
as nothing in the sums depends on the streams, the same bits on every call:
on a fresh context, repeated, and on a stream of the caller's while V is
freed and its memory used again straight after the call."""
import numpy as np
import pytest

import synth
from oracle import bip as obip
from oracle import grad as og

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("slices", [(0, 1), (1, 6), (0, 8)])
def test_sweeps_side_by_side(slices):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00756_gb300.context import BipContext
    cfg = synth.config1().replace(name="pair", ny=64, nx=64, ly=5.0, lx=5.0, nz=8, cells_y=2, cells_x=2, win=32,
                                  fy=2, fx=2, ion_slices=slices, ion_cells=(0, 1), scan_y=(10.0, 6.0, 4),
                                  scan_x=(12.0, 5.0, 4))
    sp = synth.make_specimen(cfg)
    pr = obip.make_problem(sp)
    par = og.Params(pr)
    gI = 0.2 * og.forward(pr, par) * np.random.default_rng(3).standard_normal(len(sp.scans))
    _, want = og.gradients(pr, par, dL_dI=gI)
    dev = torch.device("cuda:0")
    H = torch.tensor(sp.H, dtype=torch.complex64, device=dev)
    g = torch.tensor(gI, device=dev)
    host = torch.tensor(sp.V, dtype=torch.float32).pin_memory()
    first = None
    for _ in range(2):
        ctx = BipContext(cfg, prec="fp32")
        try:
            ctx.build(host.to(dev), sp.atoms, sp.nch)
            torch.cuda.synchronize()
            stream = torch.cuda.Stream()
            for where in (torch.cuda.current_stream(), stream, stream):
                with torch.cuda.stream(where):
                    V = host.to(dev, non_blocking=True)
                    got = ctx.grad(H, sp.scans, g, occ=False, h=False, aberr=False, V=V)["V"]
                    del V
                    torch.full((cfg.nz, cfg.ny, cfg.nx), float("nan"), device=dev)
                    out = got.cpu().numpy()
                where.synchronize()
                if first is None:
                    first = out
                    assert np.linalg.norm(out - want["V"]) < 1e-4 * np.linalg.norm(want["V"])
                assert np.array_equal(out, first)
        finally:
            ctx.close()


@pytest.mark.parametrize("safe", [0, 1])
def test_fp32_calls_can_be_captured(safe):
    """An FP32 context's coupling and derivatives (both adjoint sweeps) as a
    CUDA graph after one call as warm-up, capture-safe or not: a replay gives
    the call's bits, and the flag of a wait that ran out stays readable."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00756_gb300 import capi
    from paper_2607_00756_gb300.context import BipContext
    cfg = synth.config1()
    sp = synth.make_specimen(cfg)
    dev = torch.device("cuda:0")
    V = torch.tensor(sp.V, dtype=torch.float32, device=dev)
    H = torch.tensor(sp.H, dtype=torch.complex64, device=dev)
    g = torch.linspace(-1.0, 1.0, len(sp.scans), dtype=torch.float64, device=dev)
    ctx = BipContext(cfg, prec="fp32")
    try:
        ctx.build(V, sp.atoms, sp.nch)
        capi.bip_set_capture_safe(ctx.ctx, safe)

        def call():
            d = ctx.grad(H, sp.scans, g, occ=False, aberr=False, V=V)
            return d["V"], d["H"], ctx.coupling(H, 0)

        want = call()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
            got = call()
        graph.replay()
        torch.cuda.synchronize()
        for a, b in zip(got, want):
            a, b = (torch.view_as_real(t) if t.is_complex() else t for t in (a, b))
            assert float(b.abs().max()) > 0 and torch.equal(a, b)
        capi.bip_check_errors(ctx.ctx)
    finally:
        ctx.close()
