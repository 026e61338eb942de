"""The scan list a call is given, whatever was called before on the context:
a gradient's list does not touch the one a capture-safe context keeps for its
maps, and a captured gradient keeps its own."""
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
    from paper_2607_00756_gb300 import capi
    from paper_2607_00756_gb300.context import BipContext
    sp = synth.make_specimen(synth.config1())
    V = torch.tensor(sp.V, dtype=torch.float32, device="cuda")
    H = torch.tensor(sp.H, dtype=torch.complex64, device="cuda")
    other = sp.scans[::-1] * 0.5 + 3.0
    g = torch.linspace(-1.0, 1.0, len(sp.scans), dtype=torch.float64, device="cuda")

    def make(prec):
        ctx = BipContext(sp.cfg, prec=prec)
        ctx.build(V, sp.atoms, sp.nch)
        return ctx

    return capi, make, sp, np.ascontiguousarray(other), H, g


@pytest.mark.parametrize("prec,order,raster", [("fp32", 0, True), ("mixed", 0, True), ("mixed", 0, False), ("mixed", 1, True),
                                               ("mixed", 2, True)])
def test_map_after_a_gradient_on_other_scans(env, prec, order, raster):
    capi, make, sp, other, H, g = env
    ctx = make(prec)
    try:
        capi.bip_set_capture_safe(ctx.ctx, 1)
        ctx.set_order(order)
        ctx.set_raster_eval(raster)
        a = ctx.map(H, sp.scans).clone()
        ctx.grad(H, other, g, occ=False, aberr=False)
        b = ctx.map(H, sp.scans)
        assert torch.equal(a, b)
        # the Gram order straight after: its phase tables are of these scans
        ctx.set_order(0)
        c = ctx.map(H, sp.scans)
        capi.bip_check_errors(ctx.ctx)
        assert float((c - a).norm() / a.norm()) < 1e-3
    finally:
        ctx.close()


def test_captured_gradient_keeps_its_scans(env):
    """The host list may change (or go) after the capture, and calls on other
    scans may come between the replays."""
    capi, make, sp, other, H, g = env
    ctx = make("fp32")
    try:
        want = ctx.grad(H, sp.scans, g, occ=False, aberr=False)["H"]
        torch.cuda.synchronize()
        host = sp.scans.copy()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
            got = ctx.grad(H, host, g, occ=False, aberr=False)["H"]
        host[:] = other
        for between in (False, True):
            if between:
                ctx.grad(H, other, g, occ=False, aberr=False)
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(torch.view_as_real(got), torch.view_as_real(want))
        capi.bip_check_errors(ctx.ctx)
    finally:
        ctx.close()


@pytest.mark.parametrize("name", ["map", "sites", "grad", "cube"])
def test_host_list_may_change_when_the_call_returns(env, name):
    """A scan list in page-locked memory, from which the device copies at its
    own time, overwritten as soon as an FP32 call behind other work has
    returned."""
    capi, make, sp, other, H, g = env
    V = torch.tensor(sp.V, dtype=torch.float32, device="cuda")
    ctx = make("fp32")
    call = {"map": lambda s: ctx.map(H, s), "sites": lambda s: ctx.sites(H, s), "cube": lambda s: ctx.cube(V, H, s),
            "grad": lambda s: torch.view_as_real(ctx.grad(H, s, g, occ=False, aberr=False)["H"])}[name]
    try:
        want = call(sp.scans)
        pinned = torch.tensor(sp.scans).pin_memory()
        torch.cuda.synchronize()
        torch.cuda._sleep(400_000_000)
        got = call(pinned.numpy())
        pinned.copy_(torch.tensor(other))
        torch.cuda.synchronize()
        assert torch.equal(got, want)
        capi.bip_check_errors(ctx.ctx)
    finally:
        ctx.close()
