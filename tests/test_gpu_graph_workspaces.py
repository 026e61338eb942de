"""A captured FP32 map whose contractions are split over k, replayed after
calls on the same context whose own splits need larger workspaces: the
replay's launches still have theirs."""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_replay_after_larger_calls():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_00756_gb300 import capi
    from paper_2607_00756_gb300.context import BipContext
    from paper_2607_00756_gb300.graphs import GraphedMaps
    cfg = synth.config1()
    sp = synth.make_specimen(cfg)
    V = torch.tensor(sp.V, dtype=torch.float32, device="cuda")
    H = torch.tensor(sp.H, dtype=torch.complex64, device="cuda")
    g = torch.ones(len(sp.scans), dtype=torch.float64, device="cuda")
    ctx = BipContext(cfg, prec="fp32")
    try:
        ctx.build(V, sp.atoms, sp.nch)
        want = ctx.map(H, sp.scans).clone()
        graph = GraphedMaps([(ctx, H, sp.scans)])
        made = capi.bip_debug_allocs()[1]
        for call in (lambda: ctx.cube(V, H, sp.scans), lambda: ctx.grad(H, sp.scans, g, occ=False, V=V)):
            call()
            # what the larger calls let go would be taken by the next allocation
            filled = [torch.full((1 << 20,), 3.0, device="cuda") for _ in range(16)]
            assert torch.equal(graph.replay()[0], want)
            torch.cuda.synchronize()
            graph.check()
            assert all(bool((f == 3.0).all()) for f in filled)
        assert capi.bip_debug_allocs()[1] > made
    finally:
        ctx.close()
