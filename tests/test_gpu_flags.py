"""The give-up flag of the contractions: a wait that runs out (a give-up
limit of 1 ns) is reported whichever way the call was made, and reporting it
costs an FP32 call no wait for the stream."""
import numpy as np
import pytest

import synth
from oracle import bip as obip

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
    cfg = synth.config1()
    sp = synth.make_specimen(cfg)
    want = obip.bip_map(obip.make_problem(sp)).map
    V = torch.tensor(sp.V, dtype=torch.float32, device="cuda")
    H = torch.tensor(sp.H, dtype=torch.complex64, device="cuda")

    def make(prec):
        ctx = BipContext(cfg, prec=prec)
        ctx.build(V, sp.atoms, sp.nch)
        return ctx

    return capi, make, sp, want, V, H


def timeout(capi, call):
    with pytest.raises(capi.BipError) as e:
        call()
    assert capi.STATUS[e.value.status] == "BIP_ERR_TIMEOUT"


def right(ctx, env):
    _, _, sp, want, _, H = env
    m = ctx.map(H, sp.scans).cpu().numpy()
    return float(np.linalg.norm(m - want)) < 1e-3 * float(np.linalg.norm(want))


@pytest.mark.parametrize("prec", ["mixed", "fp32"])
def test_flag_outlives_the_next_capture_safe_call(env, prec):
    """A capture-safe map that gave up, then one that did not: the flag is
    there for bip_check_errors, once."""
    capi, make, sp, want, V, H = env
    ctx = make(prec)
    try:
        assert right(ctx, env)
        capi.bip_set_capture_safe(ctx.ctx, 1)
        capi.bip_set_wait_limit(ctx.ctx, 1)
        ctx.map(H, sp.scans)
        capi.bip_set_wait_limit(ctx.ctx, 0)
        ctx.map(H, sp.scans)
        timeout(capi, lambda: capi.bip_check_errors(ctx.ctx))
        capi.bip_check_errors(ctx.ctx)
        assert right(ctx, env)
    finally:
        ctx.close()


def test_flag_outlives_the_next_call_of_a_graph(env):
    """A graph of two FP32 calls whose first gives up at every replay: the
    second's launches leave the flag."""
    capi, make, sp, want, V, H = env
    g = torch.linspace(-1.0, 1.0, len(sp.scans), dtype=torch.float64, device="cuda")
    ctx = make("fp32")
    try:
        def calls():
            capi.bip_set_wait_limit(ctx.ctx, 1)
            ctx.grad(H, sp.scans, g, occ=False, aberr=False)
            capi.bip_set_wait_limit(ctx.ctx, 0)
            ctx.coupling(H, 0)

        ctx.grad(H, sp.scans, g, occ=False, aberr=False)
        ctx.coupling(H, 0)
        torch.cuda.synchronize()
        capi.bip_check_errors(ctx.ctx)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
            calls()
        capi.bip_check_errors(ctx.ctx)
        for _ in range(2):
            graph.replay()
            timeout(capi, lambda: capi.bip_check_errors(ctx.ctx))
        capi.bip_check_errors(ctx.ctx)
        assert right(ctx, env)
    finally:
        ctx.close()
