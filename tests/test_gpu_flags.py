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


@pytest.mark.parametrize("report", ["next call", "check_errors", "finite check", "aberrations"])
def test_fp32_give_up_is_reported(env, report):
    """An FP32 call does not wait for its launches: a wait of theirs that ran
    out is reported by the next call on the context, by bip_check_errors, or
    by the call itself where it waits for a result; once, and the context
    stays usable."""
    capi, make, sp, want, V, H = env
    ctx = make("fp32")
    try:
        assert right(ctx, env)
        capi.bip_set_wait_limit(ctx.ctx, 1)
        if report == "finite check":
            ctx.set_check_finite(1)
            timeout(capi, lambda: ctx.map(H, sp.scans))
            ctx.set_check_finite(0)
        elif report == "aberrations":
            g = torch.ones(len(sp.scans), dtype=torch.float64, device="cuda")
            timeout(capi, lambda: ctx.grad(H, sp.scans, g, occ=False, h=False))
        else:
            ctx.map(H, sp.scans)
            torch.cuda.synchronize()
        capi.bip_set_wait_limit(ctx.ctx, 0)
        if report == "next call":
            timeout(capi, lambda: ctx.map(H, sp.scans))
        elif report == "check_errors":
            timeout(capi, lambda: capi.bip_check_errors(ctx.ctx))
        capi.bip_check_errors(ctx.ctx)
        assert right(ctx, env)
    finally:
        ctx.close()


@pytest.mark.parametrize("name", ["map", "sites", "coupling", "grad", "cube", "qeels"])
def test_fp32_calls_return_with_their_work_queued(env, name):
    """Behind 0.2 s of other work on the stream a warmed-up call returns
    before that work is done."""
    from paper_2607_00756_gb300.context import BipContext
    capi, make, sp, want, V, H = env
    g = torch.ones(len(sp.scans), dtype=torch.float64, device="cuda")
    ctx = make("fp32")
    if name == "qeels":
        ctx.close()
        ctx = BipContext(synth.config1().replace(dfy=1), prec="fp32")
        ctx.build(V, sp.atoms, sp.nch)
    call = {"map": lambda: ctx.map(H, sp.scans), "sites": lambda: ctx.sites(H, sp.scans), "coupling": lambda: ctx.coupling(H, 0),
            "grad": lambda: ctx.grad(H, sp.scans, g, occ=True, aberr=False, V=V)["H"], "cube": lambda: ctx.cube(V, H, sp.scans),
            "qeels": lambda: ctx.qeels(H, sp.scans, 0)[1]}[name]
    try:
        a = call()
        torch.cuda.synchronize()
        torch.cuda._sleep(400_000_000)
        b = call()
        done = torch.cuda.Event()
        done.record()
        assert not done.query()
        torch.cuda.synchronize()
        a, b = (torch.view_as_real(t) if t.is_complex() else t for t in (a, b))
        assert torch.equal(a, b)
        capi.bip_check_errors(ctx.ctx)
    finally:
        ctx.close()


def test_map_that_gave_up_leaves_its_output(env):
    """A map that returns BIP_ERR_TIMEOUT has not written map_out."""
    capi, make, sp, want, V, H = env
    ctx = make("mixed")
    try:
        out = torch.full((len(sp.scans),), 7.0, dtype=torch.float64, device="cuda")
        capi.bip_set_wait_limit(ctx.ctx, 1)
        timeout(capi, lambda: ctx.map(H, sp.scans, out=out))
        assert torch.all(out == 7.0)
        capi.bip_set_wait_limit(ctx.ctx, 0)
        assert right(ctx, env)
    finally:
        ctx.close()
