"""The attempt loop of a small instance leaves SMs to other streams: a large context's RHS evaluations
beside it, and several small contexts beside each other, keep their pace."""
import threading
import time

import pytest
import torch

import rtbte_inputs as ri

pytestmark = pytest.mark.gpu


def _small(rt, stream):
    ctx = rt.Context(ri.toy2d(12), precision="fp64")
    ctx.upload_channels()
    ctx.set_stream(stream)
    return ctx


def _integrate(rt, ctx, y0, stream, windows):
    opt = rt.integ_options(method="bs32", t0=0.0, rtol=1e-8, atol_c=1e-15, atol_ph=1e-15)
    st, attempts, done = rt.Stats(), 0, 0
    with torch.cuda.stream(stream):
        y = y0.clone()
        while windows(done):
            y.copy_(y0)
            ctx.advance_to(0.05, y, opt, st)
            attempts += st.attempts
            done += 1
        stream.synchronize()
    return attempts


def test_a_large_rhs_keeps_its_pace_beside_a_small_integration():
    """With every SM taken for 64 attempts at a time (2 ms) an RHS of 110 us took 1.2 ms; with a part of
    them it takes less than twice its time alone."""
    import paper_2412_13402_gb300 as rt

    m = ri.graphene(120)
    s0, s1 = torch.cuda.Stream(), torch.cuda.Stream()
    big = rt.Context(m, precision="fp32")
    big.upload_channels()
    big.set_stream(s0)
    yb = torch.tensor(m.y0(), device="cuda")
    out = torch.empty_like(yb)
    small = _small(rt, s1)
    y0 = torch.tensor(small.models[0].y0(), device="cuda")
    torch.cuda.synchronize()

    def pace():
        with torch.cuda.stream(s0):
            for _ in range(20):
                big.rhs(yb, out)
            s0.synchronize()
            t0 = time.perf_counter()
            for _ in range(300):
                big.rhs(yb, out)
            s0.synchronize()
            return time.perf_counter() - t0

    alone = pace()
    stop = threading.Event()
    th = threading.Thread(target=_integrate, args=(rt, small, y0, s1, lambda n: not stop.is_set()))
    th.start()
    time.sleep(0.05)
    beside = pace()
    stop.set()
    th.join()
    assert beside < 4.0 * alone
    big.close()
    small.close()


def test_small_integrations_run_beside_each_other():
    """Four contexts on four streams take about as long as one (four times as long with every SM taken
    by each)."""
    import paper_2412_13402_gb300 as rt

    streams = [torch.cuda.Stream() for _ in range(4)]
    ctxs = [_small(rt, s) for s in streams]
    y0 = torch.tensor(ctxs[0].models[0].y0(), device="cuda")
    torch.cuda.synchronize()

    def run(n):
        bar = threading.Barrier(n + 1)

        def work(i):
            _integrate(rt, ctxs[i], y0, streams[i], lambda k: k < 1)
            bar.wait()
            _integrate(rt, ctxs[i], y0, streams[i], lambda k: k < 10)

        th = [threading.Thread(target=work, args=(i,)) for i in range(n)]
        for t in th:
            t.start()
        bar.wait()
        t0 = time.perf_counter()
        for t in th:
            t.join()
        return time.perf_counter() - t0

    assert run(4) < 2.0 * run(1)
    for c in ctxs:
        c.close()
