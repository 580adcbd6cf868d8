"""Grid-barrier waits of the one-launch attempt loop that give up: whichever CTAs notice, the call
fails with RTBTE_E_TIMEOUT and the state and time its launch started from, or gives the whole result."""
import pytest
import torch

import rtbte_inputs as ri

pytestmark = pytest.mark.gpu

E_TIMEOUT = -8


def _advance(ctx, y, t, **opts):
    """(return code, statistics) of one call."""
    import paper_2412_13402_gb300 as rt

    st = rt.Stats()
    try:
        ctx.advance_to(t, y, rt.integ_options(t0=0.0, **opts), st)
    except rt.RtbteError as e:
        return e.code, st
    return st.status, st


@pytest.mark.parametrize("n", [12, 18])  # up to 8 rows to a chunk of the error norm, and more (one more barrier)
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_a_wait_that_gives_up_fails_with_the_state_before(n, precision):
    import paper_2412_13402_gb300 as rt

    m = ri.toy2d(n)
    ctx = rt.Context(m, precision=precision)
    ctx.upload_channels()
    y0 = torch.tensor(m.y0(), device="cuda")

    def run(polls):
        ctx.set_wait_limit(polls)
        y = y0.clone()
        before = ctx.launch_count()
        rc, st = _advance(ctx, y, 0.004, method="bs32", rtol=1e-6, atol_c=1e-10, atol_ph=1e-13, h0=2e-4)
        return y, rc, st, ctx.launch_count() - before

    want, rc, ref, launches = run(-1)
    assert rc == 0 and 2 <= ref.attempts <= 64
    assert launches == 2  # the first step armed, then one launch of the attempt loop
    seen = set()
    for polls in [0, 0] + [p for p in range(1, 65) for _ in range(4)]:
        y, rc, st, _ = run(polls)
        seen.add(rc)
        assert rc in (0, E_TIMEOUT) and st.status == rc
        if rc == 0:
            assert torch.equal(y, want) and st.t == 0.004
        else:
            assert torch.equal(y, y0) and st.t == 0.0 and st.steps == 0
    assert E_TIMEOUT in seen
    y, rc, st, _ = run(-1)  # the context goes on working
    assert rc == 0 and torch.equal(y, want)
    ctx.close()


def test_a_multirate_call_reports_it_too():
    import paper_2412_13402_gb300 as rt

    m = ri.toy2d(12)
    ctx = rt.Context(m, precision="fp64")
    ctx.upload_channels()
    y0 = torch.tensor(m.y0(), device="cuda")
    y = y0.clone()
    ctx.set_wait_limit(0)
    assert _advance(ctx, y, 0.004, method="mri", h_s=0.002)[0] == E_TIMEOUT and torch.equal(y, y0)
    ctx.set_wait_limit(-1)
    assert _advance(ctx, y, 0.004, method="mri", h_s=0.002)[0] == 0
    ctx.close()
