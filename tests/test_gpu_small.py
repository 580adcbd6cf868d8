"""One-launch kernels of small single instances against the launch sequence: same RHS and same
integrations bit for bit, whatever the mask, the method, the attempts per launch and the padding."""
import numpy as np
import pytest
import torch

import rtbte_inputs as ri

pytestmark = pytest.mark.gpu

MODELS = {
    "toy6": lambda: ri.toy2d(6),        # fewer items than CTAs
    "toy11": lambda: ri.toy2d(11),      # N_q not a multiple of 4
    "toy30": lambda: ri.toy2d(30),      # 3600 rows: more than 8 rows to a chunk of the error norm
    "graphene27": lambda: ri.graphene(27, sigma_eph=0.05, sigma_pp=0.006),
    "ladder3d": lambda: ri.ladder3d(4),  # folded grid
    "graphene66": lambda: ri.graphene(66, sigma_eph=0.0075, sigma_pp=0.00075),  # lists and populations past a CTA's memory
}


def _state(m, seed):
    rng = np.random.default_rng(seed)
    y = m.y0() * (1.0 + 0.01 * rng.random(m.n_y))
    y[:m.n_c] = np.clip(y[:m.n_c], 0.0, 1.0)
    return torch.tensor(y, device="cuda")


@pytest.mark.parametrize("name", list(MODELS))
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_one_launch_rhs_equals_the_launch_sequence(name, precision):
    import paper_2412_13402_gb300 as rt

    m, other = MODELS[name](), ri.toy2d(5)
    one = rt.Context(m, precision=precision)
    one.upload_channels()
    two = rt.Context([m, other], precision=precision)  # several instances take the launch sequence
    two.upload_channels(0)
    two.upload_channels(1)
    y = _state(m, 4)
    y2 = torch.cat([y, torch.tensor(other.y0(), device="cuda")])
    for mask in range(1, 8):
        want = two.rhs(y2, parts=mask)[:m.n_y]
        assert torch.equal(one.rhs(y, parts=mask), want)
    z = y.clone()
    one.rhs(z, z)  # in place
    assert torch.equal(z, want)
    one.close()
    two.close()


@pytest.mark.parametrize("name", list(MODELS))
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("opts", [dict(method="bs32", rtol=1e-6), dict(method="zon43", rtol=1e-5),
                                  dict(method="zon43", rtol=1e-5, h0=0.02),  # the first attempts are rejected
                                  dict(method="rk4", h=5e-5), dict(method="mri", rtol=1e-5, h_s=0.002)],
                         ids=["bs32", "zon43", "rejected", "rk4", "mri"])
def test_one_launch_attempts_equal_the_launch_sequence(name, precision, opts):
    import paper_2412_13402_gb300 as rt

    m = MODELS[name]()
    ctx = rt.Context(m, precision=precision)
    ctx.upload_channels()
    got = []
    for graphs, chunk in ((True, 0), (True, 1), (False, 0)):  # one launch, one attempt a launch, the sequence
        ctx.set_graph_mode(graphs)
        y = _state(m, 9)
        st = ctx.advance_to(0.004, y, t0=0.0, atol_c=1e-9, atol_ph=1e-12, chunk=chunk, **opts)
        got.append((y, {k: st[k] for k in ("rc", "steps", "attempts", "fails", "t", "h_next", "range_violations")}))
    for y, st in got[:2]:
        assert torch.equal(y, got[2][0]) and st == got[2][1]
    assert got[0][1]["rc"] == 0
    ctx.close()
