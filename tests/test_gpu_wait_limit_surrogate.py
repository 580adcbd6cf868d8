"""Waits of the tensor-core kernels that give up: the call fails with RTBTE_E_TIMEOUT or gives the
whole result, and the kernel has let its copies and products end, so the device goes on working."""
import numpy as np
import pytest

import rtbte_inputs as ri

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

E_TIMEOUT = -8


@pytest.mark.parametrize("width,B", [(64, 17), (64, 300), (24, 300)])  # up to nine slices of 64 points to a split
def test_a_wait_that_gives_up_fails_and_leaves_the_device_working(width, B):
    import paper_2412_13402_gb300 as rt

    m = ri.graphene_small(33)
    ctx = rt.Context(m, precision="fp32")
    ctx.upload_channels()
    rng = np.random.default_rng(5)
    x = rng.standard_normal((B, 11, 11, m.nmodes)).astype(np.float32)
    t = (0.3 * rng.standard_normal(x.shape)).astype(np.float32)

    def run(polls):
        s = rt.Surrogate(ctx, width=width, capacity=1, seed=3)
        ctx.set_wait_limit(polls)
        try:
            return s.loss_grad(x, t)
        except rt.RtbteError as e:
            assert e.code == E_TIMEOUT
            return None
        finally:
            ctx.set_wait_limit(-1)
            s.close()

    want = run(-1)
    assert want is not None and run(0) is None
    for polls in [1, 2, 3, 4, 6, 8, 12, 16, 32, 64, 256] * 2:
        got = run(polls)
        if got is not None:
            assert got[0] == want[0] and np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2])
    again = run(-1)
    assert again[0] == want[0] and np.array_equal(again[1], want[1]) and np.array_equal(again[2], want[2])
    ctx.close()
