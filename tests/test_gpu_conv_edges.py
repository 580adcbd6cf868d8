"""Implicit-GEMM convolutions of the surrogate at the edges of their tiles, against the mma.sync engine
(im2col columns): sample grids down to 2 x 2, where a tap and its neighbour wrap onto the same point,
and point counts around the 128-row tile and the 64-row K slice of the weight gradients."""
import numpy as np
import pytest

import rtbte_inputs as ri

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b)))


@pytest.mark.parametrize("n,B", [(6, 1), (6, 16), (6, 32), (6, 33), (9, 7), (9, 57), (33, 1), (33, 5), (33, 17)])
def test_edges_match_the_mma_sync_engine(n, B):
    """Both engines multiply the same BF16 operands and differ in accumulation order (about 2^-22
    relative), which flips the BF16 rounding of about one activation in a thousand by 2^-8: 2^-8 *
    sqrt(1e-3) = 1.2e-4 per layer in the L2 norm, 3e-4 over the five layers and twice that again in the
    gradients, which round in both directions.  A wrong neighbour is off by order one."""
    import paper_2412_13402_gb300 as rt

    m = ri.graphene_small(n)
    ctx = rt.Context(m, precision="fp32")
    ctx.upload_channels()
    s = rt.Surrogate(ctx, width=64, capacity=1, seed=n)
    assert tuple(s.nq_s[:2]) == (n // 3, n // 3)
    rng = np.random.default_rng(100 * n + B)
    x = rng.standard_normal((B, n // 3, n // 3, m.nmodes)).astype(np.float32)
    t = (0.3 * rng.standard_normal(x.shape)).astype(np.float32)
    res = []
    for engine in (0, 1):
        s.set_gemm(engine)
        res.append(s.loss_grad(x, t))
    (l0, g0, o0), (l1, g1, o1) = res
    assert _rel(o0, o1) < 1e-3
    assert abs(l0 - l1) < 1e-3 * l1
    assert _rel(g0, g1) < 3e-3
    s.close()
    ctx.close()
