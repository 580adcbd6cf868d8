"""Device memory of a training batch: the buffers its engine reads, and no others."""
import numpy as np
import pytest

import rtbte_inputs as ri

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_implicit_convolutions_hold_no_buffers_of_the_column_engine():
    import paper_2412_13402_gb300 as rt

    m = ri.graphene(120)
    ctx = rt.Context(m, precision="fp32")
    ctx.upload_channels()
    s = rt.Surrogate(ctx, width=64, capacity=1, seed=1)
    ny, nx, C = s.nq_s[1], s.nq_s[0], m.nmodes

    def grow(B):
        x = np.zeros((B, ny, nx, C), np.float32)
        before = torch.cuda.mem_get_info()[0]
        s.loss_grad(x, x)
        return before - torch.cuda.mem_get_info()[0]

    grow(1)
    B = 256
    P = B * ny * nx
    # per point: x, t, out and its gradient in FP32 and BF16; two BF16 gradients, five FP32 gradients and five
    # activations in both precisions of 64 channels; columns of the first layer (9 C rounded up to 32)
    need = P * (C * (2 + 4 + 4 + 4 + 2) + 64 * (2 * 2 + 5 * 4 + 5 * (4 + 2)) + 2 * ((9 * C + 31) // 32 * 32))
    # whole 2 MB blocks for each buffer, and the one-sample buffers given back; a 64-channel FP32 buffer is 105 MB
    assert need - 16e6 < grow(B) < need + 64e6
    s.close()
    ctx.close()
