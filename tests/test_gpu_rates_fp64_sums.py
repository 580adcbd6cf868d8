"""Linearised ph-ph rates are FP64 sums whatever the precision of the lists and populations."""
import dataclasses

import numpy as np
import pytest
import torch

import rtbte_inputs as ri

pytestmark = pytest.mark.gpu


# populations widened in shared memory, held there in FP32 (31104 of them), read from global memory (58806)
@pytest.mark.parametrize("n,sigma", [(24, 1e-3), (72, 1e-5), (99, 1e-5)])
# 1e38: a sum of two leaves the range of FP32; small: subnormal weights beside normal ones
@pytest.mark.parametrize("scale,small", [(1.0, False), (1e-3, False), (1e38, False), (1.0, True)])
def test_rates_of_fp32_lists_are_fp64_sums(n, sigma, scale, small):
    import paper_2412_13402_gb300 as rt

    m = ri.graphene(n=n, pp_stride=1, sigma_eph=0.001, sigma_pp=sigma)
    if small:  # half of the weights below the smallest normal number
        ctx = rt.Context(m, precision="fp32")
        ctx.upload_channels()
        W = np.abs(ctx.download_channels(0, rt.RTBTE_PHPH)["W"])
        ctx.close()
        m = dataclasses.replace(m, v3_coef=m.v3_coef * 2.0 ** -126 / np.median(W[W > 0]))
    ctx = rt.Context(m, precision="fp32")
    ctx.upload_channels()
    f, N = ri.random_populations(m, 11)
    N = (N / N.max() * 2.5 * scale).astype(np.float32).astype(np.float64)  # what the FP32 copies hold
    got = ctx.phph_rates(torch.tensor(np.concatenate([f, N]), device="cuda")).cpu().numpy()
    L = ctx.download_channels(0, rt.RTBTE_PHPH)
    full, W = m.pp_full_index(), L["W"].astype(np.longdouble)
    seg = np.repeat(np.arange(2 * m.n_pp), np.diff(L["off"]))
    Nb, Nc = (N[full[L[k]]].astype(np.longdouble) for k in ("a", "b"))
    term = W * np.where(seg % 2 == 0, Nb + Nc + 1, Nc - Nb)
    if small:
        assert np.any((W > 0) & (W < 2.0 ** -126)) and np.any(W >= 2.0 ** -126)
    rows = seg // 2
    want, size, count = np.zeros(m.n_pp, np.longdouble), np.zeros(m.n_pp, np.longdouble), np.bincount(rows, minlength=m.n_pp)
    np.add.at(want, rows, term)
    np.add.at(size, rows, np.abs(W) * (Nb + Nc + 1))
    # a lane adds at most count / 32 + 32 terms (whole vectors of 4, two segments), the butterfly 5 more;
    # a term has 3 roundings
    bound = (count / 32 + 40) * 2.0 ** -53 * size
    assert np.all(np.isfinite(got)) and len(seg) > 0
    assert np.all(np.abs(got[m.n_c + full] - want) <= bound)
    ctx.close()
