"""Work units of the collision launch: every parts mask evaluates exactly the items of its parts,
whatever lies between them in the item order, for static and dynamic units and any lane count."""
import numpy as np
import pytest
import torch

import rtbte_inputs as ri

pytestmark = pytest.mark.gpu


def _models(which):
    if which == "toy":  # no ph-ph part at all
        return [ri.toy2d(7)]
    if which == "one":
        return [ri.graphene_small(24)]
    if which == "uneven":  # 4-, 8- and 16-lane groups beside each other, several instances
        return [ri.graphene(n=n, seed=n, sigma_eph=0.05, sigma_pp=0.006) for n in (24, 48, 27, 60)]
    return [ri.silicon(12)]


@pytest.mark.parametrize("which", ["toy", "one", "uneven", "silicon"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_masks_evaluate_exactly_their_parts(which, precision):
    import paper_2412_13402_gb300 as rt

    ms = _models(which)
    ctx = rt.Context(ms, precision=precision)
    for i in range(len(ms)):
        ctx.upload_channels(i)
    y = torch.tensor(np.concatenate([np.concatenate(ri.random_populations(m, 3 + i)) for i, m in enumerate(ms)]),
                     device="cuda")
    one = {p: ctx.rhs(y, parts=p) for p in (1, 2, 4)}
    for mask in (3, 5, 6, 7):
        got = ctx.rhs(y, parts=mask)
        parts = [one[p] for p in (1, 2, 4) if mask & p]
        want, size = sum(parts), sum(p.abs() for p in parts)
        # a row adds the same item partials: parts of different rows are equal bit for bit, a
        # phonon row's ph-e and ph-ph items go into one FP32 head/tail (or FP64) sum of < 2^7
        # terms whose rounding is below 2^-40 of the terms' size
        assert torch.all((got - want).abs() <= 2.0 ** -40 * size)
        if mask == 3:
            assert torch.equal(got, want)
    ctx.close()


@pytest.mark.parametrize("n,stride", [(6, 1), (24, 3), (72, 1)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_rates_equal_the_sums_over_the_lists(n, stride, precision):
    """Linearised ph-ph rates against plain sums over the downloaded list: one vector or less per
    segment, the staged populations, and (31104 FP64 populations at side 72) those in global memory."""
    import paper_2412_13402_gb300 as rt

    m = ri.graphene(n=n, pp_stride=stride, sigma_eph=0.01, sigma_pp=0.0004 if n == 72 else 0.01)
    ctx = rt.Context(m, precision=precision)
    ctx.upload_channels()
    f, N = ri.random_populations(m, 11)
    got = ctx.phph_rates(torch.tensor(np.concatenate([f, N]), device="cuda")).cpu().numpy()
    L = ctx.download_channels(0, rt.RTBTE_PHPH)
    full = m.pp_full_index()
    seg = np.repeat(np.arange(2 * m.n_pp), np.diff(L["off"]))
    Nb, Nc = N[full[L["a"]]], N[full[L["b"]]]
    term = np.where(seg % 2 == 0, Nb + Nc + 1.0, Nc - Nb)
    want, size = np.zeros(m.n_y), np.zeros(m.n_y)
    want[m.n_c + full] = np.bincount(seg // 2, L["W"] * term, m.n_pp)
    size[m.n_c + full] = np.bincount(seg // 2, np.abs(L["W"]) * (Nb + Nc + 1.0), m.n_pp)
    # the list's own weights: FP32 adds the rounding of the two populations (2^-24 each), FP64 that
    # of sums of < 2^13 terms
    assert np.all(np.abs(got - want) <= (2.0 ** -23 if precision == "fp32" else 2.0 ** -40) * size)
    assert len(seg) > 0
    ctx.close()
