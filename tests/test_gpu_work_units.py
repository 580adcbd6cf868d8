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
        assert torch.all((got - want).abs() <= 2.0 ** -40 * size.clamp(max=float(size.max())) + 0.0 * size)
        if mask == 3:
            assert torch.equal(got, want)
    ctx.close()
