"""Which launches a context takes, and the same bits on each: the one-launch kernels of small instances
with lists held in shared memory and not, and the collision launch with every tuning and with units
taken at run time.  The path is asserted by the number of launches, so that no comparison can come to
compare a path with itself."""
import dataclasses

import numpy as np
import pytest
import torch

import rtbte_inputs as ri

pytestmark = pytest.mark.gpu

SMEM = 227 * 1024  # shared memory of a CTA


def _graphene(n):
    f = (180.0 / n) ** 0.5
    return ri.graphene(n, sigma_eph=0.020 * f, sigma_pp=0.002 * f)


MODELS = {
    "toy5": lambda: ri.toy2d(5),          # fewer shares than SMs
    "toy12": lambda: ri.toy2d(12),
    "toy18": lambda: ri.toy2d(18),        # 11 rows to a chunk of the error norm
    "graphene24": lambda: _graphene(24),
    "graphene30": lambda: _graphene(30),
    "graphene42": lambda: _graphene(42),  # lists that do not fit beside the populations in FP32
    "toy70": lambda: dataclasses.replace(ri.toy2d(70), sigma_eph=3e-5),  # 157 KB of populations, short lists
    "silicon12": lambda: ri.silicon(12),
}
ALL = 7


def _state(m, seed):
    rng = np.random.default_rng(seed)
    y = m.y0() * (1.0 + 0.01 * rng.random(m.n_y))
    y[:m.n_c] = np.clip(y[:m.n_c], 0.0, 1.0)
    return torch.tensor(y, device="cuda")


def _rhs(ctx, y, launches, parts=ALL):
    before = ctx.launch_count()
    out = ctx.rhs(y, parts=parts)
    assert ctx.launch_count() - before == launches
    return out


def _make(ms, precision):
    import paper_2412_13402_gb300 as rt

    ctx = rt.Context(ms, precision=precision)
    for i in range(len(ctx.models)):
        ctx.upload_channels(i)
    return ctx


@pytest.mark.parametrize("name,precision,one_rhs,one_loop", [
    ("toy5", "fp32", True, True), ("toy5", "fp64", True, True), ("toy12", "fp64", True, True),
    ("toy18", "fp64", True, True), ("graphene24", "fp32", True, True), ("graphene42", "fp32", True, True),
    ("toy70", "fp32", True, True), ("toy70", "fp64", True, True),
    ("graphene30", "fp64", True, False), ("silicon12", "fp32", False, False), ("silicon12", "fp64", False, False)])
def test_the_path_is_the_stated_one_and_gives_the_bits_of_the_launch_sequence(name, precision, one_rhs, one_loop):
    m = MODELS[name]()
    ctx = _make(m, precision)
    y = _state(m, 3)
    want = y.clone()
    before = ctx.launch_count()
    ctx.rhs(want, want)  # in place: populations, collision sums, rows
    assert ctx.launch_count() - before == 3
    assert torch.equal(_rhs(ctx, y, 1 if one_rhs else 3), want)
    if name == "graphene42":  # the largest CTA of the loop holds the mean or more of the lists and rows (88 bytes each)
        ctas = torch.cuda.get_device_properties(0).multi_processor_count / 2
        assert (8 * int(ctx.row_entries(0).sum()) + 88 * m.n_y) / ctas + 4 * (m.n_y + m.n_pp) > SMEM
    got = []
    for graphs in (True, False):
        ctx.set_graph_mode(graphs)
        z, before = y.clone(), ctx.launch_count()
        st = ctx.advance_to(0.003, z, method="zon43", t0=0.0, rtol=1e-6, atol_c=1e-10, atol_ph=1e-13, h0=1e-3, chunk=1000)
        got.append((z, st["attempts"], st["rc"], ctx.launch_count() - before))
    assert got[0][:3][1:] == got[1][:3][1:] and torch.equal(got[0][0], got[1][0]) and got[0][2] == 0
    assert got[0][1] > 1
    if one_loop:
        assert got[0][3] == 2  # the first step armed, then one launch
    else:
        assert got[0][3] >= 10 * got[0][1]
    ctx.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_tuning_keeps_every_mask_of_the_collision_launch_bitwise(precision):
    m = MODELS["silicon12"]()
    ctx = _make(m, precision)
    y = _state(m, 8)
    before = {p: _rhs(ctx, y, 3, p) for p in range(1, 8)}
    if precision == "fp64":
        assert ctx.tuning()["static_share"] < 1.0  # units taken at run time by default
    ctx.autotune(ALL)
    tuned = ctx.tuning()
    for p in range(1, 8):
        assert torch.equal(_rhs(ctx, y, 3, p), before[p])
    ctx.autotune(3)
    ctx.autotune(4)
    assert ctx.tuning() == tuned
    for p in range(1, 8):
        assert torch.equal(_rhs(ctx, y, 3, p), before[p])
    ctx.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_units_taken_at_run_time_equal_static_ones(precision):
    """Four uneven instances (units taken at run time) against each alone (static ones, or one launch)."""
    ms = [_graphene(24), _graphene(48), ri.silicon(12), _graphene(60)]
    ctx = _make(ms, precision)
    ys = [_state(m, 20 + i) for i, m in enumerate(ms)]
    for p in (7, 3, 4):
        got, at = _rhs(ctx, torch.cat(ys), 3, p), 0
        assert ctx.tuning()["static_share"] < 1.0
        for i, m in enumerate(ms):
            one = _make(m, precision)
            assert torch.equal(got[at:at + m.n_y], one.rhs(ys[i], parts=p))
            at += m.n_y
            one.close()
    ctx.close()
