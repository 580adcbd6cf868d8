"""Timed workloads of the library, each one pass through a public entry point of
``paper_2412_13402_gb300`` on the seeded synthetic models of ``rtbte_inputs``.

A case is a dict of plain values:

  kind       "rhs"    one RHS evaluation, Context.rhs (Eq. e-ph, Eq. ph-ph)
             "erk"    one adaptive explicit Runge-Kutta window, Context.advance_to
             "mri"    one multirate (MIS) window, Context.advance_to
             "rates"  linearised mode-resolved ph-ph rates, Context.phph_rates
             "train"  Adam steps of the learned slow stage, Surrogate.train
  model      "toy" (2D, e-ph only), "graphene" (2D), "silicon" (3D, folded grid) or "ensemble"
             (several uneven graphene-like instances in one context)
  n          grid side (for the ensemble: number of instances)
  precision  collision sums in "fp32" (compensated; the default) or "fp64"
  parts      RTBTE_* bit mask of an RHS case (7: all, 3: fast part, 4: slow part)
  tune       whether the program called Context.autotune after the upload
  window     ps integrated by an "erk" / "mri" pass; h_s the MRI slow step
  steps, batch  of a "train" pass

A larger ``seed`` gives other coupling strengths, excitations and temperatures, hence other
channel weights, populations and step sequences.
"""
import math
import random

import numpy as np
import torch

import paper_2412_13402_gb300 as rt
import rtbte_inputs as ri


def _rhs(name, model, n, precision="fp32", parts=7, tune=False):
    return dict(name=name, kind="rhs", model=model, n=n, precision=precision, parts=parts, tune=tune)


def listed():
    return [
        # the smallest call: a 12x12 toy model in FP64, where a call is its kernels' latency
        _rhs("toy12_rhs_fp64", "toy", 12, precision="fp64"),
        # a parity-sized / convergence-study grid: short segments, lists that fit in L2
        _rhs("graphene63_rhs", "graphene", 63),
        # the headline evaluation: full RHS of the 180x180 workload, tuned as the README shows
        _rhs("graphene180_rhs", "graphene", 180, tune=True),
        # the FP64 mode of the precision studies and of the error-versus-cost reference
        _rhs("graphene120_rhs_fp64", "graphene", 120, precision="fp64"),
        # 3D, folded grids, dominated by long ph-ph segments
        _rhs("silicon32_rhs", "silicon", 32),
        # the batched ensemble: 64 uneven instances in one launch, short segments
        _rhs("ensemble64_rhs", "ensemble", 64),
        # adaptive Bogacki-Shampine run of the toy model: the step loop's latency
        dict(name="toy12_bs32_fp64", kind="erk", model="toy", n=12, precision="fp64", window=0.05),
        # the benchmark's window: adaptive Zonneveld 4(3) over 50 fs of the 180x180 workload
        dict(name="graphene180_zon43", kind="erk", model="graphene", n=180, precision="fp32", window=0.05),
        # multirate run, slow step 20 fs: fast and slow part masks, forced inner solves
        dict(name="graphene96_mri", kind="mri", model="graphene", n=96, precision="fp32", window=0.04, h_s=0.02),
        # batched integration with one controller per instance
        dict(name="ensemble16_zon43", kind="erk", model="ensemble", n=16, precision="fp32", window=0.02),
        # 300 K linearised ph-ph rates, the grid-convergence study's call (FP64)
        dict(name="graphene180_rates_fp64", kind="rates", model="graphene", n=180, precision="fp64"),
        # training of the learned slow stage on the 60x60 sub-lattice, minibatches of 8
        dict(name="graphene180_train", kind="train", model="graphene", n=180, precision="fp32", steps=8, batch=8),
    ]


def _log_int(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(hi, max(lo, int(round(v / step)) * step))


def draw(rng):
    """One more case of the ranges the listed ones stand for (graphene sides are multiples of
    the sub-lattice stride 3, silicon sides of the fold 2)."""
    kind = rng.choice(["rhs", "rhs", "rhs", "rhs", "erk", "erk", "mri", "rates", "train"])
    if kind == "rhs":
        model = rng.choice(["toy", "graphene", "graphene", "silicon", "ensemble"])
        precision = rng.choice(["fp32", "fp32", "fp64"])
        n = {"toy": lambda: rng.randint(6, 24), "graphene": lambda: _log_int(rng, 24, 180, 3),
             "silicon": lambda: _log_int(rng, 12, 30, 2), "ensemble": lambda: _log_int(rng, 2, 56)}[model]()
        if precision == "fp64" and model in ("graphene", "ensemble"):
            n = _log_int(rng, 24, 117, 3) if model == "graphene" else _log_int(rng, 2, 24)
        parts = 7 if model == "toy" else rng.choice([7, 7, 3, 4])
        return dict(kind="rhs", model=model, n=n, precision=precision, parts=parts, tune=False)
    if kind == "erk":
        model = rng.choice(["toy", "graphene", "graphene", "ensemble"])
        if model == "toy":
            return dict(kind="erk", model="toy", n=rng.randint(8, 20), precision="fp64",
                        window=round(rng.uniform(0.01, 0.05), 4))
        n = _log_int(rng, 24, 150, 3) if model == "graphene" else _log_int(rng, 2, 14)
        return dict(kind="erk", model=model, n=n, precision="fp32", window=round(rng.uniform(0.01, 0.05), 4))
    if kind == "mri":
        return dict(kind="mri", model="graphene", n=_log_int(rng, 24, 120, 3), precision="fp32", window=0.04,
                    h_s=rng.choice([0.01, 0.02, 0.04]))
    if kind == "rates":
        return dict(kind="rates", model="graphene", n=_log_int(rng, 48, 174, 3),
                    precision=rng.choice(["fp64", "fp64", "fp32"]))
    return dict(kind="train", model="graphene", n=_log_int(rng, 48, 174, 3), precision="fp32",
                steps=rng.randint(2, 8), batch=rng.randint(2, 8))


def _models(case, seed):
    """The case's models: coupling seeds, excitation and temperature drawn from the seed."""
    r = random.Random(seed)
    n = case["n"]
    if case["model"] == "ensemble":  # uneven sides as ri.ensemble draws them, the same for every seed
        sides = random.Random(ri.SEED_BASE + 3)
        out = []
        for _ in range(n):
            side = sides.choice(range(24, 97, 3))
            f = math.sqrt(180.0 / side)
            out.append(ri.graphene(side, seed=r.randrange(1 << 20), T=r.uniform(100.0, 500.0), E_x=r.uniform(0.1, 1.0),
                                   sigma_eph=0.020 * f, sigma_pp=0.002 * f))
        return out
    s = r.randrange(1 << 20)
    if case["model"] == "toy":
        m = ri.toy2d(n, seed=s)
        f0 = np.clip(m.f0 * r.uniform(0.7, 1.3), 0.0, 1.0)
        return [m.with_populations(f0=f0, N0=m.N0 * r.uniform(0.8, 1.2))]
    if case["model"] == "silicon":
        return [ri.silicon(n, seed=s, T=r.uniform(250.0, 350.0), E_x=r.uniform(0.15, 0.25))]
    f = math.sqrt(180.0 / n)  # broadenings widen on coarse grids, as in the ensemble
    return [ri.graphene(n, seed=s, T=r.uniform(250.0, 350.0), E_x=r.uniform(0.8, 1.0), amp=r.uniform(0.2, 0.35),
                        sigma_eph=0.020 * f, sigma_pp=0.002 * f)]


def prepare(case, seed):
    ms = _models(case, seed)
    ctx = rt.Context(ms, precision=case["precision"])
    for i in range(len(ms)):
        ctx.upload_channels(i)
    y = torch.tensor(np.concatenate([m.y0() for m in ms]), device="cuda")
    s = dict(case=case, ctx=ctx, y=y, out=torch.empty_like(y))
    if case.get("tune"):
        ctx.autotune(case["parts"])
    if case["kind"] == "erk" and case["model"] == "toy":
        s["opt"] = rt.integ_options(method="bs32", t0=0.0, rtol=1e-8, atol_c=1e-15, atol_ph=1e-15)
    elif case["kind"] == "erk":
        s["opt"] = rt.integ_options(method="zon43", t0=0.0, rtol=1e-5, atol_c=1e-9, atol_ph=1e-12)
    elif case["kind"] == "mri":
        s["opt"] = rt.integ_options(method="mri", t0=0.0, h_s=case["h_s"], rtol=1e-5, atol_c=1e-9, atol_ph=1e-12)
    elif case["kind"] == "train":
        sur = rt.Surrogate(ctx, width=64, capacity=16, seed=seed % 1000)
        z, o, t = y.clone(), rt.integ_options(method="zon43", rtol=1e-5, atol_c=1e-9, atol_ph=1e-12), 0.0
        for i in range(16):  # pairs along the method's own trajectory, 2 fs apart
            sur.collect(z, 0)
            o.t0, o.resume = t, int(i > 0)
            ctx.advance_to(t + 0.002, z, o)
            t += 0.002
        s["sur"] = sur
    return s


def run(state):
    case, ctx, y = state["case"], state["ctx"], state["y"]
    kind = case["kind"]
    if kind == "rhs":
        return ctx.rhs(y, state["out"], parts=case["parts"])
    if kind == "rates":
        return ctx.phph_rates(y)
    if kind == "train":
        loss = state["sur"].train(case["steps"], case["batch"], 1e-3)
        return [loss, state["sur"].get_params()]
    z = state["out"].copy_(y)  # the initial state, integrated in place
    ctx.advance_to(case["window"], z, state["opt"])
    return z


# ---- work ------------------------------------------------------------------------------------

_entries = {}


def _sizes(case):
    """(list bytes, entries, state rows) of one evaluation, from the case's own channel counts."""
    key = (case["model"], case["n"], case["precision"], case.get("parts", 7), case["kind"] == "rates")
    if key not in _entries:
        ms = _models(case, 1)
        ctx = rt.Context(ms, precision=case["precision"])
        for i in range(len(ms)):
            ctx.upload_channels(i)
        parts = 4 if case["kind"] == "rates" else case.get("parts", 7)
        tot = {1: 0, 2: 0, 4: 0}
        for i in range(len(ms)):
            z = ctx.sizes(i)
            for p, k in ((1, "eph_entries"), (2, "phe_entries"), (4, "pp_entries")):
                tot[p] += z[k]
        ny = ctx.n_y
        ctx.close()
        _entries[key] = (sum(v for p, v in tot.items() if parts & p), tot, ny)
    return _entries[key]


def work(case):
    """Every stored channel entry (4-byte index, 4- or 8-byte weight) and the FP64 state read once
    and the result written once; per entry 7 operations.  An integration pass reads its lists at
    every RHS evaluation (they exceed L2 at the sizes that matter); its evaluations are counted for
    the smallest step count a window takes: one attempt of 4 or 5 stages per 10 fs."""
    esize = 4 + (8 if case["precision"] == "fp64" else 4)
    if case["kind"] == "train":
        P, w, C = (case["n"] // 3) ** 2, 64, 6
        macs = P * w * (9 * C + 3 * 9 * w + w + C)
        params = w * (9 * C + 3 * 9 * w + w + C) + 5 * w + C
        per = 3 * 2 * macs * case["batch"]
        # minibatch read; weights, gradient and two moments read and written
        byts = case["batch"] * P * C * 8 + params * 4 * 7
        return {"bytes": case["steps"] * byts, "flops": case["steps"] * per}
    n, tot, ny = _sizes(case)
    if case["kind"] in ("rhs", "rates"):
        return {"bytes": n * esize + 16 * ny, "flops": 7 * n}
    if case["kind"] == "mri":
        slow = 3 * max(1, round(case["window"] / case["h_s"]))
        fast = 15 * max(1, round(case["window"] / case["h_s"]))
        e = slow * tot[4] + fast * (tot[1] + tot[2])
        return {"bytes": e * esize + 16 * ny * (slow + fast), "flops": 7 * e}
    evals = (4 if case["model"] == "toy" else 5) * max(1, round(case["window"] / 0.010))
    return {"bytes": evals * (n * esize + 16 * ny), "flops": evals * 7 * n}


# ---- the same sums in plain 64-bit torch -------------------------------------------------------

def _i64(x):
    return x - (1 << 64) if x >= (1 << 63) else x


def _shr(z, b):  # logical right shift of int64 tensors
    return (z >> b) & ((1 << (64 - b)) - 1)


def _mix64(z):
    """SplitMix64's output function on int64 tensors (two's complement wrap-around)."""
    z = z + _i64(0x9E3779B97F4A7C15)
    z = (z ^ _shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _i64(0x94D049BB133111EB)
    return z ^ _shr(z, 31)


def _mix_int(v, dev):
    return _mix64(torch.tensor(_i64(v % (1 << 64)), dtype=torch.int64, device=dev))


def _delta(e, sigma):
    return torch.exp(-(e / sigma) ** 2) / (sigma * math.sqrt(math.pi))


def _lut_index(m, key, seed, dev):
    return _shr(_mix64(key ^ _mix_int(seed, dev)), 64 - m.lut_bits)


def _eph_blocks(m, dev, span=1 << 23):
    """Kept electron-phonon channels in blocks: (process, destination, source, phonon, |g|^2 delta);
    process 0 emits a phonon leaving the destination, 1 absorbs one arriving at it."""
    k = torch.tensor(m.e_k, dtype=torch.int64, device=dev)
    eps = torch.tensor(m.e_eps, device=dev)
    band = torch.tensor(m.e_band, dtype=torch.int64, device=dev)
    omega = torch.tensor(m.ph_omega, device=dev).view(m.nmodes, m.N_q)
    lut, g2 = torch.tensor(m.lut, device=dev), torch.tensor(m.g2_coef, device=dev)
    nk, nq = m.nk, m.nq
    lin = lambda c: (c[:, 2] * nk[1] + c[:, 1]) * nk[0] + c[:, 0]  # noqa: E731
    neg = torch.stack([(-k[:, c]) % nk[c] for c in range(3)], 1)
    eid, einv = band * m.N_k + lin(k), band * m.N_k + lin(neg)
    cut, U = 3.0 * m.sigma_eph, m.nbands * m.N_k
    step = max(1, span // m.n_c)
    for d0 in range(0, m.n_c, step):
        d = torch.arange(d0, min(d0 + step, m.n_c), device=dev)
        q = torch.zeros((len(d), m.n_c), dtype=torch.int64, device=dev)
        for c in (2, 1, 0):
            t = (k[None, :, c] - k[d, None, c]) % nk[c]
            t = torch.where(t > nk[c] // 2, t - nk[c], t)
            q = q * nq[c] + torch.div(t, m.fold, rounding_mode="trunc") % nq[c]
        for nu in range(m.nmodes):
            w = omega[nu][q]
            for proc in (0, 1):
                D = (eps[d, None] - w) - eps[None, :] if proc == 0 else (eps[None, :] - w) - eps[d, None]
                i, s = torch.nonzero((D.abs() <= cut) & (w >= m.omega_cut), as_tuple=True)
                dd = d[i]
                lo, hi = torch.minimum(eid[dd], eid[s]), torch.maximum(eid[dd], eid[s])
                il, ih = torch.minimum(einv[dd], einv[s]), torch.maximum(einv[dd], einv[s])
                swap = (il < lo) | ((il == lo) & (ih < hi))
                lo, hi = torch.where(swap, il, lo), torch.where(swap, ih, hi)
                key = (lo * U + hi) * m.nmodes + nu
                g = g2[nu] * lut[_lut_index(m, key, m.g2_seed, dev)]
                yield proc, dd, s, nu * m.N_q + q[i, s], g * _delta(D[i, s], m.sigma_eph)


def _pp_blocks(m, dev, span=1 << 23):
    """Kept three-phonon channels in blocks: (process, a, b, c, |V3|^2 delta), full phonon indices;
    process 0 is a -> b + c with b <= c (weight doubled when b < c), 1 is a + c -> b (doubled)."""
    full = torch.tensor(m.pp_full_index(), device=dev)
    om = torch.tensor(m.ph_omega, device=dev)
    lut = torch.tensor(m.lut, device=dev)
    ns, st, M, nqs = m.nq_pp, m.pp_stride, m.n_pp, m.N_q_pp
    a_all = torch.arange(M, device=dev)
    q = a_all % nqs
    qc = [q % ns[0], (q // ns[0]) % ns[1], q // (ns[0] * ns[1])]
    stride = [st if m.nq[c] > 1 else 1 for c in range(3)]
    inv = torch.zeros_like(q)
    for c in (2, 1, 0):
        inv = inv * m.nq[c] + (-qc[c] * stride[c]) % m.nq[c]
    inv = (a_all // nqs) * m.N_q + inv
    wa = om[full]
    live = wa >= m.omega_cut
    cut = 3.0 * m.sigma_pp
    step = max(1, span // M)
    for a0 in range(0, M, step):
        a = torch.arange(a0, min(a0 + step, M), device=dev)
        for proc in (0, 1):
            qd = torch.zeros((len(a), M), dtype=torch.int64, device=dev)
            for c in (2, 1, 0):
                t = qc[c][a][:, None] - qc[c][None, :]
                qd = qd * ns[c] + (t if proc == 0 else -t) % ns[c]
            for nu in range(m.nmodes):
                c_ = nu * nqs + qd
                wc = wa[c_]
                D = (wa[None, :] + wc) - wa[a][:, None] if proc == 0 else (wa[a][:, None] + wc) - wa[None, :]
                keep = (D.abs() <= cut) & live[a][:, None] & live[None, :] & live[c_]
                if proc == 0:
                    keep &= c_ >= a_all[None, :]
                i, b = torch.nonzero(keep, as_tuple=True)
                aa, cc = a[i], c_[i, b]
                t, _ = torch.sort(torch.stack([full[aa], full[b], full[cc]]), dim=0)
                u, _ = torch.sort(torch.stack([inv[aa], inv[b], inv[cc]]), dim=0)
                swap = (u[0] < t[0]) | ((u[0] == t[0]) & ((u[1] < t[1]) | ((u[1] == t[1]) & (u[2] < t[2]))))
                t = torch.where(swap, u, t)
                key = (t[0] * m.n_ph + t[1]) * m.n_ph + t[2]
                v = m.v3_coef * lut[_lut_index(m, key, m.v3_seed, dev)] * _delta(D[i, b], m.sigma_pp)
                v = torch.where(b == cc, v, 2 * v) if proc == 0 else 2 * v
                yield proc, full[aa], full[b], full[cc], v


def _sum_eph(m, f, N, blocks, df, dN, parts):
    pe, pp = 2 * math.pi / ri.HBAR_EV_PS / m.N_q, 4 * math.pi / ri.HBAR_EV_PS / m.N_k
    for proc, d, s, p, g in blocks:
        if proc == 0:
            if parts & 1:
                df.index_add_(0, d, -pe * g * (f[d] * (1 - f[s]) + N[p] * (f[d] - f[s])))
            continue
        F = N[p] * (f[d] - f[s]) - f[s] * (1 - f[d])
        if parts & 1:
            df.index_add_(0, d, -pe * g * F)
        if parts & 2:
            dN.index_add_(0, p, -pp * g * F)


def _sum_pp(m, N, blocks, dN, rates=False):
    pr = 36 * math.pi / ri.HBAR_EV_PS / m.N_q_pp
    for proc, a, b, c, v in blocks:
        if rates:
            G = -(N[b] + N[c] + 1) if proc == 0 else -(N[c] - N[b])
        elif proc == 0:
            G = N[a] * (N[b] + N[c] + 1) - N[b] * N[c]
        else:
            G = N[a] * (N[c] - N[b]) - N[b] * (N[c] + 1)
        dN.index_add_(0, a, -pr * v * G)


def exact(case, seed):
    """The same quantity from the plain sums in 64 bits: for the RHS and the rates the sums
    themselves, for an integration window of a small model fixed-step RK4 on them with steps far
    below the adaptive ones.  None where that would take too long, and for training (its
    minibatches come from the library's own generator)."""
    if case["kind"] == "train":
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    ms = _models(case, seed)
    if case["kind"] in ("rhs", "rates"):
        out = []
        for m in ms:
            y = torch.tensor(m.y0(), device=dev)
            f, N = y[:m.n_c], y[m.n_c:]
            dy = torch.zeros_like(y)
            df, dN = dy[:m.n_c], dy[m.n_c:]
            parts = case.get("parts", 7)
            if case["kind"] == "rates":
                _sum_pp(m, N, _pp_blocks(m, dev), dN, rates=True)
            else:
                if parts & 3:
                    _sum_eph(m, f, N, _eph_blocks(m, dev), df, dN, parts)
                if parts & 4 and m.pp_stride > 0:
                    _sum_pp(m, N, _pp_blocks(m, dev), dN)
            out.append(dy)
        return torch.cat(out)
    if case["model"] == "ensemble" or case["n"] > 48:
        return None
    m = ms[0]
    eph = list(_eph_blocks(m, dev))
    pp = list(_pp_blocks(m, dev)) if m.pp_stride > 0 else []
    y = torch.tensor(m.y0(), device=dev)

    def rhs(y):
        dy = torch.zeros_like(y)
        _sum_eph(m, y[:m.n_c], y[m.n_c:], eph, dy[:m.n_c], dy[m.n_c:], 7)
        if pp:
            _sum_pp(m, y[m.n_c:], pp, dy[m.n_c:])
        return dy

    h = 0.0001 if case["model"] == "toy" else 0.0005
    ns = max(1, math.ceil(case["window"] / h))
    h = case["window"] / ns
    for _ in range(ns):
        k1 = rhs(y)
        k2 = rhs(y + 0.5 * h * k1)
        k3 = rhs(y + 0.5 * h * k2)
        k4 = rhs(y + h * k3)
        y = y + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
    return y
