"""What this framework is asked to do: whole collision steps on the mixed and the FP64 path, the re-bin and step of a
particle-in-cell loop, the cell sort of a freshly loaded state, the step as separate calls, and gradients through
steps. Sizes, masses, weights and time steps are those of the synthetic plasmas of the package (``workloads``), drawn
here on the GPU.

``exact`` restates the method in plain 64-bit torch (rounds of disjoint pairs over all cells at once); gradients come
from autograd through it with every draw and decision held fixed.
"""
import dataclasses
import math

import torch

import paper_2407_19151_gb300 as mcc

DEV = "cuda"
M_P = 1836.15267
M_C6 = 12.0 * 1822.888486 - 6.0
LNL = 10.0
EXACT_MOST = 150_000_000  # particles

# Plasmas: charges, masses, temperatures (per axis), decades of the log-uniform weights (lo, hi).
PLASMAS = {
    "iso": dict(q=[-1.0], m=[1.0], T=[(2.0, 1.0, 1.0)], w=[(0.0, 1.0)]),
    "equil": dict(q=[-1.0, 1.0], m=[1.0, 100.0], T=[(1.0,) * 3, (4.0,) * 3], w=[(0.0, 0.0), (1.0, 3.0)]),
    "beam": dict(q=[-1.0, -1.0, 1.0], m=[1.0, 1.0, M_P], T=[(0.01,) * 3] * 3, w=[(0.0, 3.0)] * 3),
    "diff": dict(q=[-1.0, 1.0], m=[1.0, 1836.0], T=[(1.0,) * 3, (2.0,) * 3], w=[(0.0, 1.0)] * 2),
    "three": dict(q=[-1.0, 1.0, 6.0], m=[1.0, M_P, M_C6], T=[(1.0,) * 3, (0.5,) * 3, (0.5,) * 3], w=[(0.0, 4.0)] * 3),
}


def listed():
    return [
        # the smallest call: 64 cells of one species, one FP64 step (isotropisation); launches and latency count
        dict(name="iso_f64", kind="step", plasma="iso", cells=64, mean=128, prec="f64", method="n97", steps=1, order="any"),
        # a small run on the mixed path, a few cells on every group size
        dict(name="three_small", kind="step", plasma="three", cells=100, mean=300, prec="f32", method="n97", steps=1,
             order="weight"),
        # electron-ion equilibration, TA77, tied electron weights, particles in no weight order, two steps in one call
        dict(name="equil_ta77", kind="step", plasma="equil", cells=4096, mean=512, prec="f32", method="ta77", steps=2,
             order="any"),
        # the benchmark's size: 2^18 cells, 1.34e8 particles, segments in weight order
        dict(name="three_full", kind="step", plasma="three", cells=1 << 18, mean=512, prec="f32", method="n97", steps=1,
             order="weight"),
        # relativistic beam in a plasma: power-law cell sizes, most cells small
        dict(name="beam_f32", kind="step", plasma="beam", cells=1 << 16, mean=0, prec="f32", method="n97", steps=1,
             order="any"),
        # the plain FP64 path on ordinary cells, and its relativistic form
        dict(name="three_f64", kind="step", plasma="three", cells=4096, mean=512, prec="f64", method="n97", steps=1,
             order="weight"),
        dict(name="beam_f64", kind="step", plasma="beam", cells=2048, mean=0, prec="f64", method="n97", steps=1, order="any"),
        # gradients through steps: recorded tapes on the differentiable workload, and the float variant's checkpoints
        dict(name="grad_tape", kind="grad", cells=1024, mean=512, prec="f64", method="n97", steps=2, tape=True, every=10),
        dict(name="grad_ckpt_f32", kind="grad", cells=200, mean=250, prec="f32", method="ta77", steps=3, tape=False, every=2),
        # a state loaded in random order: cell sort and the gathers that put it in binned order
        dict(name="load_sort", kind="sort", cells=1 << 16, mean=512, prec="f32", weighted=False),
        # one step of a particle-in-cell loop: push, re-bin in weight order, gather, collision step
        dict(name="pic_weight", kind="pic", cells=1 << 15, mean=512, prec="f32", order="weight"),
        # the step as separate calls (a code that looks at the pairs or the scatter itself), and the diagnostics
        dict(name="split_calls", kind="split", plasma="equil", cells=1000, mean=401, prec="f64", method="n97"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["grad", "grad", "sort", "sort", "pic", "pic", "split"])
    prec = rng.choice(["f32", "f32", "f64"])
    method = rng.choice(["n97", "n97", "ta77"])
    if kind == "step":
        plasma = rng.choice(["three", "three", "equil", "beam", "iso", "diff"])
        mean = 0 if plasma == "beam" else _log(rng, 24, 1500)
        most = (60_000_000 if prec == "f32" else 2_500_000) // (mean or 180)
        if plasma == "beam":
            most = 60_000 if prec == "f32" else 4_000
        return dict(kind=kind, plasma=plasma, cells=_log(rng, 30, most), mean=mean, prec=prec, method=method,
                    steps=rng.choice([1, 1, 2]), order=rng.choice(["weight", "any"]))
    if kind == "grad":
        mean = _log(rng, 40, 700)
        return dict(kind=kind, cells=_log(rng, 20, 400_000 // mean), mean=mean, prec=prec, method=method,
                    steps=rng.choice([1, 2, 3]), tape=prec == "f64" and rng.random() < 0.6, every=rng.choice([1, 2, 10]))
    if kind == "sort":
        mean = _log(rng, 24, 1500)
        return dict(kind=kind, cells=_log(rng, 50, 60_000_000 // mean), mean=mean, prec=prec, weighted=rng.random() < 0.5)
    if kind == "pic":
        mean = _log(rng, 60, 900)
        most = (20_000_000 if prec == "f32" else 1_500_000) // mean
        return dict(kind=kind, cells=_log(rng, 60, most), mean=mean, prec=prec, order=rng.choice(["weight", "stable"]))
    mean = _log(rng, 40, 900)
    return dict(kind=kind, plasma=rng.choice(["equil", "three"]), cells=_log(rng, 20, 600_000 // mean), mean=mean, prec=prec,
                method=method)


# ------------------------------------------------------------------------------------------------------- inputs
def _counts(plasma, cells, mean, g):
    """(cells, species) particle counts: lognormal totals (three), Poisson (equil), equal (iso, diff), power law (beam)."""
    if plasma == "three":
        z = torch.randn(cells, generator=g, device=DEV, dtype=torch.float64)
        tot = torch.round(torch.exp(math.log(mean) - 0.125 + 0.5 * z)).clamp(1, 10 * mean).long()
        base, rem = tot // 3, tot % 3
        return torch.stack([base + (rem > 0), base + (rem > 1), base], 1)
    if plasma == "equil":
        return torch.poisson(torch.full((cells, 2), mean / 2.0, device=DEV, dtype=torch.float64), generator=g).long()
    if plasma == "beam":
        k = torch.arange(16, 2049, device=DEV, dtype=torch.float64)
        cdf = torch.cumsum(k ** -1.5, 0)
        u = torch.rand(cells, generator=g, device=DEV, dtype=torch.float64) * cdf[-1]
        tot = 16 + torch.searchsorted(cdf, u).clamp(max=2032)
        nb, ne = tot // 10, (tot * 9) // 20
        return torch.stack([nb, ne, tot - nb - ne], 1)
    s = len(PLASMAS[plasma]["m"])
    return torch.full((cells, s), max(2, mean // s), device=DEV, dtype=torch.long)


def _plasma(case):
    return case.get("plasma", "three" if case["kind"] in ("sort", "pic") else "diff")


def _mean_particles(case):
    return case["cells"] * (179.0 if _plasma(case) == "beam" else float(case["mean"]))


def _inputs(case, seed):
    """The particles of a case, binned: counts, offsets, velocities, weights, time step."""
    name = _plasma(case)
    P = PLASMAS[name]
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    C, S = int(case["cells"]), len(P["m"])
    dt_ = torch.float32 if case["prec"] == "f32" else torch.float64
    # the cell sizes of a case are one sample, dealt to the cells by the seed: every seed has as many particles
    counts = _counts(name, C, case["mean"], torch.Generator(device=DEV).manual_seed(1234))
    counts = counts[torch.randperm(C, generator=g, device=DEV)]
    flat = counts.reshape(-1)
    off = torch.zeros(C * S + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(flat, 0)
    n = int(off[-1])
    sp = torch.repeat_interleave(torch.arange(S, device=DEV, dtype=torch.int32).repeat(C), flat, output_size=n)
    spl = sp.long()
    lo = torch.tensor([a for a, _ in P["w"]], device=DEV, dtype=torch.float64)
    width = torch.tensor([b - a for a, b in P["w"]], device=DEV, dtype=torch.float64)
    w = torch.pow(10.0, lo[spl] + width[spl] * torch.rand(n, generator=g, device=DEV, dtype=torch.float64))
    if case.get("order", "any") == "weight":
        by = torch.argsort(w, descending=True, stable=True)
        seg = torch.repeat_interleave(torch.arange(C * S, device=DEV, dtype=torch.int32), flat, output_size=n)
        w = w[by[torch.argsort(seg[by], stable=True)]]
        del by, seg
    v = []
    for d in range(3):
        std = torch.tensor([math.sqrt(T[d] / m) for T, m in zip(P["T"], P["m"])], device=DEV, dtype=dt_)
        x = torch.randn(n, generator=g, device=DEV, dtype=dt_) * std[spl]
        if name == "beam":
            u = torch.rand(n, generator=g, device=DEV, dtype=dt_) if d == 2 else None
            fast = math.sqrt(3.0) + (math.sqrt(99.0) - math.sqrt(3.0)) * u if d == 2 else 0.1 * x
            x = torch.where(sp == 0, fast, x)
        v.append(x.contiguous())
    w_mean = {"iso": 9.0 / math.log(10.0), "equil": 1.0, "beam": 999.0 / (3.0 * math.log(10.0)),
              "diff": 9.0 / math.log(10.0), "three": 9999.0 / (4.0 * math.log(10.0))}[name]
    n_e = (0.45 * 179.0 if name == "beam" else case["mean"] / S) * w_mean
    T_e = 4.0 / 3.0 if name == "iso" else P["T"][0][0]
    dt = 0.01 * 4.0 * math.pi * T_e ** 1.5 / (LNL * n_e)  # nu dt = 0.01 for the electrons
    return dict(C=C, S=S, n=n, counts=counts, off=off, sp=sp, v=v, w=w, dt=dt, g=g,
                species=list(zip(P["q"], P["m"])), rel=name == "beam", max_cell=int(counts.sum(1).max()))


def _params(case, x, seed):
    return mcc.Params(method=mcc.N97 if case.get("method", "n97") == "n97" else mcc.TA77, relativistic=x["rel"], dt=x["dt"],
                      seed=0x5EED0000 + int(seed), step=7)


def _grid(cells):
    nz = max(d for d in range(1, int(round(cells ** (1.0 / 3.0))) + 1) if cells % d == 0)
    m = cells // nz
    ny = max(d for d in range(1, int(m ** 0.5) + 1) if m % d == 0)
    return m // ny, ny, nz


def _positions(x, prec):
    """Each particle uniform inside its own unit cell of a periodic grid."""
    dt_ = torch.float32 if prec == "f32" else torch.float64
    nx, ny, nz = _grid(x["C"])
    cell = torch.repeat_interleave(torch.arange(x["C"], device=DEV), x["counts"].sum(1), output_size=x["n"])
    pos = []
    for i in (cell % nx, (cell // nx) % ny, cell // (nx * ny)):
        p = (i.to(torch.float64) + torch.rand(x["n"], generator=x["g"], device=DEV, dtype=torch.float64)).to(dt_)
        top = torch.nextafter((i + 1).to(dt_), torch.zeros((), device=DEV, dtype=dt_))
        pos.append(torch.minimum(p, top))
    return ((nx, ny, nz), (float(nx), float(ny), float(nz))), pos


def _shuffled(case, seed):
    x = _inputs(case, seed)
    order = torch.randperm(x["n"], generator=x["g"], device=DEV)
    cell = torch.repeat_interleave(torch.arange(x["C"], device=DEV, dtype=torch.int32), x["counts"].sum(1),
                                   output_size=x["n"])
    return x, cell[order], x["sp"][order], [a[order] for a in (*x["v"], x["w"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sort":
        x, cell, sp, arrays = _shuffled(case, seed)
        return dict(kind=kind, weighted=case["weighted"], C=x["C"], S=x["S"], cell=cell, sp=sp, arrays=arrays)
    x = _inputs(case, seed)
    p = _params(case, x, seed)
    st = dict(kind=kind, C=x["C"], S=x["S"], off=x["off"], v=x["v"], w=x["w"], species=x["species"], params=p, t=0,
              steps=case.get("steps", 1), max_cell=x["max_cell"])
    if kind == "pic":
        grid, pos = _positions(x, case["prec"])
        st["loop"] = mcc.PicLoop(*pos, *x["v"], x["w"], x["sp"], x["off"], x["C"], x["S"], grid, x["species"], LNL, p, 0.25,
                                 order=case["order"])
    elif kind == "grad":
        st["v"] = [a.requires_grad_() for a in x["v"]]
        st["w"] = x["w"].requires_grad_()
        st["lnL"] = torch.full((x["S"], x["S"]), LNL, dtype=torch.float64, requires_grad=True)
        # the cotangent of the final velocities (a loss's gradient)
        st["cot"] = [torch.randn(x["n"], generator=x["g"], device=DEV, dtype=a.dtype) for a in x["v"]]
        st["tape"], st["every"] = case["tape"], case["every"]
    return st


def run(st):
    kind, C, S = st["kind"], st["C"], st["S"]
    if kind == "sort":
        if st["weighted"]:
            perm, off = mcc.mcc_bin_weighted(st["cell"], st["sp"], st["arrays"][3], C, S)
            return perm, off, *mcc.mcc_gather_n(st["arrays"], perm)
        perm, off = mcc.mcc_bin(st["cell"], st["sp"], C, S)
        return perm, off, *[mcc.mcc_gather(a, perm) for a in st["arrays"]]
    if kind == "pic":
        corr, fail = st["loop"].step(1)
        return *st["loop"].state, st["loop"].offsets, corr, fail
    p = dataclasses.replace(st["params"], step=st["params"].step + st["t"])
    if kind == "grad":  # the same steps each time: gradients of one loss
        leaves = (*st["v"], st["w"], st["lnL"])
        out = mcc.collision_steps(*st["v"], st["w"], st["lnL"], st["off"], C, S, st["species"], p, st["steps"],
                                  max_cell=st["max_cell"], checkpoint_every=st["every"], tape=st["tape"])
        return *out, *torch.autograd.grad(out, leaves, st["cot"])
    st["t"] += st["steps"]
    v, w, off = st["v"], st["w"], st["off"]
    if kind == "step":
        corr, fail = mcc.mcc_step_fused(*v, w, off, C, S, st["species"], LNL, p, n_steps=st["steps"],
                                        max_cell=st["max_cell"])
        return *v, corr, fail
    marks = []
    for k, (a, b) in enumerate(mcc.default_interactions(S)):
        pairs = mcc.mcc_pair(off, C, S, a, b, k, p.seed, p.step)
        backup = mcc.mcc_scatter(*v, w, off, C, S, st["species"], LNL, a, b, k, pairs, p)
        marks += mcc.mcc_correct(*v, w, off, C, S, st["species"], a, b, k, p, backup)
    return *v, mcc.mcc_species_moments(*v, w, off, C, S, st["species"]), *marks


def work(case):
    """Bytes: inputs read once and outputs written once. Operations: about 150 per scatter pair (draws apart) and 60
    per particle and interaction of the correction; twice the forward's again for a gradient."""
    n, S = _mean_particles(case), len(PLASMAS[_plasma(case)]["m"])
    vb = 4 if case["prec"] == "f32" else 8
    steps = case.get("steps", 1)
    pairs = n * S / 2
    flops = steps * (150 * pairs + 60 * n * S)
    b_step = steps * n * (6 * vb + 8) + case["cells"] * (8 * S + 8)
    kind = case["kind"]
    if kind == "sort":
        return {"bytes": n * (8 + 4 + 2 * (3 * vb + 8)) + 8 * S * case["cells"], "flops": 0}
    if kind == "pic":
        return {"bytes": n * 2 * (6 * vb + 8 + 4) + 16 * S * case["cells"], "flops": flops + 12 * n}
    if kind == "grad":
        return {"bytes": n * (3 * vb + 8 + 3 * vb + 3 * vb + 3 * vb + 8), "flops": 3 * flops}
    return {"bytes": b_step, "flops": flops}


# ------------------------------------------------------------------------------------------------------- exact
def exact(case, seed):
    kind = case["kind"]
    if _mean_particles(case) > EXACT_MOST:
        return None
    if kind == "sort":
        x, cell, sp, arrays = _shuffled(case, seed)
        order = _bin(cell, sp, arrays[3] if case["weighted"] else None, x["S"])
        return None, None, *[a[order].double() for a in arrays]
    x = _inputs(case, seed)
    p = _params(case, x, seed)
    if kind == "pic":
        (n3, _), pos = _positions(x, case["prec"])
        dt_ = x["v"][0].dtype
        pos, ids = _push(pos, x["v"], n3, torch.tensor(0.25, dtype=dt_, device=DEV), dt_)
        order = _bin(ids, x["sp"], x["w"] if case["order"] == "weight" else None, x["S"])
        v, w = torch.stack([a[order] for a in x["v"]], 1).double(), x["w"][order]
        seg = ids[order].long() * x["S"] + x["sp"][order].long()
        off = torch.zeros(x["C"] * x["S"] + 1, dtype=torch.int64, device=DEV)
        off[1:] = torch.cumsum(torch.bincount(seg, minlength=x["C"] * x["S"]), 0)
        v = _step(v, w, off, x["C"], x["S"], x["species"], LNL, p, p.step)
        return *[a[order].double() for a in pos], *v.unbind(1), w, None, None, None, None
    v, w, L = torch.stack(x["v"], 1).double(), x["w"], LNL
    if kind == "grad":
        cot = [torch.randn(x["n"], generator=x["g"], device=DEV, dtype=a.dtype).double() for a in x["v"]]
        v.requires_grad_()
        w.requires_grad_()
        L = torch.full((x["S"], x["S"]), LNL, dtype=torch.float64, device=DEV, requires_grad=True)
    u = v
    for t in range(case.get("steps", 1)):
        u = _step(u, w, x["off"], x["C"], x["S"], x["species"], L, p, p.step + t)
    out = [a.detach() for a in u.unbind(1)]
    if kind == "grad":
        gv, gw, gL = torch.autograd.grad(u, (v, w, L), torch.stack(cot, 1))
        return *out, *gv.unbind(1), gw, gL
    if kind == "step":
        return *out, None, None
    mom = []
    sp = x["sp"].long()
    for s, (_, m) in enumerate(x["species"]):
        sel = sp == s
        ws, vs = w[sel], u[sel]
        mom += [ws.sum(), *(m * (ws[:, None] * vs).sum(0)), 0.5 * m * (ws * (vs * vs).sum(1)).sum(),
                torch.tensor(float(sel.sum()), device=DEV, dtype=torch.float64)]
    mom.append(torch.zeros((), device=DEV, dtype=torch.float64))
    return *out, torch.stack(mom), *[None] * (x["S"] * (x["S"] + 1))


def _weight_bits(w):
    return ~w.detach().view(torch.int64) & ~((1 << 20) - 1)


def _bin(cell, sp, w, S):
    key = cell.long() * S + sp.long()
    if w is None:
        return torch.argsort(key, stable=True)
    by = torch.argsort(_weight_bits(w) ^ torch.iinfo(torch.int64).min, stable=True)
    return by[torch.argsort(key[by], stable=True)]


def _push(pos, v, n3, dt, dt_):
    out, ids = [], []
    for x, u, n in zip(pos, v, n3):
        L = torch.tensor(float(n), dtype=dt_, device=DEV)
        y = x + u * dt
        r = y - torch.floor(y / L) * L
        r = torch.where(r < 0, r + L, r)
        r = torch.where(r >= L, r - L, r)
        y = torch.where((y >= 0) & (y < L), y, r)
        out.append(y)
        ids.append(y.int().clamp(max=n - 1))
    return out, ids[0] + n3[0] * (ids[1] + n3[1] * ids[2])


_M32 = (1 << 32) - 1


def _philox(c0, c1, c2, c3, seed):
    """Philox-4x32-10 of 64-bit tensors holding 32-bit words."""
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    m0, m1 = 0xD2511F53, 0xCD9E8D57
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
        p0, p1 = c0 * m0, c2 * m1
        c0, c1, c2, c3 = ((p1 >> 32) & _M32) ^ c1 ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ c3 ^ k1, p0 & _M32
    return c0, c1, c2, c3


def _ranges(n):
    """For counts n per cell: (cell of each entry, its index within the cell)."""
    tot = int(n.sum())
    cell = torch.repeat_interleave(torch.arange(n.numel(), device=DEV), n, output_size=tot)
    start = torch.cumsum(n, 0) - n
    return cell, torch.arange(tot, device=DEV) - start[cell]


def _permutation(p, step, inter, side, n):
    """Random order of each cell's n particles, cell after cell (local indices)."""
    cell, q = _ranges(n)
    tag = torch.full_like(q, (inter << 8) | (1 + side))
    r = _philox(q >> 1, cell, torch.full_like(q, step & _M32), tag, p.seed)
    odd = (q & 1) == 1
    hi, lo = torch.where(odd, r[2], r[0]), torch.where(odd, r[3], r[1])
    key = ((hi << 32) | (lo & ~((1 << 20) - 1)) | q) ^ torch.iinfo(torch.int64).min
    by = torch.argsort(key)
    by = by[torch.argsort(cell[by], stable=True)]
    return cell, q[by]


def _L(A):
    """coth A - 1/A."""
    B = [1 / 3, -1 / 45, 2 / 945, -1 / 4725, 2 / 93555, -1382 / 638512875, 4 / 18243225, -3617 / 162820783125,
         87734 / 38979295480125, -349222 / 1531329465290625, 310732 / 13447856940643125]
    x, s = A.clamp(max=0.5), torch.zeros_like(A)
    for b in reversed(B):
        s = s * x * x + b
    return torch.where(A < 0.5, s * x, 1.0 / torch.tanh(A) - 1.0 / A)


def _n97_A(s):
    """Root of L(A) = exp(-s), as 1 - L = 1 - exp(-s) for short lengths; bisection in ln A, then Newton."""
    y, z, small = torch.exp(-s), -torch.expm1(-s), s < 0.7

    def f(A):  # increasing in A
        G = torch.where(A < 0.5, 1.0 - _L(A), 1.0 / A - 2.0 / torch.expm1(2.0 * A))
        return torch.where(small, z - G, _L(A) - y)

    lo, hi = torch.log(y), torch.log(1.0 / z + 1.0) + 1.2
    for _ in range(48):
        mid = 0.5 * (lo + hi)
        up = f(torch.exp(mid)) < 0
        lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
    A = torch.exp(0.5 * (lo + hi))
    for _ in range(3):
        A = A - f(A) / _dL(A)
    return A


def _dL(A):
    B = [1 / 3, -3 / 45, 10 / 945, -7 / 4725, 18 / 93555, -11 * 1382 / 638512875, 52 / 18243225, -15 * 3617 / 162820783125,
         17 * 87734 / 38979295480125, -19 * 349222 / 1531329465290625, 21 * 310732 / 13447856940643125]
    x, s = A.clamp(max=0.5), torch.zeros_like(A)
    for b in reversed(B):
        s = s * x * x + b
    big = A.clamp(min=0.5)
    sh = torch.sinh(big.clamp(max=300.0))
    return torch.where(A < 0.5, s, 1.0 / (big * big) - torch.where(big < 300.0, 1.0 / (sh * sh), torch.zeros_like(A)))


def _angle(n97, s, U1, U4):
    if not n97:
        d = torch.sqrt(0.5 * s) * torch.sqrt(-2.0 * torch.log(U1)) * torch.cos(2.0 * math.pi * U4)
        den = 1.0 + d * d
        return 2.0 * d / den, 2.0 * d * d / den
    sd = s.detach()
    iso = -torch.expm1(-sd) >= 1.0
    A0 = _n97_A(torch.where(iso, torch.ones_like(sd), sd))
    A = A0 - (torch.exp(-sd) / _dL(A0)) * (s - sd)  # L(A) = exp(-s): dA/ds = -exp(-s) / L'(A)
    x = U1 * torch.expm1(-2.0 * A)
    omc = torch.where(x > -0.5, -torch.log1p(x), -torch.log((1.0 - U1) + U1 * torch.exp(-2.0 * A))) / A
    omc = torch.where(iso, 2.0 * U1, omc).clamp(0.0, 2.0)
    od = omc.detach()
    back = torch.log1p((1.0 - U1) * torch.expm1(2.0 * A0.clamp(max=300.0))) / A0
    opc = torch.where(iso, 2.0 * (1.0 - U1), torch.where(od <= 1.0, 2.0 - od, back)).clamp(0.0, 2.0)
    return torch.sqrt(omc * (opc - (omc - od))), omc


def _rotate(u, st, omc, phi):
    cp, sp = torch.cos(phi), torch.sin(phi)
    um, up = u.norm(dim=1), u[:, :2].norm(dim=1)
    ax, ay = u[:, 0] / up, u[:, 1] / up
    return torch.stack([ax * u[:, 2] * st * cp - ay * um * st * sp - u[:, 0] * omc,
                        ay * u[:, 2] * st * cp + ax * um * st * sp - u[:, 1] * omc, -up * st * cp - u[:, 2] * omc], 1)


def _gamma(u):
    return torch.sqrt(1.0 + (u * u).sum(1))


def _dgamma(a, b):
    return ((a - b) * (a + b)).sum(1) / (_gamma(a) + _gamma(b))


def _gamma_rel_m1(a, b):
    return (0.5 * (((a - b) ** 2).sum(1) - _dgamma(a, b) ** 2)).clamp(min=0.0)


def _rel_frame(a, b, ma, mb):
    """CM velocity, (gamma_C - 1)/V^2, p*, |p*| and v_rel* of a pair of proper velocities (c = 1)."""
    ga, gb = _gamma(a), _gamma(b)
    M = ma * ga + mb * gb
    V = (ma * a + mb * b) / M[:, None]
    gC = M / torch.sqrt((ma + mb) ** 2 + 2.0 * ma * mb * _gamma_rel_m1(a, b))
    co = gC * gC / (gC + 1.0)
    q = ma * mb * (gb[:, None] * (a - b) - _dgamma(a, b)[:, None] * b) / M[:, None]
    ps = q + (co * (V * q).sum(1))[:, None] * V
    pm = ps.norm(dim=1)
    vr = pm * (1.0 / (ma * torch.sqrt(1.0 + pm * pm / ma ** 2)) + 1.0 / (mb * torch.sqrt(1.0 + pm * pm / mb ** 2)))
    return V, co, ps, pm, vr


def _scatter(v, w, p, step, inter, intra, cell, k, i, j, half, rnd, sp_a, sp_b, lnL, nmin):
    """The pairs (i, j) of one interaction, rounds in order."""
    (qa, ma), (qb, mb) = sp_a, sp_b
    kappa = (qa * qb) ** 2 * lnL * p.dt / (4.0 * math.pi)
    for r in range(int(rnd.max()) + 1 if rnd.numel() else 0):
        sel = torch.nonzero(rnd == r).squeeze(1)
        a, b, kk, cc = i[sel], j[sel], k[sel], cell[sel]
        x = _philox(kk, cc, torch.full_like(kk, step & _M32), torch.full_like(kk, (inter << 8) | 3), p.seed)
        U1, U2, U3, U4 = (((t >> 9).double() + 0.5) / 8388608.0 for t in x)
        va, vb, wa, wb = v[a], v[b], w[a], w[b]
        wmax, wmin = torch.where(wa > wb, wa, wb), torch.where(wa > wb, wb, wa)
        fac = kappa * wmax * nmin[cc] * torch.where(half[sel], 0.5, 1.0)
        if p.relativistic:
            V, co, ps, pm, vr = _rel_frame(va, vb, ma, mb)
            st, omc = _angle(p.method == mcc.N97, fac / (pm * pm * vr), U1, U4)
            d = _rotate(ps, st, omc, 2.0 * math.pi * U2)
            d = d + (co * (V * d).sum(1))[:, None] * V
        else:
            mu, u = ma * mb / (ma + mb), va - vb
            um = u.norm(dim=1)
            st, omc = _angle(p.method == mcc.N97, fac / (mu * mu * um ** 3), U1, U4)
            d = mu * _rotate(u, st, omc, 2.0 * math.pi * U2)
        moves = (U3 * wmax < wmin) | (wa == wb)
        v = _put(v, a, torch.where((moves | (wa < wb))[:, None], va + d / ma, va))
        v = _put(v, b, torch.where((moves | (wb < wa))[:, None], vb - d / mb, vb))
    return v


def _put(v, idx, x):
    if v.requires_grad or x.requires_grad:
        return v.index_copy(0, idx, x)
    v[idx] = x
    return v


def _per_cell(C, cell, x):
    return torch.zeros((C,) + x.shape[1:], dtype=x.dtype, device=DEV).index_add(0, cell, x)


def _ke(rel, v):
    v2 = (v * v).sum(1)
    return v2 / (_gamma(v) + 1.0) if rel else 0.5 * v2


def _kecm(rel, m1, m2, a, b):
    if not rel:
        return 0.5 * m1 * m2 / (m1 + m2) * ((a - b) ** 2).sum(1)
    g = _gamma_rel_m1(a, b)
    return 2.0 * m1 * m2 * g / (torch.sqrt((m1 + m2) ** 2 + 2.0 * m1 * m2 * g) + m1 + m2)


def _energy_pair(rel, m1, m2, a, b, K, U):
    """The pair with its centre-of-mass energy K lowered by U at zero angle."""
    du = a - b
    if not rel:
        x = U / K
        g = (-x / (1.0 + torch.sqrt(1.0 - x)))[:, None]
        return a + (m2 / (m1 + m2))[:, None] * g * du, b - (m1 / (m1 + m2))[:, None] * g * du
    E1, E2 = m1 * _gamma(a), m2 * _gamma(b)
    A = E1 + E2 - U
    pt = m1[:, None] * a + m2[:, None] * b
    x12 = (m1 * m2)[:, None] * (_gamma(b)[:, None] * du - _dgamma(a, b)[:, None] * b)
    bv = (2.0 * A)[:, None] * (x12 + (U * m2)[:, None] * b) - (U * (2.0 * E1 - U))[:, None] * pt
    qa = 4.0 * (A * A * (du * du).sum(1) - (pt * du).sum(1) ** 2)
    qb = 4.0 * (du * bv).sum(1)
    qc = U * (2.0 * E1 - U) * (2.0 * E2 - U) * (2.0 * E1 + 2.0 * E2 - U)
    qq = -0.5 * (qb + torch.where(qb >= 0, 1.0, -1.0) * torch.sqrt((qb * qb - 4.0 * qa * qc).clamp(min=0.0)))
    r1, r2 = qq / qa, qc / qq
    al = torch.where(r1.abs() < r2.abs(), r1, r2)
    return a + (al / m1)[:, None] * du, b - (al / m2)[:, None] * du


def _absorb(v, w, p, rel, m, rho, n, D):
    """Energy pairs of one species: rho (particles in pair order, cell after cell), D the violation per cell."""
    start = torch.cumsum(n, 0) - n
    top = int(n.max())
    for ps in range(p.max_corr_passes):
        for t in range(ps % 2, top - 1, 2):
            c = torch.nonzero((D.detach() != 0) & (n > t + 1)).squeeze(1)
            if c.numel() == 0:
                if t == ps % 2 and not bool((D.detach() != 0).any()):
                    return v, D
                break
            i, j = rho[start[c] + t], rho[start[c] + t + 1]
            a, b, m1, m2, Dc = v[i], v[j], m * w[i], m * w[j], D[c]
            K = _kecm(rel, m1, m2, a, b)
            ok = K.detach() > 0
            if not bool(ok.all()):
                c, i, j, a, b, m1, m2, Dc, K = (z[ok] for z in (c, i, j, a, b, m1, m2, Dc, K))
            cap = p.fE * K
            last = Dc.detach().abs() < cap.detach()
            U = torch.where(last, Dc, torch.sign(Dc.detach()) * cap)
            a, b = _energy_pair(rel, m1, m2, a, b, K, U)
            v = _put(_put(v, i, a), j, b)
            D = _put(D, c, torch.where(last, torch.zeros_like(Dc), Dc - U))
    return v, D


def _correct(v, vb, w, p, C, intra, sides, active):
    """Moment correction of one interaction: sides = [(mass, idx, cell, order, n)] of its one or two species."""
    rel = p.relativistic
    num, den = 0.0, 0.0
    for m, idx, cell, _, _ in sides:
        num = num + _per_cell(C, cell, (m * w[idx])[:, None] * (v[idx] - vb[idx]))
        den = den + _per_cell(C, cell, m * w[idx] ** 2)
    B = num / torch.where(den > 0, den, torch.ones_like(den))[:, None]
    dE, Es, wbar = 0.0, [], []
    for m, idx, cell, _, n in sides:
        x, y = v[idx] - B[cell] * w[idx][:, None], vb[idx]
        v = _put(v, idx, x)
        d = ((x - y) * (x + y)).sum(1)
        d = d / (_gamma(x) + _gamma(y)) if rel else 0.5 * d
        dE = dE + _per_cell(C, cell, m * w[idx] * d)
        Es.append(_per_cell(C, cell, m * w[idx] * _ke(rel, x)))
        wbar.append(_per_cell(C, cell, w[idx]) / n.clamp(min=1))
    Ds = [dE]
    fail = torch.zeros(C, dtype=torch.bool, device=DEV)
    if not intra:
        can = [s[4] >= 2 for s in sides]
        both = can[0] & can[1]
        f = wbar[0] * Es[0] / torch.where(both, wbar[0] * Es[0] + wbar[1] * Es[1], torch.ones_like(dE))
        zero = torch.zeros_like(dE)
        D0 = torch.where(both, f * dE, torch.where(can[0], dE, zero))
        Ds = [D0, torch.where(both, dE - D0, torch.where(can[0], zero, torch.where(can[1], dE, zero)))]
        fail = ~can[0] & ~can[1] & (dE != 0) & active
    for (m, idx, cell, order, n), D, E in zip(sides, Ds, Es):
        D = torch.where((D.detach().abs() <= 2.0 ** -47 * E.detach()) | fail | ~active, torch.zeros_like(D), D)
        v, D = _absorb(v, w, p, rel, m, order, n, D)
        fail = fail | (D.detach() != 0)
    if bool(fail.any()):
        for _, idx, cell, _, _ in sides:
            back = idx[fail[cell]]
            v = _put(v, back, vb[back])
    return v


def _step(v, w, off, C, S, species, lnL, p, step):
    """One collision step, every interaction in order; v is (particles, 3) in 64 bits."""
    counts = (off[1:] - off[:-1]).view(C, S)
    starts = off[:-1].view(C, S)
    seg = torch.repeat_interleave(torch.arange(C * S, device=DEV), counts.reshape(-1), output_size=int(off[-1]))
    wk = _weight_bits(w) ^ torch.iinfo(torch.int64).min
    if not (v.requires_grad or w.requires_grad):
        v = v.clone()
    for inter, (a, b) in enumerate(mcc.default_interactions(S)):
        intra = a == b
        na, nb = counts[:, a], counts[:, b]
        active = na >= 2 if intra else (na > 0) & (nb > 0)
        sides, perms = [], []
        for side, s in enumerate((a,) if intra else (a, b)):
            n = torch.where(active, counts[:, s], torch.zeros_like(na))
            cell, q = _permutation(p, step, inter, side, n)
            perm = starts[cell, s] + q
            by = torch.argsort(wk[perm], stable=True)  # descending weight, ties in the random order
            order = perm[by[torch.argsort(seg[perm][by], stable=True)]]
            idx = starts[cell, s] + _ranges(n)[1]
            sides.append((species[s][1], idx, cell, order, n))
            perms.append((perm, torch.cumsum(n, 0) - n))
        vb = v.clone() if not v.requires_grad else v
        if intra:
            odd = (na & 1) == 1
            npairs = torch.where(active, torch.where(odd, (na + 3) // 2, na // 2), torch.zeros_like(na))
            cell, k = _ranges(npairs)
            o = odd[cell]
            trip = o & (k < 3)
            first = torch.where(trip, k, torch.where(o, 2 * k - 3, 2 * k))
            second = torch.where(trip, (k + 1) % 3, first + 1)
            perm, st = perms[0]
            i, j = perm[st[cell] + first], perm[st[cell] + second]
            rnd, nmin = torch.where(trip, k, torch.zeros_like(k)), (na - 1).double()
        else:
            lo, hi = torch.minimum(na, nb), torch.maximum(na, nb)
            cell, k = _ranges(torch.where(active, hi, torch.zeros_like(hi)))
            m = k % lo[cell]
            big = (na >= nb)[cell]
            i = perms[0][0][perms[0][1][cell] + torch.where(big, k, m)]
            j = perms[1][0][perms[1][1][cell] + torch.where(big, m, k)]
            trip, rnd, nmin = torch.zeros_like(k, dtype=torch.bool), k // lo[cell], lo.double()
        L = lnL[a, b] if torch.is_tensor(lnL) else lnL
        v = _scatter(v, w, p, step, inter, intra, cell, k, i, j, trip, rnd, species[a], species[b], L, nmin)
        v = _correct(v, vb, w, p, C, intra, sides, active)
    return v
