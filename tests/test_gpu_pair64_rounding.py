"""Rounding of the FP64 pair kinematics: velocity changes of single pairs against extended precision, beside the same formulas
in plain double (numpy). One particle of each pair is at rest, so that its velocity after the scatter is the change itself,
not rounded into a larger one. Every operation of the device's form is corrected to about half a unit of the last place, so
its rms error is that of plain double up to the spread of the samples: at most 1.1 times (uncorrected reciprocal roots
give 1.13 to 1.24)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2407_19151_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N = 20000
SEED, STEP, LNL = 0x1234567, 6, 10.0


def _philox():
    return np.array([O.philox4x32_10([0, c, STEP, 3], [SEED, 0]) for c in range(N)], dtype=np.uint32)


def _turn(k, T):
    """cos and sin of 2 pi (k + 1/2) 2^-23, the angle reduced to the nearest quarter turn in whole numbers."""
    h = 2 * k.astype(np.int64) + 1  # in 2^-24 of a turn
    q = (h + (1 << 21)) >> 22
    a = (h - (q << 22)).astype(np.longdouble) * (8 * np.arctan(np.longdouble(1)) / (1 << 24))
    c, s = np.cos(a), np.sin(a)
    q = q % 4
    cs = np.where(q == 0, c, np.where(q == 1, -s, np.where(q == 2, -c, s)))
    sn = np.where(q == 0, s, np.where(q == 1, c, np.where(q == 2, -s, -c)))
    return cs.astype(T), sn.astype(T)


def _angle(method, s, r, T):
    U1 = ((r[:, 0] >> 9).astype(T) + T(0.5)) * T(2.0 ** -23)
    if method == W.TA77:
        d = np.sqrt(T(0.5) * s) * (np.sqrt(T(-2) * np.log(U1)) * _turn(r[:, 3] >> 9, T)[0])
        den = T(1) + d * d
        return T(2) * d / den, T(2) * d * d / den
    A = T(-1) / np.expm1(-s)  # e^-2A vanishes over the sampled lengths (s < 0.01: A > 100)
    o = -np.log1p(-U1) / A
    return np.sqrt(o * (T(2) - o)), o


def _rotate(u, um, st, omc, cp, sp, T):
    up = np.sqrt(u[0] * u[0] + u[1] * u[1])
    ax, ay = u[0] / up, u[1] / up
    return [ax * u[2] * st * cp - ay * um * st * sp - u[0] * omc, ay * u[2] * st * cp + ax * um * st * sp - u[1] * omc,
            -up * st * cp - u[2] * omc]


def _change(method, rel, kappa, u, r, T):
    """Velocity change of the first particle of a pair of unit masses (c = 1); the first moves at u, the second is at rest."""
    u = [x.astype(T) for x in u]
    cp, sp = _turn(r[:, 1] >> 9, T)
    u2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    if not rel:
        um = np.sqrt(u2)
        st, omc = _angle(method, kappa.astype(T) * T(4) / (u2 * um), r, T)
        return [T(0.5) * x for x in _rotate(u, um, st, omc, cp, sp, T)]
    g = np.sqrt(T(1) + u2)
    M = g + T(1)
    V = [x / M for x in u]
    dg = u2 / (g + T(1))
    grm1 = np.maximum(T(0.5) * (u2 - dg * dg), T(0))
    gC = M / np.sqrt(T(4) + T(2) * grm1)
    cb = gC * gC / (gC + T(1))
    q = [x / M for x in u]
    Vq = V[0] * q[0] + V[1] * q[1] + V[2] * q[2]
    p = [a + cb * Vq * b for a, b in zip(q, V)]
    p2 = p[0] * p[0] + p[1] * p[1] + p[2] * p[2]
    pm = np.sqrt(p2)
    st, omc = _angle(method, kappa.astype(T) / (p2 * (pm * (T(2) / np.sqrt(T(1) + p2)))), r, T)
    d = _rotate(p, pm, st, omc, cp, sp, T)
    Vd = V[0] * d[0] + V[1] * d[1] + V[2] * d[2]
    return [a + cb * Vd * b for a, b in zip(d, V)]


@pytest.mark.parametrize("method", [W.TA77, W.N97])
@pytest.mark.parametrize("rel", [False, True])
def test_rounding_of_pairs(method, rel):
    import paper_2407_19151_gb300 as mcc
    rng = np.random.default_rng(17)
    u = rng.normal(size=(3, N))
    um = np.sqrt((u ** 2).sum(0))
    s = np.exp(rng.uniform(np.log(1e-7), np.log(1e-2), N))
    if rel:
        pm = np.sqrt((np.sqrt(1 + um ** 2) - 1) / 2)
        kappa = s * pm ** 3 * 2 / np.sqrt(1 + pm ** 2)
    else:
        kappa = s * um ** 3 / 4
    w = np.repeat(kappa, 2)  # the weight carries kappa: q = 1 and lnL dt / (4 pi eps0^2 dV) = 1
    off = torch.arange(0, 2 * N + 1, 2, dtype=torch.int64, device="cuda")
    pi, pj, _ = mcc.mcc_pair(off, N, 1, 0, 0, 0, SEED, STEP)
    pi = pi[::2].cpu().numpy()
    v = np.zeros((3, 2 * N))
    v[:, pi] = u  # the first particle of each pair moves
    dv = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in v]
    par = mcc.Params(method=method, relativistic=rel, dt=4 * np.pi / LNL, c=1.0, seed=SEED, step=STEP, correct=False)
    mcc.mcc_step_fused(*dv, torch.from_numpy(w).cuda(), off, N, 1, [(1.0, 1.0)], LNL, par, max_cell=2)
    mcc.sync_status(0)
    got = np.stack([x.cpu().numpy() for x in dv])[:, 4 * np.arange(N) + 1 - pi]
    k = (LNL * (4 * np.pi / LNL)) / (4.0 * np.pi) * w[::2]  # as the library forms it
    r = _philox()
    exact = -np.stack(_change(method, rel, k, u, r, np.longdouble))  # the second particle loses what the first gains
    plain = -np.stack(_change(method, rel, k, u, r, np.float64))
    rms = lambda x: float(np.sqrt((((x - exact) ** 2).sum(0) / (exact ** 2).sum(0)).mean()))  # noqa: E731
    mine, theirs = rms(got), rms(plain)
    print(f"rms error of a pair's change: {mine:.3e}, plain double {theirs:.3e}")
    assert theirs < 4e-16
    assert mine <= 1.1 * theirs
