"""Coulomb logarithms that are accepted but odd: negative (no scattering under N97, whose 1 - e^-s is then negative), zero, infinite
and not a number (isotropic), on both precisions, against the oracle on the same inputs."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2407_19151_gb300 import workloads as W

from _parity import F32_TOL, F64_TOL, device_state, gpu_velocities, oracle_state, velocity_error

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lnL", [-10.0, 0.0, np.inf, np.nan])
def test_scatter_order_nxn(lnL):
    import paper_2407_19151_gb300 as mcc
    wl = W.three_species(n_cells=20, mean_count=12.0, precision="f64")
    kw = dict(method=W.N97, dt=wl.dt, seed=wl.seed, step=4, correct=False, pairing=1)
    v, w, off = device_state(wl, "f64")
    mcc.mcc_step_fused(*v, w, off, wl.n_cells, 3, list(zip(wl.q, wl.m)), lnL, mcc.Params(**kw))
    mcc.sync_status(0)
    st = oracle_state(wl, "f64")
    before = st.v().copy()
    O.step(st, wl.q, wl.m, np.full((3, 3), lnL), O.Params(**kw), n_steps=1)
    got = gpu_velocities(v)
    if lnL <= 0:
        np.testing.assert_array_equal(got, before)
    assert velocity_error(got, st.v(), wl.offsets).max() < F64_TOL


@pytest.mark.parametrize("rel", [False, True])
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("lnL", [-10.0, -1e-3, 0.0, np.inf, np.nan])
def test_scatter(lnL, prec, rel):
    import paper_2407_19151_gb300 as mcc
    wl = W.relativistic_beam(n_cells=20, count_hi=200, precision=prec) if rel else \
        W.three_species(n_cells=20, mean_count=60.0, precision=prec)
    kw = dict(method=W.N97, relativistic=rel, dt=wl.dt, c=wl.c, seed=wl.seed, step=4, correct=False)
    v, w, off = device_state(wl, prec)
    mcc.mcc_step_fused(*v, w, off, wl.n_cells, 3, list(zip(wl.q, wl.m)), lnL, mcc.Params(**kw))
    mcc.sync_status(0)
    st = oracle_state(wl, prec)
    before = st.v().copy()
    O.step(st, wl.q, wl.m, np.full((3, 3), lnL), O.Params(**kw), n_steps=1)
    got = gpu_velocities(v)
    assert np.isfinite(got).all()
    if lnL <= 0:
        np.testing.assert_array_equal(got, before)
    # (isotropic: many large angles in a row, a few times the small-angle bound on the mixed path)
    assert velocity_error(got, st.v(), wl.offsets).max() < (F64_TOL if prec == "f64" else 4 * F32_TOL)


def test_ta77_not_a_number_stays_one():
    import paper_2407_19151_gb300 as mcc
    wl = W.three_species(n_cells=5, mean_count=60.0, precision="f64")
    v, w, off = device_state(wl, "f64")
    p = mcc.Params(method=W.TA77, dt=wl.dt, seed=1, correct=False)
    mcc.mcc_step_fused(*v, w, off, wl.n_cells, 3, list(zip(wl.q, wl.m)), float("nan"), p)
    mcc.sync_status(0)
    st = oracle_state(wl, "f64")
    O.step(st, wl.q, wl.m, np.full((3, 3), np.nan), O.Params(method=W.TA77, dt=wl.dt, seed=1, correct=False), n_steps=1)
    np.testing.assert_array_equal(np.isnan(gpu_velocities(v)), np.isnan(st.v()))
