"""Kernel forms at the sizes where they change: the count of listed enthalpy
tiles (by the solve kernel up to 1152 tiles, by a list above), the stamps of a
context whose fields are loaded again after an odd number of steps, the
reduction's FP32-pair sums, and what the adjoints' forward runs read of tiles
that the next step's pass may already take.
"""
import numpy as np
import pytest

import lbm_workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build()
    import paper_1503_08406_gb300 as P
    return P


def _f32(w):
    for k in ("phi", "K", "T0", "fl0"):
        setattr(w, k, getattr(w, k).astype(np.float32).astype(np.float64))
    return w


# one row of tiles, 1 to 1153 of them; many listed (a noisy temperature field)
@pytest.mark.parametrize("nx", [32, 33, 36864, 36865, 36896])
def test_listed_tiles_counted_or_listed(P, oracle_mod, nx):
    w = _f32(W.periodic_box(nx, ny=12))
    lat = P.Lattice(w.nx, w.ny, **w.params)
    lat.set_fields(w.phi, w.K, w.T0, w.fl0)
    lat.step(5)
    assert lat.status() == 0
    o = oracle_mod.Oracle(w.nx, w.ny, **w.params)
    o.set_fields(w.phi, w.K, w.T0, w.fl0)
    o.step(5)
    got, exp = lat.macros(), o.macros()
    for k in ("ux", "uy", "T", "fl"):   # the short-run bar of the parity tests
        assert np.abs(got[k] - exp[k]).max() < 2e-5 * np.abs(exp[k]).max(), k


@pytest.mark.parametrize("lead", [1, 2, 3])
def test_fields_loaded_again_leave_no_stamps(P, lead):
    """A context stepped, then loaded with fields whose front lies elsewhere,
    continues as a new one does."""
    a, b = W.melted_cavity(96, melted_cols=70), W.melted_cavity(96, melted_cols=20)
    used, new = (P.Lattice(96, 96, **b.params) for _ in range(2))
    used.set_fields(a.phi, a.K, a.T0, a.fl0)
    for _ in range(lead):
        used.step(1)
    for lat in (used, new):
        lat.set_fields(b.phi, b.K, b.T0, b.fl0)
        lat.step(7)
    for x, y in zip(used.get_state(), new.get_state()):
        assert np.array_equal(x.view(np.uint32), y.view(np.uint32))


@pytest.mark.parametrize("steps", [4, 5])
@pytest.mark.parametrize("over", [{}, {"storage": "fp16"}, {"flow_walls": 1},
                                  {"sigma_solid": 0.5}, {"T_l": 0.1}])
def test_reduce_equals_fp64_sums_of_the_state(P, steps, over):
    w = W.melted_cavity(77)
    p = {**w.params, **over}
    lat = P.Lattice(77, 77, **p)
    lat.set_fields(w.phi, w.K, w.T0, w.fl0)
    lat.step(steps)
    _check_sums(lat, w, p)


def test_reduce_beyond_fp32_range(P):
    """Deviations whose FP32 sum overflows, not their FP64 sum."""
    w = W.melted_cavity(40)
    lat = P.Lattice(40, 40, **w.params)
    lat.set_fields(w.phi, w.K, w.T0, w.fl0)
    f, g, fl = lat.get_state()
    f[:, 5, 5] = 3e38
    lat.set_state(f, g, fl)
    _check_sums(lat, w, w.params)


def _check_sums(lat, w, p):
    """Against the same sums of the checkpoint in FP64 (T is the FP32 sum of its
    populations); both add at most 1e4 terms of one sign in FP64, each within
    2^-48 of exact: 1e-12 covers it."""
    f, g, fl = lat.get_state()
    got = lat.reduce()
    inside = np.zeros_like(fl, dtype=bool)
    inside[1:-1, 1:-1] = True
    T = g[0]
    for i in range(1, 5):
        T = T + g[i]
    fl = fl.astype(np.float64)
    sl, ss = p["sigma"], p.get("sigma_solid") or p["sigma"]
    a = w.phi.astype(np.float32).astype(np.float64) * np.float64(np.float32(
        p["dT"] / (p["sigma"] * p["St"]))) * np.float32(sl) / (
            np.float32(ss) + fl * (np.float64(np.float32(sl)) - np.float32(ss)))
    mass = (1.0 + f.astype(np.float64).sum(0))[inside].sum()
    heat = (T.astype(np.float64) + a * fl)[inside].sum()
    assert abs(got["mass"] - mass) <= 1e-12 * abs(mass)
    assert abs(got["enthalpy"] - heat) <= 1e-12 * abs(heat)
    assert abs(got["melt_frac"] - fl[inside].mean()) <= 1e-12


def _cavity_with_far_walls(flow):
    """The front 140 nodes from the hot wall, so that the wall's tiles and most
    of the liquid are away from it."""
    w = W.adjoint_cavity(256, source_n=256, melted=0.55) if flow else W.adjoint_slab(512, 64)
    if not flow:
        x = np.arange(w.nx)[None, :]
        w.T0[:, :] = np.where(x < 140, 1.0 - x / 140.0, -1.0)
        w.fl0[:, :] = np.where(w.T0 > 0.3, 1.0, np.where(w.T0 < -0.3, 0.0, 0.5))
    return w


@pytest.mark.parametrize("flow", [0, 1])
def test_nusselt_objective_reads_every_step(P, flow):
    """J is the mean of the hot-wall Nusselt number after each step (the same
    FP64 sum in another order: 1e-11), whichever schedule the forward run has."""
    w = _cavity_with_far_walls(flow)
    lat = P.Lattice(w.nx, w.ny, **w.params)
    lat.set_fields(w.phi, w.K, w.T0, w.fl0, w.wall_T_left)
    nus = []
    for _ in range(20):
        lat.step(1)
        nus.append(lat.reduce()["nu_hot"])
    runs = []
    for every in (0, 5):
        lat.set_fields(w.phi, w.K, w.T0, w.fl0, w.wall_T_left)
        run = lat.adjoint_coupled if flow else lat.adjoint
        runs.append(run(20, "nusselt", checkpoint_every=every))
        assert abs(runs[-1][0] - np.mean(nus)) <= 1e-11 * abs(np.mean(nus))
    for a, b in zip(runs[0][1:], runs[1][1:]):   # same states, same bits
        assert np.array_equal(a, b)
