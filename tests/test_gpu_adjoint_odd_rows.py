"""Adjoints on a periodic y axis of odd length, where the last row of the band
meets the first: gradients against the FP64 reference, and the same bits from
every repeat and every checkpoint spacing (each lists the band's nodes in an
order of its own).
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
    for k in ("phi", "K", "T0", "fl0", "wall_T_left"):
        setattr(w, k, getattr(w, k).astype(np.float32).astype(np.float64))
    return w


def _run(P, w, steps, objective, every):
    lat = P.Lattice(w.nx, w.ny, **w.params)
    lat.set_fields(w.phi, w.K, w.T0, w.fl0, w.wall_T_left)
    out = (lat.adjoint_coupled if w.params["flow"] else lat.adjoint)(
        steps, objective, checkpoint_every=every)
    assert lat.status() == 0
    return out


def _same_bits(P, w, steps, objective):
    runs = [_run(P, w, steps, objective, every) for every in (0, 0, 0, 7, 1)]
    for r in runs[1:]:
        for a, b in zip(runs[0][1:], r[1:]):
            assert np.isfinite(a).all() and np.abs(a).max() > 0
            assert np.array_equal(a, b)
    return runs[0]


def _check(got, ref, names, tol=1e-3):   # the bars of the adjoints' other tests
    assert abs(got[0] - ref[0]) < 1e-4 * abs(ref[0])
    for name, g, e in zip(names, got[1:], ref[1:]):
        assert np.abs(g - e).max() < tol * np.abs(e).max(), name


@pytest.mark.parametrize("objective", ["melt", "nusselt"])
@pytest.mark.parametrize("ny", [3, 5])
def test_conduction_odd_rows(P, oracle_mod, ny, objective):
    from oracle.adjoint_ref import ConductionRef
    w = _f32(W.adjoint_slab(40, ny, seed=2))
    got = _same_bits(P, w, 400, objective)
    ref = ConductionRef(w.nx, w.ny, w.params).gradients(400, w.T0, w.fl0, w.phi, w.wall_T_left,
                                                        objective=objective)
    _check(got, ref, ("phi", "Tw"))


def _mushy(w):
    """Every node between solid and liquid: the band is the whole interior."""
    rng = np.random.default_rng(3)
    p = w.params
    mid, half = 0.5 * (p["T_s"] + p["T_l"]), 0.5 * (p["T_l"] - p["T_s"])
    w.T0 = mid + 0.5 * half * rng.uniform(-1, 1, (w.ny, w.nx))
    w.fl0 = (w.T0 - p["T_s"]) / (p["T_l"] - p["T_s"])
    return _f32(w)


# bands solved in shared memory (up to 4096 nodes) and beyond it
@pytest.mark.parametrize("nx,ny", [(40, 99), (200, 101)])
def test_conduction_wide_band_odd_rows(P, nx, ny):
    _same_bits(P, _mushy(W.adjoint_slab(nx, ny)), 21, "melt")


@pytest.mark.parametrize("ny", [23, 24])
def test_coupled_channel(P, oracle_mod, ny):
    """The small melted cavity as a channel periodic in y, odd and even."""
    from oracle.coupled_ref import CoupledRef
    w = W.melted_cavity(24)
    w.ny = ny
    w.phi, w.K, w.T0, w.fl0 = (a[:ny].copy() for a in (w.phi, w.K, w.T0, w.fl0))
    w.params = {**w.params, "T_s": 0.1, "T_l": 0.4,
                "bc": ("dirichlet", "dirichlet", "periodic", "periodic")}
    w.wall_T_left = 1.0 + 0.1 * np.sin(2 * np.pi * np.arange(ny) / ny)
    w = _f32(w)
    got = _same_bits(P, w, 40, "melt")
    ref = CoupledRef(w.nx, w.ny, w.params).gradients(40, w.T0, w.fl0, w.phi, w.K, w.wall_T_left,
                                                     "melt")
    _check(got, ref, ("phi", "lnK", "Tw"))


def test_coupled_wide_band_odd_rows(P):
    w = W.adjoint_cavity(128)
    w.ny = 127
    w.phi, w.K, w.T0, w.fl0 = (a[:127].copy() for a in (w.phi, w.K, w.T0, w.fl0))
    w.params = {**w.params, "bc": ("dirichlet", "dirichlet", "periodic", "periodic")}
    w.wall_T_left = np.ones(127)
    _same_bits(P, _mushy(w), 15, "melt")
