"""The liquid fraction at which a node carries flow, at and beyond full melt:
with f_act = 1 fully liquid nodes flow, above 1 none does, in both stream-collide
kernels (whose bits are the same) and in every storage.
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


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("f_act", [1.0, 1.0000001192092896, 2.0])
@pytest.mark.parametrize("steps", [8, 9])
def test_flow_threshold_at_full_melt(P, storage, f_act, steps):
    w = W.melted_cavity(128, melted_cols=100)   # whole tiles of liquid away from the walls
    runs = []
    for variant in (1, 2):
        lat = P.Lattice(w.nx, w.ny, **{**w.params, "storage": storage, "f_act": f_act,
                                       "kernel_variant": variant})
        lat.set_fields(w.phi, w.K, w.T0, w.fl0)
        lat.step(steps)
        assert lat.status() == 0 and lat.kernel_variant() == variant
        m = lat.macros()
        assert (np.abs(m["ux"]).max() > 0) == (f_act <= 1.0)
        runs.append(lat.get_state())
        if f_act > 1.0:   # nothing moves: the populations stay at rest
            assert not np.any(runs[-1][0])
    for a, b in zip(*runs):
        assert np.array_equal(a, b)
