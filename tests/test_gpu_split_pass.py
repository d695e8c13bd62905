"""Steps of a CUDA graph, whose stream-collide pass is split into the tiles away
from the last step's front (run beside its enthalpy kernels) and those near it,
against the same steps taken one by one, whose pass is whole: the same bits.
"""
import numpy as np
import pytest

import lbm_workloads as W

pytestmark = pytest.mark.gpu

STEPS = 69   # a 64-step graph and shorter ones, from both parities


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__
    __graft_entry__.build()
    import paper_1503_08406_gb300 as P
    return P


def _run(P, w, chunks, **over):
    lat = P.Lattice(w.nx, w.ny, **{**w.params, **over})
    lat.set_fields(w.phi, w.K, w.T0, w.fl0, w.wall_T_left)
    for n in chunks:
        lat.step(n)
    assert lat.status() == 0
    return lat.get_state()


def _same(a, b):
    for k, (x, y) in enumerate(zip(a, b)):
        diff = np.flatnonzero(x.view(np.uint32) != y.view(np.uint32))
        assert diff.size == 0, (("f", "g", "fl")[k], diff.size, diff[:8])


def _check_split(P, w, **over):
    # (35: an odd number, so that the second graph starts from the other parity)
    _same(_run(P, w, (35, STEPS - 35), **over), _run(P, w, [1] * STEPS, **over))


def _strip_box(nx, ny, cx, cy):
    """A periodic box, solid but for the nodes within 4 of column cx and of row cy
    (None: no such strip), across the edge of the lattice where they lie there."""
    w = W.periodic_box(nx, ny=ny)
    yy, xx = np.mgrid[0:ny, 0:nx]
    far = lambda a, c, n: np.minimum(abs(a - c), n - abs(a - c))
    liquid = np.zeros((ny, nx), dtype=bool)
    if cx is not None:
        liquid |= far(xx, cx, nx) <= 4
    if cy is not None:
        liquid |= far(yy, cy, ny) <= 4
    rng = np.random.default_rng(nx + ny)
    w.T0 = np.where(liquid, 0.8, -0.2) + 0.05 * rng.standard_normal((ny, nx))
    w.fl0 = liquid.astype(np.float64)
    return w


# a last tile of 1 to 7 nodes on a periodic axis: the enthalpy regions of the tile
# before it, of itself and of tile 0 reach through it
@pytest.mark.parametrize("nx,ny,cx,cy", [
    (129, 100, 0, None), (129, 100, 120, None), (129, 100, 128, None), (135, 64, 6, None),
    (100, 131, None, 2), (64, 131, None, 122), (133, 130, 131, 1)])
@pytest.mark.parametrize("flow", [0, 1])
def test_narrow_last_tile_of_a_periodic_axis(P, nx, ny, cx, cy, flow):
    w = _strip_box(nx, ny, cx, cy)
    over = {"flow": flow} if flow else {"flow": 0, "tau_T": 0.8}
    _check_split(P, w, **over)


def test_narrow_last_tiles_of_a_mapped_lattice(P):
    """1419 tiles: the near map and the tiles across both edges."""
    _check_split(P, _strip_box(4099, 323, 2, 321))
