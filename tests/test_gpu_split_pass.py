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
        assert np.isfinite(x).all()
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


# ---- the forms of the near-tile pass ------------------------------------------
#
# Ordinary loads: asking every tile, by flags (up to 1152 enthalpy tiles) or the near
# map; from the list, above eight 32x8 tiles for each of the solve's CTAs (two per
# SM, so 2432 of them on 152 SMs).  Tensor maps: asking, or from the list as soon as
# the solve has fewer CTAs than tiles.

def _cavity(nx, ny):
    """A walled cavity whose front winds through many tiles, their surroundings
    overlapping."""
    w = W.melted_cavity(64)
    w.nx, w.ny = nx, ny
    w.params = {**w.params, "H": float(ny)}
    rng = np.random.default_rng(nx * ny)
    w.phi = 0.35 + 0.2 * rng.random((ny, nx))
    w.K = W.kozeny_carman_K(w.phi, 1e-4 * ny * ny)
    yy, xx = np.mgrid[0:ny, 0:nx]
    m = nx * (0.4 + 0.15 * np.sin(5 * np.pi * yy / ny))
    w.fl0 = (xx < m).astype(np.float64)
    w.T0 = np.where(xx < m, 1.0 - xx / (2.0 * m), 0.0)
    w.T0[:, 0], w.fl0[:, 0] = 1.0, 1.0
    return w


@pytest.mark.parametrize("nx,ny,over", [
    (1000, 704, {}),                                        # 704 tiles, counted by the solve
    (1000, 704, {"flow": 0, "tau_T": 0.8}),
    (1000, 704, {"storage": "fp16"}), (1000, 704, {"storage": "bf16"}),
    (1000, 704, {"flow_walls": 1}), (1000, 704, {"flow_walls": 1, "storage": "fp16"}),
    (1000, 704, {"flow_front": 1, "flow_walls": 1, "storage": "bf16"}),
    (1024, 1024, {}), (1024, 1024, {"storage": "fp16"}),
    (1240, 1000, {}),                                       # 1248 tiles: list and near map
    (1240, 1000, {"storage": "bf16", "flow_front": 1}),
    (320, 300, {}),                                         # 100 tiles: one CTA each
    (640, 600, {"storage": "fp16", "flow_walls": 1})])      # 380 tiles: asks every tile
def test_walled_lattices(P, nx, ny, over):
    w = _cavity(nx, ny)
    one = _run(P, w, [1] * STEPS, kernel_variant=1, **over)
    for variant in (1, 2):
        _same(_run(P, w, (35, STEPS - 35), kernel_variant=variant, **over), one)


# (1002: rows that no tensor map fits)
@pytest.mark.parametrize("over", [{}, {"storage": "fp16"}])
def test_walled_lattice_without_tensor_maps(P, over):
    _check_split(P, _cavity(1002, 701), **over)


# periodic boxes above 2432 tiles of 32x8; one, two and three enthalpy tiles across,
# where a tile is reached from both sides, and narrow last tiles along them
@pytest.mark.parametrize("nx,ny", [(1024, 640), (1280, 1024), (30, 20000), (40, 20000),
                                   (72, 8200), (9000, 72), (40, 20003), (20005, 40)])
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_periodic_boxes(P, nx, ny, storage):
    w = _strip_box(nx, ny, nx // 2 if nx >= ny else None, 3 if ny > nx else None)
    rng = np.random.default_rng(7)   # and 40 melted spots, beside one another here and there
    for _ in range(40):
        x, y = rng.integers(nx), rng.integers(ny)
        w.T0[y:y + 6, x:x + 6] = 0.8
        w.fl0[y:y + 6, x:x + 6] = 1.0
    _check_split(P, w, storage=storage)


def test_flow_walls_16_bit(P, oracle_mod):
    """Extrapolated walls with 16-bit storage against the FP64 oracle: the parity
    cavity and the bars of the storage tests, whose rounding is the same (a wall node
    stores its populations like any other)."""
    w = W.parity_cavity(256)
    for k in ("phi", "K", "T0", "fl0"):
        setattr(w, k, getattr(w, k).astype(np.float32).astype(np.float64))
    o = oracle_mod.Oracle(w.nx, w.ny, **{**w.params, "flow_walls": 1})
    o.set_fields(w.phi, w.K, w.T0, w.fl0)
    o.step(1000)
    exp = o.macros()
    for storage, bar in (("fp16", dict(ux=0.03, uy=0.03, T=3e-3, fl=1e-2)),
                         ("bf16", dict(ux=0.2, uy=0.2, T=2e-2, fl=5e-2))):
        lat = P.Lattice(w.nx, w.ny, **{**w.params, "flow_walls": 1, "storage": storage})
        lat.set_fields(w.phi, w.K, w.T0, w.fl0)
        lat.step(1000)
        assert lat.status() == 0
        got = lat.macros()
        for k, b in bar.items():
            assert np.abs(got[k] - exp[k]).max() < b * np.abs(exp[k]).max(), (storage, k)
