"""Tiles that overhang the grid and tiles cut into slabs: the automatic choice
on grids that 4 x 4 x 32 and 8 x 8 x 8 do not divide, and on grids of so few
tiles that each is cut along x, against the FP64 oracle and against the same
run on tiles that divide the grid."""
import numpy as np
import pytest

from gpu_helpers import Case, by_id, rel_l2
from paper_2101_12149_gb300 import inputs, pic

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [pic.FP64, pic.FP32_MIXED])
@pytest.mark.parametrize("n,order", [
    ((9, 7, 11), 3),      # 8 x 8 x 8, one cell over along x, z not a multiple of 4 (no TMA, scalar flush)
    ((13, 10, 40), 1),    # order 1: 4 x 4 x 32 overhanging (FP32-mixed: halo 1), z a multiple of 4 (TMA)
    ((18, 6, 62), 2),     # 4 x 4 x 32 overhanging in y and z
    ((5, 6, 33), 3),      # one cell in the last z tile
    ((17, 24, 9), 2),     # 8 x 8 x 8 overhanging in x and z
    ((5, 5, 5), 3),       # one tile larger than the grid, its halo more than one period
    ((16, 16, 16), 1),    # 8 tiles in slabs of one plane
    ((8, 12, 64), 3),     # 12 tiles of 4 x 4 x 32 in slabs of one plane
    ((32, 32, 32), 2),    # 64 tiles in halves
])
def test_overhanging_tiles_and_slabs_match_the_oracle(precision, n, order):
    c = Case(n, order, 2, 0.3, 211, precision=precision, field_scale=0.5)
    c.ctx.step(3)
    c.oracle_steps(3)
    e = c.errors()
    if precision == pic.FP64:
        assert max(e.values()) < 1e-11, e
    else:
        assert e["EB"] < 2e-5 and e["J"] < 2e-4 and e["pos"] < 1e-6 and e["mom"] < 2e-5, e


@pytest.mark.parametrize("sort_every", [1, 2])
def test_overhanging_tiles_equal_dividing_tiles(sort_every):
    """Graph replays, a sort cadence, coarse and random reorders, the adjoint
    and the charge density on overhanging tiles: as on tiles of 2 x 1 x 2 cells,
    which divide the grid (only the order of additions differs)."""
    n = (10, 9, 34)
    out = []
    for tile in ((0, 0, 0), (2, 1, 2)):
        c = Case(n, 2, 2, 0.3, 223, field_scale=0.1, tile=tile, sort_every=sort_every, stream=torch.cuda.Stream())
        c.ctx.step(5)
        for shift in (4, pic.ORDER_RANDOM, 0):
            c.ctx.sort_particles(shift)
            c.ctx.step(2)
        rho = c.ctx.charge_density()
        loss, _, du = c.ctx.step_adjoint(4, 2)
        out.append((c.ctx.get_fields(), by_id(c.ctx.get_particles()), np.asarray(rho), loss, np.asarray(du)))
    a, b = out
    assert rel_l2(a[0], b[0]) < 1e-11
    for k in pic.PARTICLE_KEYS:
        assert rel_l2(a[1][k], b[1][k]) < 1e-10, k
    assert rel_l2(a[2], b[2]) < 1e-10 and abs(a[3] - b[3]) < 1e-10 * abs(b[3]) and rel_l2(a[4], b[4]) < 1e-9


@pytest.mark.parametrize("n,dividing", [((10, 6, 37), (2, 2, 1)), ((6, 10, 70), (2, 2, 2))])
def test_window_on_overhanging_tiles(n, dividing):
    """Moving window: removal, shift and injection with the last z tile overhanging."""
    out = []
    for tile in ((0, 0, 0), dividing):
        c = pic.Context(n, order=2, window_speed=1.0, tile=tile)
        c.set_window_plasma(2, 0.05, 10.0, 8.0)
        parts = inputs.uniform_plasma(5, n, 2, sigma_u=0.3)
        F = np.zeros((9,) + n)
        F[:6] = inputs.random_fields(7, n, 0.05)[:6]
        c.set_fields(F)
        c.load_particles(-1.0, 1.0, parts)
        c.step(9)
        c.step(6)
        got = c.get_particles()
        o = np.argsort(got["id"])
        out.append((c.get_fields(), {k: got[k][o] for k in got}))
    a, b = out
    assert np.array_equal(a[1]["id"], b[1]["id"])
    assert rel_l2(a[0], b[0]) < 1e-11
    for k in pic.PARTICLE_KEYS:
        assert np.linalg.norm(a[1][k] - b[1][k]) < 1e-10 * (1 + np.linalg.norm(b[1][k])), k


@pytest.mark.parametrize("n,order,tile,moves", [
    ((9, 7, 11), 1, (0, 0, 0), 0),
    ((10, 9, 34), 2, (0, 0, 0), 0),
    ((9, 12, 13), 3, (0, 0, 0), 0),
    ((8, 8, 64), 3, (0, 0, 0), 0),
    ((16, 16, 16), 2, (2, 2, 2), 0),
    ((10, 9, 34), 2, (0, 0, 0), 3),   # three pushes since the sort: particles beyond their slab's box
])
def test_fp32_mixed_adjoint_on_tiles_against_fp64(n, order, tile, moves):
    """The FP32-mixed reverse sweep adds the gather's adjoint by tiles; FP64
    does so particle by particle.  dL/du within 1e-3, as the 64^3 workload's
    bound between the two precisions."""
    out = []
    for precision in (pic.FP64, pic.FP32_MIXED):
        c = Case(n, order, 3, 0.4, 229, field_scale=0.05, tile=tile, precision=precision)
        c.ctx.set_external_drive(0.07, 2 * np.pi / n[0])
        for _ in range(moves):
            c.ctx.gather_push()
        loss, dA, du = c.ctx.step_adjoint(5, 2)
        out.append((loss, dA, np.asarray(du)))
    a, b = out
    assert abs(a[0] - b[0]) < 1e-4 * abs(a[0])
    assert abs(a[1] - b[1]) < 1e-3 * abs(a[1])
    assert rel_l2(b[2], a[2]) < 1e-3
