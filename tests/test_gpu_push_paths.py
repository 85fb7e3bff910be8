"""The push paths of the bit-parallel region discharge: rounds the graph warp
runs alone, crowded layers handed to the whole block, BFS layers past the
masks, and switches between them inside one round, on tiles of every shape.

Each result is compared with Dinic and, bit for bit, with the generic kernel
(kernel_variant 1), which runs the same rounds vertex by vertex."""
import numpy as np
import pytest

from gen import grids
from gen.grids import GridInstance
from helpers import assert_parity, gpu_solve, opts
from paper_1109_1146_gb300.mf import arcs_of

pytestmark = pytest.mark.gpu


def _random(dims, conn, seed, **kw):
    """grids.random_grid, also on the stencils of Sec. 7.1 (links leaving the grid removed)."""
    if conn < 100:
        return grids.random_grid(dims, conn, seed, **kw)
    X, Y, _ = dims
    base = grids.random_grid(dims, 4, seed, **kw)
    nl = np.concatenate([grids.random_grid(dims, 4, seed + h, **kw).nlink[:1] for h in range(arcs_of(conn) // 2)])
    nl = nl.reshape(-1, Y, X)
    for h, (dx, dy) in enumerate(((1, 0), (0, 1)) + grids.PAPER_DISPLACEMENTS[2:arcs_of(conn) // 2]):
        nl[h, max(0, Y - dy):, :] = 0
        nl[h, :, max(0, X - dx):] = 0
    return GridInstance(dims, conn, base.cs, base.ct, nl.reshape(len(nl), -1))


def _serpentine(X, Y, Z, conn):
    """One corridor that runs through every voxel of each z layer (capacity 3 along it, 0 across), the source at
    its start and the sink at its end: one tile's BFS has as many layers as the tile has vertices."""
    H = arcs_of(conn) // 2
    n = X * Y * Z
    cs, ct = np.zeros((Z, Y, X), np.int32), np.zeros((Z, Y, X), np.int32)
    nl = np.zeros((H, Z, Y, X), np.int32)
    nl[0, :, :, :X - 1] = 3
    for y in range(Y - 1):
        nl[1, :, y, X - 1 if y % 2 == 0 else 0] = 3
    cs[:, 0, 0] = 7
    cs[:, Y // 2, X // 2] = 2
    ct[:, Y - 1, X - 1 if Y % 2 else 0] = 9
    return GridInstance((X, Y, Z), conn, cs.reshape(n), ct.reshape(n), nl.reshape(H, n))


def _crowded(X, Y, Z, conn, step):
    """Excess everywhere, sinks on every step-th column: layers with many vertices in every row."""
    inst = _random((X, Y, Z), conn, 7, cmax=60, tmax=20, p_zero=0.1)
    x = np.arange(inst.n) % X
    cs = np.where(x % step == 0, 0, 5 + inst.cs).astype(np.int32)
    ct = np.where(x % step == 0, 400, 0).astype(np.int32)
    return GridInstance(inst.dims, conn, cs, ct, inst.nlink)


SHAPES = [((70, 37, 1), 4, (32, 32, 1)), ((64, 64, 1), 8, (32, 32, 1)), ((33, 50, 1), 4, (32, 16, 1)),
          ((64, 31, 1), 8, (32, 16, 1)), ((128, 40, 1), 4, (64, 32, 1)), ((100, 65, 1), 8, (64, 32, 1)),
          ((64, 64, 1), 4, (64, 64, 1)), ((65, 130, 1), 8, (64, 64, 1)), ((40, 19, 9), 6, (32, 8, 4)),
          ((64, 16, 8), 6, (32, 8, 8)), ((33, 9, 10), 6, (32, 4, 4)), ((64, 17, 5), 6, (32, 8, 2)),
          ((50, 33, 9), 6, (32, 16, 8)), ((70, 37, 1), 108, (32, 32, 1)), ((64, 64, 1), 112, (32, 32, 1)),
          ((33, 50, 1), 116, (32, 32, 1)), ((40, 65, 1), 124, (32, 32, 1)), ((67, 40, 1), 128, (32, 32, 1))]


@pytest.mark.parametrize("dims,conn,tile", SHAPES)
@pytest.mark.parametrize("kind", ["serpentine", "crowded2", "crowded9", "crowded32", "sparse"])
def test_same_as_generic_and_dinic(dims, conn, tile, kind):
    if kind == "serpentine":
        inst = _serpentine(*dims, conn)
    elif kind == "sparse":
        inst = _random(dims, conn, 3, cmax=4, tmax=300, p_zero=0.6)
    else:
        inst = _crowded(*dims, conn, int(kind[7:]))
    got = gpu_solve(inst, tile=tile)
    assert_parity(inst, got)
    ref = gpu_solve(inst, tile=tile, opts=opts(kernel_variant=1))
    for k in ("res", "tres", "exc", "lab"):
        assert np.array_equal(got[k], ref[k]), k
    for k in ("sweeps", "discharges", "rounds", "flow_value"):
        assert getattr(got["stats"], k) == getattr(ref["stats"], k), k


def test_many_regions_same_as_generic():
    # above the number of regions from which five 32x8x4 regions share an SM (a build of its own)
    inst = grids.random_grid((256, 250, 120), 6, 12, cmax=9, tmax=120, p_zero=0.5)
    got = gpu_solve(inst)
    ref = gpu_solve(inst, opts=opts(kernel_variant=1))
    assert got["flow"] == ref["flow"]
    for k in ("smin", "smax", "res", "tres", "exc", "lab"):
        assert np.array_equal(got[k], ref[k]), k
    assert got["stats"].rounds == ref["stats"].rounds


@pytest.mark.parametrize("Z", [40, 262, 281])
def test_halo_labels_far_apart(Z):
    # two columns of regions joined at the top only: the halo of a low region holds labels near 0 (the
    # sinks beside it) and near twice the height, so the next stage lies past the 64 labels kept as bits
    X, Y = 64, 8
    nl = np.zeros((3, Z, Y, X), np.int32)
    nl[1, :, :Y - 1, :] = 2
    nl[2, :Z - 1] = 4
    nl[0, Z - 1, :, :X - 1] = 40
    cs, ct = np.zeros((Z, Y, X), np.int32), np.zeros((Z, Y, X), np.int32)
    cs[:6, ::3, 3:32:4] = 5
    ct[0, :, 32:] = 2
    inst = GridInstance((X, Y, Z), 6, cs.reshape(-1), ct.reshape(-1), nl.reshape(3, -1))
    got = gpu_solve(inst, tile=(32, 8, 4))
    assert_parity(inst, got)
    ref = gpu_solve(inst, tile=(32, 8, 4), opts=opts(kernel_variant=1))
    for k in ("res", "tres", "exc", "lab"):
        assert np.array_equal(got[k], ref[k]), k
    assert got["stats"].rounds == ref["stats"].rounds
