"""mf_solve enqueues up to four sweeps before it waits.  Its state is that of
single mf_sweep calls, also where a sweep that is not the first of such a
window hits the round cap, and the grid goes on from there alike."""
import numpy as np
import pytest

from gen import grids
from gen.grids import GridInstance
from helpers import assert_parity, opts
from paper_1109_1146_gb300 import Grid, mf
from paper_1109_1146_gb300.mf import arcs_of

pytestmark = pytest.mark.gpu


def _state(g):
    res, tres, exc = g.get_residual()
    lab, dinf = g.get_labels()
    return {"res": res, "tres": tres, "exc": exc, "lab": lab, "dinf": dinf}


def _same(a, b):
    for k in a:
        assert np.array_equal(a[k], b[k]), k


def _grid(inst, tile):
    g = Grid(inst.dims, inst.conn, tile=tile)
    g.set_caps(inst.cs, inst.ct, inst.nlink)
    return g


SCHEDULES = [{}, {"global_relabel_period": 0}, {"global_relabel_period": 3, "global_relabel_first": 2},
             {"global_relabel_period": 2, "partial_discharge": 1}, {"boundary_relabel_period": 3, "global_relabel_period": 0}]


@pytest.mark.parametrize("kw", SCHEDULES)
@pytest.mark.parametrize("make,tile", [(lambda: grids.segmentation_2d(150, 101, 2, conn=4), (32, 32, 1)),
                                       (lambda: grids.segmentation_2d(131, 140, 3, conn=8, hard_seed_frac=0.03), (32, 16, 1)),
                                       (lambda: grids.volume_3d(70, 31, 17, 4), (32, 8, 4))])
def test_windows_equal_single_sweeps(make, tile, kw):
    inst = make()
    with _grid(inst, tile) as a, _grid(inst, tile) as b:
        stats = a.solve(opts(**kw))
        got = dict(_state(a), flow=a.flow_value(), smin=a.get_cut(0), smax=a.get_cut(1))
        b.begin(opts(**kw))
        sweeps = 1
        while b.sweep() != 0:
            sweeps += 1
        b.finish()
        assert stats.sweeps == sweeps
        _same(_state(a), _state(b))
    assert_parity(inst, got)


def _relay(conn, rows, slices, mids):
    """Excess on the last column of the first 32-wide tile moves on by one tile a sweep, in one round each, through
    `mids` tiles of straight corridors; the tile after them has sinks behind a random network."""
    X, n = 32 * (2 + mids), 32 * (2 + mids) * rows * slices
    x1 = 32 * (1 + mids)
    cs, ct = np.zeros((slices, rows, X), np.int32), np.zeros((slices, rows, X), np.int32)
    nl = np.zeros((arcs_of(conn) // 2, slices, rows, X), np.int32)
    base = grids.random_grid((32, rows, slices), 4 if conn > 100 else conn, 11, cmax=9, tmax=60, p_zero=0.5)
    own = base.nlink.reshape(-1, slices, rows, 32)
    cs[:, :, 31] = 50
    nl[0, :, :, 31:x1] = 60
    nl[:len(own), :, :, x1:] = own
    ct[:, :, x1:] = np.where(base.ct > 40, base.ct, 0).reshape(slices, rows, 32)
    return GridInstance((X, rows, slices), conn, cs.reshape(n), ct.reshape(n), nl.reshape(len(nl), n))


@pytest.mark.parametrize("mids", [0, 1, 2])
@pytest.mark.parametrize("conn,rows,slices,tile", [(4, 32, 1, (32, 32, 1)), (8, 20, 1, (32, 32, 1)), (6, 8, 4, (32, 8, 4)),
                                                   (108, 32, 1, (32, 32, 1))])
def test_round_cap_in_a_later_sweep_of_a_window(conn, rows, slices, tile, mids):
    inst = _relay(conn, rows, slices, mids)
    o = opts(max_rounds=2, global_relabel_period=0)
    with _grid(inst, tile) as a, _grid(inst, tile) as b:
        with pytest.raises(mf.MFError) as e:
            a.solve(o)
        assert e.value.status == mf.MF_EROUNDLIMIT
        b.begin(o)
        for s in range(1 + mids):
            assert b.sweep() > 0, s
        with pytest.raises(mf.MFError) as e:
            b.sweep()
        assert e.value.status == mf.MF_EROUNDLIMIT
        _same(_state(a), _state(b))
        assert a.solve(o, check=False).sweeps == 2 + mids
        # both go on from the error
        for _ in range(3):
            r = []
            for g in (a, b):
                try:
                    r.append(g.sweep())
                except mf.MFError as err:
                    r.append((err.status,))
            assert r[0] == r[1]
            _same(_state(a), _state(b))
            if r[0] == 0:
                break
        # and a solve with the default cap is exact
        a.solve(opts())
        got = dict(_state(a), flow=a.flow_value(), smin=a.get_cut(0), smax=a.get_cut(1))
    assert_parity(inst, got)
