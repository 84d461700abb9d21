"""The marching kernels on the work that grids of up to 1.4 M nodes otherwise do by tiles: boundary
input per step and in the persistent run (which imposes it and meets at a barrier of its own),
enclosed grids, recorded runs and the expiry of a ring wait inside the persistent run. Rows per
warp set by the caller make a small grid march; results equal the tiles' bit for bit.
"""
import numpy as np
import pytest

from paper_1410_0753_gb300 import CliffsError, CliffsGrid, ERR_TIMEOUT, cliffs_inject_wait_expiry
from tests.test_gpu_tiles import _grid, _result, _same
from workloads import Nest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("edges", [(0, 1, 2, 3), (1, 2), (3,)])
@pytest.mark.parametrize("kw", [dict(), dict(alternate=1), dict(coords=0), dict(open_edges=1)])
@pytest.mark.parametrize("nx,ny", [(70, 64), (121, 33)])
def test_boundary_input_marching_and_by_tiles(nx, ny, kw, edges):
    rng = np.random.default_rng(8)
    times = 7.0 + np.cumsum(rng.uniform(0.5, 1.5, 30))
    outs = []
    for march in (0, 1):
        for persistent in (False, True):
            g, eta = _grid(nx, ny, **kw)
            if march:
                g.set_rows_per_warp(7)
            g.set_initial(eta)
            r = np.random.default_rng(9)
            for e in range(4):
                vals = 0.1 * r.standard_normal((30, 3, ny if e < 2 else nx))
                if e in edges:
                    g.set_boundary_input(e, times, vals)
            g.set_boundary_clock(0.0, stop_at_end=True)
            g.step(5, persistent=persistent)
            g.step(1000, persistent=persistent)          # ends with the records
            outs.append([np.array(g.steps_done), *_result(g)])
            g.close()
    assert 5 < outs[0][0] < 1000
    for o in outs[1:]:
        _same(outs[0], o)


@pytest.mark.parametrize("kw", [dict(), dict(coords=0, alternate=1)])
def test_enclosed_grids_marching_and_by_tiles(kw):
    outs = []
    for march in (0, 1):
        for persistent in (False, True):
            g, eta = _grid(150, 90, nests=[Nest(*p) for p in _nests(kw)], bndout=2, **kw)
            if march:
                g.set_rows_per_warp(11)
            g.set_initial(eta)
            g.step(15, persistent=persistent)
            outs.append(_result(g) + [g.boundary(m, e) for m in range(2) for e in range(4)])
            g.close()
    for o in outs[1:]:
        _same(outs[0], o)


def _nests(kw):
    """two enclosed grids in the coordinates of _grid(150, 90), the first across window edges"""
    x0, y0, dx, dy = (0.0, 0.0, 50.0, 40.0) if kw.get("coords", 1) == 1 else (10.0, 40.0, 1 / 600.0, 1 / 600.0)
    return [(x0 + 51.3 * dx, y0 + 20.5 * dy, dx / 3, dy / 3, 60, 45), (x0 + 3 * dx, y0 + 2 * dy, dx / 2, dy / 2, 20, 21)]


@pytest.mark.parametrize("every", [1, 4])
@pytest.mark.parametrize("alternate", [0, 1])
def test_recorded_gradient_marching_and_by_tiles(alternate, every):
    outs = []
    for march in (0, 1):
        g, eta = _grid(130, 70, alternate=alternate)
        if march:
            g.set_rows_per_warp(9)
        g.set_initial(eta)
        g.adjoint_record(every)
        g.step(7)
        g.step(6)
        seed = np.random.default_rng(4).standard_normal((7, 4)).astype(np.float32)
        outs.append(_result(g) + [g.adjoint_recorded(seed), *g.adjoint_velocity()])
        g.close()
    assert np.abs(outs[0][-3]).max() > 0
    _same(outs[0], outs[1])


def test_ring_wait_expiry_inside_the_persistent_marching_run():
    """Every ring slot of the run waits for bytes that never come, for at most 2 M cycles: the run
    ends with a timeout status and the grid goes on working."""
    outs = []
    for inject in (0, 1):
        g, eta = _grid(130, 70, batch=3)
        g.set_rows_per_warp(9)
        fields = np.stack([eta, 0.5 * eta, 0.25 * eta])
        g.set_initial(fields)
        if inject:
            cliffs_inject_wait_expiry(g.h, 2_000_000)
            with pytest.raises(CliffsError) as e:
                g.step(10, persistent=True)
            assert e.value.code == ERR_TIMEOUT
            g.set_initial(fields)
        g.step(10, persistent=True)
        outs.append([r for b in range(3) for r in _result(g, b)])
        g.close()
    _same(outs[0], outs[1])
