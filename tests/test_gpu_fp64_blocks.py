"""FP64 blocks, lists and detector at the edges of their rules, against the oracle: grids on
either side of the sizes where the blocks of a tile (304 tiles) and the kernels of the end of
step (1024 tiles) change, and the limiter on rough states."""
import numpy as np
import pytest

import oracle
from paper_2010_02003_gb300 import inputs

pytestmark = pytest.mark.gpu


def scales(b):
    h = np.abs(b[0]).max()
    q = max(np.abs(b[3]).max(), np.abs(b[6]).max(), h * np.sqrt(9.8 * h))
    return np.array([h, h, h, q, q, q, q, q, q])[:, None, None]


@pytest.mark.parametrize("scheme", ["dg2", "fv2"])
@pytest.mark.parametrize("nx,ny", [(608, 128), (609, 128), (17, 300), (1024, 256), (1025, 256)])
def test_steps_at_the_sizes_where_blocks_and_lists_change(nx, ny, scheme):
    from paper_2010_02003_gb300 import binding as B

    case = inputs.hump(nx=nx, ny=ny, eta=-1.0, dam_eta=1.0, dam_radius=0.3 * min(nx, ny),
                       amp=0.3, width2=float(min(nx, ny)) ** 2)
    kw = {"dg2": {}, "fv2": {"scheme": B.DG2_SCHEME_FV2}}[scheme]
    o = oracle.Oracle(nx, ny, case.dx, case.dy, cfl=case.cfl, scheme=scheme)
    o.set_dem(case.z_corner, None, case.n_uniform, case.eta_corner)
    s = B.solver_from_case(case, **kw)
    every = B.solver_from_case(case, skip_dry_tiles=False, **kw)
    for k in range(6):
        if k == 3:  # restarted: the flags come with the state
            for x in (s, every):
                x.set_state(x.state(), x.time()[0])
        dt = o.step()
        s.step(dt)
        every.step(dt)
    a, b = s.state(), o.state()
    assert (np.abs(a - b) / scales(b)).max() <= 1e-12
    assert np.array_equal(a, every.state()) and s.mass() == every.mass()
    n, active = s.tile_stats()[:2]
    assert n == -(-nx // 32) * -(-ny // 8) and 0 < active <= n


@pytest.mark.parametrize("size", [1e-5, 1e-2, 1.0, 30.0])
def test_limiter_on_rough_states(size):
    """One DG2-LL step from random states whose components jump by orders of magnitude from
    cell to cell, so that Eq. 6 fires in many cells and is near its threshold in some."""
    from paper_2010_02003_gb300 import binding as B

    nx, ny, dx = 61, 43, 0.2
    rng = np.random.default_rng(11)
    z = 0.02 * rng.standard_normal((ny + 1, nx + 1))
    u = np.zeros((9, ny, nx))
    u[0] = 0.2 + 3.0 * rng.random((ny, nx))
    u[1:3] = 0.3 * u[0] * rng.uniform(-1.0, 1.0, (2, ny, nx))
    for k in range(3, 9):
        u[k] = size * 10.0 ** rng.uniform(-4.0, 0.0, (ny, nx)) * rng.choice([-1.0, 1.0], (ny, nx))
    o = oracle.Oracle(nx, ny, dx, dx, cfl=0.33, limiter=True)
    o.set_dem(z, None, 0.03, None)
    o.set_state(u, 0.0)
    s = B.Solver(nx, ny, dx, variant=B.DG2_LL, cfl=0.33)
    s.set_dem(z, n_uniform=0.03)
    s.set_state(u, 0.0)
    limited = o.limit(u)
    assert (limited != u).mean() > 0.02
    s.step(o.step(1e-4))
    a, b = s.state(), o.state()
    assert (np.abs(a - b) / scales(b)).max() <= 1e-12
