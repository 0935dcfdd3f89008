"""State in and out over the host boundary: exact round trips on ragged grids, in both
precisions, and refusal of non-finite values without touching the state."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def make(nx, ny, precision, **kw):
    from paper_2010_02003_gb300 import binding as B

    s = B.Solver(nx, ny, 2.0, precision=precision, **kw)
    rng = np.random.default_rng(nx * 100 + ny)
    s.set_dem(rng.uniform(0.0, 20.0, (ny + 1, nx + 1)), n_uniform=0.03)
    planes = rng.standard_normal((9, ny, nx))
    planes[0] = rng.uniform(0.0, 2.0, (ny, nx))
    planes[3] *= 10.0 ** rng.integers(-42, 3, (ny, nx))   # FP32 denormals among them
    return s, planes


def expected32(s, planes):
    """The FP32 form's modes of `planes` (eta0 as hi + lo) taken back to FP64 depth modes."""
    z = s.topo()
    out = planes.astype(np.float32).astype(np.float64)
    e0 = planes[0] + z[0]
    hi = e0.astype(np.float32).astype(np.float64)
    lo = (e0 - hi).astype(np.float32).astype(np.float64)
    out[0] = (hi - z[0]) + lo
    for k in (1, 2):
        out[k] = (planes[k] + z[k]).astype(np.float32).astype(np.float64) - z[k]
    return out


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 41), (37, 1), (32, 8), (33, 9), (31, 7), (130, 67)])
def test_round_trip_is_exact(nx, ny, precision):
    s, planes = make(nx, ny, precision)
    s.set_state(planes, 3.0)
    want = expected32(s, planes) if precision else planes
    assert np.array_equal(s.state(), want)
    assert s.time()[0] == 3.0
    m, ledger = s.mass()
    assert m == ledger and abs(m - 4.0 * want[0].sum()) <= 1e-13 * nx * ny * m
    s.set_state(s.state(), 4.0)     # what came out goes in again
    assert np.array_equal(s.state(), expected32(s, want) if precision else want)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("plane,value", [(0, np.nan), (4, np.inf), (8, -np.inf)])
def test_non_finite_values_are_refused_and_the_state_kept(plane, value, precision):
    from paper_2010_02003_gb300 import binding as B

    s, planes = make(35, 11, precision)
    s.set_state(planes, 1.0)
    before = s.state()
    worse = planes.copy()
    worse[plane, 10, 34] = value
    worse[8, 10, 34] = np.nan
    with pytest.raises(B.Dg2Error, match=f"value {plane * 35 * 11 + 35 * 11 - 1}"):
        s.set_state(worse, 2.0)
    assert np.array_equal(s.state(), before) and s.time()[0] == 1.0
    s.set_state(planes, 2.0)
    assert np.array_equal(s.state(), before) and s.time()[0] == 2.0
