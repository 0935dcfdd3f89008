"""The flags that a state set with dg2_set_state carries: the first step from it equals that of
a solver that computes every tile, also with films, depths below zero and slopes on dry ground.
A film of tol_dry counts as dry by its average, but beside a wall of the bed its face depth,
formed as eta - z, may round to more."""
import numpy as np
import pytest

from paper_2010_02003_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = 1e-5


def state(nx, ny, scheme):
    """Patches of what a cell can hold, far apart on a dry, rough bed."""
    u = np.zeros((9, ny, nx))

    def patch(k):
        j, i = int((0.1 + 0.8 * (k * 0.37 % 1.0)) * ny), int((k + 0.5) / 10 * nx)
        return slice(j, j + 3), slice(i, i + 5)

    u[(0, *patch(0))] = 0.7                     # water
    u[(0, *patch(1))] = 0.5 * TOL               # a film that counts as dry
    u[(0, *patch(2))] = TOL                     # at the tolerance
    u[(0, *patch(9))] = TOL * (1.0 - 1e-4 * np.arange(15.0).reshape(3, 5))
    u[(0, *patch(3))] = -0.3                    # below zero, above the check at -1 m
    u[(0, *patch(4))] = -1e-9
    u[(3, *patch(5))] = 0.2                     # discharge on dry ground
    u[(6, *patch(6))] = -1e-40
    if scheme == "dg2":
        u[(1, *patch(7))] = 0.4                 # slopes on dry ground
        u[(5, *patch(8))] = 1e-3
    u[0, ny - 1, nx - 1] = 0.2                  # the last cell
    return u


CASES = [("dg2", 0, 0), ("dg2", 1, 0), ("dg2", 0, 1), ("dg2", 1, 1), ("fv2", 0, 0), ("fv1", 0, 0)]


@pytest.mark.parametrize("scheme,variant,precision", CASES)
@pytest.mark.parametrize("nx,ny", [(333, 171), (1030, 270)])
def test_uploaded_states_step_as_if_every_tile_were_computed(scheme, variant, precision, nx, ny):
    check(scheme, variant, precision, nx, ny)


def test_uploaded_states_on_the_wide_fp32_tiles():
    check("dg2", 0, 1, 4099, 2047)              # above 2^23 cells: tiles of 32 x 8


def check(scheme, variant, precision, nx, ny):
    from paper_2010_02003_gb300 import binding as B

    kw = {"variant": variant, "precision": precision}
    if scheme != "dg2":
        kw["scheme"] = {"fv2": B.DG2_SCHEME_FV2, "fv1": B.DG2_SCHEME_FV1}[scheme]
    z = 0.05 * np.random.default_rng(3).standard_normal((ny + 1, nx + 1)).cumsum(axis=1)
    case = inputs.Case(name="", nx=nx, ny=ny, dx=2.0, dy=2.0, z_corner=z, eta_corner=None,
                       manning=None, n_uniform=0.03, bc=(inputs.WALL, inputs.OPEN) * 2)
    some, every = (B.solver_from_case(case, skip_dry_tiles=k, **kw) for k in (True, False))
    u = state(nx, ny, scheme)
    for s in (some, every):
        s.set_state(u, 5.0)
    n, active = some.tile_stats()[:2]
    assert 0 < active < n
    assert some.time() == every.time() and some.mass() == every.mass()
    for _ in range(4):
        some.step()
        every.step()
        assert some.time() == every.time() and some.mass() == every.mass()
        a, b = some.state(), every.state()
        assert np.array_equal(a, b), [int((x != y).sum()) for x, y in zip(a, b)]
        for _ in range(3):                      # and again from a state that steps have made
            some.step()
        for s in (every, some):
            s.set_state(some.state(), some.time()[0])


@pytest.mark.parametrize("scheme", ["dg2", "fv2", "fv1"])
def test_a_depth_below_minus_one_metre_is_met_by_the_first_step(scheme):
    from paper_2010_02003_gb300 import binding as B

    kw = {} if scheme == "dg2" else {"scheme": {"fv2": B.DG2_SCHEME_FV2,
                                                "fv1": B.DG2_SCHEME_FV1}[scheme]}
    s = B.Solver(70, 40, 1.0, **kw)
    s.set_dem(np.zeros((41, 71)), n_uniform=0.03)
    u = np.zeros((9, 40, 70))
    u[0, 20, 50] = -1.5
    s.set_state(u, 0.0)
    with pytest.raises(B.Dg2Error) as e:
        s.step(0.1, want_dt=True)
    assert e.value.code == B.DG2_E_NONFINITE
