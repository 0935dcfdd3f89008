"""An ensemble call that ends with an error leaves its healthy members ready to go on alone:
the tiles that their own steps compute are those of the states the ensemble left them in.

The failing member is dry, with cells of 0.1 m, a Courant number of 40 and an inflow that
starts after 20 steps of the 1 s cap: its first wet steps are hundreds of times too long and
its state becomes non-finite, after the other member's water has crossed several tiles.  Only
floating-point arithmetic on finite inputs happens on the GPU: nothing here can fault or hang it."""
import numpy as np
import pytest

from paper_2010_02003_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [0, 1], ids=["NL", "LL"])
@pytest.mark.parametrize("call", ["run_to", "autotune"])
def test_healthy_member_goes_on_alone_after_the_ensemble_failed(call, variant):
    from paper_2010_02003_gb300 import binding as B

    # a patch of water in one 16 x 8 tile of a dry basin of 20 x 20 tiles
    case = inputs.hump(nx=320, ny=160, eta=-1.0, amp=0.0)
    start = np.zeros((9, case.ny, case.nx))
    start[0, 82:88, 162:174] = 2.0
    healthy = B.solver_from_case(case, variant=variant, precision=B.DG2_FP32)
    every = B.solver_from_case(case, variant=variant, precision=B.DG2_FP32, skip_dry_tiles=False)
    for s in (healthy, every):
        s.set_state(start, 0.0)
    assert healthy.tile_stats()[1] == 9          # the tile of the patch and those around it
    flat = inputs.hump(nx=40, ny=24, dx=0.1, eta=-1.0, amp=0.0)
    failing = B.solver_from_case(flat, variant=variant, precision=B.DG2_FP32, cfl=40.0, dt_max=1.0)
    failing.add_inflow(inputs.WEST, 0.0, 2.4, [0.0, 20.0, 21.0], [0.0, 0.0, 50.0])
    ens = B.Ensemble([healthy, failing])
    with pytest.raises(B.Dg2Error, match="non-finite") as e:
        if call == "run_to":
            ens.run_to(1e4)
        else:
            ens.autotune(1e4, steps_per_trial=4)
    assert e.value.code == B.DG2_E_NONFINITE
    n = healthy.steps()
    assert n >= 32
    for _ in range(n):
        every.step()
    assert np.array_equal(healthy.state(), every.state())
    moved = healthy.state()[0][96:].max()
    assert moved > 0.0                           # beyond the tiles around the patch's
    for _ in range(3):
        healthy.step()
        every.step()
        assert healthy.time() == every.time()
        assert np.array_equal(healthy.state(), every.state())
