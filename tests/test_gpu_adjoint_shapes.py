"""The adjoint on grids that are long and narrow: a channel along y gives what the same channel
along x gives, transposed (the blocks of its kernels are not square, and a launch's grid takes
at most 65535 blocks along y)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# planes of a state after the axes are exchanged: h, h1x, h1y, qx, qx1x, qx1y, qy, qy1x, qy1y
SWAP = [0, 2, 1, 6, 8, 7, 3, 5, 4]


def channel(length, width, seed):
    """Topography modes, state and Manning n of a rough, moving channel along x."""
    rng = np.random.default_rng(seed)
    x = np.arange(length)[None, :] + 0.3 * np.arange(width)[:, None]
    z = np.stack([0.1 * np.sin(x / 7.0), 0.02 * rng.uniform(-1.0, 1.0, x.shape),
                  0.02 * rng.uniform(-1.0, 1.0, x.shape)])
    u = 0.02 * rng.uniform(-1.0, 1.0, (9, width, length))
    u[0] += 0.6 + 0.1 * np.sin(x / 11.0)
    u[3] += 0.4 + 0.1 * np.cos(x / 5.0)
    u[6] += 0.1
    return z, u, rng.uniform(0.02, 0.06, x.shape)


def build(z, u, n, ydir, gauges, nsteps, dt=0.02):
    """An FP64 adjoint problem of the channel along x, or turned to run along y."""
    import torch
    from paper_2010_02003_gb300 import binding as B

    if ydir:
        z, u = z[[0, 2, 1]].transpose(0, 2, 1), u[SWAP].transpose(0, 2, 1)
        n, gauges = n.T, gauges[:, ::-1]
    ny, nx = n.shape
    p = B.dg2_default_params()
    nbytes = B.dg2_adj_workspace_bytes(nx, ny, 2, len(gauges), nsteps)
    ws = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    a = B.dg2_adj_create(nx, ny, 1.0, 1.0, p, 2, len(gauges), nsteps,
                         (ws.data_ptr() + 255) // 256 * 256, nbytes,
                         torch.cuda.current_stream().cuda_stream)
    B.dg2_adj_set_problem(a, z, u, 0.0, n, B.DG2_SOUTH if ydir else B.DG2_WEST, 0.0,
                          float(min(nx, ny)), [0.0, 1.0], [0.3, 0.5], gauges)
    B.dg2_adj_set_schedule(a, np.full(nsteps, dt), [nsteps], np.full((1, len(gauges)), 0.4))
    return a, ws, (nx, ny)


def solve(*args):
    from paper_2010_02003_gb300 import binding as B

    a, ws, (nx, ny) = build(*args)
    loss, gn, gq = B.dg2_adj_gradient(a, nx, ny, 2)
    B.dg2_adj_destroy(a)
    return loss, gn, gq


def compare(length, width, nsteps):
    z, u, n = channel(length, width, 100 * width + length % 97)
    # gauges in the first, a middle and the last cell
    gauges = np.array([[0.4, 0.3], [length // 2 + 0.6, width // 2 + 0.2],
                       [length - 0.3, width - 0.4]])
    loss, gn, gq = solve(z, u, n, False, gauges, nsteps)
    loss_t, gn_t, gq_t = solve(z, u, n, True, gauges, nsteps)
    # both orders of the same sums over a few smooth steps: rounding, 1e-12 as for parity
    assert loss > 0.0 and abs(loss_t - loss) <= 1e-12 * loss
    assert np.abs(gn).max() > 0.0 and np.abs(gq).max() > 0.0
    assert np.abs(gn_t.T - gn).max() <= 1e-12 * np.abs(gn).max()
    assert np.abs(gq_t - gq).max() <= 1e-12 * np.abs(gq).max()


def test_more_rows_of_tiles_than_a_launch_has_along_y():
    compare(8 * 65535 + 1, 1, 2)


# widths either side of those at which the forward stage's tiles change, with lengths that end
# inside a tile, at its end and one cell past it
@pytest.mark.parametrize("length", [1, 63, 64, 65, 127, 128, 129, 300])
@pytest.mark.parametrize("width", [1, 2, 3, 4, 5])
def test_narrow_grids_give_the_transposed_result(length, width):
    compare(length, width, 3)


@pytest.mark.parametrize("width", [1, 2, 3])
def test_a_narrow_grid_takes_no_longer_along_y(width):
    """Least time of the forward steps of some 260 000 cells, along y and along x.  Tiles of
    16 x 8 cells kept 1 to 3 of 16 lanes at work along y: 4.9, 4.5 and 3.1 times."""
    import torch
    from paper_2010_02003_gb300 import binding as B

    length = 262144 // width
    z, u, n = channel(length, width, 5)
    best = []
    for ydir in (False, True):
        a, ws, _ = build(z, u, n, ydir, np.array([[0.5, 0.5]]), 8)
        t = []
        for _ in range(6):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            B.dg2_adj_forward(a, 1, 1)
            e1.record()
            torch.cuda.synchronize()
            t.append(e0.elapsed_time(e1))
        best.append(min(t[1:]))
        B.dg2_adj_destroy(a)
    assert best[1] <= 2.0 * best[0], best
