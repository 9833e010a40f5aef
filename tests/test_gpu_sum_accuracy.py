"""The plane profile against exact sums of the FP32 fields it adds, to the accuracy
of FP64 additions: every term (density, velocity, exact product) enters a sum of
53 bits or more, so a column is off by at most one FP64 rounding an addition on
the longest path from a cell to the result (a thread's partial sums, the block's
tree, the blocks of a plane)."""
import math

import numpy as np
import pytest
import torch

from paper_2009_04352_gb300 import lbm, workload

pytestmark = pytest.mark.gpu

W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)[:, None, None, None]


def _fsum(a):
    return math.fsum(np.asarray(a, dtype=np.float64).ravel())


def _check_profile(ch, additions):
    rho, u = ch.moments()
    out = torch.empty((ch.ny, lbm.K_STATS), dtype=torch.float64, device="cuda")
    lbm.lbm_plane_profile_noalloc(ch.handle, out.data_ptr())
    ch.sync()
    got = out.cpu().numpy()
    r, (ux, uy, uz) = rho.astype(np.float64), u.astype(np.float64)
    cols = [r, ux, uy, uz, ux * ux, uy * uy, uz * uz, ux * uy, r * ux, r * uy, r * uz]
    for y in range(ch.ny):
        for k, c in enumerate(cols):
            assert abs(got[y, k] - _fsum(c[:, y])) <= additions * 2.0 ** -53 * _fsum(np.abs(c[:, y])), (y, k)


@pytest.mark.parametrize("precision,rho", [(lbm.FP32, 0.3), (lbm.FP32, 1e9), (lbm.FP32, 1e-5), (lbm.FP32, -3.0),
                                           (lbm.FP16_SHIFTED, 0.3), (lbm.FP16_SHIFTED, 3000.0)])
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("nx", [63, 62, 64])
def test_profile_at_densities_away_from_one(nx, mixed, precision, rho):
    """Densities whose distance from 1 is no FP32 number (above 2^24) or outweighs
    them (below 1/2), alone and beside ordinary ones."""
    case = workload.CASES["c1"].with_(nx=nx, ny=4, nz=32, wall=lbm.WALL_BB)
    ch = lbm.Channel.from_case(case, precision=precision)
    r = np.random.RandomState(5)
    level = np.where(mixed & (r.rand(1, 32, 4, nx) < 0.1), 1.0, rho)
    ch.set_populations(W * level * (1.0 + 0.1 * r.rand(19, 32, 4, nx)))
    # a tile or two a block, at most 64 blocks a plane, five plus four levels of the block
    _check_profile(ch, 80)
    ch.close()


@pytest.mark.parametrize("precision,layout", [(lbm.FP32, lbm.PULL2), (lbm.FP32, lbm.AA), (lbm.FP16_SHIFTED, lbm.PULL2)])
@pytest.mark.parametrize("nx", [1, 2, 4, 66])
def test_profile_of_uniform_planes(nx, precision, layout):
    """Equal cells: every partial sum of a plane is off the same way, so nothing averages out."""
    case = workload.derive_channel("uniform", nx, 304, 1200, 640.0)
    ch = lbm.Channel.from_case(case, precision=precision, layout=layout)
    ch.init_channel(workload.u_mean_profile(case), 0.0, 3)
    ch.step(1)
    # three additions for the words of a block's sum, its share of the error-free runs, at most 30 blocks a plane
    _check_profile(ch, 48)
    ch.close()


@pytest.mark.parametrize("speed", [1e-22, 1e-27, 1e-33])
@pytest.mark.parametrize("nx", [63, 64])
def test_profile_of_tiny_velocities(nx, speed):
    """Products whose rounding error FP32 cannot hold, beside cells at rest."""
    case = workload.CASES["c1"].with_(nx=nx, ny=4, nz=32, wall=lbm.WALL_BB, force=(0.0, 0.0, 0.0))
    f = np.zeros((19, 32, 4, nx))
    f[1:] = speed * np.random.RandomState(6).rand(18, 32, 4, nx) * (np.random.RandomState(7).rand(32, 4, nx) < 0.7)
    # an upload of W + f would round f away: the stored deviations go into a caller's buffer
    buf = torch.zeros(lbm.lbm_population_bytes(nx, 4, 32, lbm.FP32), dtype=torch.uint8, device="cuda")
    sx = (nx + 31) // 32 * 32
    ch = lbm.Channel.from_buffers(case, [buf], layout=lbm.AA)
    view = buf[:19 * 32 * 4 * sx * 4].view(torch.float32).view(19, 32, 4, sx)
    view[..., :nx] = torch.from_numpy(f.astype(np.float32)).cuda()
    torch.cuda.synchronize()
    assert ch.moments()[1].any()
    _check_profile(ch, 80)
    ch.close()


@pytest.mark.parametrize("layout", [lbm.PULL2, lbm.AA])
@pytest.mark.parametrize("nx", [1, 2, 3, 66])
def test_conservation_of_spread_magnitudes(nx, layout):
    """One large population among many that its FP32 sum holds no bit of; with one block a
    plane every thread adds the same terms in the same order."""
    ny, nz = 2432, 160
    case = workload.CASES["c1"].with_(nx=nx, ny=ny, nz=nz, wall=lbm.WALL_BB)
    if nx == 66:
        case = case.with_(nz=48)
        nz = 48
    ch = lbm.Channel.from_case(case, layout=layout)
    z = np.where(np.arange(nz) % 16 == 0, 1.0, 5.893394927625195e-08)
    ch.set_populations(np.broadcast_to(W + z[None, :, None, None], (19, nz, ny, nx)))
    fb = z.astype(np.float32).astype(np.float64) * (nx * ny)
    total = ch.conservation()
    # three additions for the words of a block's sums, the directions, ten blocks a thread and eight levels in the
    # last reduction, and the error-free runs' share; the cells' rest mass is added last
    assert abs(total[0] - (19 * math.fsum(fb) + case.cells)) <= 64 * 2.0 ** -53 * 19 * math.fsum(fb) + 2.0 ** -52 * total[0]
    for k in range(3):
        assert abs(total[1 + k]) <= 64 * 2.0 ** -53 * 19 * math.fsum(fb)
    ch.close()
