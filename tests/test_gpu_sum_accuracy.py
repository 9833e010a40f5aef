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
