"""Sums and fields of the current state against exact sums of the exported
populations: every width of the gather (one, two and four cells a thread), both
layouts and phases, all walls, row tails, and runs longer than one compensated
sum. The bound is the kernel's own: a run of 32 additions keeps its residual in
FP32, so it is off by at most 32 half ulps x 2^-24 of the run's sum (2^-44), and
the FP64 sums behind it add less."""
import math

import numpy as np
import pytest
import torch

from paper_2009_04352_gb300 import lbm, workload

pytestmark = pytest.mark.gpu

W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)[:, None, None, None]
E = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
              (1, 0, 1), (-1, 0, -1), (0, 1, 1), (0, -1, -1), (1, -1, 0), (-1, 1, 0), (1, 0, -1), (-1, 0, 1), (0, 1, -1),
              (0, -1, 1)])
BOUND = 2.0 ** -43


def _fsum(a):
    return math.fsum(np.asarray(a, dtype=np.float64).ravel())


@pytest.mark.parametrize("steps", [0, 1, 2])
@pytest.mark.parametrize("layout", [lbm.PULL2, lbm.AA])
@pytest.mark.parametrize("precision", [lbm.FP32, lbm.FP16_SHIFTED])
@pytest.mark.parametrize("nx,ny,nz,wall", [(37, 6, 5, 1), (1, 8, 3, 0), (130, 5, 4, 0), (132, 5, 3, 2), (300, 3, 2, 1),
                                           (4, 2, 5, 1), (2, 40, 2300, 1), (132, 5, 3, 3), (512, 4, 3, 0)])
def test_sums_and_moments(nx, ny, nz, wall, precision, layout, steps):
    if wall == lbm.WALL_WFB_NODE and layout == lbm.AA:
        pytest.skip("wall nodes run on two lattices")
    case = workload.derive_channel("sums", nx, ny, nz, 640.0, wall=wall).with_(force=(2e-6, 1e-7, -1e-6))
    ch = lbm.Channel.from_case(case, precision=precision, layout=layout)
    ch.init_channel(workload.u_mean_profile(case), 0.01, 3)
    ch.step(steps)
    fb = (ch.populations() - W).astype(np.float32).astype(np.float64)   # the stored deviations, exactly

    total = ch.conservation()
    want = [_fsum(fb)] + [_fsum(E[:, k][:, None, None, None] * fb) for k in range(3)]
    scale = _fsum(np.abs(fb))
    assert abs(total[0] - case.cells - want[0]) <= BOUND * scale + 2.0 ** -52 * case.cells
    for k in range(3):
        assert abs(total[1 + k] - want[1 + k]) <= BOUND * scale

    # moments: host and device copies, with and without the wide stores
    rho, u = ch.moments()
    n = case.cells
    for off in (0, 1):
        buf = torch.full((4 * n + 1,), float("nan"), dtype=torch.float32, device="cuda")
        lbm.lbm_moments(ch.handle, buf[off:].data_ptr(), buf[off + n:].data_ptr(), 1)
        got = buf[off:off + 4 * n].cpu().numpy()
        assert np.array_equal(got[:n], rho.ravel()) and np.array_equal(got[n:], u.ravel())
    r64 = 1.0 + fb.sum(axis=0)
    F = np.array(case.force)
    u64 = np.stack([(np.tensordot(E[:, k].astype(float), fb, 1) + 0.5 * F[k]) / r64 for k in range(3)])
    assert np.max(np.abs(rho - r64)) <= 2.0 ** -20 * np.max(r64)    # a dozen FP32 roundings of values near 1
    assert np.max(np.abs(u - u64)) <= 2.0 ** -20 * max(np.max(np.abs(fb)), 1e-30) * 19

    prof = torch.empty((ny, lbm.K_STATS), dtype=torch.float64, device="cuda")
    lbm.lbm_plane_profile_noalloc(ch.handle, prof.data_ptr())
    ch.sync()
    prof = prof.cpu().numpy()
    r, (ux, uy, uz) = rho.astype(np.float64), u.astype(np.float64)
    cols = [r, ux, uy, uz, ux * ux, uy * uy, uz * uz, ux * uy, r * ux, r * uy, r * uz]
    for y in range(ny):
        for k, c in enumerate(cols):
            assert abs(prof[y, k] - _fsum(c[:, y])) <= BOUND * _fsum(np.abs(c[:, y])), (y, k)
    ch.close()


def test_finite_sums_beyond_fp32_stay_finite():
    """Populations near the top of FP32 overflow an FP32 sum, not the FP64 one."""
    case = workload.CASES["c1"].with_(nx=64, ny=4, nz=40, wall=lbm.WALL_BB)
    ch = lbm.Channel.from_case(case)
    f = np.broadcast_to(W, (19, 40, 4, 64)).copy()
    f[0] = 3e38
    ch.set_populations(f)
    total = ch.conservation()
    assert abs(total[0] - float(np.float32(3e38)) * case.cells) <= 1e-12 * total[0]
    f[0, 3, 1, 5] = np.nan
    ch.set_populations(f)
    with pytest.raises(lbm.LbmError) as ei:
        ch.conservation()
    assert ei.value.code == lbm.LBM_ERR_DIVERGED
    ch.close()


@pytest.mark.parametrize("layout", [lbm.PULL2, lbm.AA])
@pytest.mark.parametrize("precision", [lbm.FP32, lbm.FP16_SHIFTED])
@pytest.mark.parametrize("nx", [66, 130, 192, 258, 322, 386, 452, 520, 151, 301])
def test_sampled_sums_match_the_profile(nx, precision, layout):
    """Rows of every number of warps a CTA takes (one to four) and several CTAs a
    row: the fused sums of a sampled step against the profile of the state it
    starts from (FP32 warp sums: a few 1e-7 of the column)."""
    case = workload.derive_channel("rows", nx, 9, 7, 640.0)
    ch = lbm.Channel.from_case(case, precision=precision, layout=layout)
    ch.init_channel(workload.u_mean_profile(case), workload.noise_amplitude(case), 9)
    prof = torch.empty((9, lbm.K_STATS), dtype=torch.float64, device="cuda")
    for _ in range(2):
        lbm.lbm_plane_profile_noalloc(ch.handle, prof.data_ptr())
        ch.set_stats_every(1)
        ch.step(1)
        st, _, n = ch.plane_stats(reset=True)
        assert n == 1
        want = prof.cpu().numpy()
        assert np.all(np.abs(st - want) <= 1e-6 * np.max(np.abs(want), axis=0))
    ch.close()
