"""Steps replayed from the library's graphs against the same steps launched one
by one, bitwise, on both sides of the lines at which the graph's launches change:
wall rows as a parallel branch, planes walked backwards in every other step, and
the even AA step of the four-cell kernel as one launch. Single launches always
run all rows forwards, so any row left out, done twice or read too early shows.
"""
import pytest
import torch

from paper_2009_04352_gb300 import lbm, workload

pytestmark = pytest.mark.gpu

CASES = [  # nx, ny, nz, precision, layout, collision, wall
    (96, 48, 56, lbm.FP32, lbm.PULL2, 0, 1), (96, 48, 57, lbm.FP32, lbm.PULL2, 0, 1),   # 2^18 cells between them
    (96, 3, 911, lbm.FP32, lbm.PULL2, 1, 1), (96, 2, 1366, lbm.FP32, lbm.PULL2, 0, 0),  # one interior row, none
    (160, 64, 64, lbm.FP32, lbm.PULL2, 0, 1), (162, 64, 70, lbm.FP32, lbm.PULL2, 1, 3),  # alternating order
    (160, 64, 130, lbm.FP32, lbm.AA, 0, 1), (130, 67, 151, lbm.FP32, lbm.AA, 1, 2),
    (256, 64, 82, lbm.FP16_SHIFTED, lbm.PULL2, 0, 1), (252, 65, 83, lbm.FP16_SHIFTED, lbm.PULL2, 1, 1),
    (130, 66, 152, lbm.FP16_SHIFTED, lbm.PULL2, 0, 0), (256, 64, 162, lbm.FP16_SHIFTED, lbm.AA, 0, 1),
    (256, 64, 162, lbm.FP16_SHIFTED, lbm.AA, 1, 0), (256, 128, 256, lbm.FP16_SHIFTED, lbm.AA, 0, 1),
    (512, 256, 256, lbm.FP32, lbm.PULL2, 0, 1),   # 2^25 cells
]


def _run(case, precision, layout, mrt, chunks):
    ch = lbm.Channel.from_case(case, precision=precision, layout=layout)
    if mrt:
        ch.set_les(lbm.COLLISION_MRT, case.u_tau, 26.0)
    ch.init_channel(workload.u_mean_profile(case), workload.noise_amplitude(case), 7)
    for n in chunks:
        ch.step(n)
    rho, u = ch.moments(device=True)
    tau = torch.from_numpy(ch.wall_stress())
    ch.close()
    return rho, u, tau


@pytest.mark.parametrize("nx,ny,nz,precision,layout,mrt,wall", CASES)
def test_graph_steps_match_single_steps(nx, ny, nz, precision, layout, mrt, wall):
    case = workload.derive_channel("order", nx, ny, nz, 640.0, wall=wall)
    want = _run(case, precision, layout, mrt, [1] * 35)
    got = _run(case, precision, layout, mrt, [16, 3, 16])   # graphs of either start phase
    for a, b in zip(want, got):
        assert torch.equal(a, b)
