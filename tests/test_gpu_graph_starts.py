"""Graphs of every length and start phase against single launches, bit for bit in the
stored state: the four-step graph from phase 1 (an odd number of steps, then four
to eight), the graph of a sampled step and the plain steps after it from either
phase, on grids with and without the wall-row branch and the alternating order of
the planes; and uploads of FP16 populations, staged a few directions at a time."""
import numpy as np
import pytest
import torch

from paper_2009_04352_gb300 import lbm, workload

pytestmark = pytest.mark.gpu

CASES = [  # nx, ny, nz, precision, layout, collision, wall
    (64, 32, 32, lbm.FP32, lbm.PULL2, 0, 1), (63, 12, 14, lbm.FP32, lbm.AA, 0, 1),          # one launch a step
    (96, 48, 57, lbm.FP32, lbm.PULL2, 0, 1), (64, 32, 34, lbm.FP32, lbm.AA, 1, 1),          # two, planes forwards
    (66, 12, 14, lbm.FP16_SHIFTED, lbm.PULL2, 0, 0), (66, 40, 26, lbm.FP16_SHIFTED, lbm.AA, 0, 1),
    (129, 40, 32, lbm.FP16_SHIFTED, lbm.PULL2, 1, 1), (64, 16, 16, lbm.FP16_SHIFTED, lbm.AA, 0, 1),
    (160, 64, 64, lbm.FP32, lbm.PULL2, 0, 1), (162, 64, 70, lbm.FP32, lbm.PULL2, 1, 3),     # planes in alternating order
    (161, 64, 72, lbm.FP32, lbm.PULL2, 0, 1), (160, 64, 130, lbm.FP32, lbm.AA, 0, 1),
    (256, 64, 82, lbm.FP16_SHIFTED, lbm.PULL2, 0, 1), (252, 65, 83, lbm.FP16_SHIFTED, lbm.PULL2, 1, 1),
    (256, 64, 162, lbm.FP16_SHIFTED, lbm.AA, 0, 1), (256, 128, 256, lbm.FP16_SHIFTED, lbm.AA, 1, 1),
]


def _run(case, precision, layout, mrt, every, chunks):
    nbytes = lbm.lbm_population_bytes(case.nx, case.ny, case.nz, precision)
    bufs = [torch.zeros(nbytes, dtype=torch.uint8, device="cuda") for _ in range(1 if layout == lbm.AA else 2)]
    ch = lbm.Channel.from_buffers(case, bufs, precision=precision, layout=layout)
    if mrt:
        ch.set_les(lbm.COLLISION_MRT, case.u_tau, 26.0)
    ch.init_channel(workload.u_mean_profile(case), workload.noise_amplitude(case), 7)
    ch.set_stats_every(every)
    for n in chunks:
        ch.step(n)
    sums = ch.plane_stats()
    tau = ch.wall_stress()
    ch.close()
    sx = (case.nx + 31) // 32 * 32
    dtype = torch.float16 if precision == lbm.FP16_SHIFTED else torch.float32
    state = bufs[0 if layout == lbm.AA else sum(chunks) % 2][:19 * case.nz * case.ny * sx * dtype.itemsize]
    return state.view(dtype).view(19, case.nz, case.ny, sx)[..., :case.nx], tau, sums


@pytest.mark.parametrize("every,chunks", [(0, [16, 3, 6, 16]), (0, [1, 8, 24]), (0, [1, 12, 16]), (6, [3, 33]), (7, [3, 40]), (7, [4, 1, 40])])
@pytest.mark.parametrize("nx,ny,nz,precision,layout,mrt,wall", CASES)
def test_graphs_of_either_start(nx, ny, nz, precision, layout, mrt, wall, every, chunks):
    case = workload.derive_channel("starts", nx, ny, nz, 640.0, wall=wall)
    want, want_tau, want_sums = _run(case, precision, layout, mrt, every, [1] * sum(chunks))
    got, tau, sums = _run(case, precision, layout, mrt, every, chunks)
    assert torch.isfinite(want).all() and torch.equal(got, want)
    assert np.array_equal(tau, want_tau)
    assert all(np.array_equal(a, b) for a, b in zip(sums, want_sums))


@pytest.mark.parametrize("layout", [lbm.PULL2, lbm.AA])
@pytest.mark.parametrize("nx,ny,nz,wall", [(64, 6, 5, 1), (66, 5, 7, 0), (63, 4, 9, 1), (1, 2, 3, 0), (40, 5, 6, 3)])
def test_fp16_upload_round_trip(nx, ny, nz, wall, layout):
    if wall == lbm.WALL_WFB_NODE and layout == lbm.AA:
        pytest.skip("wall nodes run on two lattices")
    case = workload.derive_channel("upload", nx, ny, nz, 640.0, wall=wall)
    ch = lbm.Channel.from_case(case, precision=lbm.FP16_SHIFTED, layout=layout)
    w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)[:, None, None, None]
    r = np.random.RandomState(4)
    for steps in (0, 1, 2):   # into either lattice or phase
        ch.step(steps)
        f = w * (1.0 + 0.3 * r.randn(19, nz, ny, nx))
        ch.set_populations(f)
        assert np.array_equal(ch.populations(), (f - w).astype(np.float16).astype(np.float64) + w)
    ch.close()
