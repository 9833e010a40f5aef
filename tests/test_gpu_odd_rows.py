"""Plain steps on rows of an odd number of cells (two cells a thread) against
sampled steps of the same run, which the one-cell kernel takes: the same
populations and wall stress, bit for bit."""
import numpy as np
import pytest

from paper_2009_04352_gb300 import lbm, workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mrt", [False, True])
@pytest.mark.parametrize("layout", [lbm.PULL2, lbm.AA])
@pytest.mark.parametrize("precision", [lbm.FP32, lbm.FP16_SHIFTED])
@pytest.mark.parametrize("nx,ny,nz,wall", [  # 2^17 cells and more run two cells a thread, the last case does not
    (1, 1024, 128, 1), (3, 2, 21846, 0), (5, 3, 8739, 2), (61, 43, 50, 1), (63, 46, 46, 0), (65, 64, 32, 1),
    (127, 3, 345, 2), (129, 32, 32, 1), (257, 30, 17, 0), (255, 33, 40, 1), (31, 65, 65, 0)])
def test_odd_rows_match_the_one_cell_kernel(nx, ny, nz, wall, precision, layout, mrt):
    case = workload.derive_channel("odd", nx, ny, nz, 640.0, wall=wall).with_(force=(2e-6, 1e-7, -1e-6))
    out = []
    for every in (1, 0):
        ch = lbm.Channel.from_case(case, precision=precision, layout=layout)
        assert ch.kernel == lbm.KERNEL_CELL
        if mrt:
            ch.set_les(lbm.COLLISION_MRT, case.u_tau, 26.0)
        ch.init_channel(workload.u_mean_profile(case), 0.01, 5)
        ch.set_stats_every(every)
        got = []
        for n in (1, 2, 16):   # single launches of either start phase, then a graph
            ch.step(n)
            got += [ch.populations(), ch.wall_stress()]
        out.append(got)
        ch.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("mrt", [False, True])
@pytest.mark.parametrize("layout", [lbm.PULL2, lbm.AA])
@pytest.mark.parametrize("precision", [lbm.FP32, lbm.FP16_SHIFTED])
@pytest.mark.parametrize("nx,ny,nz,wall", [  # both sides of 2^18 cells, and of 2^20 for rows of three warps against two
    (33, 3, 2700, 1), (61, 2, 2200, 0), (63, 65, 64, 2), (63, 66, 64, 1), (127, 48, 43, 1), (129, 48, 48, 0), (257, 32, 33, 1),
    (67, 126, 124, 1), (67, 128, 124, 1)])
def test_odd_rows_of_larger_grids(nx, ny, nz, wall, precision, layout, mrt):
    test_odd_rows_match_the_one_cell_kernel(nx, ny, nz, wall, precision, layout, mrt)
