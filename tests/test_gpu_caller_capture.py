"""lbm_step and lbm_batch_step inside a stream capture of the caller's own, after one
step outside it: the replayed capture advances the state as single steps do,
also when the sampling interval changed since."""
import numpy as np
import pytest
import torch

from paper_2009_04352_gb300 import lbm, workload

pytestmark = pytest.mark.gpu

FORMS = [  # nx, ny, nz, precision, layout
    (64, 32, 32, lbm.FP32, lbm.PULL2), (64, 64, 64, lbm.FP32, lbm.PULL2), (64, 32, 32, lbm.FP16_SHIFTED, lbm.PULL2),
    (64, 32, 34, lbm.FP32, lbm.AA), (64, 16, 16, lbm.FP16_SHIFTED, lbm.AA), (63, 12, 14, lbm.FP32, lbm.PULL2),
]


def _start(target, case):
    target.init_channel(workload.u_mean_profile(case), workload.noise_amplitude(case), 11)


@pytest.mark.parametrize("every", [0, 1, 5, 6])
@pytest.mark.parametrize("nx,ny,nz,precision,layout", FORMS)
def test_steps_in_a_capture(nx, ny, nz, precision, layout, every):
    case = workload.derive_channel("capture", nx, ny, nz, 640.0)
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    a = lbm.Channel.from_case(case, precision=precision, layout=layout, stream=stream.cuda_stream)
    b = lbm.Channel.from_case(case, precision=precision, layout=layout)
    for ch in (a, b):
        _start(ch, case)
        ch.set_stats_every(3)
        ch.step(4)
    b.set_stats_every(every)
    a.sync()
    with torch.cuda.graph(graph, stream=stream):
        a.set_stats_every(every)
        a.step(13)
        a.step(23)
    graph.replay()
    torch.cuda.synchronize()
    for _ in range(36):
        b.step(1)
    assert np.array_equal(a.populations(), b.populations())
    assert np.array_equal(a.wall_stress(), b.wall_stress())
    for got, want in zip(a.plane_stats(), b.plane_stats()):
        assert np.array_equal(got, want)
    # the handle steps on outside the capture, with graphs of the new interval
    a.step(40)
    for _ in range(40):
        b.step(1)
    assert np.array_equal(a.populations(), b.populations())
    assert np.array_equal(a.plane_stats()[0], b.plane_stats()[0])
    a.close()
    b.close()


@pytest.mark.parametrize("form", [lbm.BATCH_PERSISTENT, lbm.BATCH_MEMBER_GRIDS])
@pytest.mark.parametrize("precision", [lbm.FP32, lbm.FP16_SHIFTED])
@pytest.mark.parametrize("every", [0, 5])
def test_batch_steps_in_a_capture(every, precision, form):
    cases = [workload.derive_channel(f"m{i}", *s, 640.0) for i, s in enumerate(((32, 8, 16), (48, 12, 10), (64, 16, 32)))]
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    a, b = lbm.Batch(cases, precision=precision, stream=stream.cuda_stream), lbm.Batch(cases, precision=precision)
    for batch in (a, b):
        batch.set_form(form)
        for m, c in zip(batch.members, cases):
            _start(m, c)
        batch.set_stats_every(3)
        batch.step(4)
    b.set_stats_every(every)
    a.sync()
    with torch.cuda.graph(graph, stream=stream):
        a.set_stats_every(every)
        a.step(13)
        a.step(23)
    graph.replay()
    torch.cuda.synchronize()
    for _ in range(36):
        b.step(1)
    for x, y in zip(a.members, b.members):
        assert np.array_equal(x.populations(), y.populations())
    a.close()
    b.close()
