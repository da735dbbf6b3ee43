"""What the library says about its launches: one timing record per launch, also where a
chunk has two; and a failed launch leaves no error behind for other contexts."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2303_01471_gb300 import qhd

SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152


def loaded(shape, batch=1, stream=None):
    sim = qhd.QHD(shape, batch=batch, stream=stream)
    sim.set_potential(np.zeros((batch, *shape)))
    sim.set_schedule(qhd.Schedule())
    sim.reset_state()
    return sim


def test_one_timing_record_per_launch_of_a_batch_of_both_forms():
    sim = loaded((128, 128), 3 * SMS + 5)
    sim.timing_enable(1)
    before = sim.launch_count()
    sim.evolve(0.1, 0.01)
    got = sim.timing_read()
    assert sim.launch_count() - before == 3 == got["prep"][1] + got["whole"][1] and got["whole"][1] == 2
    sim.close()


@pytest.mark.parametrize("shape", [(64,), (16, 16), (64, 64), (4, 32, 32)], ids=lambda s: "x".join(map(str, s)))
def test_failed_launch_leaves_no_error_behind(shape):
    """A launch into a stream whose capture has been broken off fails on the host; a
    context on another stream works on."""
    rt = ctypes.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0])
    side = torch.cuda.Stream()
    a, b = loaded(shape, stream=side), loaded(shape)
    torch.cuda.synchronize()
    s, graph = ctypes.c_void_p(side.cuda_stream), ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(s, 1) == 0          # thread-local mode
    assert rt.cudaStreamSynchronize(s) != 0              # not allowed there: breaks the capture off
    assert a.lib.qhd_evolve(a.ctx, 0.1, 0.01) == qhd.QHD_ERR_CUDA
    assert rt.cudaStreamEndCapture(s, ctypes.byref(graph)) != 0 and not graph.value
    rt.cudaGetLastError()
    b.set_potential(np.zeros((1, *shape)))
    b.evolve(0.1, 0.01)
    assert b.observables(0.1)[0].norm == pytest.approx(1.0, abs=1e-6)
    b.close()
    a.close()
