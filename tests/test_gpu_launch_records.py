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
