"""set_potential's minimiser, range and non-finite check over the numbers of partial
results at which they are reduced on the device or on the host
(csrc/qhd_host.cu): one partial per instance, 6080 and 6400 in all."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2303_01471_gb300 import qhd


@pytest.mark.parametrize("shape,batch", [((8, 8), 7000), ((128, 64), 190), ((128, 64), 200)])
def test_minimiser_and_nonfinite_check(shape, batch):
    rng = np.random.default_rng(4)
    f = np.round(rng.uniform(0.0, 50.0, (batch, *shape)))  # many ties: the lowest index counts
    sim = qhd.QHD(shape, batch=batch)
    fd = torch.from_numpy(f).cuda()
    sim.set_potential(fd)
    sim.reset_state()
    for b, o in enumerate(sim.observables(0.1)):
        want = np.unravel_index(np.argmin(f[b]), shape)
        assert o.x_star[:2] == tuple(i / n for i, n in zip(want, shape))
        assert o.e_f == pytest.approx(f[b].mean(), rel=1e-6)
    for value in (float("nan"), float("inf"), float("-inf")):
        fd[batch - 1, -1, -1] = value
        with pytest.raises(qhd.QHDError, match="instance %d: 1 non-finite" % (batch - 1)):
            sim.set_potential(fd)
    sim.close()
