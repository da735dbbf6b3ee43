"""P_succ counts mesh points strictly nearer than the radius: the uniform state on a
power-of-two mesh gives count / G exactly, with the radius on a mesh distance, one
unit in the last place above it, and between distances (csrc/qhd_kernels.cu compares
squared distances); and set_potential's minimiser over one and many partials."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2303_01471_gb300 import qhd


@pytest.mark.parametrize("shape", [(16,), (8, 16), (4, 8, 16)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("radius", [0.125, np.nextafter(0.125, 1.0), np.sqrt(0.125 ** 2 + 0.25 ** 2), 0.3, 1e-200, 10.0])
def test_strict_radius(shape, radius):
    at = tuple(n // 2 for n in shape)
    f = np.ones(shape)
    f[at] = 0.0
    sim = qhd.QHD(shape)
    sim.set_potential(f)
    sim.reset_state()
    obs = sim.observables(float(radius))[0]
    axes = np.meshgrid(*[np.arange(n) / n for n in shape], indexing="ij")
    r2 = np.zeros(shape)
    for d in range(len(shape) - 1, -1, -1):  # the library's order of summation
        r2 = r2 + (axes[d] - at[d] / shape[d]) ** 2
    amp = np.float64(np.float32(1.0 / np.sqrt(f.size)))
    assert obs.p_succ == pytest.approx(np.count_nonzero(np.sqrt(r2) < radius) * amp ** 2, rel=1e-12)
    sim.close()


@pytest.mark.parametrize("shape,batch", [((8, 8), 3), ((128, 64), 40)])
def test_minimiser_lowest_index_on_ties(shape, batch):
    rng = np.random.default_rng(3)
    f = np.round(rng.uniform(0.0, 50.0, (batch, *shape)))  # many ties
    sim = qhd.QHD(shape, batch=batch)
    sim.set_potential(f)
    sim.reset_state()
    for b, o in enumerate(sim.observables(0.1)):
        want = np.unravel_index(np.argmin(f[b]), shape)
        assert o.x_star[:2] == tuple(i / n for i, n in zip(want, shape))
    sim.close()
