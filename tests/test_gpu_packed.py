"""The packed line FFT's plans (csrc/qhd_packed.cuh) and the plane engine built on
them (csrc/qhd_plane2.cuh) against the FP64 oracle.

Launches over more than 2^20 points transform lines of 128, 256 and 1024 points
with 16 points per thread instead of 8; batches just above that line run that
plan at every tile width (1 to 32 pairs of columns) and as rows.  Tolerance per
amplitude: the short-run bound of tests/test_gpu_parity.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle
import workloads
from paper_2303_01471_gb300 import qhd
from test_gpu_parity import compare, to_oracle_sched

# (shape, instances): just over 2^20 points each
LARGE = [((1024, 2), 513), ((1024, 16), 65), ((16, 1024), 65), ((128, 8), 1025), ((4, 128, 2), 1025),
         ((256, 16, 4), 65), ((2, 16, 256), 129), ((128, 16, 16), 33)]


IDS = dict(ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))


def run_and_compare(shape, batch, picked, own_phi=False):
    insts = {b: workloads.gaussian_wells(50 + b, shape, K=4) for b in picked}
    f = np.broadcast_to(insts[0].f, (batch, *shape)).copy()
    for b in picked:
        f[b] = insts[b].f
    sim = qhd.QHD(shape, batch=batch)
    sim.set_potential(torch.from_numpy(f).cuda())
    scheds = [qhd.Schedule(c_phi=2.0 + 0.1 * (b % 3) if own_phi else 2.0) for b in range(batch)]
    sim.set_schedule(scheds)
    sim.reset_state()
    n = 20
    sim.evolve(n * 0.01, 0.01)
    obs = sim.observables(0.1)
    for b in picked:
        psi_o = oracle.evolve(insts[b].f, oracle.uniform_state(shape), 0.0, 0.01, n, to_oracle_sched(scheds[b]))
        compare(sim.psi[b].cpu().numpy().astype(np.complex128), obs[b], insts[b].f, psi_o, steps=n)
    ctas = sim.cluster_ctas()
    sim.close()
    return ctas


@pytest.mark.parametrize("shape,batch", LARGE, **IDS)
def test_sixteen_point_plan_matches_oracle(shape, batch):
    run_and_compare(shape, batch, sorted({0, batch // 2, batch - 1}))


# every 2-D mesh of the one-CTA form, in batches of two waves and a few instances
# more (those run on clusters): first and last of each part
@pytest.mark.parametrize("shape,own_phi", [((n0, n1), k % 2 == 0) for k, (n0, n1) in enumerate(
    [(32, 32), (32, 64), (32, 128), (32, 256), (64, 32), (64, 64), (64, 128), (64, 256), (128, 32), (128, 64),
     (128, 128)])], **IDS)
def test_one_cta_per_instance_matches_oracle(shape, own_phi):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sim = qhd.QHD(shape, batch=8 * sms)
    assert sim.cluster_ctas() == 1
    sim.close()
    batch = 8 * sms + 5
    ctas = run_and_compare(shape, batch, [0, sms, 8 * sms - 1, 8 * sms + 4], own_phi)
    assert ctas == 1


# the plane pass of 3-D meshes whose planes the all-shapes parity test leaves out
@pytest.mark.parametrize("shape", [(2, 32, 128), (2, 32, 256), (2, 64, 32), (2, 64, 64), (2, 64, 256), (2, 128, 64),
                                   (2, 128, 128), (2, 128, 256), (2, 256, 32), (2, 256, 128)], **IDS)
def test_plane_pass_matches_oracle(shape):
    run_and_compare(shape, 3, [0, 2], own_phi=True)
