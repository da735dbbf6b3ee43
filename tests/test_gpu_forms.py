"""Which 2-D instances of a batch run in one CTA each (csrc/qhd_plane.cu): batches of
both forms, first and last instance of each part against the FP64 oracle, and batches
that the choice leaves to the clusters.  The launches per chunk say which ran: the
step tables, then one launch per form."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle
import workloads
from paper_2303_01471_gb300 import qhd
from test_gpu_parity import compare, to_oracle_sched

SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152


# whole waves of the one-CTA form (1, 2 and 4 instances per SM) and five more instances
@pytest.mark.parametrize("shape,per_sm,waves", [((128, 128), 1, 3), ((128, 64), 2, 1), ((128, 32), 4, 1)])
@pytest.mark.parametrize("own_phi", [False, True], ids=["shared-kinetic", "own-kinetic"])
def test_batch_of_both_forms_matches_oracle(shape, per_sm, waves, own_phi):
    solo = SMS * per_sm * waves
    batch = solo + 5
    picked = [0, solo - 1, solo, batch - 1]
    insts = {b: workloads.gaussian_wells(50 + b, shape, K=4) for b in picked}
    f = np.broadcast_to(insts[0].f, (batch, *shape)).copy()
    for b in picked:
        f[b] = insts[b].f
    sim = qhd.QHD(shape, batch=batch)
    sim.set_potential(torch.from_numpy(f).cuda())
    scheds = [qhd.Schedule(c_phi=2.0 + 0.1 * (b % 3) if own_phi else 2.0) for b in range(batch)]
    sim.set_schedule(scheds)
    sim.reset_state()
    before = sim.launch_count()
    sim.evolve(0.2, 0.01)
    assert sim.cluster_ctas() == 1 and sim.launch_count() - before == 3
    obs = sim.observables(0.1)
    for b in picked:
        psi_o = oracle.evolve(insts[b].f, oracle.uniform_state(shape), 0.0, 0.01, 20, to_oracle_sched(scheds[b]))
        compare(sim.psi[b].cpu().numpy().astype(np.complex128), obs[b], insts[b].f, psi_o, steps=20)
    sim.close()


# per SM: fewer instances than the one-CTA form gains from, or a mesh that gains nothing
@pytest.mark.parametrize("shape,batch,ctas", [((32, 32), SMS, 2), ((32, 32), SMS + 8, 2), ((64, 32), SMS // 2, 2),
                                              ((128, 32), SMS // 2 + 1, 4), ((128, 128), SMS // 2 + 1, 4),
                                              ((64, 256), 2 * SMS, 2), ((64, 64), SMS, 1), ((128, 128), SMS, 1)])
def test_small_batches_keep_their_clusters(shape, batch, ctas):
    sim = qhd.QHD(shape, batch=batch)
    assert sim.cluster_ctas() == ctas
    sim.close()
