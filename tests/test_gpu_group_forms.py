"""A batched group over contexts whose own form is one CTA per instance (or that and
clusters): with the default split every context gets the bits of its own qhd_evolve,
beside contexts that go through the group's queue."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle
import workloads
from paper_2303_01471_gb300 import qhd
from test_gpu_parity import compare

SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152


def make_ctx(n, batch, seed):
    f, _ = workloads.batch_fast_on_device([("wells", seed + b) for b in range(batch)], (n, n), "cuda", K=4)
    sim = qhd.QHD((n, n), batch=batch)
    sim.set_potential(f)
    sim.set_schedule([qhd.Schedule(c_phi=2.0 + 0.1 * (b % 3)) for b in range(batch)])
    sim.reset_state()
    return sim, f


# 64^2 all in one CTA each, 128^2 in both forms, 256^2 on clusters; chunks that overlap
# the step tables and chunks that do not
@pytest.mark.parametrize("steps", [20, 40])
def test_default_group_matches_each_context_bit_for_bit(steps):
    sizes = [(64, 2 * SMS + 3), (128, 3 * SMS + 5), (256, 3)]
    sims, refs = [], []
    for n, batch in sizes:
        for to in (sims, refs):
            to.append(make_ctx(n, batch, 10 * n))
    assert [s.cluster_ctas() for s, _ in sims] == [1, 1, 8]
    grp = qhd.Group([s for s, _ in sims])
    assert grp.info()["sub"] == {64: 1, 128: 1, 256: 8}
    for _ in range(2):                                  # the second pass replays the graph
        for s, _ in sims:
            s.reset_state()
        grp.evolve(steps * 0.01, 0.01)
    assert grp.status() == qhd.QHD_OK and grp.info()["captures"] == 1
    for (s, f), (r, _) in zip(sims, refs):
        r.evolve(steps * 0.01, 0.01)
        torch.cuda.synchronize()
        assert torch.equal(s.psi, r.psi) and s.time() == r.time()
    (s, f), n = sims[1], 128
    obs = s.observables(0.1)
    for b in (0, 3 * SMS - 1, 3 * SMS, 3 * SMS + 4):
        fb = f[b].cpu().numpy()
        psi_o = oracle.evolve(fb, oracle.uniform_state((n, n)), 0.0, 0.01, steps, oracle.Schedule(c_phi=2.0 + 0.1 * (b % 3)))
        compare(s.psi[b].cpu().numpy().astype(np.complex128), obs[b], fb, psi_o, steps=steps)
    grp.close()
    for s, _ in sims + refs:
        s.close()


def test_explicit_splits_and_the_injected_timeout():
    a, f = make_ctx(64, 2 * SMS, 7)
    with pytest.raises(qhd.QHDError) as ei:
        qhd.Group([a], qhd.GroupConfig.make((1, 0, 0), 0, 0))
    assert ei.value.status == qhd.QHD_ERR_INVALID_ARG
    grp = qhd.Group([a], qhd.GroupConfig.make((4, 0, 0), 0, 0))
    grp.evolve(0.2, 0.01)
    assert grp.status() == qhd.QHD_OK and grp.info()["sub"][64] == 4
    psi_o = oracle.evolve(f[0].cpu().numpy(), oracle.uniform_state((64, 64)), 0.0, 0.01, 20, oracle.Schedule(c_phi=2.0))
    compare(a.psi[0].cpu().numpy().astype(np.complex128), a.observables(0.1)[0], f[0].cpu().numpy(), psi_o, steps=20)
    grp.close()
    grp = qhd.Group([a])
    a.reset_state()
    grp.evolve(0.2, 0.01)
    assert grp.status() == qhd.QHD_OK
    grp.inject_wait_timeout(True)                       # reaches the contexts beside the queue too
    a.reset_state()
    grp.evolve(0.2, 0.01)
    assert grp.status() == qhd.QHD_ERR_TIMEOUT
    grp.close()
    a.close()
