"""Kernels whose launch overlaps the end of the kernel before (csrc/qhd_launch.cuh)
read nothing that kernel writes before it is complete."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import workloads
from test_gpu_parity import align_global_phase
from paper_2303_01471_gb300 import qhd

REL_TOL = 1e-12   # same kernels, same block counts: identical up to FP64 rounding order


def test_static_observables_queued_back_to_back():
    """qhd_observables_static calls on one stream with nothing waiting in between, the
    mesh, the box and x* changing from call to call, against the context path: each
    call's set-up kernel writes what its reduction reads, in one array for all calls."""
    lib = qhd.load()
    radius = 0.3
    configs = []
    for seed, (shape, lo, hi) in enumerate([((64,), (0.0,), (1.0,)), ((64, 128), (-1.0, 0.0), (1.0, 2.0)),
                                            ((8, 16, 4), (0.0, -0.5, 0.0), (1.0, 0.5, 2.0)),
                                            ((64, 128), (0.0, 0.0), (1.0, 1.0))]):
        d = len(shape)
        inst = workloads.gaussian_wells(70 + seed, shape, K=4)
        sim = qhd.QHD(shape, lo=lo, hi=hi)
        sim.set_potential(inst.f)
        psi = np.random.default_rng(seed).normal(size=(1, *shape, 2)).astype(np.float32)
        sim.psi.copy_(torch.view_as_complex(torch.from_numpy(psi / np.linalg.norm(psi))).reshape(sim.psi.shape))
        configs.append({"d": d, "n": (ctypes.c_int64 * d)(*shape), "lo": (ctypes.c_double * d)(*lo),
                        "hi": (ctypes.c_double * d)(*hi), "psi": sim.psi.clone(), "f": torch.from_numpy(inst.f).cuda(),
                        "ref": sim.observables(radius)[0]})
        sim.close()
    p = [c["ref"].p_succ for c in configs]
    assert all(abs(p[k] - p[k - 1]) > 1e-3 for k in range(len(p)))   # another call's table would show
    out = torch.full((200, 3), float("nan"), dtype=torch.float64, device="cuda")
    stream = torch.cuda.current_stream()
    torch.cuda.synchronize()
    for call in range(out.shape[0]):
        c = configs[call % len(configs)]
        xs = (ctypes.c_double * 3)(*c["ref"].x_star)
        assert lib.qhd_observables_static(c["d"], c["n"], c["lo"], c["hi"], 1, ctypes.c_void_p(c["psi"].data_ptr()),
                                          ctypes.c_void_p(c["f"].data_ptr()), xs, radius,
                                          ctypes.c_void_p(out[call].data_ptr()), None,
                                          ctypes.c_void_p(stream.cuda_stream)) == qhd.QHD_OK
    stream.synchronize()
    for call, got in enumerate(out.cpu().numpy()):
        ref = configs[call % len(configs)]["ref"]
        assert got == pytest.approx(np.array([ref.norm, ref.e_f, ref.p_succ]), rel=REL_TOL, abs=1e-300), call


# 200 steps of some 40 FP32 roundings each, in two runs, add up at random: sqrt(2 * 200 * 40)
# of half an ulp is 4e-6 of an amplitude; five times that
ROUNDING = 2e-5


@pytest.mark.parametrize("own_kinetic", [False, True], ids=["shared-kinetic", "own-kinetic"])
@pytest.mark.parametrize("shape", [(64,), (1024,), (16, 16), (512, 4), (16, 16, 16), (8, 32, 32)],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_one_step_calls_match_one_call(shape, own_kinetic):
    """Every call of one step builds its kinetic tables in the kernel before the passes
    that read them, where the call before had its own: 200 calls queued without a
    synchronisation against one call of 200 steps."""
    insts = [workloads.gaussian_wells(80 + b, shape, K=4) for b in range(3)]
    states = []
    for calls in (1, 200):
        sim = qhd.QHD(shape, batch=3)
        sim.set_potential(np.stack([i.f for i in insts]))
        sim.set_schedule([qhd.Schedule(c_phi=2.0 + (0.3 * b if own_kinetic else 0.0)) for b in range(3)])
        sim.reset_state()
        for _ in range(calls):
            sim.evolve(2.0 / calls, 0.01)
        states.append(sim.psi.cpu().numpy().astype(np.complex128))
        sim.close()
    for a, b in zip(*states):
        assert np.max(np.abs(align_global_phase(b, a) - a)) <= ROUNDING * np.abs(a).max()


# one launch of up to 16 blocks, of up to one block per SM, of more, and of one-warp
# blocks in several waves: where a pass releases the next differs (csrc/qhd_launch.cuh);
# chunks of 32 and of 33 steps: the whole-run kernels overlap or not
@pytest.mark.parametrize("shape,batch", [((16, 16), 1), ((256, 16), 1), ((512, 64), 4), ((512, 64), 16), ((4, 1024), 300),
                                         ((64, 64), 8), ((128, 128), 200), ((256, 256), 8), ((64, 64, 64), 1), ((64,), 64)],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
@pytest.mark.parametrize("steps", [32, 33])
def test_repeated_runs_are_the_same_bits(shape, batch, steps):
    """A pass that reads what the one before has not finished writing differs from run
    to run: six runs queued without a synchronisation in between, each from a fresh
    state, leave the same bits."""
    sim = qhd.QHD(shape, batch=batch)
    f = torch.rand((batch, *shape), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    sim.set_potential(f)
    sim.set_schedule(qhd.Schedule())
    states = []
    for _ in range(6):
        sim.reset_state()
        sim.evolve(steps * 0.01, 0.01)
        states.append(sim.psi.clone())
    assert all(torch.equal(s, states[0]) for s in states[1:])
    assert abs(sim.observables()[-1].norm - 1.0) < 1e-5
    sim.close()
