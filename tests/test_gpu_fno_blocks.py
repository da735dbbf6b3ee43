"""Block shapes of the surrogate's tensor-core kernels: several instances per block
in the axis-0 stages with a remainder, hidden widths that are no multiple of 32 in
the weight gradients.  A batch gives each instance the bits it gets alone;
gradients agree with the FP32 path to BF16 accuracy (5e-2 per block, as in
tests/test_gpu_fno.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2303_01471_gb300 import fno
from test_gpu_fno import dev, perturbed_params, tiny_batch


# 2432 = 4 instances x 4 blocks on each of 152 SMs: just above it, with 1 to 3 instances left over
@pytest.mark.parametrize("n,modes,hidden,batch", [(16, 8, 48, 305), (32, 16, 128, 154), (32, 8, 32, 307)])
def test_block_shapes(n, modes, hidden, batch):
    cfg = fno.FNOConfig(n=n, width=32, modes=modes, layers=2, hidden=hidden, act_bf16=True)
    f, sigma, pt = tiny_batch(11, B=batch, n=n)
    params = torch.from_numpy(perturbed_params(cfg, 12))
    fd, sd, pd = dev(f, torch.float64), dev(sigma, torch.float32), dev(pt, torch.float32)
    net = fno.FNO(cfg, batch_max=batch, params=params)
    many = net.forward(fd, sd)
    for b in (0, 3, 4, batch - 1):
        assert torch.equal(many[b], net.forward(fd[b:b + 1].contiguous(), sd[b:b + 1].contiguous())[0])
    net.close()
    grads = {}
    for bf16 in (True, False):
        net = fno.FNO(fno.FNOConfig(**{**cfg.__dict__, "act_bf16": bf16}), batch_max=batch, train=True, params=params)
        net.loss_grad(fd, sd, pd)
        grads[bf16] = net.grad.cpu().numpy().astype(np.float64)
        net.close()
    for name, (o, k) in fno.param_layout(cfg).items():
        if k and name != "p2_b":
            g16, g32 = grads[True][o:o + k], grads[False][o:o + k]
            assert np.linalg.norm(g16 - g32) <= 5e-2 * np.linalg.norm(g32), name
