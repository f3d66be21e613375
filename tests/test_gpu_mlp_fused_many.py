"""The fused training kernel with more networks than it has blocks: a block trains one network
after the other, and the later ones find nothing of the earlier ones.  Bit for bit the parameters,
moments and last gradient of the separate kernels (rt_mlp_train_step), for networks that a block
takes first, second and last."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    import paper_cs_0703028_gb300 as m
    return m


# a ragged tile, and two with a ragged last one; an odd number of steps, so that a network ends in
# the other half of what a block keeps twice
@pytest.mark.parametrize("batch,n_steps", [(37, 3), (200, 3), (128, 1)])
def test_networks_taken_one_after_the_other(rt, batch, n_steps):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n_nets, n = 2 * sms + 17, 2 * batch
    gen = torch.Generator(device="cuda").manual_seed(batch)
    u = torch.rand(n_nets, n, 4, generator=gen, device="cuda")
    lo, hi = [7.6, 600.0, 0.5, 0.01], [7.601, 2200.0, 5.0, 0.3]
    raw = (torch.tensor(lo, device="cuda") + u * torch.tensor([b - a for a, b in zip(lo, hi)], device="cuda")).contiguous()
    target = (4.0 + torch.sin(6.0 * u[..., 0]) + u[..., 1] * u[..., 2]).contiguous()
    params = torch.from_numpy(np.stack([synth.mlp_init(b, spread_biases=True) for b in range(n_nets)])).cuda().reshape(-1)
    norms = rt.norms_tensor([lo] * n_nets, [hi] * n_nets, [4.0] * n_nets, [1.2] * n_nets)
    a = rt.MlpEnsembleTrainer(params.clone(), norms)
    a.steps(raw, target, batch, 2e-3, 2e-3, 6, n_steps, 6 + n_steps)
    for b in (0, 16, 17, sms - 1, sms, sms + 16, 2 * sms - 1, 2 * sms, 2 * sms + 16):
        s = slice(b * rt.RT_MLP_NPARAM, (b + 1) * rt.RT_MLP_NPARAM)
        t = rt.MlpTrainer(params[s].clone(), rt.make_norm(lo, hi, 4.0, 1.2))
        t.step_no = 5
        for i in range(n_steps):
            q = (5 + i) % 2 * batch
            t.step(raw[b, q:q + batch], target[b, q:q + batch], 2e-3)
        for x, y in ((a.params, t.params), (a.m, t.m), (a.v, t.v), (a.grad, t.grad)):
            assert torch.equal(x[s], y), b
    assert int(a.status) == 0
