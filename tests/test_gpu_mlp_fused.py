"""Training steps of one 128-sample tile, or of several for enough networks, run in one fused
kernel: bit for bit the parameters, moments and last gradient of the separate forward, backward and Adam kernels
(rt_mlp_train_step, which keeps them)."""
import math

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    import paper_cs_0703028_gb300 as m
    return m


# one sample, ragged rows of a warp and of the tile, a full tile; several networks and batches;
# more steps than one launch takes, from the middle of a schedule (bias corrections not yet 1);
# batches of two and three tiles with a ragged last one
@pytest.mark.parametrize("n_nets,batch,n_batches,n_steps,first", [(1, 1, 2, 3, 1), (2, 33, 1, 3, 1), (1, 64, 3, 4, 7), (3, 127, 2, 3, 200),
                                                                  (2, 128, 3, 5, 20000), (1, 40, 2, 243, 1), (40, 129, 2, 2, 3), (50, 300, 1, 2, 1)])
def test_fused_steps_equal_separate_kernels(rt, n_nets, batch, n_batches, n_steps, first):
    import torch
    n = batch * n_batches
    gen = torch.Generator(device="cuda").manual_seed(n_nets * 1000 + batch)
    u = torch.rand(n_nets, n, 4, generator=gen, device="cuda")
    lo, hi = [7.6, 600.0, 0.5, 0.01], [7.601, 2200.0, 5.0, 0.3]
    raw = (torch.tensor(lo, device="cuda") + u * torch.tensor([b - a for a, b in zip(lo, hi)], device="cuda")).contiguous()
    target = (4.0 + torch.sin(6.0 * u[..., 0]) + u[..., 1] * u[..., 2]).contiguous()
    params = torch.from_numpy(np.stack([synth.mlp_init(b, spread_biases=True) for b in range(n_nets)])).cuda().reshape(-1)
    norms = rt.norms_tensor([lo] * n_nets, [hi] * n_nets, [4.0] * n_nets, [1.2] * n_nets)
    a = rt.MlpEnsembleTrainer(params.clone(), norms)
    losses = torch.zeros(n_steps, dtype=torch.float32, device="cuda")
    a.steps(raw, target, batch, 2e-3, 2e-3, first, n_steps, first + n_steps, losses=losses)
    per_step = torch.zeros(n_nets, n_steps, device="cuda")
    for b in range(n_nets):
        norm = rt.make_norm(lo, hi, 4.0, 1.2)
        t = rt.MlpTrainer(params[b * rt.RT_MLP_NPARAM:(b + 1) * rt.RT_MLP_NPARAM].clone(), norm)
        t.step_no = first - 1
        for i in range(n_steps):
            q = (first - 1 + i) % n_batches * batch
            per_step[b, i] = t.step(raw[b, q:q + batch], target[b, q:q + batch], 2e-3)[0]
        s = slice(b * rt.RT_MLP_NPARAM, (b + 1) * rt.RT_MLP_NPARAM)
        for x, y in ((a.params, t.params), (a.m, t.m), (a.v, t.v), (a.grad, t.grad)):
            assert torch.equal(x[s], y)
    assert int(a.status) == 0
    # losses are binary32 sums over the networks in any order: n_nets roundings
    assert torch.allclose(losses, per_step.mean(0), rtol=1e-6 * n_nets)
    assert math.isfinite(float(losses.sum()))
