"""A TD step beside rollouts that append to its ring: all parts of a sample (s,
a, r, terminal, and both networks' s') come from one ring entry, whatever the
step counter does meanwhile.

With lr = 0 nothing but the seed and the step counter decides a step's samples,
so each step that ran beside the rollouts has the loss and the gradient, bit
for bit, of a step that runs alone with the counter at one of the values it
passed through (the ring never wraps: completed slots keep their contents).  One
cluster (a batch of one tile) or one CTA takes all tiles, so that one reading of
the counter covers the step."""

import numpy as np
import pytest
import torch

from workloads.configs import base_params
from workloads.maps import make_map

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,steps,n_roll,ctas", [(16, 400, 400, 0), (40, 400, 400, 1), (2048, 40, 160, 1)])
def test_samples_come_from_one_entry_beside_rollouts(batch, steps, n_roll, ctas):
    from paper_2305_04180_gb300 import QNet, Replay, Sim

    n, K, first = 16, 1, 3
    sim = Sim(dict(base_params(), seed=9), [make_map(3, 128)], np.zeros(n, np.int32))
    sim.reset()
    actor = QNet(sim.obs_dim, 16, seed=1)
    q = QNet(sim.obs_dim, batch, seed=2)
    q.set_params(3.0 * q.get_params("online"), "target")
    q.set_grid_limit(learner=ctas)
    rp = Replay(first + n_roll * K + 1, n, sim.obs_dim, reserve=1)
    eps = torch.full((n,), 0.5, device="cuda")
    for _ in range(first):
        sim.rollout(K, policy="eps_q", qnet=actor, eps=eps, replay=rp)
    loss = torch.zeros((steps, 1), device="cuda")
    grad = torch.zeros((steps, q.n_params), device="cuda")

    def td(i, loss, grad, stream=None):
        q.train_step(rp, batch, lr=0.0, target_every=0, seed=100 + i, loss=loss, grad=grad, stream=stream)

    sa, sl = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for i in range(steps):
        for _ in range(n_roll // steps):
            sim.rollout(K, policy="eps_q", qnet=actor, eps=eps, replay=rp, stream=sa)
        td(i, loss[i], grad[i], sl)
    torch.cuda.synchronize()
    last = rp.steps_recorded()
    assert last == first + (n_roll // steps) * steps * K and torch.isfinite(grad).all()

    empty = [np.zeros((0, sim.obs_dim)), np.zeros((0, sim.obs_dim)), np.zeros(0), np.zeros(0), np.zeros(0)]
    at = torch.zeros(steps, dtype=torch.int64, device="cuda")  # a counter value that gives the step's result
    loss1, grad1 = torch.zeros_like(loss), torch.zeros_like(grad)
    for c in range(first, last + 1, K):
        rp.write(0, *empty, steps_recorded=c)
        for i in range(steps):
            td(i, loss1[i], grad1[i])
        at[(grad1 == grad).all(1) & (loss1 == loss).all(1)] = c
    assert (at > 0).all(), f"{int((at == 0).sum())} of {steps} steps mix entries"
    assert at.unique().numel() > 1  # the counter did move while the steps ran
