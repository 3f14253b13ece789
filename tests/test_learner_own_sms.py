"""The learner under ``sg_qnet_set_grid_limit`` runs as single CTAs that take a
tile's three forwards in turn: the same parameters, moments, target, loss and
gradient, bit for bit, as the clusters of an unlimited learner, at the edges of
both tile sizes and of the batch that separates them."""

import numpy as np
import pytest
import torch

from tests._helpers import bits

pytestmark = pytest.mark.gpu


def _ring(n_in, slots=40, n=64, seed=3):
    from paper_2305_04180_gb300 import Replay

    rng = np.random.default_rng(seed)
    rp = Replay(slots, n, n_in)
    m = slots * n
    rp.write(0, rng.normal(size=(m, n_in)), rng.normal(size=(m, n_in)), rng.integers(0, 5, m), rng.normal(size=m),
             rng.random(m) < 0.2, steps_recorded=slots)
    return rp


def _run(batch, n_in, arch, limit, rp, steps=5):
    from paper_2305_04180_gb300 import QNet

    q = QNet(n_in, batch, seed=4, arch=arch)
    q.set_params(2.0 * q.get_params("online"), "target")
    q.set_grid_limit(learner=limit)
    out = []
    for i in range(steps):
        loss, grad = torch.zeros(1, device="cuda"), torch.zeros(q.n_params, device="cuda")
        q.train_step(rp, batch, lr=1e-3, target_every=2, seed=7, loss=loss, grad=grad)
        out += [loss.cpu().numpy(), grad.cpu().numpy()]
    m, v, st = q.optimizer_state()
    assert st == steps and np.isfinite(out[-1]).all()
    x = torch.randn(33, n_in, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    return out + [q.get_params("online"), q.get_params("target"), m, v, q.forward(x).cpu().numpy()]


@pytest.mark.parametrize("batch,n_in,arch,limits", [
    (1, 37, "dueling", (1,)), (16, 32, "paper", (1, 2)), (17, 69, "dueling", (1, 2)), (256, 37, "paper", (1, 3, 8)),
    (300, 53, "dueling", (2, 7)), (2047, 37, "dueling", (5, 127)), (2048, 69, "dueling", (1, 2, 8, 15)),
    (2049, 32, "paper", (1, 16)), (4096, 37, "dueling", (6, 100))])
def test_limited_learner_is_bit_identical(batch, n_in, arch, limits):
    rp = _ring(n_in)
    want = _run(batch, n_in, arch, 0, rp)
    for limit in limits:
        for a, b in zip(want, _run(batch, n_in, arch, limit, rp)):
            assert np.array_equal(bits(a), bits(b)), limit


@pytest.mark.parametrize("batch", [40, 2100])
def test_action_outside_the_table_changes_nothing(batch):
    from paper_2305_04180_gb300 import QNet, Replay

    rng = np.random.default_rng(5)
    m = 40 * 64
    rp = Replay(40, 64, 37)
    rp.write(0, rng.normal(size=(m, 37)), rng.normal(size=(m, 37)), np.full(m, 5), rng.normal(size=m), np.zeros(m),
             steps_recorded=40)
    q = QNet(37, batch, seed=4)
    q.set_grid_limit(learner=3)
    before = q.get_params("online"), q.optimizer_state()
    loss = torch.zeros(1, device="cuda")
    q.train_step(rp, batch, lr=1e-3, target_every=2, seed=7, loss=loss)
    after = q.get_params("online"), q.optimizer_state()
    assert np.isnan(loss.item()) and after[1][2] == 0
    assert np.array_equal(bits(before[0]), bits(after[0])) and np.array_equal(bits(before[1][0]), bits(after[1][0]))


def test_limited_learner_overlaps_a_rollout():
    """A learner on 12 SMs beside a rollout on the others: about the time of one
    after the other (0.96 of it), where a learner that finds no SMs to run on until
    the rollout ends takes 1.6 times as long."""
    from paper_2305_04180_gb300 import Sim
    from paper_2305_04180_gb300.trainer import ColorTrainer
    from workloads.configs import DR_RANGES, base_params
    from workloads.maps import make_map

    n, K = 65536, 32
    sim = Sim(base_params(**DR_RANGES), [make_map(1 + i, 366) for i in range(32)], (np.arange(n) % 32).astype(np.int32))
    sim.reset()
    tr = ColorTrainer(sim, batch=4096, slots=K + 8, learn_start=0, two_streams=True, max_rollout_k=K, seed=5)
    sim.rollout(K, policy="eps_q", qnet=tr.actor, eps=tr.eps, replay=tr.replay)
    graphs = [tr.capture_iteration(K, 16, concurrent=False), tr.capture_iteration(K, 16, learner_sms=12)]
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
    ratio = []
    for _ in range(7):
        ev[0].record(tr.s_actor)
        for i, g in enumerate(graphs):
            for _ in range(3):
                g.launch(tr.s_actor)
            ev[i + 1].record(tr.s_actor)
        torch.cuda.synchronize()
        ratio.append(ev[1].elapsed_time(ev[2]) / ev[0].elapsed_time(ev[1]))
    assert sim.status() == 0 and np.isfinite(tr.loss.item())
    assert np.median(ratio) < 1.15, ratio
