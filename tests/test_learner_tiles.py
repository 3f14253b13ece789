"""``sg_td_train_step`` at the edges of its tiles: 16-sample tiles (one, a
remainder, 16 and 17 of them, the largest batch), 128-sample tiles (the
smallest batch, a remainder), every input width class, both networks.  Loss and
gradient against the float64 oracle's bf16 recipe; the update against the
oracle's Adam; and every copy of the weights that the update writes (BF16
image, tensor-core operands, target) against those of a fresh network given
the same parameters, bit for bit."""

import numpy as np
import pytest
import torch

from oracle import qnet as OQ
from tests._helpers import ring_sample_entries

pytestmark = pytest.mark.gpu

SLOTS, ENVS = 7, 301


def _theta(seed, n_in, arch):
    p = OQ.init_params(seed, n_in, arch)
    return OQ.flatten({k: v * 2.0 for k, v in p.items()}).astype(np.float32)


@pytest.mark.parametrize("batch,n_in,arch", [
    (1, 37, "dueling"), (15, 32, "paper"), (16, 48, "dueling"), (17, 69, "dueling"), (256, 33, "paper"),
    (257, 37, "dueling"), (2047, 69, "paper"), (2048, 37, "dueling"), (2049, 32, "paper"), (2176, 69, "dueling"),
    (7000, 53, "dueling")])
def test_td_step_at_tile_edges(batch, n_in, arch):
    from paper_2305_04180_gb300 import QNet, Replay

    rng = np.random.default_rng(batch)
    cap = SLOTS * ENVS
    ring = (rng.uniform(-1, 1, (cap, n_in)).astype(np.float32), rng.uniform(-1, 1, (cap, n_in)).astype(np.float32),
            rng.integers(0, 5, cap).astype(np.uint8), (2.0 * rng.normal(size=cap)).astype(np.float32),
            (rng.uniform(size=cap) < 0.1).astype(np.uint8))
    rp = Replay(SLOTS, ENVS, n_in, reserve=2)
    steps = 3 if batch % 2 else 40  # a ring that is still filling, and a full one
    rp.write(0, *ring, steps_recorded=steps)
    q = QNet(n_in, batch, 0, arch=arch)
    on, tg = _theta(1, n_in, arch), _theta(2, n_in, arch)
    q.set_params(on, "online")
    q.set_params(tg, "target")
    loss, grad = torch.zeros(1, device="cuda"), torch.zeros(q.n_params, device="cuda")
    kw = dict(gamma=0.98, seed=5, loss=loss, grad=grad)
    q.train_step(rp, batch, lr=0.0, **kw)
    g0 = grad.cpu().numpy().astype(np.float64)
    idx = ring_sample_entries(5, 0, batch, steps, SLOTS, ENVS, 2)
    bt = {k: v[idx].astype(np.int64 if k == "a" else np.float64)
          for k, v in zip(("s", "s2", "a", "r", "term"), ring)}
    ref_loss, ref = OQ.td_loss_grad(OQ.unflatten(on.astype(np.float64), n_in, arch),
                                    OQ.unflatten(tg.astype(np.float64), n_in, arch), bt, 0.98, bf16=True)
    # the bounds of the repository's other TD tests: float32 sums, and values that
    # round to a neighbouring BF16 on one side
    assert abs(float(loss.item()) - ref_loss) <= 1e-2 * max(abs(ref_loss), 0.1)
    ref, at = OQ.flatten(ref), 0
    for name, shape in OQ.param_shapes(n_in, arch):
        sl = slice(at, at + int(np.prod(shape)))
        assert np.linalg.norm(g0[sl] - ref[sl]) <= 6e-2 * max(np.linalg.norm(ref[sl]), 1e-12), name
        at = sl.stop
    assert at == g0.size
    # the update, a target step
    q.train_step(rp, batch, lr=1e-3, target_every=1, **kw)
    assert np.array_equal(grad.cpu().numpy(), g0.astype(np.float32))
    th, m, v = OQ.adam_step(on.astype(np.float64), g0, np.zeros_like(g0), np.zeros_like(g0), 1, lr=1e-3)
    got = q.get_params("online")
    assert np.max(np.abs(got - th)) <= 2e-6
    assert np.array_equal(q.get_params("target"), got)
    st = q.state_dict()
    assert st["steps"] == 1 and np.allclose(st["m"], m, rtol=1e-5, atol=1e-12)
    # the next step and the batched forward read every copy the update wrote
    fresh = QNet(n_in, batch, 0, arch=arch)
    fresh.load_state_dict(st)
    obs = torch.from_numpy(ring[0][:130]).cuda()
    assert torch.equal(q.forward(obs), fresh.forward(obs))
    out = []
    for net in (q, fresh):
        for _ in range(2):
            net.train_step(rp, batch, lr=1e-3, target_every=3, **kw)
        out.append((loss.clone(), grad.clone(), net.state_dict()))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    for k in ("online", "target", "m", "v"):
        assert np.array_equal(out[0][2][k], out[1][2][k]), k
    assert out[0][2]["steps"] == 3 and np.array_equal(out[0][2]["target"], out[0][2]["online"])
