"""The small fused actor where its envs per CTA change (one env per CTA up to
one per SM, eight and nine, 16), with 8- and 16-row network tiles: the same
trajectories, ring and final state as with 32 envs per CTA, bit for bit."""

import numpy as np
import pytest
import torch

from oracle import qnet as OQ
from workloads import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 16, 152, 153, 1216, 1217, 2432])
@pytest.mark.parametrize("dyn", [0, 2])
def test_actor_env_spread_agrees(n, dyn):
    from paper_2305_04180_gb300 import QNet, Replay, Sim

    w = workload("qnet4096", n_envs=n)
    p = dict(w.params, t_max=9)
    if dyn:
        p.update(n_dyn=dyn, dyn_radius=6.0, dyn_speed_lo=10.0, dyn_speed_hi=100.0, dyn_keepout=20.0)
    out = []
    for rows in (16, 32):
        s = Sim(p, w.maps(), w.env_map)
        q = QNet(s.obs_dim, 16, 0)
        q.set_params((OQ.flatten(OQ.init_params(4, s.obs_dim)) * 3.0).astype(np.float32))
        q.set_rollout_rows(rows)
        rp = Replay(5, n, s.obs_dim)
        s.reset()
        seq = dict(obs_seq=torch.empty((6, n, s.obs_dim), device="cuda"), rew_seq=torch.empty((6, n), device="cuda"),
                   act_seq=torch.empty((6, n), dtype=torch.uint8, device="cuda"),
                   done_seq=torch.empty((6, n), dtype=torch.uint8, device="cuda"))
        eps = torch.full((n,), 0.2, device="cuda")
        for _ in range(3):
            s.rollout(6, policy="eps_q", qnet=q, eps=eps, replay=rp, **seq)
        assert s.status() == 0 and rp.steps_recorded() == 18
        out.append([v.cpu().numpy() for v in seq.values()] + list(s.get_state()) + list(rp.read(0, rp.capacity)))
    for a, b in zip(*out):
        assert np.array_equal(a.view(np.uint32) if a.dtype == np.float32 else a,
                              b.view(np.uint32) if b.dtype == np.float32 else b)
