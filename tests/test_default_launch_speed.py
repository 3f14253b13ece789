"""``sg_sim_rollout`` before any launch is set is not slower than one warp per
env (SG_ROLLOUT_GRID): at the sizes where its choice turns from one form to
another, with and without moving obstacles."""

import numpy as np
import pytest
import torch

from workloads.configs import DR_RANGES, DYN_RANGES, base_params
from workloads.maps import make_map

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,K,dyn", [
    (256, 2, False), (1024, 2, False), (2048, 4, False), (4096, 12, False), (4096, 16, False), (8192, 16, False),
    (16384, 18, False), (2048, 8, True), (3000, 24, True), (4096, 16, True), (4096, 56, True), (8192, 32, True),
    (16384, 32, True), (16384, 72, True)])
def test_default_is_not_slower_than_grid(n, K, dyn):
    """The median over rounds that time both in turn; 8% covers their spread
    (under 2%) and the flat part of the line between two forms.  Where a form
    is the wrong one it takes 15% or more longer."""
    from paper_2305_04180_gb300 import Sim

    maps = [make_map(1 + i, 366) for i in range(32)]
    p = base_params(**(dict(DR_RANGES, **DYN_RANGES) if dyn else {}))
    sims = [Sim(p, maps, (np.arange(n) % 32).astype(np.int32)) for _ in range(2)]
    sims[1].set_launch("grid")
    obs = sims[0].new_obs()
    seq = dict(obs_seq=torch.empty((K, n, sims[0].obs_dim), device="cuda"), rew_seq=torch.empty((K, n), device="cuda"),
               act_seq=torch.empty((K, n), dtype=torch.uint8, device="cuda"),
               done_seq=torch.empty((K, n), dtype=torch.uint8, device="cuda"))
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
    reps = max(3, 60000 // (n * K // 8 + 1))
    for s in sims:
        s.reset()
        s.rollout(64, obs=obs)
    ratio = []
    for _ in range(9):
        ev[0].record()
        for i, s in enumerate(sims):
            for _ in range(reps):
                s.rollout(K, obs=obs, **seq)
            ev[i + 1].record()
        torch.cuda.synchronize()
        ratio.append(ev[0].elapsed_time(ev[1]) / ev[1].elapsed_time(ev[2]))
    assert np.median(ratio) < 1.08, ratio
