"""``sg_sim_rollout`` before any launch is set: the library's choice by env
count and K gives the results of one warp per env (SG_ROLLOUT_GRID, itself
compared with the oracle elsewhere) bit for bit, at the sizes where one form
ends and the next begins, and leaves the reported launch alone."""

import numpy as np
import pytest
import torch

from tests._helpers import bits
from workloads.configs import DR_RANGES, base_params
from workloads.maps import make_map, random_tiny_map

pytestmark = pytest.mark.gpu

DISCS = dict(n_dyn=2, dyn_radius=6.0, dyn_speed_lo=10.0, dyn_speed_hi=200.0, dyn_keepout=20.0)


@pytest.mark.parametrize("n,K,kw", [
    (1, 1, {}), (16, 33, {}), (152, 32, {}), (153, 31, {}), (1024, 3, {}), (1024, 4, {}), (4864, 18, {}),
    (4864, 19, {}), (4865, 32, {}), (300, 64, DISCS), (5000, 33, DISCS), (100, 40, dict(march_step=0.37)),
    (200, 40, dict(march_sectors=1))])
def test_default_rollout_matches_grid(n, K, kw):
    from paper_2305_04180_gb300 import Sim

    p = base_params(n_beams=64, t_max=25, **DR_RANGES)
    p.update(kw)
    maps = [make_map(41, 128), make_map(42, 200, 90)]
    if not kw.get("n_dyn"):
        maps.append(random_tiny_map(43, 61, 47, 0.1))
    rng = np.random.default_rng(n)
    env_map = rng.integers(0, len(maps), n).astype(np.int32)
    beams = rng.choice([2, 27, 33, 64], n).astype(np.int32)
    out = []
    for launch in (None, dict(kernel="grid")):
        g = Sim(p, maps, env_map, beams)
        assert g.launch_config()["kernel"] == "grid"
        if launch:
            g.set_launch(**launch)
        g.reset()
        seq = dict(obs_seq=torch.empty((K, n, g.obs_dim), device="cuda"), rew_seq=torch.empty((K, n), device="cuda"),
                   act_seq=torch.empty((K, n), dtype=torch.uint8, device="cuda"),
                   done_seq=torch.empty((K, n), dtype=torch.uint8, device="cuda"))
        for _ in range(2):
            obs = g.rollout(K, obs=g.new_obs(), **seq)
        assert g.status() == 0
        out.append([obs.cpu().numpy()] + [v.cpu().numpy() for v in seq.values()] + list(g.get_state()))
    for a, b in zip(*out):
        same = np.array_equal(bits(a), bits(b)) if a.dtype == np.float32 else np.array_equal(a, b)
        assert same
