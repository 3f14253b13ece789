"""The pipelined rollout with a helper warp (one env per CTA and 15 observation
warps, or 7 with moving obstacles), sliced in time: segments of an odd and an even
number of 32-step chunks, a short last chunk or a whole one, and more items than
resident CTAs, so that a segment continues a state that another CTA stored.  Bit
for bit the rollout of one warp per env."""

import numpy as np
import pytest
import torch

from workloads.configs import DR_RANGES, base_params
from workloads.maps import make_map

pytestmark = pytest.mark.gpu

DISCS = dict(n_dyn=3, dyn_radius=6.0, dyn_speed_lo=10.0, dyn_speed_hi=200.0, dyn_keepout=20.0)
HELPED = {"discs": (DISCS, dict(warps_per_block=8, obs_warps=7)),
          "discs, 15": (DISCS, dict(warps_per_block=16, obs_warps=15)),
          "plain": ({}, dict(warps_per_block=16, obs_warps=15)),
          "march": (dict(march_step=0.6), dict(warps_per_block=16, obs_warps=15))}


@pytest.mark.parametrize("form", list(HELPED))
@pytest.mark.parametrize("segment,K", [(32, 33), (32, 64), (32, 300), (64, 65), (64, 159), (64, 256), (96, 97),
                                       (96, 290)])
def test_sliced_helper_matches_grid(form, segment, K):
    from paper_2305_04180_gb300 import Sim

    kw, launch = HELPED[form]
    n = 700
    p = base_params(n_beams=40, t_max=45, **DR_RANGES)
    p.update(kw)
    maps = [make_map(31, 128), make_map(33, 200, 90)]
    env_map = (np.arange(n) % 2).astype(np.int32)
    out = []
    for cfg in (dict(kernel="grid"), dict(kernel="pipe", order="map", segment=segment, **launch)):
        g = Sim(p, maps, env_map)
        g.set_launch(**cfg)
        g.reset()
        seq = dict(obs_seq=torch.zeros((K, n, g.obs_dim), device="cuda"), rew_seq=torch.zeros((K, n), device="cuda"),
                   act_seq=torch.zeros((K, n), dtype=torch.uint8, device="cuda"),
                   done_seq=torch.zeros((K, n), dtype=torch.uint8, device="cuda"))
        for _ in range(2):
            obs = g.rollout(K, obs=g.new_obs(), **seq)
        assert g.status() == 0
        out.append([obs, *seq.values()] + [torch.from_numpy(x.view(np.int32)) for x in g.get_state()])
    assert (out[0][4] != 0).any()  # episodes end
    for a, b in zip(*out):
        assert torch.equal(a.view(torch.int32) if a.dtype == torch.float32 else a,
                           b.view(torch.int32) if b.dtype == torch.float32 else b)
