"""``sg_sim_step`` with a march step other than one cell: its forms (one and two
envs per warp, the kernel pair, eight envs per warp) give a one-step rollout's
values bit for bit at the sizes where one ends and the next begins, and a step of
few envs is not held up by envs that wait for one another in a warp."""

import numpy as np
import pytest
import torch

from tests._helpers import bits
from workloads.configs import DR_RANGES, base_params
from workloads.maps import make_map, random_tiny_map

pytestmark = pytest.mark.gpu

DISCS = dict(n_dyn=2, dyn_radius=6.0, dyn_speed_lo=10.0, dyn_speed_hi=200.0, dyn_keepout=20.0)


def _sims(n, kw, beams=64):
    from paper_2305_04180_gb300 import Sim

    p = base_params(n_beams=beams, t_max=5, **DR_RANGES)
    p.update(kw)
    maps = [make_map(41, 128), make_map(42, 200, 90)]
    if not kw.get("n_dyn"):
        maps.append(random_tiny_map(43, 61, 47, 0.1))
    env_map = np.random.default_rng(n).integers(0, len(maps), n).astype(np.int32)
    out = []
    for _ in range(2):
        s = Sim(p, maps, env_map)
        s.set_launch("grid")
        s.reset()
        out.append(s)
    return out


# an env per warp up to 32 an SM (0: that many)
@pytest.mark.parametrize("n", [1, 0, 8191, 8192, 65561, (1 << 20) + 1])
@pytest.mark.parametrize("kw", [dict(march_step=0.37, range_max=60.0), dict(march_step=2.0),
                                dict(march_step=0.5, **DISCS)])
def test_forms_match_a_one_step_rollout(n, kw):
    n = n or 32 * torch.cuda.get_device_properties(0).multi_processor_count
    a, b = _sims(n, kw, beams=33)
    act = torch.empty((1, n), dtype=torch.uint8, device="cuda")
    rew, done = torch.empty((1, n), device="cuda"), torch.empty((1, n), dtype=torch.uint8, device="cuda")
    for _ in range(6):  # past the truncation at step 5
        want = b.rollout(1, obs=b.new_obs(), act_seq=act, rew_seq=rew, done_seq=done)
        obs, r, d = a.step(act[0])
        assert torch.equal(d, done[0])
        assert torch.equal(r.view(torch.int32), rew[0].view(torch.int32))
        assert torch.equal(obs.view(torch.int32), want.view(torch.int32))
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(bits(x), bits(y)) if x.dtype == np.float32 else np.array_equal(x, y)
    assert a.status() == 0


@pytest.mark.parametrize("n,march_step", [(16, 2.0), (300, 2.0), (1024, 2.0), (4096, 2.0), (1024, 0.5)])
def test_few_envs_take_no_longer_than_one_per_warp(n, march_step):
    """The rollout kernel of one warp per env does the same work in one step:
    twice its time is far from what the step takes when its warps hold one env
    each (0.9 to 1.1), and far below what eight envs in a warp's turn take (2.5 to 4)."""
    a, b = _sims(n, dict(march_step=march_step, t_max=2000), beams=32)
    act = torch.zeros(n, dtype=torch.uint8, device="cuda")
    obs, rew, done = a.new_obs(), torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda")
    e0, e1, e2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
    ratio = []
    for _ in range(9):
        e0.record()
        for _ in range(40):
            a.step(act, obs, rew, done)
        e1.record()
        for _ in range(40):
            b.rollout(1, obs=obs)
        e2.record()
        torch.cuda.synchronize()
        ratio.append(e0.elapsed_time(e1) / e1.elapsed_time(e2))
    assert np.median(ratio) < 2.0, ratio
