"""A launch that is read and set again stays the launch it was: also the one of a
simulator whose launch was never set, where each rollout chooses by its size."""

import numpy as np
import pytest
import torch

from workloads.configs import base_params
from workloads.maps import make_map

pytestmark = pytest.mark.gpu

PIPE = dict(kernel="pipe", warps_per_block=8, obs_warps=3, order="map")


def _ms(s, obs, K=1000):
    out = []
    for _ in range(4):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        s.rollout(K, obs=obs)
        b.record()
        torch.cuda.synchronize()
        out.append(a.elapsed_time(b))
    return min(out[1:])


def test_read_and_set_again_changes_nothing():
    from paper_2305_04180_gb300 import Sim

    s = Sim(base_params(), [make_map(1, 128)], np.zeros(16, np.int32))
    s.reset()
    obs = s.new_obs()
    unset = s.launch_config()
    ms = _ms(s, obs)
    s.set_launch(**unset)
    assert s.launch_config() == unset
    # one warp per env takes 10 times as long here as what the library chooses
    assert _ms(s, obs) < 3 * ms
    s.set_launch("grid")
    grid = s.launch_config()
    assert grid != unset and grid["kernel"] == "grid"
    slow = _ms(s, obs)
    assert slow > 3 * ms
    s.set_launch(**grid)
    assert s.launch_config() == grid and _ms(s, obs) > 3 * ms
    s.set_launch(**PIPE)
    pipe = s.launch_config()
    s.set_launch(**pipe)
    assert s.launch_config() == pipe
    s.set_launch(**unset)
    assert s.launch_config() == unset and _ms(s, obs) < 3 * ms


def test_the_autotuners_keys_are_enough():
    from paper_2305_04180_gb300 import Sim
    from paper_2305_04180_gb300.autotune import KEYS

    s = Sim(base_params(), [make_map(1, 128)], np.zeros(16, np.int32))
    unset = s.launch_config()
    s.set_launch(**PIPE)
    s.set_launch(**{k: unset[k] for k in KEYS})
    assert s.launch_config() == unset
