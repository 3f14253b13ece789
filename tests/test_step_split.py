"""``sg_sim_step`` over its launch forms: one env per warp, several, and the
motion / finish kernel pair of large batches, at the sizes where one ends and
the next begins, over mixed maps (poses outside a map among them), uneven
beams, march steps and sector counts that take the general march, and moving
obstacles.  Bit for bit against the strict-float32 oracle."""

import numpy as np
import pytest
import torch

from oracle.sim import OracleSim
from tests._helpers import bits, gpu_state_to_oracle, oracle_state_to_gpu
from workloads.configs import DR_RANGES, base_params
from workloads.maps import empty_map, make_map, random_tiny_map

pytestmark = pytest.mark.gpu

DISCS = dict(n_dyn=3, dyn_radius=6.0, dyn_speed_lo=10.0, dyn_speed_hi=200.0, dyn_keepout=20.0)


@pytest.mark.parametrize("n,kw", [
    (1, {}), (152, {}), (153, {}), (4864, {}), (4865, {}), (8191, {}), (8192, {}), (8195, dict(march_sectors=1)),
    (8223, dict(march_sectors=32)), (8192, dict(march_step=0.37, range_max=60.0)),
    (8193, dict(march_step=2.0)), (700, DISCS), (8200, DISCS)])
def test_step_forms_match_oracle(n, kw):
    from paper_2305_04180_gb300 import Sim

    p = base_params(n_beams=64, t_max=40, **DR_RANGES)
    p.update(kw)
    maps = [make_map(31, 128), random_tiny_map(32, 61, 47, 0.1), make_map(33, 200, 90), make_map(34, 366)]
    if not kw.get("n_dyn"):
        maps += [empty_map(20, 9), random_tiny_map(35, 1, 1, 1.0)]  # starts outside the map
    rng = np.random.default_rng(n)
    env_map = rng.integers(0, len(maps), n).astype(np.int32)
    beams = rng.choice([2, 27, 32, 33, 64], n).astype(np.int32)
    g = Sim(p, maps, env_map, beams)
    o = OracleSim(p, maps, env_map, beams, prec="f32")
    g.reset()
    o.reset()
    term = torch.zeros((n, g.obs_dim), device="cuda")
    done_seen = 0
    for t in range(6):
        state = g.get_state()
        f, u = state[:2]
        if t == 3:  # spread the poses over the maps, some near truncation
            w = np.array([m.shape[1] for m in maps])[env_map]
            h = np.array([m.shape[0] for m in maps])[env_map]
            f[0], f[1] = rng.uniform(-3, w + 3), rng.uniform(-3, h + 3)
            f[2] = rng.uniform(-3.1, 3.1, n)
            u[0] = rng.integers(30, 40, n)
            g.set_state(*state)
        o.set_state(*gpu_state_to_oracle(*state))
        a = rng.integers(0, 5, n).astype(np.uint8)
        obs, rew, done = g.step(torch.from_numpy(a).cuda(), term_obs=term)
        oobs, orew, odone, oterm = o.step(a)
        d = done.cpu().numpy()
        assert np.array_equal(d, odone), t
        assert np.array_equal(bits(rew.cpu().numpy()), bits(orew)), t
        assert np.array_equal(bits(obs.cpu().numpy()), bits(oobs)), t
        assert np.array_equal(bits(term.cpu().numpy()[d != 0]), bits(oterm[d != 0])), t
        got = g.get_state()
        of, ou, ob, *od = o.state()
        gf, gu = oracle_state_to_gpu(of, ou, ob, u[2] + 1)
        assert np.array_equal(bits(got[0]), bits(gf)) and np.array_equal(got[1], gu), t
        if od:
            assert np.array_equal(bits(got[2]), bits(od[0])), t
        done_seen += int((d != 0).sum())
    assert g.status() == 0 and done_seen > 0
