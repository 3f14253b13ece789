"""What the performance of this library is measured on.

Every case is one call (or one call per pass) that a user of the vectorized
simulator, its fused actor or its learner makes, on inputs made from a seed.
Kinds:

* ``step``      ``Sim.step``: one vectorized step with the caller's actions.
* ``rollout``   ``Sim.rollout`` with random actions: K steps in one call,
                every step's observation, action, reward and flags returned.
* ``q_rollout`` ``Sim.rollout`` with the eps-greedy Q-network actor, the
                transitions written to a replay ring.
* ``forward``   ``QNet.forward``: batched Q-values.
* ``td``        ``QNet.train_step``: one double-DQN step from a replay ring.

Sizes come from the workloads of this repository (16 envs on one map; 1,024
domain-randomised envs on 32 maps; one map per env with 16 to 64 beams;
4,096 and 65,536 envs under the Q-network; batches of 256 and 4,096).
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2305_04180_gb300 import QNet, Replay, Sim

# The robot and the randomisation ranges of the repository's workloads.
ACTIONS = ((0.36, 1.0), (18.0, 1.0), (18.0, 0.0), (18.0, -1.0), (0.36, -1.0))
BASE = dict(n_beams=32, fov=float(np.float32(1.5 * math.pi)), range_max=100.0, march_step=1.0, robot_radius=10.0,
            goal_radius=20.0, near_dist=30.0, t_max=2000, start_offset=30.0, start_jitter=5.0, dt_lo=0.1, dt_hi=0.1,
            k_lo=0.6, k_hi=0.6, cap_lo=1.0, cap_hi=1.0, sigma_lo=0.0, sigma_hi=0.0, delay_lo=0, delay_hi=0,
            v_nom=18.0, w_nom=1.0, actions=ACTIONS, seed=42)
RANDOMISED = dict(dt_lo=0.05, dt_hi=0.2, delay_lo=0, delay_hi=2, k_lo=0.6, k_hi=1.0, cap_lo=0.5, cap_hi=1.5,
                  sigma_lo=0.0, sigma_hi=2.0)
OBSTACLES = dict(dyn_radius=8.0, dyn_speed_lo=4.0, dyn_speed_hi=30.0, dyn_keepout=60.0)

# Launch configurations of the random rollout that users of the autotuner get
# ("default": a simulator whose launch was never set).
LAUNCHES = {
    "default": None,
    "pipe": dict(kernel="pipe", warps_per_block=8, obs_warps=7, order="map"),
    "pipe-sliced": dict(kernel="pipe", warps_per_block=8, obs_warps=7, order="map", segment=512),
}

ACTION_ROWS = 64  # distinct action vectors that step passes walk through
GAMMA = 0.98


def _sim_case(name, kind, envs, **kw):
    c = dict(name=name, kind=kind, envs=envs, steps=1, maps=32, side=366, beams=32, mixed=False, dr=True, dyn=0,
             launch="default", arch="dueling")
    c.update(kw)
    return c


def listed():
    return [
        # the paper's own scale: 16 copies of one map, an external policy
        # stepping them one call at a time (latency of the smallest call)
        _sim_case("step-16", "step", 16, maps=1, dr=False),
        # an external policy on a GPU-sized batch of randomised envs
        _sim_case("step-65536", "step", 65536),
        # 16 envs on one map, 1,000 random steps, launch never configured
        _sim_case("rollout-16", "rollout", 16, steps=1000, maps=1, dr=False),
        # data collection, 1,024 randomised envs, the autotuner's launch
        _sim_case("rollout-1024", "rollout", 1024, steps=2000, launch="pipe-sliced"),
        # uneven batch: a map of 128 to 1,024 cells a side per env, 16 to 64 beams
        _sim_case("rollout-uneven-2048", "rollout", 2048, steps=64, maps=2048, beams=64, mixed=True, dr=False,
                  launch="pipe"),
        # moving obstacles, 4 discs per env
        _sim_case("rollout-discs-1024", "rollout", 1024, steps=500, dyn=4, launch="pipe-sliced"),
        # the paper's actor: 16 envs, 27 beams, its 256-128-5 network, short chunks
        _sim_case("actor-16", "q_rollout", 16, steps=8, maps=16, beams=27, arch="paper"),
        # the fused actor on a mid-size batch
        _sim_case("actor-4096", "q_rollout", 4096, steps=32, dr=False),
        # the full-size actor: mixed maps, 16 to 64 beams
        _sim_case("actor-65536", "q_rollout", 65536, steps=32, maps=256, beams=64, mixed=True),
        # Q-values of a large batch of stored observations (evaluation, relabelling)
        dict(name="forward-1M", kind="forward", rows=1 << 20, inputs=37, arch="dueling"),
        # the paper's learner step: batch 256 from a 1M-transition ring
        dict(name="learn-256", kind="td", batch=256, inputs=37, slots=256, ring_envs=4096, arch="dueling"),
        # the full-size learner step
        dict(name="learn-4096", kind="td", batch=4096, inputs=69, slots=64, ring_envs=16384, arch="dueling"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["step", "step", "rollout", "rollout", "q_rollout", "q_rollout", "forward", "td", "td"])
    if kind == "forward":
        return dict(kind=kind, rows=_log_int(rng, 1, 1 << 20), inputs=rng.choice([32, 37, 53, 69]),
                    arch=rng.choice(["dueling", "paper"]))
    if kind == "td":
        return dict(kind=kind, batch=_log_int(rng, 16, 4096), inputs=rng.choice([32, 37, 53, 69]),
                    slots=rng.choice([32, 64]), ring_envs=_log_int(rng, 64, 8192),
                    arch=rng.choice(["dueling", "paper"]))
    envs = _log_int(rng, 16, {"step": 65536, "rollout": 1024, "q_rollout": 40000}[kind])
    maps = min(envs, rng.choice([1, 16, 32, 64]))
    c = _sim_case("", kind, envs, maps=maps, beams=rng.choice([16, 27, 32, 48, 64]), mixed=rng.random() < 0.3,
                  dr=rng.random() < 0.7, dyn=rng.choice([0, 0, 0, 4]), side=rng.choice([256, 366, 512]))
    if kind == "rollout":
        c["steps"] = _log_int(rng, 32, 1000)
        c["launch"] = rng.choice(["default", "pipe", "pipe-sliced"])
    if kind == "q_rollout":
        c["steps"] = rng.randint(4, 24)
        c["arch"] = rng.choice(["dueling", "paper"])
        c["dyn"] = 0
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs

def _map(rng, side):
    """Border walls, 20 rectangles of 5 to 40 cells, 10 discs of radius 3 to
    15, the areas around start and goal cleared (1 = occupied)."""
    g = np.zeros((side, side), np.uint8)
    for rw, rh, fx, fy in zip(rng.integers(5, 41, 20), rng.integers(5, 41, 20), rng.random(20), rng.random(20)):
        x, y = 1 + int(fx * (side - 2 - rw)), 1 + int(fy * (side - 2 - rh))
        g[y:y + rh, x:x + rw] = 1
    discs = [(int(r), 1 + r + fx * (side - 2 - 2 * r), 1 + r + fy * (side - 2 - 2 * r), 1)
             for r, fx, fy in zip(rng.integers(3, 16, 10), rng.random(10), rng.random(10))]
    for r, x, y, v in discs + [(25, 30.0, 30.0, 0), (25, side - 30.0, side - 30.0, 0)]:
        x0, x1, y0, y1 = max(0, int(x - r) - 1), int(x + r) + 2, max(0, int(y - r) - 1), int(y + r) + 2
        box = g[y0:y1, x0:x1]
        yy = np.arange(y0, y0 + box.shape[0])[:, None] + 0.5 - y
        xx = np.arange(x0, x0 + box.shape[1])[None, :] + 0.5 - x
        box[xx * xx + yy * yy <= r * r] = v
    g[0, :] = g[-1, :] = g[:, 0] = g[:, -1] = 1
    return g


def _sim_inputs(case, seed):
    """Parameters, maps, env -> map, beams per env (host values)."""
    rng = np.random.default_rng([seed, 1])
    p = dict(BASE, n_beams=case["beams"], seed=seed)
    if case["dr"]:
        p.update(RANDOMISED)
    if case["dyn"]:
        p.update(OBSTACLES, n_dyn=case["dyn"])
    n, m = case["envs"], case["maps"]
    sides = rng.choice([128, 256, 366, 512, 1024], m) if case["mixed"] else np.full(m, case["side"])
    if case["mixed"] and case["kind"] != "rollout":
        sides = np.maximum(sides, 256)
    if case["dyn"]:
        sides = np.maximum(sides, 256)
    maps = [_map(rng, int(s)) for s in sides]
    beams = None
    if case["mixed"]:
        beams = rng.choice([b for b in (16, 32, 64) if b <= case["beams"]], n).astype(np.int32)
    return p, maps, (np.arange(n) % m).astype(np.int32), beams


def _start_state(case, p, maps, env_map, seed):
    """A batch of envs in the middle of their episodes: poses uniform over the
    free cells of each map, moving, parameters from their ranges.  f [9, n]
    (x, y, phi, v_l, v_a, dt, K, cap, sigma), u [4, n] (episode step, episode,
    steps since reset, last two actions | delay << 16)."""
    rng = np.random.default_rng([seed, 2])
    n = case["envs"]
    x, y = np.zeros(n), np.zeros(n)
    for m, g in enumerate(maps):
        at = np.flatnonzero(env_map == m)
        free = np.flatnonzero(g == 0)
        cell = free[rng.integers(0, free.size, at.size)]
        x[at], y[at] = cell % g.shape[1], cell // g.shape[1]
    f = np.empty((9, n), np.float32)
    f[0], f[1] = x + rng.uniform(0.1, 0.9, n), y + rng.uniform(0.1, 0.9, n)
    f[2] = rng.uniform(-math.pi, math.pi, n) * 0.999
    f[3], f[4] = rng.uniform(0.0, 18.0, n), rng.uniform(-1.0, 1.0, n)
    for row, k in ((5, "dt"), (6, "k"), (7, "cap"), (8, "sigma")):
        f[row] = rng.uniform(p[k + "_lo"], p[k + "_hi"], n) if p[k + "_hi"] > p[k + "_lo"] else p[k + "_lo"]
    u = np.empty((4, n), np.uint32)
    u[0] = rng.integers(2, p["t_max"], n)
    u[1] = rng.integers(0, 100, n)
    u[2] = u[0]
    u[3] = (rng.integers(0, 5, n) | rng.integers(0, 5, n) << 8
            | rng.integers(p["delay_lo"], p["delay_hi"] + 1, n) << 16)
    d = None
    if case["dyn"]:
        d = np.empty((4 * case["dyn"], n), np.float32)
        w = np.array([g.shape[1] for g in maps])[env_map]
        for o in range(case["dyn"]):
            d[4 * o], d[4 * o + 1] = rng.uniform(10, w - 10), rng.uniform(10, w - 10)
            d[4 * o + 2], d[4 * o + 3] = rng.uniform(-20, 20, n), rng.uniform(-20, 20, n)
    return f, u, d


def _net(arch, n_in, seed):
    """A network's parameters in the library's flat order (float32): uniform
    in +-1/sqrt(fan_in), W1 b1 W2 b2 W3 b3."""
    rng = np.random.default_rng([seed, 3])
    h2, out = (256, 6) if arch == "dueling" else (128, 5)
    parts = []
    for rows, cols in ((256, n_in), (h2, 256), (out, h2)):
        b = 1.0 / math.sqrt(cols)
        parts += [rng.uniform(-b, b, (rows, cols)).astype(np.float32), rng.uniform(-b, b, rows).astype(np.float32)]
    return parts


def _flat(parts):
    return np.concatenate([q.ravel() for q in parts])


def _obs_batch(rows, n_in, seed):
    """Observations as the simulator gives them: normalised ranges (many at
    the limit), then goal frame, heading and velocities."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    o = torch.rand((rows, n_in), generator=gen, device="cuda")
    o[:, :n_in - 5] = (o[:, :n_in - 5] * 1.5).clamp_(max=1.0)
    o[:, n_in - 5:] = o[:, n_in - 5:] * 2.0 - 1.0
    return o


def _ring(case, seed):
    """A full ring's transitions (device tensors s, s2, a, r, term)."""
    cap = case["slots"] * case["ring_envs"]
    s = _obs_batch(cap, case["inputs"], seed)
    s2 = s + 0.05 * (_obs_batch(cap, case["inputs"], seed + 1) - 0.5)
    gen = torch.Generator(device="cuda").manual_seed(seed + 2)
    a = torch.randint(0, 5, (cap,), generator=gen, device="cuda", dtype=torch.uint8)
    t = torch.rand(cap, generator=gen, device="cuda")
    r = torch.rand(cap, generator=gen, device="cuda") * 1.5 - 0.5
    r = torch.where(t < 0.02, torch.full_like(r, -10.0), torch.where(t > 0.995, torch.full_like(r, 75.0), r))
    term = ((t < 0.02) | (t > 0.995)).to(torch.uint8)
    return s, s2, a, r, term


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind, case=case)
    if kind == "forward":
        q = QNet(case["inputs"], 256, 0, arch=case["arch"])
        q.set_params(_flat(_net(case["arch"], case["inputs"], seed)))
        st.update(net=q, obs=_obs_batch(case["rows"], case["inputs"], seed))
        return st
    if kind == "td":
        q = QNet(case["inputs"], case["batch"], 0, arch=case["arch"])
        q.set_params(_flat(_net(case["arch"], case["inputs"], seed)), "online")
        q.set_params(_flat(_net(case["arch"], case["inputs"], seed + 1)), "target")
        ring = Replay(case["slots"], case["ring_envs"], case["inputs"])
        ring.write(0, *[v.cpu().numpy() for v in _ring(case, seed)], steps_recorded=case["slots"])
        st.update(net=q, ring=ring, seed=seed, loss=torch.zeros(1, device="cuda"),
                  grad=torch.zeros(q.n_params, device="cuda"))
        return st
    p, maps, env_map, beams = _sim_inputs(case, seed)
    sim = Sim(p, maps, env_map, beams)
    n, K, D = case["envs"], case["steps"], sim.obs_dim
    sim.reset(seed)
    f, u, d = _start_state(case, p, maps, env_map, seed)
    sim.set_state(f, u, d)
    st.update(sim=sim, obs=sim.new_obs())
    if kind == "step":
        acts = np.random.default_rng([seed, 4]).integers(0, 5, (ACTION_ROWS, n)).astype(np.uint8)
        st.update(acts=torch.from_numpy(acts).cuda(), at=0, rew=torch.empty(n, device="cuda"),
                  done=torch.empty(n, dtype=torch.uint8, device="cuda"))
        return st
    if case["launch"] != "default":
        sim.set_launch(**LAUNCHES[case["launch"]])
    st.update(act_seq=torch.empty((K, n), dtype=torch.uint8, device="cuda"),
              rew_seq=torch.empty((K, n), device="cuda"),
              done_seq=torch.empty((K, n), dtype=torch.uint8, device="cuda"))
    if kind == "rollout":
        st.update(obs_seq=torch.empty((K, n, D), device="cuda"))
    else:
        q = QNet(D, 256, 0, arch=case["arch"])
        q.set_params(_flat(_net(case["arch"], D, seed)))
        eps = torch.linspace(0.01, 0.3, n, device="cuda")
        slots = max(2 * K, min(256, (1 << 21) // n))
        st.update(net=q, eps=eps, ring=Replay(slots, n, D, K))
    return st


def run(st):
    kind = st["kind"]
    if kind == "forward":
        return st["net"].forward(st["obs"])
    if kind == "td":
        st["net"].train_step(st["ring"], st["case"]["batch"], gamma=GAMMA, lr=1e-4, target_every=200, seed=st["seed"],
                             loss=st["loss"], grad=st["grad"])
        return dict(loss=st["loss"], grad=st["grad"])
    sim = st["sim"]
    if kind == "step":
        a = st["acts"][st["at"] % ACTION_ROWS]
        st["at"] += 1
        obs, rew, done = sim.step(a, obs=st["obs"], rew=st["rew"], done=st["done"])
        return dict(obs=obs, rew=rew, done=done)
    seqs = dict(act_seq=st["act_seq"], rew_seq=st["rew_seq"], done_seq=st["done_seq"])
    if kind == "rollout":
        sim.rollout(st["case"]["steps"], obs=st["obs"], obs_seq=st["obs_seq"], **seqs)
        return dict(obs=st["obs"], obs_seq=st["obs_seq"], **seqs)
    sim.rollout(st["case"]["steps"], policy="eps_q", qnet=st["net"], eps=st["eps"], replay=st["ring"], obs=st["obs"],
                **seqs)
    return dict(obs=st["obs"], **seqs)


def _net_flops(arch, n_in):
    h2, out = (256, 6) if arch == "dueling" else (128, 5)
    return 2 * (n_in * 256 + 256 * h2 + h2 * out), n_in * 256 + 256 + 256 * h2 + h2 + h2 * out + out


def work(case):
    kind = case["kind"]
    if kind == "forward":
        fl, params = _net_flops(case["arch"], case["inputs"])
        return {"bytes": 4 * (case["rows"] * (case["inputs"] + 5) + params), "flops": fl * case["rows"]}
    if kind == "td":
        # three forwards, the weight gradients and the hidden layers'
        # backpropagation; parameters, both moments and the gradient once
        fl, params = _net_flops(case["arch"], case["inputs"])
        back = 2 * fl - 2 * case["inputs"] * 256
        return {"bytes": case["batch"] * (8 * case["inputs"] + 6) + 4 * params * (1 + 3 + 3 + 1),
                "flops": case["batch"] * (3 * fl + back)}
    n, K, B = case["envs"], case["steps"], case["beams"]
    D = B + 5
    side = 700 if case["mixed"] else case["side"]
    state = n * (52 + 16 * case["dyn"])
    maps = case["maps"] * side * side // 8
    # a beam's direction, its hit distance and (when randomised) its noise
    flops = n * K * B * (60 if case["dr"] else 30)
    if kind == "step":
        return {"bytes": maps + 2 * state + n * (1 + 4 * D + 5), "flops": flops}
    if kind == "rollout":
        return {"bytes": maps + 2 * state + 4 * n * D + n * K * (4 * D + 6), "flops": flops}
    fl, params = _net_flops(case["arch"], D)
    return {"bytes": maps + 2 * state + 4 * (n * D + params + n) + n * K * (8 * D + 6 + 6), "flops": flops + n * K * fl}


# ------------------------------------------------------- values in 64 bits

def _q64(parts, s):
    """Q-values, hidden activations and head outputs in float64 (torch)."""
    W1, b1, W2, b2, W3, b3 = parts
    z1 = s @ W1.T + b1
    h1 = z1.clamp(min=0)
    z2 = h1 @ W2.T + b2
    h2 = z2.clamp(min=0)
    o = h2 @ W3.T + b3
    return o if o.shape[1] == 5 else o[:, :1] + o[:, 1:] - o[:, 1:].mean(1, keepdim=True)


def _parts64(arch, n_in, seed, grad=False):
    return [torch.from_numpy(q).cuda().double().requires_grad_(grad) for q in _net(arch, n_in, seed)]


_M64 = (1 << 64) - 1


def _mix(z):
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & _M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & _M64
    return z ^ (z >> 31)


def _at(s, c):
    """SplitMix64 of counter c under seed s (Python integers)."""
    return _mix((s + (c + 1) * 0x9E3779B97F4A7C15) & _M64)


def _wrap(v):
    """An unsigned 64-bit constant as the int64 of the same bits."""
    return v - (1 << 64) if v >= 1 << 63 else v


def _shr(z, k):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _at_t(s, c):
    """SplitMix64 over int64 tensors (bit patterns)."""
    z = s + (c + 1) * _wrap(0x9E3779B97F4A7C15)
    z = (z ^ _shr(z, 30)) * _wrap(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _wrap(0x94D049BB133111EB)
    return z ^ _shr(z, 31)


def _u_hi(h):
    return _shr(h, 40).double() * 2.0 ** -24


def _u_mid(h):
    return (_shr(h, 16) & 0xFFFFFF).double() * 2.0 ** -24


class _Step64:
    """One vectorized step without obstacles in float64 (torch)."""

    def __init__(self, case, seed):
        self.p, maps, env_map, beams = _sim_inputs(case, seed)
        dev = "cuda"
        self.n, self.B, self.seed = case["envs"], case["beams"], seed
        self.W = torch.tensor([g.shape[1] for g in maps], device=dev)[torch.from_numpy(env_map).to(dev).long()]
        off = np.cumsum([0] + [g.size for g in maps])
        self.off = torch.tensor(off[:-1], device=dev)[torch.from_numpy(env_map).to(dev).long()]
        self.grid = torch.from_numpy(np.concatenate([g.ravel() for g in maps])).to(dev)
        nb = np.full(self.n, self.B) if beams is None else beams
        self.nb = torch.from_numpy(nb.astype(np.int64)).to(dev)
        f, u, _ = _start_state(case, self.p, maps, env_map, seed)
        self.f = torch.from_numpy(f).to(dev).double()
        self.u = torch.from_numpy(u.astype(np.int64)).to(dev)
        self.env = torch.arange(self.n, device=dev)
        Wd = self.W.double()
        so = self.p["start_offset"]
        self.gx, self.D, self.so = Wd - so, (Wd - 2 * so) * math.sqrt(2.0), so

    def occupied(self, ix, iy):
        """Occupied or outside, for cells [n, m]."""
        W = self.W[:, None]
        out = (ix < 0) | (iy < 0) | (ix >= W) | (iy >= W)
        at = self.off[:, None] + torch.where(out, 0, iy * W + ix)
        return out | (self.grid[at] != 0)

    def scan(self, x, y, phi, sigma, ep, step):
        """Normalised ranges [n, B] and the nearest noise-free range."""
        p, n, B = self.p, self.n, self.B
        j = torch.arange(B, device="cuda").double()[None]
        beta = phi[:, None] + j * (p["fov"] / (self.nb[:, None] - 1).double()) - p["fov"] / 2
        ux, uy = -torch.cos(beta), -torch.sin(beta)
        K = int(math.floor(p["range_max"] / p["march_step"]))
        hit = torch.full((n, B), K + 1, device="cuda")
        for k in range(K, 0, -1):
            t = k * p["march_step"]
            o = self.occupied(torch.floor(x[:, None] + t * ux).long(), torch.floor(y[:, None] + t * uy).long())
            hit = torch.where(o, k, hit)
        r = (hit.double() * p["march_step"]).clamp(max=p["range_max"])
        live = j < self.nb[:, None]
        near = torch.where(live, r, p["range_max"]).amin(1)
        key = _at_t(_at_t(torch.full_like(self.env, _wrap(_at(self.seed, 2))), self.env), (ep << 32) | step)
        h = _at_t(key[:, None], torch.arange(B, device="cuda")[None])
        u1 = (_shr(h, 40) + 1).double() * 2.0 ** -24
        z = torch.sqrt(-2.0 * torch.log(u1)) * torch.cos(2.0 * math.pi * _u_mid(h))
        r = torch.where(sigma[:, None] > 0, (r + sigma[:, None] * z).clamp(0.0, p["range_max"]), r)
        return torch.where(live, r / p["range_max"], 1.0), near

    def extras(self, x, y, phi, vl, va):
        dx, dy = self.gx - x, self.gx - y
        c, s = torch.cos(phi), torch.sin(phi)
        fwd, left = -(dx * c + dy * s), s * dx - c * dy
        alpha = torch.atan2(left, fwd)
        e = torch.stack([fwd / self.D, left / self.D, alpha / math.pi, vl / self.p["v_nom"], va / self.p["w_nom"]], 1)
        return e, alpha, torch.sqrt(dx * dx + dy * dy)

    def step(self, a):
        p = self.p
        x, y, phi, vl, va, dt, K, cap, sigma = self.f
        q0, q1, d = self.u[3] & 255, (self.u[3] >> 8) & 255, self.u[3] >> 16
        ah = torch.where(d == 0, a, torch.where(d == 1, q0, q1))
        table = torch.tensor(ACTIONS, device="cuda", dtype=torch.float64)[ah]
        vl = K * vl + (1 - K) * table[:, 0] * cap
        va = K * va + (1 - K) * table[:, 1] * cap
        x, y = x - dt * vl * torch.cos(phi), y - dt * vl * torch.sin(phi)
        phi = phi + dt * va
        phi = torch.where(phi >= math.pi, phi - 2 * math.pi, torch.where(phi < -math.pi, phi + 2 * math.pi, phi))
        ep, step = self.u[1], self.u[0] + 1
        r = p["robot_radius"]
        m = int(math.ceil(r)) + 1
        o = torch.arange(-m, m + 1, device="cuda")
        ox, oy = o.repeat(o.numel())[None], o.repeat_interleave(o.numel())[None]
        cx, cy = torch.floor(x).long()[:, None] + ox, torch.floor(y).long()[:, None] + oy
        W = self.W[:, None]
        inside = (cx >= 0) & (cy >= 0) & (cx < W) & (cy < W)
        close = (cx + 0.5 - x[:, None]) ** 2 + (cy + 0.5 - y[:, None]) ** 2 <= r * r
        Wd = self.W.double()
        col = (inside & close & self.occupied(cx, cy)).any(1) | (x < 0) | (y < 0) | (x >= Wd) | (y >= Wd)
        e, alpha, d1 = self.extras(x, y, phi, vl, va)
        arrive, trunc = d1 <= p["goal_radius"], step >= p["t_max"]
        obs, near = self.scan(x, y, phi, sigma, ep, step)
        g = self.gx - self.so
        d2 = (g * (y - self.so) - g * (x - self.so)).abs() / self.D
        rew = (0.3 * (1 - d1 / self.D) + 0.1 * (1 - 2 * d2 / self.D) + 0.3 * (vl > 0.5 * p["v_nom"] * cap).double()
               + 0.3 * (1 - alpha.abs() / math.pi) - 0.1 * (near < p["near_dist"]).double())
        rew = torch.where(col, -10.0, torch.where(arrive, 75.0, rew))
        done = col.long() | arrive.long() << 1 | trunc.long() << 2
        obs = torch.cat([obs, e], 1)
        # a new episode for the envs that are done
        pre = _at_t(_at_t(torch.full_like(self.env, _wrap(_at(self.seed, 1))), self.env), ep + 1)
        u = [_u_hi(_at_t(pre, torch.full_like(pre, k))) for k in range(8)]
        J = p["start_jitter"]
        sig = p["sigma_lo"] + u[4] * (p["sigma_hi"] - p["sigma_lo"])
        bx, by = self.so - J + 2 * J * u[5], self.so - J + 2 * J * u[6]
        bphi, zero = -math.pi + 2 * math.pi * u[7], torch.zeros_like(x)
        eb = self.extras(bx, by, bphi, zero, zero)[0]
        ob, _ = self.scan(bx, by, bphi, sig, ep + 1, torch.zeros_like(step))
        obs = torch.where((done != 0)[:, None], torch.cat([ob, eb], 1), obs)
        return dict(obs=obs, rew=rew, done=None)


def exact(case, seed):
    """What ``run`` returns for these inputs, in 64 bits.  Rollouts have no
    such value: where one rounding moves a hit, a collision or a greedy
    action, the trajectory that follows is another one."""
    kind = case["kind"]
    if kind == "forward":
        with torch.no_grad():
            return _q64(_parts64(case["arch"], case["inputs"], seed),
                        _obs_batch(case["rows"], case["inputs"], seed).double())
    if kind == "step" and not case["dyn"]:
        acts = np.random.default_rng([seed, 4]).integers(0, 5, (ACTION_ROWS, case["envs"]))
        return _Step64(case, seed).step(torch.from_numpy(acts[0].astype(np.int64)).cuda())
    if kind == "td":
        s, s2, a, r, term = _ring(case, seed)
        slots, n = case["slots"], case["ring_envs"]
        key = _at(_at(seed, 4), 0)
        at = []
        for i in range(case["batch"]):
            j = _at(_at(key, i), 0) % (slots * n)
            at.append(((slots - 1 - j // n) % slots) * n + j % n)
        at = torch.tensor(at, device="cuda")
        on = _parts64(case["arch"], case["inputs"], seed, grad=True)
        with torch.no_grad():
            pick = _q64(on, s2[at].double()).argmax(1, keepdim=True)
            q2 = _q64(_parts64(case["arch"], case["inputs"], seed + 1), s2[at].double()).gather(1, pick)[:, 0]
            y = r[at].double() + GAMMA * (1.0 - term[at].double()) * q2
        q = _q64(on, s[at].double()).gather(1, a[at].long()[:, None])[:, 0]
        loss = torch.nn.functional.huber_loss(q, y, delta=1.0)
        loss.backward()
        return dict(loss=loss.detach().reshape(1), grad=torch.cat([w.grad.reshape(-1) for w in on]))
    return None
