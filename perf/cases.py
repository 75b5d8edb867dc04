"""The calls a user of the simulator makes, as cases that can be timed and compared.

A case is a dict of plain values; `listed()` names twelve, `draw(rng)` gives more
of the same ranges, `prepare(case, seed)` makes what a program holds before the
call (an environment handle in mid-episode, device buffers, a ring of commands),
`run(state)` is one call through the package's public entry points, and
`exact(case, seed)` restates the same call in 64-bit torch without the package.

Fields of a case: form ("step": one control step per call, "rollout": T steps
per call, "grad": the differentiable rollout with its gradients), envs, swarm
(drones per env, 0: uneven sizes 1..64), K (observed neighbours), T, training
(every scenario type with downwash), contacts (of "grad": "smooth" or
"discrete"), ckpt (steps between checkpoints)."""
import math

import numpy as np
import torch

from paper_2306_09537_gb300.env import QuadSwarmEnv, RolloutFn

PHYS = ("floor", "walls", "motor_noise", "obs_noise", "dr", "auto_reset")
WEIGHTS = {"pos": -1.0, "spin": -0.1, "hit_floor": -1.0, "hit_wall": -1.0, "hit_ceil": -1.0, "hit_quad": -1.0}
SCENARIOS = ("single", "static", "dynamic", "swap", "shrink_expand", "swarm_vs_swarm", "pursuit_lissajous",
             "pursuit_bezier")
UNEVEN = np.array([1, 2, 4, 8, 16, 32, 64])
RING = 16  # command tensors a stepping program cycles through
EPISODE = 1500


def listed():
    def case(name, form, envs, swarm, K, T=1, training=False, contacts="", ckpt=0):
        return {"name": name, "form": form, "envs": envs, "swarm": swarm, "K": K, "T": T, "training": training,
                "contacts": contacts, "ckpt": ckpt}

    return [
        # one drone under a controller or in an evaluation: the smallest call, all launch and latency
        case("step_1x1", "step", 1, 1, 0),
        # a policy's training step on single drones at the usual batch (the headline size)
        case("step_8192x1", "step", 8192, 1, 0),
        # the same on swarms of eight that observe six neighbours
        case("step_2048x8", "step", 2048, 8, 6),
        # large-batch training: the state streams through memory on every call
        case("step_1048576x1", "step", 1 << 20, 1, 0),
        # a horizon of recorded or sampled commands (replay, sampling-based control) at the usual batch
        case("rollout_8192x1_t100", "rollout", 8192, 1, 0, 100),
        # the same at the largest batch: the whole chip computes
        case("rollout_1048576x1_t32", "rollout", 1 << 20, 1, 0, 32),
        # horizons of swarms of eight
        case("rollout_2048x8_t64", "rollout", 2048, 8, 6, 64),
        # every training scenario with downwash, ragged: an odd count of swarms of seven
        case("rollout_training_1999x7_t64", "rollout", 1999, 7, 6, 64, training=True),
        # environments of mixed swarm sizes in one batch (1 to 64 drones each)
        case("rollout_uneven_4096_t32", "rollout", 4096, 0, 6, 32),
        # the largest teams
        case("rollout_256x128_t16", "rollout", 256, 128, 6, 16),
        # trajectory optimisation: loss, gradients of every command and of the initial states
        case("grad_smooth_1024x8_t128", "grad", 1024, 8, 6, 128, contacts="smooth", ckpt=16),
        # the same through the simulator's own contacts on a larger batch and a shorter horizon
        case("grad_contacts_8192x8_t64", "grad", 8192, 8, 6, 64, contacts="discrete", ckpt=16),
    ]


def draw(rng):
    form = rng.choice(["step", "step", "rollout", "rollout", "grad"])
    grad = form == "grad"
    uneven = not grad and rng.random() < 0.2
    swarm = 0 if uneven else rng.choice([1, 1, 1, 2, 3, 5, 6, 8, 8, 8, 11, 16, 24, 32] + ([] if grad else [50, 64, 100, 128]))
    size = 10 if uneven else swarm
    drones = math.exp(rng.uniform(0.0, math.log(1 << 16 if grad else 1 << 20 if size == 1 else 1 << 17)))
    envs = max(1, int(drones / size))
    most = (1 << 22 if grad else 1 << 25) // (envs * size * max(1, size // 4))  # no costlier than the largest listed case
    T = 1 if form == "step" else max(1, min(int(math.exp(rng.uniform(math.log(4), math.log(128)))), most))
    training = not grad and size > 1 and rng.random() < 0.3
    K = 0 if size == 1 else rng.choice([2, 6, 6, 6, 8])
    return {"form": form, "envs": envs, "swarm": swarm, "K": K, "T": T, "training": training,
            "contacts": rng.choice(["smooth", "discrete"]) if grad else "", "ckpt": rng.choice([4, 8, 16, 32]) if grad else 0}


def _sizes(case):
    if case["swarm"]:
        return np.full(case["envs"], case["swarm"], dtype=np.int32)
    p = UNEVEN.astype(np.float64) ** -0.38
    return np.random.RandomState(case["envs"]).choice(UNEVEN, size=case["envs"], p=p / p.sum()).astype(np.int32)


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _inputs(case, seed):
    """States of drones in flight, per-env parameters (+-20%), goals, episode phases, scenario records and commands, float32."""
    dev = _device()
    gen = torch.Generator(device=dev).manual_seed(seed)
    sizes = torch.from_numpy(_sizes(case)).to(dev).long()
    E, D, T = case["envs"], int(sizes.sum()), case["T"]
    env_of = torch.repeat_interleave(torch.arange(E, device=dev), sizes)

    def uniform(*shape, lo=0.0, hi=1.0):
        return lo + (hi - lo) * torch.rand(*shape, generator=gen, device=dev)

    nominal = torch.tensor([0.028, 1.657e-5, 1.666e-5, 2.926e-5, 2.0, 0.04, 0.046], device=dev)
    params = nominal * uniform(E, 7, lo=0.8, hi=1.2)
    goals = torch.stack([uniform(E, lo=-5, hi=5), uniform(E, lo=-5, hi=5), uniform(E, lo=0, hi=10)], 1)
    lo, hi = torch.tensor([-4.9, -4.9, 0.1], device=dev), torch.tensor([4.9, 4.9, 9.9], device=dev)
    if case["swarm"] == 1:
        x = lo + (hi - lo) * uniform(D, 3)
    else:  # a swarm gathers around its goal
        x = torch.minimum(torch.maximum(goals[env_of] + uniform(D, 3, lo=-2.0, hi=2.0), lo), hi)
        x += torch.where((x == lo) | (x == hi), (lo + hi) * 0.5 - x, torch.zeros_like(x)) * uniform(D, 3, hi=0.3)
    q = torch.nn.functional.normalize(torch.randn(D, 4, generator=gen, device=dev), dim=1)
    a, b, c, d = q.unbind(1)
    R = torch.stack([1 - 2 * (c * c + d * d), 2 * (b * c - d * a), 2 * (b * d + c * a), 2 * (b * c + d * a),
                     1 - 2 * (b * b + d * d), 2 * (c * d - b * a), 2 * (b * d - c * a), 2 * (c * d + b * a),
                     1 - 2 * (b * b + c * c)], 1)
    hover = (1.0 / params[:, 4])[env_of, None].expand(D, 4)
    state = torch.cat([x, uniform(D, 3, lo=-1, hi=1), R, uniform(D, 3, lo=-1, hi=1), hover.sqrt(),
                       torch.zeros(D, 4, device=dev), hover], 1).contiguous()
    # episodes in every phase, none ending during the first pass
    phase = torch.randint(0, EPISODE - T, (E,), generator=gen, device=dev, dtype=torch.int32)
    tick = torch.randint(0, 1 << 20, (E,), generator=gen, device=dev, dtype=torch.int32)
    records = None
    if case["training"]:
        kind = torch.randint(0, len(SCENARIOS), (E,), generator=gen, device=dev)
        f = torch.randint(0, 5, (E, 2), generator=gen, device=dev)
        word = torch.randint(0, 1 << 16, (E, 2), generator=gen, device=dev)
        switch = torch.randint(EPISODE // 4, 3 * EPISODE // 4 + 1, (E,), generator=gen, device=dev)
        half = torch.tensor([3.5, 3.5, 3.5], device=dev)
        mid = torch.tensor([0.0, 0.0, 5.0], device=dev)
        chase = (kind == 6)[:, None]
        c0 = mid + torch.where(chase, torch.ones_like(half), half) * uniform(E, 3, lo=-1, hi=1)
        c1 = torch.where(chase, half * uniform(E, 3, lo=0.5, hi=1.0), mid + half * uniform(E, 3, lo=-1, hi=1))
        freq, turn = 0.1 * uniform(E, 3, lo=0.5, hi=1.5) * chase, uniform(E, 3) * chase
        records = torch.cat([kind[:, None], f, switch[:, None], word[:, :1], c0, c1, freq, turn, word[:, 1:]], 1).float().contiguous()
    actions = torch.rand(RING if case["form"] == "step" else T, D, 4, generator=gen, device=dev)
    return {"sizes": sizes, "env_of": env_of, "state": state, "params": params.contiguous(), "goals": goals.contiguous(),
            "phase": phase, "tick": tick, "records": records, "actions": actions}


def prepare(case, seed):
    i = _inputs(case, seed)
    grad = case["form"] == "grad"
    feats = ("dr", "motor_noise") + (("smooth",) if case["contacts"] == "smooth" else ("floor", "walls", "collisions")) if grad \
        else PHYS + (("collisions",) if case["swarm"] != 1 else ()) + (("downwash",) if case["training"] else ())
    env = QuadSwarmEnv(case["envs"], case["swarm"] or _sizes(case), case["K"], feats, seed=seed, weights=WEIGHTS,
                       scenarios=SCENARIOS if case["training"] else ())
    env.set_state(i["state"], i["params"], i["goals"], i["phase"], i["tick"])
    if i["records"] is not None:
        env.set_scenario(i["records"])
    s = {"form": case["form"], "env": env, "actions": i["actions"]}
    if case["form"] == "step":
        s.update(ring=list(i["actions"]), at=0)
    elif case["form"] == "rollout":
        T, dev = case["T"], env.device
        s.update(obs=torch.empty(T, env.D, env.obs_dim, device=dev), reward=torch.empty(T, env.D, device=dev),
                 done=torch.empty(T, env.E, dtype=torch.uint8, device=dev))
    else:
        s.update(actions=i["actions"].requires_grad_(), x0=i["state"].requires_grad_(), ckpt=case["ckpt"])
    return s


def run(state):
    if state["form"] == "step":
        at = state["at"]
        state["at"] = (at + 1) % RING
        obs, reward, done = state["env"].step(state["ring"][at])
        return {"obs": obs, "reward": reward, "done": done}
    if state["form"] == "rollout":
        obs, reward, done = state["env"].rollout(state["actions"], state["obs"], state["reward"], state["done"])
        return {"obs": obs, "reward": reward, "done": done}
    loss = RolloutFn.apply(state["actions"], state["x0"], state["env"], state["ckpt"])
    grad_actions, grad_x0 = torch.autograd.grad(loss.sum(), (state["actions"], state["x0"]))
    return {"loss": loss.detach(), "grad_actions": grad_actions, "grad_x0": grad_x0}


def work(case):
    sizes = _sizes(case).astype(np.float64)
    E, D, T, pairs = len(sizes), sizes.sum(), case["T"], float((sizes * (sizes - 1)).sum())
    obs = 18 + 6 * case["K"]
    state = 2 * D * 30 * 4 + E * (7 + 3 + 2 + 2) * 4  # drones and counters in and out, parameters and goals in
    if case["form"] == "grad":  # commands, initial states and d loss in; loss and gradients out
        return {"bytes": D * 4.0 * (2 * 4 * T + 2 * 30 + 2) + E * 44.0, "flops": 3.0 * T * (1080 * D + 25 * pairs)}
    return {"bytes": state + T * (D * 4.0 * (4 + obs + 1) + E), "flops": T * (1080.0 * D + 25 * pairs)}


# ---------------------------------------------------------------- the same calls in 64 bits
F = np.float32
DT, G, KAPPA, MU = float(F(0.005)), float(F(9.81)), float(F(0.006)), float(F(0.3))
NOISE_DECAY, NOISE_FRAC, HIT_DECAY, OMEGA = float(F(0.9)), float(F(0.02)), float(F(0.8)), 40.0
HIT_V, HIT_W, SEE_X, SEE_V, SEE_W = float(F(0.2)), 0.5, float(F(5e-3)), float(F(1e-2)), float(F(1.75e-4))
ROOM = (5.0, 5.0, 10.0)
DW_K1, DW_K2, DW_B1, DW_H, DW_A, DW_W = float(F(2.4525)), -2.0, 1.0, 0.5, float(F(0.1)), 1.0
MOTOR, OBS, COLL, WALL, DOWNWASH, WAYPOINT, SWAP = 3, 4, 5, 6, 9, 12, 13
SUBSTEPS = 2
WORD = 0xFFFFFFFF


def _philox(c0, c1, c2, seed):
    """Philox4x32-10 (Salmon et al., SC'11) of counters (c0, c1, c2, 0), int64 tensors holding 32-bit words."""
    def mul(m, x):
        p, q = m * (x & 0xFFFF), m * (x >> 16)
        return (q + (p >> 16)) >> 16, (((q & 0xFFFF) << 16) + p) & WORD

    k0, k1 = seed & WORD, seed >> 32
    x0, x1 = torch.broadcast_tensors(c0, c1)
    x2, x3 = torch.full_like(x0, c2), torch.zeros_like(x0)
    for _ in range(10):
        (h0, l0), (h1, l1) = mul(0xD2511F53, x0), mul(0xCD9E8D57, x2)
        x0, x1, x2, x3 = h1 ^ x1 ^ k0, l1, h0 ^ x3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & WORD, (k1 + 0xBB67AE85) & WORD
    return [(2 * (x >> 9) + 1).double() / 2 ** 24 for x in (x0, x1, x2, x3)], x0


def _normals(u, v):
    rho = torch.sqrt(-2 * torch.log(u))
    return [rho * torch.cos(2 * math.pi * v), rho * torch.sin(2 * math.pi * v)]


class _Sim:
    def __init__(self, case, seed, x0=None):
        i = self.i = _inputs(case, seed)
        self.case, self.seed, self.dev = case, seed, _device()
        s = i["state"].double() if x0 is None else x0
        self.x, self.v, self.R, self.w = s[:, 0:3], s[:, 3:6], s[:, 6:15].reshape(-1, 3, 3), s[:, 15:18]
        self.uf, self.eps = s[:, 18:22], s[:, 22:26]
        e = i["env_of"]
        m, ix, iy, iz, t2w, tau, arm = i["params"].double().unbind(1)
        self.m, self.arm, self.inertia = m[e], arm[e], torch.stack([ix, iy, iz], 1)[e]
        self.fmax, self.lag = (0.25 * m * G * t2w)[e, None], -torch.expm1(-DT / tau)[e, None]
        self.noise = (NOISE_FRAC * m * G * 0.25)[e, None]
        self.tick, self.ep = i["tick"].long(), i["phase"].long()
        self.id = torch.arange(len(e), device=self.dev)
        off = torch.cumsum(i["sizes"], 0) - i["sizes"]
        self.groups = [(int(n), off[i["sizes"] == n][:, None] + torch.arange(int(n), device=self.dev))
                       for n in torch.unique(i["sizes"]).tolist()]
        self.goal = i["goals"].double()[e]

    def block(self, tag, sub, blk, of=None):
        ids = self.id if of is None else of
        return _philox(self.tick[self.i["env_of"][ids]], ids, (tag << 16) | (sub << 8) | blk, self.seed)[0]

    def six(self, tag, sub, of):
        a, b = self.block(tag, sub, 0, of), self.block(tag, sub, 1, of)
        return torch.stack(_normals(a[0], a[1]) + _normals(a[2], a[3]) + _normals(b[0], b[1]), 1)

    def physics(self, u, sub):
        """One 200 Hz substep; returns (hit floor, hit wall, hit ceiling)."""
        smooth = self.case["contacts"] == "smooth"
        q = self.block(MOTOR, sub, 0)
        n = torch.stack(_normals(q[0], q[1]) + _normals(q[2], q[3]), 1)
        acc = self.penalty() if smooth else None
        self.uf = self.uf + self.lag * (u - self.uf)
        self.eps = NOISE_DECAY * self.eps + self.noise * n
        f0, f1, f2, f3 = (self.fmax * self.uf ** 2 + self.eps).unbind(1)
        T, sa = f0 + f1 + f2 + f3, self.arm * math.sqrt(0.5)
        torque = torch.stack([sa * (f0 + f1 - f2 - f3), sa * (f1 + f2 - f0 - f3), KAPPA * (f1 + f3 - f0 - f2)], 1)
        thrust, mg = self.R[:, :, 2] * T[:, None], self.m * G
        down = torch.tensor([0.0, 0.0, -G], dtype=torch.float64, device=self.dev)
        a = thrust / self.m[:, None] + down
        v0 = self.v
        if smooth:
            a = a + acc
        else:  # resting on the floor: friction against the thrust at rest or the motion
            flo = (self.x[:, 2] <= 0) & (thrust[:, 2] < mg)
            fric, fxy, vxy = MU * (mg - thrust[:, 2]), thrust[:, :2], v0[:, :2]
            still = (vxy == 0).all(1)
            nf = torch.sqrt(torch.where((fxy == 0).all(1), 1.0, (fxy ** 2).sum(1)))
            held = fxy * torch.where(nf > fric, 1 - fric / nf, torch.zeros_like(nf))[:, None]
            nv = torch.sqrt(torch.where(still, 1.0, (vxy ** 2).sum(1)))
            fxy = torch.where(still[:, None], held, fxy - (fric / nv)[:, None] * vxy)
            rest = torch.cat([fxy / self.m[:, None], torch.zeros_like(a[:, :1])], 1)
            a = torch.where(flo[:, None], rest, a)
            v0 = torch.where(flo[:, None], torch.cat([v0[:, :2], torch.zeros_like(v0[:, :1])], 1), v0)
        wdot = (torque - torch.linalg.cross(self.w, self.inertia * self.w)) / self.inertia
        v = v0 + DT * a
        if not smooth:
            stop = flo & ~still & ((v[:, :2] * v0[:, :2]).sum(1) < 0)
            v = torch.where(stop[:, None], torch.cat([torch.zeros_like(v[:, :2]), v[:, 2:]], 1), v)
        x = self.x + DT * v
        w = torch.clamp(self.w + DT * wdot, -OMEGA, OMEGA)
        # R <- polar factor of R (I + dt [w]x): the rotation about w by atan(dt |w|), re-orthonormalised
        c = torch.rsqrt(1 + DT * DT * (w * w).sum(1))[:, None, None]
        z = torch.zeros_like(w[:, 0])
        W = torch.stack([z, -w[:, 2], w[:, 1], w[:, 2], z, -w[:, 0], -w[:, 1], w[:, 0], z], 1).reshape(-1, 3, 3)
        RW = self.R @ W
        M = self.R + DT * c * RW + (DT * c) ** 2 / (1 + c) * (RW @ W)
        R = 1.5 * M - 0.5 * M @ (M.transpose(1, 2) @ M)
        if smooth:
            self.x, self.v, self.w, self.R = x, v, w, R
            return None
        hit = (x[:, 2] <= 0) & (v[:, 2] < 0)
        keep = torch.tensor([1.0, 1.0, 0.0], dtype=torch.float64, device=self.dev)
        x, v, w = torch.where(hit[:, None], x * keep, x), torch.where(hit[:, None], 0.0, v), torch.where(hit[:, None], 0.0, w)
        heading = torch.where(hit[:, None], R[:, :2, 0], torch.tensor([1.0, 0.0], dtype=torch.float64, device=self.dev))
        heading = heading / torch.sqrt((heading ** 2).sum(1, keepdim=True))
        cs, sn, one = heading[:, 0], heading[:, 1], torch.ones_like(z)
        up = torch.stack([cs, -sn, z, sn, cs, z, z, z, one], 1).reshape(-1, 3, 3)
        R = torch.where(hit[:, None, None], up, R)
        lim = torch.tensor(ROOM, dtype=torch.float64, device=self.dev)
        over, under = x > lim, (x < -lim) & torch.tensor([True, True, False], device=self.dev)
        out = (over & (v > 0)) | (under & (v < 0))
        x, v = torch.where(over, lim, torch.where(under, -lim, x)), torch.where(out, 0.0, v)
        at = out.any(1).nonzero()[:, 0]
        if len(at):
            n = self.six(WALL, sub, at)
            v, w = v.index_put((at,), HIT_DECAY * (v[at] + HIT_V * n[:, :3])), w.index_put((at,), w[at] + HIT_W * n[:, 3:])
        self.x, self.v, self.w, self.R = x, v, w, R
        return hit, out[:, :2].any(1), out[:, 2]

    def penalty(self):
        """Softplus penalties of floor, walls, ceiling and pairs."""
        def sp(p):
            return torch.nn.functional.softplus(p, beta=200.0, threshold=60.0)
        k, x = 20.0 * G, self.x
        lim = torch.tensor(ROOM, dtype=torch.float64, device=self.dev)
        low = torch.tensor([-5.0, -5.0, 0.0], dtype=torch.float64, device=self.dev)
        acc = k * (sp(low - x) - sp(x - lim))
        for n, ix in self.groups:
            if n > 1:
                r = x[ix][:, :, None] - x[ix][:, None]
                own = torch.eye(n, dtype=torch.bool, device=self.dev)
                d = torch.sqrt((r * r).sum(-1) + own)
                psi = torch.where(own, torch.zeros_like(d), k * sp(2 * self.arm[ix][:, :, None] - d) / d)
                acc = acc.index_put((ix.reshape(-1),), (psi[..., None] * r).sum(2).reshape(-1, 3), accumulate=True)
        return acc

    def pairs(self):
        """Collisions and downwash of every env; returns the drones that hit another."""
        hit_any = torch.zeros(len(self.id), dtype=torch.bool, device=self.dev)
        x, v = self.x, self.v
        for n, ix in self.groups:
            if n == 1:
                continue
            flat = ix.reshape(-1)
            r = x[ix][:, None] - x[ix][:, :, None]  # [env, i, j] = x_j - x_i
            own = torch.eye(n, dtype=torch.bool, device=self.dev)
            key, thr = (r * r).sum(-1), (2 * self.arm[ix][:, :, None]) ** 2
            hit = (key < thr) & ~own
            hit_any[flat] = hit.any(2).reshape(-1)
            rv = v[ix][:, None] - v[ix][:, :, None]  # v_j - v_i
            act = hit & ((rv * r).sum(-1) < 0)
            nrm = -r / torch.sqrt(key + own)[..., None]
            dv = torch.where(act[..., None], (rv * nrm).sum(-1, keepdim=True) * nrm, torch.zeros_like(r)).sum(2).reshape(-1, 3)
            at = act.any(2).reshape(-1).nonzero()[:, 0]
            if len(at):
                d = flat[at]
                k = self.six(COLL, 0, d)
                self.v = self.v.index_put((d,), HIT_DECAY * (self.v[d] + dv[at] + HIT_V * k[:, :3]))
                self.w = self.w.index_put((d,), self.w[d] + HIT_W * k[:, 3:])
            if self.case["training"]:
                dz = r[..., 2]
                above = ((r[..., :2] ** 2).sum(-1) < thr) & (dz > 0) & (dz < DW_H) & ~own
                az = -(torch.where(above, DW_K1 * (DW_K2 * dz + DW_B1), torch.zeros_like(dz))).sum(2).reshape(-1)
                at = above.any(2).reshape(-1).nonzero()[:, 0]
                if len(at):
                    d, T = flat[at], SUBSTEPS * DT
                    k = self.six(DOWNWASH, 0, d)
                    push = DW_A * k[:, :3] + torch.stack([torch.zeros_like(az[at])] * 2 + [az[at]], 1)
                    self.v = self.v.index_put((d,), self.v[d] + T * push)
                    self.w = self.w.index_put((d,), self.w[d] + T * DW_W * k[:, 3:])
        return hit_any

    def neighbours(self):
        """[D, 6 K]: relative position and velocity of the K nearest, ties to the lower index, zeros where there is none."""
        K = self.case["K"]
        out = torch.zeros(len(self.id), K, 6, dtype=torch.float64, device=self.dev)
        for n, ix in self.groups:
            k = min(K, n - 1)
            if k == 0:
                continue
            x32 = self.x[ix].float()
            key = ((x32[:, None] - x32[:, :, None]) ** 2).sum(-1)
            key = key.masked_fill(torch.eye(n, dtype=torch.bool, device=self.dev), math.inf)
            near = key.sort(dim=2, stable=True).indices[:, :, :k]  # [env, i, k]
            s = torch.cat([self.x, self.v], 1)[ix]
            pick = torch.gather(s[:, None].expand(-1, n, -1, -1), 2, near[..., None].expand(-1, -1, -1, 6))
            out[ix.reshape(-1), :k] = (pick - s[:, :, None]).reshape(-1, k, 6)
        return out.flatten(1)

    def step(self, action):
        """One control step: (observation, reward)."""
        f = torch.clamp(action.double(), 0, 1)
        ground, wall, ceil = (torch.zeros(len(self.id), dtype=torch.bool, device=self.dev) for _ in range(3))
        for sub in range(SUBSTEPS):
            h, s, c = self.physics(torch.sqrt(f), sub)
            ground, wall, ceil = ground | h, wall | s, ceil | c
        quad = self.pairs()
        goal = self.goals(self.ep + 1) if self.case["training"] else self.goal
        a, b, c = (self.block(OBS, 0, k) for k in range(3))
        u = [2 * t - 1 for t in a + b[:2]]
        see = torch.stack(u[:3], 1) * SEE_X, torch.stack(u[3:6], 1) * SEE_V, \
            torch.stack(_normals(b[2], b[3]) + _normals(c[0], c[1])[:1], 1) * SEE_W
        obs = torch.cat([self.x - goal + see[0], self.v + see[1], self.R.reshape(-1, 9), self.w + see[2], self.neighbours()], 1)
        reward = -(self.x - goal).norm(dim=1) - float(F(0.1)) * self.w.norm(dim=1)
        reward = reward - ground.double() - wall.double() - ceil.double() - quad.double()
        self.tick, self.ep = self.tick + 1, self.ep + 1
        return obs, reward

    def goals(self, tau):
        """Every drone's goal at control step tau [E] of its episode (the eight scenario types)."""
        out = self.goal.clone()
        rec = self.i["records"].double()
        word = rec[:, 4].long() | (rec[:, 17].long() << 16)
        for n, ix in self.groups:
            e = self.i["env_of"][ix[:, 0]]
            r, t, seed, i = rec[e], tau[e].double(), word[e], torch.arange(n, device=self.dev)
            kind, late, c0, c1 = r[:, 0].long(), tau[e] >= r[:, 3].long(), r[:, 5:8], r[:, 8:11]
            g = self.goal[ix].clone()

            def place(form, k, of):  # offsets of slots k [env, i] in formations form [env]
                every = torch.stack([_formation(q, k, of) for q in range(5)])
                return every[form, torch.arange(len(e), device=self.dev)]

            plain = i.expand(len(e), n)
            first, second = place(r[:, 1].long(), plain, n), place(r[:, 2].long(), plain, n)
            lat, c0e, c1e = late[:, None, None], c0[:, None], c1[:, None]
            scale = 1 - 0.5 * (1 - torch.cos(2 * math.pi * t / 400)) / 2
            keys = _philox(seed[:, None], i[None], SWAP << 16, self.seed)[1]
            before = (keys[:, None] < keys[:, :, None]) | ((keys[:, None] == keys[:, :, None]) & (i[None] < i[:, None]))
            swapped = place(r[:, 1].long(), before.sum(2), n)
            n0 = (n + 1) // 2
            team = (i >= n0).long()
            form = torch.where(late, r[:, 2].long(), r[:, 1].long())
            versus = torch.cat([place(form, plain[:, :n0], n0)] + ([place(form, plain[:, n0:] - n0, n - n0)] if n > n0 else []), 1)
            side = (team[None] ^ late[:, None].long())[..., None] == 1
            p = r[:, 11:14] * (SUBSTEPS * DT) * t[:, None] + r[:, 14:17]
            liss = (c1 * torch.sin(2 * math.pi * p) + c0)[:, None]
            seg = tau[e] // 300
            s = ((tau[e] - 300 * seg).double() / 300)[:, None]
            box = torch.tensor([3.5, 3.5, 7.0], dtype=torch.float64, device=self.dev)
            wp = []
            for j in range(-1, 3):
                q = torch.stack(_philox(seed, seg + j + 1, WAYPOINT << 16, self.seed)[0][:3], 1)
                wp.append(torch.cat([2 * box[:2] * q[:, :2] - box[:2], box[2] * q[:, 2:] + 1.5], 1))
            p1, p2 = wp[1] + (wp[2] - wp[0]) / 6, wp[2] - (wp[3] - wp[1]) / 6
            bez = ((1 - s) ** 3 * wp[1] + 3 * (1 - s) ** 2 * s * p1 + 3 * (1 - s) * s ** 2 * p2 + s ** 3 * wp[2])[:, None]
            choices = [g, c0e + first, torch.where(lat, c1e + second, c0e + first), c0e + torch.where(lat, swapped, first),
                       c0e + scale[:, None, None] * first, torch.where(side, c1e, c0e) + versus, liss.expand_as(g), bez.expand_as(g)]
            out[ix.reshape(-1)] = torch.stack(choices)[kind, torch.arange(len(e), device=self.dev)].reshape(-1, 3)
        return out


def _formation(form, k, n):
    """Offsets from the centre of goal slots k of n goals half a metre apart: circle, grid, sphere, cylinder, cube."""
    s, k, z = 0.5, k, torch.zeros_like(k, dtype=torch.float64)

    def root(p):
        m = 1
        while m ** p < n:
            m += 1
        return m

    def ring(at, of):
        r, a = min(s * of / (2 * math.pi), 4.0), 2 * math.pi * at.double() / of
        return r * torch.cos(a), r * torch.sin(a)

    if form == 0:
        return torch.stack([*ring(k, n), z], -1)
    if form == 1:
        m = root(2)
        return torch.stack([s * ((k % m) - 0.5 * (m - 1)), s * ((k // m) - 0.5 * (-(-n // m) - 1)), z], -1)
    if form == 2:
        r, a = s * math.sqrt(n / (4 * math.pi)), (2 * k + 1).double() / n
        turn = ((k * math.floor(2 ** 32 * (3 - math.sqrt(5)) / 2)) & WORD).double() / 2 ** 32 * 2 * math.pi
        rho = torch.sqrt(a * (2 - a))
        return torch.stack([r * rho * torch.cos(turn), r * rho * torch.sin(turn), r * (1 - a)], -1)
    if form == 3:
        L = 1
        while 4 * L * L < n:
            L += 1
        m = -(-n // L)
        return torch.stack([*ring(k % m, m), s * ((k // m) - 0.5 * (-(-n // m) - 1))], -1)
    m = root(3)
    return torch.stack([s * ((k % m) - 0.5 * (m - 1)), s * ((k // m) % m - 0.5 * (m - 1)),
                        s * ((k // (m * m)) - 0.5 * (-(-n // (m * m)) - 1))], -1)


def exact(case, seed):
    if case["form"] != "grad":
        sim, obs, reward = _Sim(case, seed), [], []
        for t in range(case["T"]):
            o, r = sim.step(sim.i["actions"][t])
            obs.append(o)
            reward.append(r)
        if case["form"] == "step":
            return {"obs": obs[0], "reward": reward[0], "done": None}
        return {"obs": torch.stack(obs), "reward": torch.stack(reward), "done": None}
    i = _inputs(case, seed)
    x0, actions = i["state"].double().requires_grad_(), i["actions"].double().requires_grad_()
    with torch.enable_grad():
        sim = _Sim(case, seed, x0)
        loss = torch.zeros(len(sim.id), dtype=torch.float64, device=sim.dev)
        for t in range(case["T"]):
            f = torch.clamp(actions[t], 0, 1)
            for sub in range(SUBSTEPS):
                sim.physics(torch.sqrt(f), sub)
            if case["contacts"] == "discrete":
                sim.pairs()
            loss = loss + ((sim.x - sim.goal) ** 2).sum(1) + float(F(1e-3)) * (f * f).sum(1)
            sim.tick = sim.tick + 1
        grad_actions, grad_x0 = torch.autograd.grad(loss.sum(), (actions, x0), materialize_grads=True)
    return {"loss": loss.detach(), "grad_actions": grad_actions, "grad_x0": grad_x0}
