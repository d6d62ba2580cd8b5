"""Performance cases of the roll-out engine: what a user has it do, through its public entry points.

Each case is one of four kinds of call:

  forward   ws_policy_forward_noalloc on a batch of observations
  rollout   ws_reset, ws_rollout and the post-passes (returns; forces on the landscape), the records fetched
            into the trainer's device tensors
  train     one training iteration: weights in, roll-out, A2C update or PPO epochs, weights out
  serve     one client's request through the server: submit, wait for each chunk, read it, acknowledge it

The environments are the control env (and the acrobot, its sibling), the economy with uneven agent counts and the
Gaussian-sum landscape; paths are the batched FP32 path and the BF16 tensor-core path.
"""
import math

import numpy as np
import torch

from paper_2408_00930_gb300 import warpsci as W

ENV = {"control": W.WS_ENV_CONTROL, "economy": W.WS_ENV_ECONOMY, "landscape": W.WS_ENV_LANDSCAPE,
       "acrobot": W.WS_ENV_ACROBOT}
PATH = {"fp32": W.WS_PATH_BATCHED_FP32, "bf16": W.WS_PATH_BATCHED_BF16}
EPISODE = {"control": 200, "economy": 540, "landscape": 1000, "acrobot": 500}
GAMMA, SIGMA, CLIP = 0.99, 0.05, 0.1
LR, EPS, C_V, C_E = 0.05, 0.2, 0.5, 0.01
KEEP_K = 2 ** 64 - 1


def listed():
    return [
        # a few agents' policy step inside another program's captured graph: the smallest call
        dict(name="forward_small", kind="forward", rows=300, inp=16, h0=128, h1=128, out=20),
        # the largest batch the allocation-free forward takes at the 256-unit policy
        dict(name="forward_large", kind="forward", rows=8192, inp=4, h0=256, h1=256, out=2),
        # the small control workload: 1,000 envs, horizon 200, all in FP32; launch-bound
        dict(name="control_small_fp32", kind="rollout", env="control", path="fp32", envs=1000, steps=200, hidden=64),
        # the same workload on the BF16 path as a trainer client sees it, chunk by chunk from the server
        dict(name="serve_small_bf16", kind="serve", env="control", path="bf16", envs=1000, steps=200, hidden=64),
        # the control workload at scale on the tensor cores: two chunks of 50 steps and their returns
        dict(name="control_large_bf16", kind="rollout", env="control", path="bf16", envs=131072, steps=100, hidden=256),
        # the same envs and policy in full FP32
        dict(name="control_large_fp32", kind="rollout", env="control", path="fp32", envs=131072, steps=10, hidden=256),
        # one chunk of the multi-agent economy: 8 to 256 agents per env and a planner
        dict(name="economy_bf16", kind="rollout", env="economy", path="bf16", envs=2048, steps=50, hidden=128),
        # one chunk of the reaction landscape and the forces of its transitions, on the tensor cores
        dict(name="landscape_bf16", kind="rollout", env="landscape", path="bf16", envs=8192, steps=50, hidden=256,
             dim=24, gauss=4096),
        # the landscape in full FP32 (the reference path of the energy), with forces
        dict(name="landscape_fp32", kind="rollout", env="landscape", path="fp32", envs=8192, steps=4, hidden=256,
             dim=24, gauss=4096),
        # one actor-critic iteration on a chunk of the control workload at scale (6.55 M rows)
        dict(name="train_a2c_bf16", kind="train", algo="a2c", env="control", path="bf16", envs=131072, steps=50,
             hidden=256),
        # one PPO iteration of the small control workload in FP32: 200,000 rows, two epochs
        dict(name="train_ppo_fp32", kind="train", algo="ppo", env="control", path="fp32", envs=1000, steps=200,
             hidden=64),
        # one PPO iteration of the economy: agents' and planner's pairs, uneven envs
        dict(name="train_ppo_economy", kind="train", algo="ppo", env="economy", path="bf16", envs=2048, steps=8,
             hidden=128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "rollout", "rollout", "rollout", "train", "train", "serve"])
    if kind == "forward":
        c = dict(kind=kind, inp=rng.choice([4, 6, 16, 24]), out=rng.choice([2, 3, 10, 20, 48]))
        c["h0"], c["h1"] = rng.choice([32, 64, 100, 128, 256]), rng.choice([32, 64, 100, 128, 256])
        c["rows"] = _log(rng, 1, (1 << 22) // (c["h0"] + c["h1"]))
        return c
    path = rng.choice(["fp32", "bf16"])
    if kind == "serve":
        return dict(kind=kind, env="control", path=path, envs=_log(rng, 256, 16384), steps=rng.choice([100, 130, 150, 200]),
                    hidden=rng.choice([64, 128] if path == "fp32" else [64, 128, 256]))
    env = rng.choice(["control", "control", "acrobot", "economy", "landscape", "landscape"])
    c = dict(kind=kind, env=env, path=path)
    fp32 = path == "fp32"
    if env in ("control", "acrobot"):
        c["envs"] = _log(rng, 256, 131072)
        c["hidden"] = rng.choice([64, 100, 128, 256] if fp32 else [64, 128, 256])
        c["steps"] = rng.randint(5, 20 if fp32 else 100)
    elif env == "economy":
        c["envs"] = _log(rng, 64, 2048)
        c["hidden"] = 128
        c["steps"] = rng.randint(2, 8 if fp32 else 50)
    else:
        c["envs"] = _log(rng, 256, 8192)
        c["hidden"] = 256 if not fp32 else rng.choice([64, 100, 256])
        c["dim"] = rng.choice([8, 16, 24])
        c["gauss"] = rng.choice([256, 1000, 1024, 4096]) if fp32 else rng.choice([256, 1024, 4096])
        c["steps"] = rng.randint(2, 5 if fp32 else 50)
    if kind == "train":
        c["algo"] = rng.choice(["a2c", "ppo"])
        c["steps"] = min(c["steps"], 16 if env in ("control", "acrobot") else 4 if env == "economy" else 8)
    return c


# ---- shapes -----------------------------------------------------------------------------------------------
def _io(c):
    """Observation width, action width (words), policy output width."""
    d = c.get("dim", 0)
    return {"control": (4, 1, 2), "acrobot": (6, 1, 3), "economy": (16, 1, 20), "landscape": (d, d, 2 * d)}[c["env"]]


def _agents(c, seed=None):
    """Agents per env, U{8..256} by the case; a seed only reorders them, so that every seed has the same slots."""
    a = np.random.default_rng(c["envs"]).integers(8, 257, c["envs"]).astype(np.int32)
    return a if seed is None else np.random.default_rng(seed).permutation(a)


def _slots(c):
    return int(_agents(c).sum()) + c["envs"] if c["env"] == "economy" else c["envs"]


def _params(widths):
    return sum(a * b + b for a, b in zip(widths, widths[1:]))


def _nets(c):
    """(widths, rows per step) of each policy."""
    obs, _, out = _io(c)
    h = c["hidden"]
    if c["env"] == "economy":
        return [((16, h, h, 20), _slots(c) - c["envs"]), ((16, h, h, 10), c["envs"])]
    return [((obs, h, h, out), c["envs"])]


def _fields(c):
    """Records a trainer reads: (field, shape of a step, type)."""
    obs, act, _ = _io(c)
    s = _slots(c)
    f = [("obs", W.WS_F_OBS, (obs, s), torch.float32),
         ("action", W.WS_F_ACTION, (act, s) if c["env"] == "landscape" else (s,),
          torch.float32 if c["env"] == "landscape" else torch.int32),
         ("logp", W.WS_F_LOGP, (s,), torch.float32),
         ("reward", W.WS_F_REWARD, (s,), torch.float32),
         ("done", W.WS_F_DONE, (s,), torch.uint8)]
    if c["env"] == "economy":
        f.append(("wealth", W.WS_F_WEALTH, (s,), torch.int64))
    if c["env"] == "landscape":
        f.append(("energy", W.WS_F_ENERGY, (s,), torch.float32))
    if c["kind"] == "rollout":
        f.append(("return", W.WS_F_RETURN, (s,), torch.float32))
        if c["env"] == "landscape":
            f.append(("force", W.WS_F_FORCE, (act, s), torch.float32))
    return f


def _bytes(t):
    return t.numel() * t.element_size()


# ---- the calls --------------------------------------------------------------------------------------------
def prepare(case, seed):
    c = case
    if c["kind"] == "forward":
        g = torch.Generator(device="cuda").manual_seed(seed)
        widths = (c["inp"], c["h0"], c["h1"], c["out"])
        parts = []
        for a, b in zip(widths, widths[1:]):
            k = 1 / math.sqrt(a)
            parts.append((torch.rand(a * b + b, device="cuda", generator=g) * 2 - 1) * k)
        obs = torch.randn(c["rows"], c["inp"], device="cuda", generator=g)
        out = torch.empty(c["rows"], c["out"], device="cuda")
        return dict(case=c, obs=obs, params=torch.cat(parts), out=out)
    if c["kind"] == "serve":
        q, keep = W.make_request(ENV[c["env"]], PATH[c["path"]], c["envs"], c["steps"], 50, EPISODE[c["env"]],
                                 c["hidden"], c["hidden"], seed=seed % (1 << 30) + 1)
        # room for the request's state, its FP32 scratch and its ring of two chunks
        budget = (64 << 20) + c["envs"] * (100 * 40 + 8 * c["hidden"] + 512)
        chunks = [min(50, c["steps"] - t) for t in range(0, c["steps"], 50)]
        np_type = {torch.float32: np.float32, torch.int32: np.int32, torch.uint8: np.uint8}
        out = [{n: np.empty((t,) + shape, np_type[dt]) for n, _, shape, dt in _fields(c)} for t in chunks]
        return dict(case=c, request=q, keep=keep, server=W.Server(budget), out=out)
    kw = dict(param_seed=seed % (1 << 30) + 1, gamma=GAMMA)
    if c["env"] == "economy":
        kw["agents_per_env"] = _agents(c, seed)
    if c["env"] == "landscape":
        kw.update(dim=c["dim"], n_gauss=c["gauss"], noise_sigma=SIGMA, step_clip=CLIP)
        if c["kind"] == "rollout":
            kw["flags"] = W.WS_FLAG_FORCE
    if c["kind"] == "train":
        kw["flags"] = W.WS_FLAG_TRAIN
    r = W.Rollout(ENV[c["env"]], PATH[c["path"]], c["envs"], c["steps"], EPISODE[c["env"]], c["hidden"], c["hidden"],
                  **kw)
    s = dict(case=c, rollout=r, seed=seed % (1 << 30) + 7)
    if c["kind"] == "rollout":
        s["out"] = {n: (f, torch.empty((c["steps"],) + shape, dtype=dt, device="cuda"))
                    for n, f, shape, dt in _fields(c)}
    else:
        sizes = {"params": sum(_params(w) for w, _ in _nets(c)),
                 "critic": sum(_params(w[:3] + (1,)) for w, _ in _nets(c))}
        field = {"params": W.WS_F_PARAMS, "critic": W.WS_F_CRITIC}
        for n, size in sizes.items():
            start = torch.from_numpy(r.fetch_raw(field[n], 4 * size).view(np.float32).copy()).cuda()
            s[n] = (field[n], start, torch.empty_like(start))
        s["ret"] = torch.empty(c["steps"], _slots(c), device="cuda")
    return s


def _ok(status, where):
    if status != W.WS_OK:
        raise W.WarpSciError(status, where)


def run(state):
    c = state["case"]
    if c["kind"] == "forward":
        _ok(W.ws_policy_forward_noalloc(state["obs"].data_ptr(), c["rows"], state["params"].data_ptr(), c["inp"],
                                        c["h0"], c["h1"], c["out"], state["out"].data_ptr(),
                                        torch.cuda.current_stream().cuda_stream), "ws_policy_forward_noalloc")
        return state["out"]
    if c["kind"] == "serve":
        s = state["server"]
        status, rid = s.submit(state["request"])
        _ok(status, "ws_server_submit")
        for k, out in enumerate(state["out"]):
            _ok(s.wait_chunk(rid, k), "ws_server_wait_chunk")
            for name, field, _, _ in _fields(c):
                _ok(s.fetch(rid, field, k, out[name]), "ws_server_fetch")
            _ok(s.ack(rid, k), "ws_server_ack")
        _ok(s.release(rid), "ws_server_release")
        return state["out"]
    r, n = state["rollout"], c["steps"]
    if c["kind"] == "rollout":
        r.reset(state["seed"])
        r.rollout(n)
        r.returns(n)
        if c["env"] == "landscape":
            r.forces(n)
        for field, dst in state["out"].values():
            r.fetch_device(field, 0, n, dst)
        return {name: dst for name, (_, dst) in state["out"].items()}
    for name in ("params", "critic"):
        field, start, _ = state[name]
        r._ok(W.ws_load(r.ctx, field, start.data_ptr(), _bytes(start), 1, KEEP_K), "ws_load")
    r.reset(state["seed"])
    r.rollout(n)
    if c["algo"] == "a2c":
        r._ok(W.ws_a2c_update(r.ctx, n, LR, C_V, C_E), "ws_a2c_update")
    else:
        r.advantages(n)
        for _ in range(2):
            r._ok(W.ws_ppo_update(r.ctx, n, LR, EPS, C_V, C_E), "ws_ppo_update")
    r.fetch_device(W.WS_F_RETURN, 0, n, state["ret"])
    out = {"return": state["ret"]}
    for name in ("params", "critic"):
        field, _, end = state[name]
        r.fetch_device(field, 0, 0, end)
        out[name] = end
    return out


# ---- what a pass cannot do without ------------------------------------------------------------------------
def work(case):
    c = case
    mlp = lambda w: 2 * sum(a * b for a, b in zip(w, w[1:]))  # noqa: E731
    if c["kind"] == "forward":
        w = (c["inp"], c["h0"], c["h1"], c["out"])
        return {"bytes": 4 * (c["rows"] * (c["inp"] + c["out"]) + _params(w)), "flops": c["rows"] * mlp(w)}
    size = {torch.float32: 4, torch.int32: 4, torch.uint8: 1, torch.int64: 8}
    record = sum(size[t] * int(np.prod(shape)) for _, _, shape, t in _fields(c))
    t, nets = c["steps"], _nets(c)
    flops = t * sum(rows * mlp(w) for w, rows in nets)
    if c["env"] == "landscape":  # distance, exponent and sum of every env-Gaussian pair; the force's sum with it
        per = 3 * c["dim"] + 4 + (3 * c["dim"] + 4 + 2 * c["dim"] if c["kind"] == "rollout" else 0)
        flops += t * c["envs"] * c["gauss"] * per
    weights = 4 * sum(_params(w) for w, _ in nets)
    if c["kind"] == "train":
        epochs = 1 if c["algo"] == "a2c" else 2
        both = sum(rows * (mlp(w) + mlp(w[:3] + (1,))) for w, rows in nets)
        flops += t * both * 3 * epochs
        weights *= 4 * epochs
        record += epochs * 4 * (sum(_io(c)[:2]) + 3) * _slots(c)  # each epoch reads the rows it learns from
    return {"bytes": t * record + weights, "flops": flops}


# ---- the same in 64 bits ------------------------------------------------------------------------------------
def _u32(x):
    return x & 0xFFFFFFFF


def _philox(seed, c0, c1, c2, c3):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors that hold 32-bit words."""
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        a, b = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = _u32(b >> 32) ^ c1 ^ k0, _u32(b), _u32(a >> 32) ^ c3 ^ k1, _u32(a)
        k0, k1 = _u32(k0 + 0x9E3779B9), _u32(k1 + 0xBB67AE85)
    return c0, c1, c2, c3


def _draw(seed, c0, env, agent, tag, sub=0):
    i = torch.arange(1, device="cuda")
    z = torch.zeros(torch.broadcast_shapes(*(torch.as_tensor(v).shape for v in (c0, env, agent, sub))),
                    dtype=torch.int64, device="cuda") + i[0]
    return _philox(seed, z + c0, z + env, z + agent, z + (tag << 24) + sub)


def _u01(w):
    return (w >> 8).double() * 2.0 ** -24


def _between(w, lo, hi):
    """U(lo, hi) as one FP32 multiply-add, which 64 bits hold exactly before the one rounding."""
    lo, hi = np.float32(lo), np.float32(hi)
    return (float(np.float32(hi - lo)) * _u01(w) + float(lo)).float().double()


def _normals(w):
    a, b, c, d = w
    rad = lambda u: torch.sqrt(-2 * torch.log(((u >> 8) + 1).double() * 2.0 ** -24))  # noqa: E731
    return (rad(a) * torch.cos(2 * math.pi * _u01(b)), rad(a) * torch.sin(2 * math.pi * _u01(b)),
            rad(c) * torch.cos(2 * math.pi * _u01(d)), rad(c) * torch.sin(2 * math.pi * _u01(d)))


def _init_net(seed, widths, pid):
    layers = []
    for l, (a, b) in enumerate(zip(widths, widths[1:])):
        n = a * b + b
        bound = float(np.float32(1) / np.sqrt(np.float32(a)))
        w = _draw(seed, torch.arange(-(-n // 4), device="cuda"), l, pid, 4)
        v = _between(torch.stack(w, 1).reshape(-1)[:n], -bound, bound)
        layers.append((v[:a * b].view(a, b).clone(), v[a * b:].clone()))
    return layers


def _mlp(net, x):
    for w, b in net[:-1]:
        x = torch.tanh(x @ w + b)
    return x @ net[-1][0] + net[-1][1]


def _flat(net):
    return torch.cat([t.reshape(-1) for layer in net for t in layer])


def _control(c, pseed, rseed):
    """The control env's records in 64 bits: lists over steps of obs, action, logp, done."""
    n, net = c["envs"], _init_net(pseed, (4, c["hidden"], c["hidden"], 2), 0)
    env = torch.arange(n, device="cuda")
    start = lambda k: torch.stack([_between(w, -0.05, 0.05) for w in _draw(rseed, k, env, 0, 1)])  # noqa: E731
    s, t = start(0xFFFFFFFF), torch.zeros(n, dtype=torch.int64, device="cuda")
    got = {"obs": [], "action": [], "logp": [], "done": []}
    for k in range(c["steps"]):
        logp = torch.log_softmax(_mlp(net, s.T), 1)
        a = (_u01(_draw(rseed, k, env, 0, 0)[0]) >= logp[:, 0].exp()).long()
        x, v, th, w = s
        u = 20.0 * a - 10.0
        nxt = torch.stack([x + 0.02 * v, v + 0.02 * (u - 0.5 * x - 0.1 * v), th + 0.02 * w,
                           w + 0.02 * (9.8 * torch.sin(th) - 0.3 * torch.cos(th) * u)])
        t = t + 1
        done = (nxt[0].abs() > 2.4) | (nxt[2].abs() > 0.21) | (t >= EPISODE["control"])
        got["obs"].append(s)
        got["action"].append(a)
        got["logp"].append(logp.gather(1, a[:, None])[:, 0])
        got["done"].append(done)
        s, t = torch.where(done, start(k), nxt), torch.where(done, 0, t)
    return {k: torch.stack(v) for k, v in got.items()}, net


def _returns(reward, done):
    g, out = torch.zeros_like(reward[0]), []
    for r, d in zip(reward.flip(0), done.flip(0)):
        g = r + float(np.float32(GAMMA)) * torch.where(d, 0.0, g)
        out.append(g)
    return torch.stack(out[::-1])


def _exact_landscape(c, pseed, rseed):
    n, D, M = c["envs"], c["dim"], c["gauss"]
    net = _init_net(pseed, (D, c["hidden"], c["hidden"], 2 * D), 0)
    m, env = torch.arange(M, device="cuda"), torch.arange(n, device="cuda")
    four = lambda f: torch.stack([w for j in range(0, D, 4) for w in f(j // 4)], 0)  # noqa: E731
    centre = four(lambda q: [_between(w, -3, 3) for w in _draw(pseed, m, 0, 0, 5, q)])[:D].T
    z = _normals(_draw(pseed, m, 0, 0, 5, 64))
    width, amp = torch.exp(float(np.float32(0.3)) * z[0]), z[2]

    def field(x):
        energy, force = [], []
        for y in x.split(64):
            d = y[:, None, :] - centre
            e = amp * torch.exp(-d.square().sum(2) / (2 * width * width))
            energy.append(e.sum(1))
            force.append(torch.einsum("nm,nmd->nd", e / (width * width), d))
        return torch.cat(energy), torch.cat(force)

    def noise(k, sub):
        return float(np.float32(SIGMA)) * _normals(_draw(rseed, k, env, 0, 3, sub))[0]

    x = four(lambda q: [_between(w, -3, 3) for w in _draw(rseed, 0xFFFFFFFF, env, 0, 1, q)])[:D].T
    seen = field(x)[0] + noise(0xFFFFFFFF, 1)
    got = {k: [] for k in ("obs", "action", "logp", "reward", "energy", "force")}
    for k in range(c["steps"]):
        o = _mlp(net, x)
        ls = o[:, D:].clamp(-5, 2)
        z = four(lambda q: _normals(_draw(rseed, k, env, 0, 0, q)))[:D].T
        clip = float(np.float32(CLIP))
        dx = (o[:, :D] + ls.exp() * z).clamp(-clip, clip)
        e, f = field(x + dx)
        now = e + noise(k, 0)
        for name, v in (("obs", x.T), ("action", dx.T), ("reward", seen - now), ("energy", e), ("force", f.T),
                        ("logp", (-0.5 * z * z - ls - 0.5 * math.log(2 * math.pi)).sum(1))):
            got[name].append(v)
        x, seen = x + dx, now
    got = {k: torch.stack(v) for k, v in got.items()}
    got["done"] = None
    got["return"] = _returns(got["reward"], torch.zeros_like(got["reward"], dtype=torch.bool))
    return got


def _exact_train(c, pseed, rseed):
    rec, net = _control(c, pseed, rseed)
    crit = _init_net(pseed, (4, c["hidden"], c["hidden"], 1), 2)
    ret = _returns(torch.ones_like(rec["logp"]), rec["done"])
    x, a = rec["obs"].transpose(1, 2).reshape(-1, 4), rec["action"].reshape(-1)
    g, old = ret.reshape(-1), rec["logp"].reshape(-1)
    with torch.no_grad():
        held = g - _mlp(crit, x)[:, 0]
    eps = float(np.float32(EPS))
    for _ in range(1 if c["algo"] == "a2c" else 2):
        ps = [t.requires_grad_() for layer in net + crit for t in layer]
        lp = torch.log_softmax(_mlp(net, x), 1)
        v = _mlp(crit, x)[:, 0]
        la = lp.gather(1, a[:, None])[:, 0]
        if c["algo"] == "a2c":
            pg = -(g - v).detach() * la
        else:
            rho = torch.exp(la - old)
            pg = -torch.minimum(rho * held, rho.clamp(1 - eps, 1 + eps) * held)
        loss = (pg + float(np.float32(C_E)) * (lp.exp() * lp).sum(1) + C_V * (g - v).square()).mean()
        grads = torch.autograd.grad(loss, ps)
        new = [(p - float(np.float32(LR)) * d).detach() for p, d in zip(ps, grads)]
        net, crit = list(zip(new[0:6:2], new[1:6:2])), list(zip(new[6::2], new[7::2]))
        net, crit = [tuple(l) for l in net], [tuple(l) for l in crit]
    return {"return": ret, "params": _flat(net), "critic": _flat(crit)}


def exact(case, seed):
    c = case
    if c["kind"] == "forward":
        s = prepare(c, seed)
        widths, p, x = (c["inp"], c["h0"], c["h1"], c["out"]), s["params"].double(), s["obs"].double()
        for i, (a, b) in enumerate(zip(widths, widths[1:])):
            x = x @ p[:a * b].view(a, b) + p[a * b:a * b + b]
            x, p = torch.tanh(x) if i < 2 else x, p[a * b + b:]
        return x
    # BF16 policies decide actions by their own rounding, and the acrobot's and the economy's paths fork with
    # the first draw that falls the other way: no value in 64 bits is theirs.
    if c["path"] != "fp32" or c["kind"] == "serve" or c["env"] in ("economy", "acrobot"):
        return None
    pseed, rseed = seed % (1 << 30) + 1, seed % (1 << 30) + 7
    if c["env"] == "landscape":
        return _exact_landscape(c, pseed, rseed) if c["kind"] == "rollout" else None
    if c["kind"] == "train":
        return _exact_train(c, pseed, rseed) if c["envs"] * c["steps"] * c["hidden"] <= 1 << 26 else None
    rec, _ = _control(c, pseed, rseed)
    one = torch.ones_like(rec["logp"])
    return {"obs": rec["obs"], "action": None, "logp": rec["logp"], "reward": one, "done": None,
            "return": _returns(one, rec["done"])}
