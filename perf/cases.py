"""Performance cases: what programs have this library do, each through its Python entry points.

A case is a dict of plain values:
  kind     "step"     one Env.step per pass (an agent that looks at every observation)
           "step_n"   one Env.step_n call of `steps` steps (rollouts with known actions); with "packed"
                      the frames come one bit per pixel (Env.step_n_packed)
           "host"     one Env.step_host per pass into pinned host buffers; with "packed" Env.step_host_packed
           "forward"  one Policy.forward of n observations; with "u8" Policy.forward_u8 on byte frames
           "rollout"  one Policy.rollout of `steps` steps: the network acts on the device
           "server"   `requests` requests submitted at once to a Server and waited for
  game     which programs the instances run (see _games)
  launch   "" = as created, or "block x instances-per-warp x steps-per-launch" with the letters p
           (persistent queue) and b (balanced waves) behind it: a shape found by an earlier tuning run
"""
import math

import numpy as np
import torch

from paper_2510_01764_gb300 import octax
from paper_2510_01764_gb300 import workloads as W

_SERVER_BUDGET = 256 << 20  # device bytes for the server's resident instances (about 60,000)


def listed():
    return [
        # a debugging or evaluation loop: the smallest documented configuration, one call per step
        _case("step-64-template", "step", "template", 64),
        # an odd-sized mixed-game trainer on the three shooter levels, sticky actions and no-op resets
        _case("step-1001-shooter-wrapped", "step", "shooter-wrapped", 1001),
        # the ordinary training loop: 16,384 instances, one call per step, library defaults
        _case("step-16384-template", "step", "template", 16384),
        # a 32-step rollout behind the usual wrappers, in a tuned launch shape
        _case("rollout-16384-wrapped", "step_n", "wrapped", 16384, steps=32, launch="256x7x32b"),
        # packed frames for a learner that unpacks them, ragged size, library defaults
        _case("packed-12289-shooter", "step_n", "shooter", 12289, steps=16, packed=True),
        # 16 ROMs of uneven size and speed: one persistent graph-replayed launch per 16 frames
        _case("batch-65536-16roms", "step_n", "batch", 65536, steps=8, launch="64x16x4p"),
        # random programs: divergent control flow, memory written everywhere; the largest call
        _case("random-262144", "step_n", "random", 262144, steps=4, launch="128x16x16"),
        # Super-CHIP frames (8 KB each), library defaults
        _case("schip-8192", "step_n", "schip", 8192, steps=8),
        # a trainer whose learner lives on the host: pinned buffers over the host link
        _case("host-4096-template", "host", "template", 4096),
        # re-evaluating a minibatch of observations with the network
        _case("forward-16384", "forward", "template", 16384),
        # acting on the device: the network picks every action of an 8-step rollout
        _case("policy-rollout-2048", "rollout", "template", 2048, steps=8),
        # a wave of unrelated step requests to the server
        _case("server-48-requests", "server", "batch", 4096, requests=48),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step_n", "step_n", "host", "forward", "rollout", "server"])

    def size(lo, hi):  # log-uniform, odd as often as even
        return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))

    launch = ""
    if kind == "step":
        return _case("", kind, rng.choice(["template", "shooter", "shooter-wrapped", "wrapped", "batch", "random"]),
                     size(64, 65536))
    if kind == "step_n":
        game = rng.choice(["template", "wrapped", "shooter", "batch", "random", "schip"])
        n = size(64, 8192 if game == "schip" else 131072)
        most = max(1, min(64, 1048576 // n // (4 if game == "schip" else 1)))
        if rng.random() < 0.5:
            launch = rng.choice(["64x16x4p", "128x16x16", "256x7x32b", "128x8x8"])
        if game == "schip" and launch in ("256x7x32b", "128x16x16"):
            launch = "128x8x8"
        return _case("", kind, game, n, steps=size(1, most), packed=rng.random() < 0.3, launch=launch)
    if kind == "host":
        return _case("", kind, rng.choice(["template", "shooter"]), size(64, 8192), packed=rng.random() < 0.5)
    if kind == "forward":
        return _case("", kind, "template", size(64, 32768), u8=rng.random() < 0.3)
    if kind == "rollout":
        n = size(64, 8192)
        return _case("", kind, rng.choice(["template", "wrapped"]), n, steps=size(1, min(32, 65536 // n)))
    return _case("", kind, "batch", size(256, 4096), requests=size(4, 64))


def _case(name, kind, game, n, steps=1, packed=False, u8=False, launch="", requests=0):
    c = {"name": name, "kind": kind, "game": game, "n": n, "steps": steps, "packed": packed, "u8": u8,
         "launch": launch, "requests": requests}
    if not name:
        del c["name"]
    return c


def _games(game, n):
    """(GameSpecs, game of each instance or None, steps to play before the inputs are representative)."""
    if game == "template":
        return W.cfg_scale().games, None, 128
    if game == "wrapped":  # until episodes end at different times
        return W.cfg_wrappers().games, None, 3072 if n <= 32768 else 1024
    if game in ("shooter", "shooter-wrapped"):
        games = W.cfg_shooter().games
        if game == "shooter-wrapped":
            games = [W.replace(g, sticky_prob=0.25, max_noops=30) for g in games]
        return games, (np.arange(n) % 3).astype(np.uint16), 320
    if game == "batch":
        w = W.cfg_batch(n_envs=max(n, 16))
        return w.games, w.game_of_env[:n], 128
    if game == "random":
        w = W.cfg_divergence(n_envs=n)
        return w.games[:min(64, n)], w.game_of_env, 32
    if game == "schip":
        return W.cfg_schip().games, None, 128
    raise ValueError(game)


def _actions(gen, games, *shape):
    return torch.randint(0, games[0].n_actions, shape, dtype=torch.uint8, device="cuda", generator=gen)


def _env(case, seed, gen):
    games, goe, warm = _games(case["game"], case["n"])
    env = octax.Env(games, case["n"], game_of_env=goe, seed=seed)
    if case["launch"]:
        block, ipw, spl = case["launch"].rstrip("pb").split("x")
        env.set_launch(block=int(block), inst_per_warp=int(ipw), steps_per_launch=int(spl),
                       persistent=int("p" in case["launch"]), balance=int("b" in case["launch"]))
    # Play on with random actions, so that scores, timers, written memory and episode ends are as in a running
    # program (in chunks whose outputs take at most 1 GB).
    chunk = max(1, min(32, (1 << 20) // case["n"]))
    out = None
    for _ in range(-(-warm // chunk)):
        out = env.step_n_packed(_actions(gen, games, chunk, case["n"]), out)
    return env, games, out[0][-1].clone()


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n, T, kind = case["n"], case["steps"], case["kind"]
    if kind == "server":
        return _prepare_server(case, seed)
    env, games, words = _env(case, seed, gen)
    s = {"case": case, "env": env, "words": words}
    dev = "cuda"
    if kind in ("step", "host"):
        host = {"pin_memory": True} if kind == "host" else {"device": dev}
        acts = _actions(gen, games, n)
        s["actions"] = acts.cpu().pin_memory() if kind == "host" else acts
        obs = (torch.empty((n,) + env.packed_obs_shape, dtype=torch.int64, **host) if case["packed"]
               else torch.empty(env.obs_shape, dtype=torch.uint8, **host))
        s["out"] = (obs, torch.empty(n, dtype=torch.float32, **host), torch.empty(n, dtype=torch.uint8, **host))
    elif kind == "step_n":
        s["actions"] = _actions(gen, games, T, n)
        obs = (torch.empty((T, n) + env.packed_obs_shape, dtype=torch.int64, device=dev) if case["packed"]
               else torch.empty((T,) + env.obs_shape, dtype=torch.uint8, device=dev))
        s["out"] = (obs, torch.empty((T, n), dtype=torch.float32, device=dev),
                    torch.empty((T, n), dtype=torch.uint8, device=dev))
    else:
        s["params"] = W.policy_params(seed, games[0].n_actions + 1)
        s["policy"] = octax.Policy(s["params"], n)
        s["seed"] = seed
        if case["u8"]:
            s["frames"] = _bits(words).to(torch.uint8)
    return s


def _bits(words):
    """int64 [n, 4, 32] -> 0/1 [n, 4, 32, 64]."""
    return (words.unsqueeze(-1) >> torch.arange(64, device=words.device)) & 1


def _prepare_server(case, seed):
    games, _, _ = _games(case["game"], case["n"])
    rng = np.random.default_rng(seed)
    server = octax.Server(games, memory_budget_bytes=_SERVER_BUDGET, block=128, inst_per_warp=16)
    items, sizes = [], _request_sizes(case)
    for game, n, T in sizes:
        acts = rng.integers(0, 4, size=(T, n), dtype=np.uint8)
        out = (torch.empty((T, n, 4, 32, 64), dtype=torch.uint8, device="cuda"),
               torch.empty((T, n), dtype=torch.float32, device="cuda"),
               torch.empty((T, n), dtype=torch.uint8, device="cuda"))
        items.append((game, acts, int(rng.integers(1 << 32)), out))
    torch.cuda.synchronize()
    return {"case": case, "server": server, "items": items}


def _request_sizes(case):
    """(game, instances, steps) of each request: 1 .. n instances log-uniform, 1-8 steps, from the case alone."""
    rng = np.random.default_rng(case["n"] * 1000 + case["requests"])
    return [(int(rng.integers(0, 16)), int(np.exp(rng.uniform(0, np.log(case["n"] + 1)))), int(rng.integers(1, 9)))
            for _ in range(case["requests"])]


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "step":
        return s["env"].step(s["actions"], s["out"])
    if kind == "step_n":
        f = s["env"].step_n_packed if case["packed"] else s["env"].step_n
        return f(s["actions"], s["out"])
    if kind == "host":
        f = s["env"].step_host_packed if case["packed"] else s["env"].step_host
        return f(s["actions"], s["out"])
    if kind == "forward":
        if case["u8"]:
            return s["policy"].forward_u8(s["frames"], seed=s["seed"])
        return s["policy"].forward(s["words"], seed=s["seed"])
    if kind == "rollout":
        return s["policy"].rollout(s["env"], case["steps"], s["words"], seed=s["seed"]) + (s["words"],)
    ids = s["server"].submit_batch(s["items"])
    s["server"].wait_batch(ids)
    # the requests' own output tensors, by size (64 results at most are kept apart)
    return [t for it in s["items"][:21] for t in it[3]]


def work(case):
    """Bytes: actions in, observations, rewards and flags out, the instance state once in and once out; the
    network's weights are few. Flops: the network's multiply-adds, counted twice."""
    n, T, kind = case["n"], case["steps"], case["kind"]
    net = 2.0 * (15 * 15 * 32 * 128 + 6 * 6 * 64 * 512 + 4 * 4 * 64 * 576 + 1024 * 512 + 256 * 6)
    schip = case["game"] == "schip"
    words, state = (128, 1100) if schip else (32, 340)
    frames = 4 * words * (8 if case["packed"] else 64)
    if kind == "forward":
        return {"bytes": n * ((8192 if case["u8"] else 1024) + 25.0), "flops": n * net}
    if kind == "rollout":
        return {"bytes": n * (2.0 * 1024 + 2 * state + T * 30.0), "flops": T * n * net}
    if kind == "server":
        return {"bytes": float(sum(k * (8198 * t + state) for _, k, t in _request_sizes(case))), "flops": 0.0}
    return {"bytes": float(n * (T * (frames + 6) + 2 * state)), "flops": 0.0}


def exact(case, seed):
    """The network in 64 bits for the forward cases; the emulator's outputs are whole numbers."""
    if case["kind"] != "forward":
        return None
    s = prepare(case, seed)
    p = {k: torch.from_numpy(np.asarray(v)).cuda().double() for k, v in s["params"].items()}
    F = torch.nn.functional
    logits, values = [], []
    for x in _bits(s["words"]).split(2048):
        x = x.transpose(2, 3).double()  # [n, frame, x, y]
        x = F.relu(F.conv2d(x, p["w1"], p["b1"], stride=(4, 2)))
        x = F.relu(F.conv2d(x, p["w2"], p["b2"], stride=2))
        x = F.relu(F.conv2d(x, p["w3"], p["b3"])).flatten(1)  # (channel, x, y)
        logits.append(F.relu(x @ p["wa1"].T + p["ba1"]) @ p["wa2"].T + p["ba2"])
        values.append(F.relu(x @ p["wc1"].T + p["bc1"]) @ p["wc2"] + p["bc2"])
    return torch.cat(logits), torch.cat(values), None
