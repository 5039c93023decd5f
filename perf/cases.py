"""Performance cases: the work a user of this library has it do, over the
range of sizes, rules and precisions it is used for.

Four kinds of call:

  run         a whole experiment in one or many worlds: reset from a seed, n
              steps, then the records, the final state, and the last step's
              logits and actions.  With "watch", the records are read back
              after every step (eco_step_read), as a monitor does.
  policy      one policy pass (observe, MLP, sample) over a population whose
              world and weights the caller supplied.
  checkpoint  the whole state and every agent's parameters saved from one
              handle and restored into another, whose next policy pass is
              returned: checkpoint and resume, and the exchange of traits
              with an outer population algorithm.
  claims      eco_move_claims_noalloc on the caller's own device arrays.

Sizes are the named workloads' (workloads.py), the bench's and the tests';
draw() spreads over the ranges between them.
"""
import math

import numpy as np
import torch

from paper_2510_18221_gb300 import eco, workloads


def listed():
    return [
        # One move-claim resolution for a host framework that keeps its own
        # world: the smallest call, a few launches.
        {"name": "claims-512", "kind": "claims", "side": 512, "agents": 12000},
        # The small workload as configured: 100 steps of a 64x64 world,
        # bound by the latency of a step, not by bytes.
        {"name": "small-run-fp32", "kind": "run", "base": "small", "worlds": 1, "side": 64, "slots": 256, "alive": 200,
         "precision": "fp32", "steps": 100, "watch": False, "sparse": False},
        # One policy pass over an odd number of agents, weights as the
        # caller wrote them (evaluation of a given population).
        {"name": "policy-bf16", "kind": "policy", "side": 254, "slots": 5003, "alive": 4001, "patch_k": 11, "hidden": 64,
         "form": "plain", "n_hidden": 1, "vision": "channels", "precision": "bf16"},
        # The mid workload as configured: 1000 steps, full-precision weights.
        {"name": "mid-run-fp32", "kind": "run", "base": "mid", "worlds": 1, "side": 512, "slots": 16384, "alive": 12000,
         "precision": "fp32", "steps": 1000, "watch": False, "sparse": False},
        # The mid workload in FP8, every step's records watched from the
        # host.
        {"name": "mid-watch-fp8", "kind": "run", "base": "mid", "worlds": 1, "side": 512, "slots": 16384, "alive": 12000,
         "precision": "fp8", "steps": 300, "watch": True, "sparse": False},
        # Checkpoint and resume of a mid-rules world (256x256).
        {"name": "checkpoint-bf16", "kind": "checkpoint", "side": 256, "slots": 2048, "alive": 1500, "precision": "bf16"},
        # The paper-scale world: its founders' population, and past step 100
        # the smaller one that lives on regrowth.
        {"name": "paper-run-bf16", "kind": "run", "base": "paper", "worlds": 1, "side": 1024, "slots": 65536, "alive": 50000,
         "precision": "bf16", "steps": 500, "watch": False, "sparse": False},
        # The same world with the input-sparse kernel family, which a user
        # with one-hot vision chooses for speed.
        {"name": "paper-sparse-bf16", "kind": "run", "base": "paper", "worlds": 1, "side": 1024, "slots": 65536, "alive": 50000,
         "precision": "bf16", "steps": 300, "watch": False, "sparse": True},
        # The paper's rules, policy form and RGB vision at the paper's scale.
        {"name": "ecology-run-bf16", "kind": "run", "base": "ecology", "worlds": 1, "side": 1024, "slots": 65536, "alive": 50000,
         "precision": "bf16", "steps": 100, "watch": False, "sparse": False},
        # The same with terrain: flowing water and three resources.
        {"name": "terrain-run-bf16", "kind": "run", "base": "terrain", "worlds": 1, "side": 1024, "slots": 65536, "alive": 50000,
         "precision": "bf16", "steps": 100, "watch": False, "sparse": False},
        # The large workload's 683-128-128-9 FP8 policies, on a world whose
        # masters leave room for others on the card.
        {"name": "largenet-run-fp8", "kind": "run", "base": "large", "worlds": 1, "side": 1024, "slots": 65536, "alive": 50000,
         "precision": "fp8", "steps": 200, "watch": False, "sparse": False},
        # Many uneven worlds advanced together (self-averaging studies).
        {"name": "batched-run-bf16", "kind": "run", "base": "batched", "worlds": 16, "side": 0, "slots": 0, "alive": 0,
         "precision": "bf16", "steps": 100, "watch": False, "sparse": False},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _even(v):
    return max(32, int(round(v / 2.0)) * 2)


def draw(rng):
    kind = rng.choice(["run"] * 7 + ["policy"] * 2 + ["checkpoint", "claims"])
    prec = rng.choice(["fp32", "bf16", "fp8"])
    if kind == "claims":
        side = _even(_log(rng, 32, 1024))
        return {"kind": kind, "side": side, "agents": max(1, int(side * side * _log(rng, 0.01, 0.3)))}
    if kind == "policy":
        side = _even(_log(rng, 64, 512))
        alive = max(16, min(12000, int(side * side * _log(rng, 0.02, 0.2))))
        form = rng.choice(["plain", "paper"])
        return {"kind": kind, "side": side, "slots": int(alive * rng.uniform(1.0, 1.4)), "alive": alive,
                "patch_k": rng.choice([3, 5, 7, 9, 11, 13]), "hidden": rng.choice([32, 64, 64]), "form": form,
                "n_hidden": rng.choice([1, 2, 3]) if form == "paper" else 1, "vision": rng.choice(["channels", "rgb"]),
                "precision": prec}
    if kind == "checkpoint":
        alive = int(_log(rng, 200, 1500))
        return {"kind": kind, "side": _even(_log(rng, 128, 512)), "slots": int(alive * rng.uniform(1.05, 1.4)), "alive": alive,
                "precision": prec}
    if rng.random() < 0.2:
        return {"kind": kind, "base": "batched", "worlds": rng.randint(2, 8 if prec == "fp32" else 16), "side": 0, "slots": 0, "alive": 0,
                "precision": prec, "steps": int(_log(rng, 16, 100)), "watch": False, "sparse": False}
    base = rng.choice(["small", "mid", "mid", "paper", "paperform", "ecology", "terrain"])
    side = _even(_log(rng, 32, 128) if base == "small" else _log(rng, 128, 1024))
    alive = max(16, min(25000 if prec == "fp32" else 50000, int(side * side * _log(rng, 0.02, 0.15))))
    sparse = base in ("mid", "paper", "paperform") and rng.random() < 0.25
    return {"kind": kind, "base": base, "worlds": 1, "side": side, "slots": int(alive * rng.uniform(1.1, 1.5)), "alive": alive,
            "precision": prec, "steps": int(_log(rng, 16, 200)), "watch": rng.random() < 0.25, "sparse": sparse}


# ---------------------------------------------------------------------------
# run
# ---------------------------------------------------------------------------

def _worlds(case, seed):
    if case["base"] == "batched":
        return workloads.batched(case["worlds"], seed=0, base_seed=seed, precision=case["precision"])
    return [workloads.get(case["base"], side=case["side"], slots=case["slots"], init_alive=case["alive"],
                          precision=case["precision"], seed=seed)]


def _prepare_run(case, seed):
    env = eco.Env(_worlds(case, seed), policy_variant=-1 if case["sparse"] else 0)
    env.reset_seed(seed)
    env.prepare()
    return {"case": case, "env": env, "seed": seed}


def _run_run(s):
    case, env = s["case"], s["env"]
    env.reset_seed(s["seed"])
    if case["watch"]:
        seen = np.zeros((case["steps"] + 1, eco.ECO_N_STATS), np.int64)
        for t in range(case["steps"]):
            seen[t] = eco.eco_step_read(env.h, 1)[1][0]
        total, last = eco.eco_read_stats(env.h, 1)
        seen[case["steps"]] = last[0]
        out = {"total": total, "last": seen}
    else:
        env.step(case["steps"])
        total, last = eco.eco_read_stats(env.h, env.n_envs)
        out = {"total": total, "last": last}
    if env.n_envs == 1:
        out["state"] = env.read_state(0)
    out["policy"] = [env.read_policy_io(e) for e in range(env.n_envs)]
    return out


# ---------------------------------------------------------------------------
# policy: a world and weights made from the seed alone
# ---------------------------------------------------------------------------

def _policy_world(case):
    return workloads.get("mid", side=case["side"], slots=case["slots"], init_alive=0, patch_k=case["patch_k"],
                         hidden=case["hidden"], policy_form=case["form"], n_hidden=case["n_hidden"],
                         vision=case["vision"], precision=case["precision"])


def _policy_state(case, seed):
    rng = np.random.default_rng(seed)
    side, S, K = case["side"], case["slots"], case["alive"]
    N = side * side
    wall = (rng.random(N) < 0.02).astype(np.uint8)
    food = ((rng.random(N) < 0.05) & (wall == 0)).astype(np.uint8)
    cells = rng.permutation(np.flatnonzero(wall == 0))[:K]
    slots = np.sort(rng.permutation(S)[:K])
    occ = np.full(N, -1, np.int32)
    occ[cells] = slots
    alive = np.zeros(S, np.uint8)
    x, y = np.zeros(S, np.int32), np.zeros(S, np.int32)
    alive[slots] = 1
    x[slots], y[slots] = cells % side, cells // side
    return {"food": food, "wall": wall, "occ": occ, "alive": alive, "x": x, "y": y,
            "facing": rng.integers(0, 4, S).astype(np.uint8), "energy": rng.integers(1, 200, S).astype(np.int32),
            "colour": rng.random((S, 3)).astype(np.float32)}


def _shape(case):
    """(D, H, A, hidden layers, input biases, paper form) of a policy case."""
    paper = case["form"] == "paper"
    return 3 * case["patch_k"] ** 2 + 8, case["hidden"], 9, case["n_hidden"] if paper else 1, 3 if paper else 1, paper


def _policy_params(case, seed):
    """[slots][P] FP32 in logical order: normals over sqrt(fan-in), small
    biases, and in the paper form a log-temperature."""
    D, H, A, layers, ns, paper = _shape(case)
    g = torch.Generator(device="cuda").manual_seed(seed)
    S = case["slots"]
    gain = 2.0 if paper else 1.0

    def normal(n, sd):
        return torch.randn(S, n, generator=g, device="cuda") * sd

    parts = [normal(H * D, math.sqrt(gain / D)), normal(ns * H, 0.05)]
    for _ in range(layers):
        parts += [normal(H * H, math.sqrt(gain / H)), normal(H, 0.05)]
    parts += [normal(A * H, math.sqrt(gain / H)), normal(1 if paper else A, 0.05)]
    return torch.cat(parts, dim=1)


def _prepare_policy(case, seed):
    env = eco.Env(_policy_world(case))
    env.reset_seed(seed)
    env.write_state(0, _policy_state(case, seed))
    params = _policy_params(case, seed)
    for a in range(0, case["slots"], 1024):
        env.write_params(0, a, params[a:a + 1024].cpu().numpy())
    env.prepare()
    return {"case": case, "env": env}


def _run_policy(s):
    s["env"].policy_only(1)
    logits, act = s["env"].read_policy_io(0)
    return {"logits": logits, "actions": act}


def _observe(case, st):
    """Observations [slots][D] in 64 bits: the k x k patch turned so that the
    facing is up, three channels per cell, then energy, the one-hot facing
    and three zeros."""
    side, k, S = case["side"], case["patch_k"], case["slots"]
    dx, dy = np.array([0, 1, 0, -1]), np.array([-1, 0, 1, 0])
    f = st["facing"].astype(np.int64)
    right = (f + 1) % 4
    rows, cols = np.divmod(np.arange(k * k), k)
    ahead, aside = k // 2 - rows, cols - k // 2
    cx = (st["x"][:, None] + ahead * dx[f][:, None] + aside * dx[right][:, None]) % side
    cy = (st["y"][:, None] + ahead * dy[f][:, None] + aside * dy[right][:, None]) % side
    c = cy * side + cx
    agent, wall, food = st["occ"][c] >= 0, st["wall"][c] != 0, st["food"][c] != 0
    if case["vision"] == "rgb":
        patch = np.zeros((S, k * k, 3))
        patch[..., 1] = food
        patch[wall] = 0.5
        patch[agent] = st["colour"].astype(np.float64)[st["occ"][c][agent]]
    else:
        patch = np.stack([food, agent, wall], axis=-1).astype(np.float64)
    scalars = np.zeros((S, 8))
    scalars[:, 0] = st["energy"] / 200.0
    scalars[np.arange(S), 1 + f] = 1.0
    return np.concatenate([patch.reshape(S, -1), scalars], axis=1)


def _streamed(w, precision):
    """The values of weight rows [..., in] as the precision holds them."""
    if precision == "bf16":
        return w.bfloat16().double()
    if precision == "fp8":
        s = w.abs().amax(-1, keepdim=True) / 448.0
        s = torch.where(s == 0, torch.ones_like(s), s)
        return (w / s).to(torch.float8_e4m3fn).double() * s.double()
    return w.double()


def _exact_policy(case, seed):
    D, H, A, layers, ns, paper = _shape(case)
    st = _policy_state(case, seed)
    obs = torch.from_numpy(_observe(case, st)).cuda()
    p = _policy_params(case, seed)
    act = torch.relu if paper else torch.tanh
    out = torch.zeros(case["slots"], A, dtype=torch.float64, device="cuda")
    for a in range(0, case["slots"], 256):
        q, x = p[a:a + 256], obs[a:a + 256]
        n, at = q.shape[0], 0

        def take(*shape):
            nonlocal at
            v = q[:, at:at + math.prod(shape)].reshape(n, *shape)
            at += math.prod(shape)
            return v

        def times(w, h):
            return torch.einsum("noi,ni->no", _streamed(w, case["precision"]), h)

        w, b = take(H, D), take(ns, H)
        h = act(times(w, x) + b.double().sum(1))
        for _ in range(layers):
            w, b = take(H, H), take(H)
            h = act(times(w, h) + b.double())
        logits = times(take(A, H), h)
        out[a:a + 256] = logits * torch.exp(-take(1).double()) if paper else logits + take(A).double()
    out[torch.from_numpy(st["alive"] == 0).cuda()] = 0.0    # never computed
    return {"logits": out, "actions": None}


# ---------------------------------------------------------------------------
# checkpoint
# ---------------------------------------------------------------------------

def _prepare_checkpoint(case, seed):
    w = workloads.get("mid", side=case["side"], slots=case["slots"], init_alive=case["alive"], precision=case["precision"],
                      seed=seed)
    env, other = eco.Env(w), eco.Env(w)
    for e in (env, other):
        e.reset_seed(seed)
        e.prepare()
    env.step(16)
    return {"case": case, "env": env, "other": other}


def _run_checkpoint(s):
    env, other = s["env"], s["other"]
    state, params = env.read_state(0), env.read_params(0)
    other.write_state(0, state)
    other.write_params(0, 0, params)
    other.policy_only(1)
    logits, act = other.read_policy_io(0)
    return {"state": state, "params": params, "logits": logits, "actions": act}


# ---------------------------------------------------------------------------
# claims
# ---------------------------------------------------------------------------

def _prepare_claims(case, seed):
    rng = np.random.default_rng(seed)
    side, n = case["side"], case["agents"]
    cells = rng.choice(side * side, size=n, replace=False).astype(np.int32)
    blocked = (rng.random(side * side) < 0.02).astype(np.uint8)
    blocked[cells] = 1

    def dev(a):
        return torch.from_numpy(a).cuda()

    return {"side": side, "n": n, "seed": seed & 0xFFFFFFFF, "pos": dev(cells), "blocked": dev(blocked),
            "act": dev(rng.integers(0, 9, n).astype(np.uint8)), "facing": dev(rng.integers(0, 4, n).astype(np.uint8)),
            "facing_out": torch.empty(n, dtype=torch.uint8, device="cuda"),
            "pos_out": torch.empty(n, dtype=torch.int32, device="cuda"),
            "moved": torch.empty(n, dtype=torch.uint8, device="cuda")}


def _run_claims(s):
    eco.eco_move_claims_noalloc(s["side"], s["n"], s["pos"].data_ptr(), s["act"].data_ptr(), s["facing"].data_ptr(),
                                s["blocked"].data_ptr(), s["seed"], 7, s["facing_out"].data_ptr(),
                                s["pos_out"].data_ptr(), s["moved"].data_ptr(), torch.cuda.current_stream().cuda_stream)
    return s["facing_out"], s["pos_out"], s["moved"]


def prepare(case, seed):
    kinds = {"run": _prepare_run, "policy": _prepare_policy, "checkpoint": _prepare_checkpoint, "claims": _prepare_claims}
    return kinds[case["kind"]](case, seed)


def run(state):
    if "pos" in state:
        return _run_claims(state)
    return {"run": _run_run, "policy": _run_policy, "checkpoint": _run_checkpoint}[state["case"]["kind"]](state)


def exact(case, seed):
    # The other kinds' numbers are whole, copies of their inputs, or the end
    # of a long run, which no plain 64-bit formula gives in a few seconds.
    return _exact_policy(case, seed) if case["kind"] == "policy" else None


# ---------------------------------------------------------------------------
# work: bytes and operations of one pass
# ---------------------------------------------------------------------------

def _net(w):
    """(parameters, weights, streamed bytes, input weights) of one agent."""
    nch = 4 if w.get("rules") == "terrain" else 3
    D, H, A = nch * w["patch_k"] ** 2 + w["n_scalars"], w["hidden"], w["n_actions"]
    paper = w.get("policy_form") == "paper"
    layers = w.get("n_hidden", 1) if paper else 1
    ns = (1 + (w["n_scalars"] >= 8) + (w["patch_k"] > 0)) if paper else 1
    nw = D * H + layers * H * H + A * H
    nb = ns * H + layers * H + (1 if paper else A)
    es = {"fp32": 4, "bf16": 2, "fp8": 1}[w["precision"]]
    rows = (H + layers * H + A) if es == 1 else 0
    return nw + nb, nw, nw * es + 4 * (nb + rows), D * H


def _agent_steps(w, steps):
    """Agents alive summed over the steps, about: the founders live on their
    first energy, then the world feeds a part of them."""
    if w.get("rules", "simple") != "simple":
        per = 0.5 * min(steps, 48) + 0.05 * max(0, min(steps, 100) - 48)
    else:
        per = 0.98 * min(steps, 72) + 125 * (1 - math.exp(-max(0, min(steps, 260) - 72) / 125)) + 0.2 * max(0, steps - 260)
    return w["init_alive"] * per


def work(case):
    if case["kind"] == "claims":
        return {"bytes": 13 * case["agents"] + case["side"] ** 2, "flops": 0}
    if case["kind"] == "run":
        total, flops = 0.0, 0.0
        for w in _worlds(case, 0):
            P, nw, stream, n_in = _net(w)
            n = _agent_steps(w, case["steps"])
            if case["sparse"]:      # the rows of nonzero inputs, about 20 of them
                share = 20.0 / (n_in / w["hidden"])
                skip = n_in * (1 - share)
                stream, nw = stream - skip * stream / P, nw - skip
            fresh = w["slots"] * (4 * P + (0 if case["precision"] == "fp32" else stream))   # the reset's weights
            total += fresh + n * stream + case["steps"] * w["side"] ** 2 + 10 * w["side"] ** 2 + 64 * w["slots"]
            flops += 2.0 * nw * n
        return {"bytes": total, "flops": flops}
    if case["kind"] == "policy":
        _, nw, stream, _ = _net(_policy_world(case))
        return {"bytes": case["alive"] * (stream + 3 * case["patch_k"] ** 2) + case["slots"] * 37, "flops": 2.0 * nw * case["alive"]}
    P, nw, stream, _ = _net(workloads.get("mid", precision=case["precision"]))
    return {"bytes": case["slots"] * (2 * 4 * P + (0 if case["precision"] == "fp32" else stream)) + case["alive"] * stream
            + 2 * 6 * case["side"] ** 2 + 2 * 45 * case["slots"], "flops": 2.0 * nw * case["alive"]}
