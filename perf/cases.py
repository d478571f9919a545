"""What the speed of this framework is measured on: a list of calls that its users make, and draws of more of them.

The framework steps batches of CartPole environments. Its users call it in five ways, and each is a `kind` here:

  step     one fused step with actions that the user's own program chose (an agent outside the library)
  loop     many single steps with hashed actions issued from one call (the paper's host loop)
  rollout  T steps in one launch, under hashed actions, a policy or supplied actions, with or without per-step outputs
  chunk    the same from a saved batch of states in the middle of its episodes (collection of training data and planning;
           the call advances a batch in place, so the saved one is copied first)
  host     one step between page-locked HOST buffers

Sizes are those of inputs.py's workloads, or smaller and odd ones of the same sort. The per-op ladder is not here: it is the
slow end of a comparison, and nobody steps environments with it to get work done. Results do not depend on the execution
strategy, bit for bit, so every case is compared exactly.
"""
import math

import numpy as np
import torch

from paper_2301_13062_b200 import binding as cp
from paper_2301_13062_b200 import inputs

#: policies by name: (kind, multiply-adds per evaluation, tanh per evaluation)
POLICIES = {
    "random": (cp.CP_POLICY_RANDOM, 0, 0),
    "linear": (cp.CP_POLICY_LINEAR, 8, 0),
    "mlp16": (cp.CP_POLICY_MLP, 96, 16),
    "mlp32": (cp.CP_POLICY_MLP32, 192, 32),
    "mlp64": (cp.CP_POLICY_MLP64, 384, 64),
    "deep": (cp.CP_POLICY_MLP_DEEP, 352, 32),
    "per_env": (cp.CP_POLICY_LINEAR_PER_ENV, 8, 0),
    "given": (cp.CP_POLICY_RANDOM, 0, 0),  # actions are data
}
OUTPUTS = {
    "returns": (),  # per-environment returns and episode counts alone
    "stream": ("reward_stream", "done_bits"),
    "actions": ("reward_stream", "done_bits", "action_bits"),
    "full": ("reward_stream", "done_bits", "action_bits", "trajectory"),
}
DEVICE = "cuda"


def _rollout(name, n, T, policy="random", outputs="returns", limit=0, contracted=False, starts=False, kind="rollout"):
    return {"name": name, "kind": kind, "n": n, "T": T, "policy": policy, "outputs": outputs, "limit": limit,
            "contracted": contracted, "starts": starts}


def listed():
    return [
        # An agent outside the library steps a small batch: one launch per step, latency and host cost are all there is.
        {"name": "step_agent", "kind": "step", "n": 4099, "given": True, "limit": 500, "aligned": False},
        # A large batch held in a plain [4, n] tensor of an odd n: planes that do not start on 16 bytes. Memory-bound.
        {"name": "step_ragged", "kind": "step", "n": 5_000_011, "given": True, "limit": 0, "aligned": False},
        # The per-step workload (65,536 environments through single launches), the whole chip synchronised at each step.
        {"name": "step_loop", "kind": "loop", "n": 65_536, "T": 200},
        # One step for a caller whose arrays live in page-locked host memory.
        {"name": "step_host", "kind": "host", "n": 500_000, "given": True},
        # The paper's own shape: few environments, a long horizon; the latency of one step.
        _rollout("paper", 2048, 10_000),
        # Evaluation of a network on few environments under CartPole-v1's 500-step limit.
        _rollout("eval_network", 4096, 500, "mlp64", limit=500),
        # Population search: a linear policy of its own for every environment, scored over one limited episode and more.
        _rollout("population", 20_011, 500, "per_env", limit=500),
        # Collection of training data with a network: everything that a learner reads, from environments in mid-episode.
        _rollout("collect", 50_001, 128, "mlp16", outputs="full", limit=500, kind="chunk"),
        # Recorded actions and start states played again: the paper's baseline reads its random values from memory.
        _rollout("replay", 200_003, 250, "given", starts=True),
        # The headline workload: a batch that fills the chip, hashed actions.
        _rollout("headline", 1_048_576, 500),
        # The write-heavy workload: a linear policy, reward plane and done bits of every step.
        _rollout("linear_stream", 1_048_576, 400, "linear", outputs="stream"),
        # The largest: a network policy inside the rollout of 16.8 M environments.
        _rollout("network_large", 16_777_216, 200, "mlp16"),
    ]


def _cost(policy):
    return 60 + 2 * POLICIES[policy][1] + 20 * POLICIES[policy][2]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step", "step", "loop", "host", "rollout", "rollout", "rollout", "rollout", "chunk", "chunk"])
    if kind == "step":
        n = log(1_000, 16_000_000)
        aligned = rng.random() < 0.5
        return {"kind": kind, "n": n // 4 * 4 if aligned else n, "given": rng.random() < 0.7,
                "limit": rng.choice([0, 0, 500]), "aligned": aligned}
    if kind == "loop":
        return {"kind": kind, "n": log(1_000, 500_000), "T": log(20, 400)}
    if kind == "host":
        return {"kind": kind, "n": log(2_000, 4_000_000), "given": rng.random() < 0.7}
    policy = rng.choice(["random", "random", "linear", "mlp16", "mlp32", "mlp64", "deep", "per_env", "given", "given"])
    outputs = rng.choice(["returns", "returns", "stream", "actions", "full"])
    starts = policy == "given" and rng.random() < 0.5
    n, T = log(500, 4_000_000), log(4, 2_000)
    # no more arithmetic than the largest listed case, no more than 2 GB of per-step data
    per_step = {"returns": 0, "stream": 5, "actions": 5, "full": 21}[outputs] + (16 if starts else 0) + 1
    most = min(16_777_216 * 200 * _cost("mlp16") / 2 / _cost(policy), 2e9 / per_step)
    T = max(4, min(T, int(most / n)))
    n = max(500, min(n, int(most / T)))
    return {"kind": kind, "n": n, "T": T, "policy": policy, "outputs": outputs, "limit": rng.choice([0, 200, 500]),
            "contracted": rng.random() < 0.2, "starts": starts}


def _words(n):
    return (n + 31) // 32


def _live_states(n, g, device):
    """States of the sort that running environments hold: mostly well inside the termination box, some close to leaving it."""
    half = torch.tensor([2.0, 1.2, 0.19, 1.4], device=device).reshape(4, 1)
    return (torch.rand(4, n, generator=g, device=device) * 2 - 1) * half


def _weights(case, seed, device):
    kind = POLICIES[case["policy"]][0]
    if case["policy"] == "per_env":
        g = torch.Generator(device).manual_seed(seed * 7 + 3)
        return 0.5 * torch.randn(10, case["n"], generator=g, device=device)
    return inputs.policy_weights(kind, seed * 7 + 3) if kind != cp.CP_POLICY_RANDOM else None


def _data(case, seed, device):
    """The inputs of a case, made from the seed alone."""
    g = torch.Generator(device).manual_seed(int(seed))
    n, T = case["n"], case.get("T", 1)
    d = {"seed": (int(seed) * 2654435761 + 97) & 0xFFFFFFFF, "t0": 0}
    if case["kind"] in ("step", "loop", "host", "chunk"):
        d["planes"] = _live_states(n, g, device)
        d["t0"] = 1 + int(seed) % 5000
    if case["kind"] == "chunk" or (case["kind"] == "step" and case["limit"]):
        # steps already taken: some environments reach the limit in this call
        d["ep_len"] = torch.randint(0, max(1, (case["limit"] or 500) - 1), (n,), generator=g, device=device, dtype=torch.int32)
    if case["kind"] in ("step", "host") and case["given"]:
        d["action"] = torch.randint(0, 2, (n,), generator=g, device=device, dtype=torch.uint8)
    if case.get("policy") == "given":
        d["bits"] = torch.randint(-2**31, 2**31, (T, _words(n)), generator=g, device=device, dtype=torch.int64).to(torch.int32)
    if case.get("starts"):
        d["starts"] = torch.rand(T, 4, n, generator=g, device=device) * 0.1 - 0.05
    if "policy" in case:
        d["weights"] = _weights(case, int(seed), device)
    return d


def prepare(case, seed):
    d = _data(case, seed, DEVICE)
    n, T = case["n"], case.get("T", 1)
    s = {"case": case, "d": d}

    def empty(*shape, dtype=torch.float32):
        return torch.empty(*shape, dtype=dtype, device=DEVICE)

    if case["kind"] == "host":
        s["in"] = d["planes"].cpu().pin_memory()
        s["action"] = d["action"].cpu().pin_memory() if case["given"] else None
        s["out"] = (torch.empty(4, n).pin_memory(), torch.empty(n).pin_memory(),
                    torch.empty(n, dtype=torch.uint8).pin_memory())
        return s
    if case["kind"] == "step":
        stride = (n + 3) // 4 * 4 if case["aligned"] else n
        planes = torch.zeros(4, stride, device=DEVICE)
        planes[:, :n] = d["planes"]
        out = torch.zeros(4, stride, device=DEVICE)
        s["from"], s["to"] = cp.cp_wrap(planes, n, d["seed"], t=d["t0"]), cp.cp_wrap(out, n, d["seed"])
        s["out"] = (out, empty(n), empty(n, dtype=torch.uint8))
        s["ep_len"] = torch.empty_like(d["ep_len"]) if case["limit"] else None
        return s
    if case["kind"] in ("loop", "chunk"):
        s["planes"] = torch.empty_like(d["planes"])
        s["batch"] = cp.cp_wrap(s["planes"], n, d["seed"], t=d["t0"])
    if case["kind"] == "loop":
        s["out"] = (s["planes"], empty(n), empty(n, dtype=torch.uint8))
        return s
    if case["kind"] == "chunk":
        s["ep_len"] = torch.empty_like(d["ep_len"])
    s["policy"] = cp.policy(POLICIES[case["policy"]][0], d["weights"])
    r = {"ep_return_sum": empty(n), "ep_count": empty(n, dtype=torch.int32), "totals": empty(2, dtype=torch.int64)}
    shapes = {"reward_stream": ((T, n), torch.float32), "done_bits": ((T, _words(n)), torch.int32),
              "action_bits": ((T, _words(n)), torch.int32), "trajectory": ((T, 4, n), torch.float32)}
    for key in OUTPUTS[case["outputs"]]:
        r[key] = empty(*shapes[key][0], dtype=shapes[key][1])
    if case["kind"] == "rollout":
        r["final_state"] = empty(4, n)
    s["returns"] = r
    s["options"] = {"max_episode_steps": case["limit"], "action_bits_in": d.get("bits"), "start_states_in": d.get("starts"),
                    "arithmetic": cp.CP_ARITH_CONTRACTED if case["contracted"] else cp.CP_ARITH_EXACT}
    return s


def run(state):
    case, d = state["case"], state["d"]
    if case["kind"] == "host":
        cp.cp_step_host(case["n"], d["seed"], d["t0"], state["in"], state["action"], *state["out"])
        return state["out"]
    if case["kind"] == "step":
        out, reward, done = state["out"]
        if not case["limit"]:
            cp.cp_step(state["from"], d.get("action"), state["to"], reward, done)
            return state["out"]
        state["ep_len"].copy_(d["ep_len"])
        cp.cp_step_ex(state["from"], d.get("action"), state["to"], reward, done, state["ep_len"], case["limit"])
        return (*state["out"], state["ep_len"])
    if case["kind"] == "loop":
        state["planes"].copy_(d["planes"])
        cp.cp_set_time(state["batch"], d["t0"])
        cp.cp_step_repeat(state["batch"], case["T"], *state["out"][1:])
        return state["out"]
    returns = state["returns"]
    returns["totals"].zero_()
    if case["kind"] == "rollout":
        cp.cp_rollout_ex(n_envs=case["n"], T=case["T"], seed=d["seed"], policy=state["policy"], **state["options"], **returns)
        return returns
    state["planes"].copy_(d["planes"])
    state["ep_len"].copy_(d["ep_len"])
    cp.cp_set_time(state["batch"], d["t0"])
    cp.cp_rollout_ex(T=case["T"], state=state["batch"], ep_len=state["ep_len"], policy=state["policy"], **state["options"], **returns)
    return {**returns, "planes": state["planes"], "ep_len": state["ep_len"]}


def work(case):
    """Floating-point operations of the step as it is defined (43, and the policy's), each input and output once."""
    n, T = case["n"], case.get("T", 1)
    if case["kind"] in ("step", "host"):
        return {"bytes": n * (37 + (1 if case["given"] else 0) + (8 if case.get("limit") else 0)), "flops": 43 * n}
    if case["kind"] == "loop":  # every single step reads and writes the batch
        return {"bytes": 37 * n * T, "flops": 43 * n * T}
    _, madds, tanhs = POLICIES[case["policy"]]
    per_step = {"returns": 0, "stream": 4.125, "actions": 4.25, "full": 20.25}[case["outputs"]]
    if case["policy"] == "given":
        per_step += 0.125 + (0.7 if case["starts"] else 0)  # an episode lasts about 22 steps under coin-flip actions
    once = 8 + (40 if case["policy"] == "per_env" else 0) + (16 if case["kind"] == "rollout" else 40)
    return {"bytes": n * (T * per_step + once), "flops": n * T * (43 + 2 * madds + 8 * tanhs)}


def tolerance(case):
    return "exact"


# ---- the same results from float64 torch, from the definitions alone ----
M32 = 0xFFFFFFFF


def _mix(h):
    h = h ^ (h >> 16)
    h = (h * 0x6A09E667) & M32
    h = h ^ (h >> 15)
    h = (h * 0xBB67AE85) & M32
    return h ^ (h >> 16)


class _Stream:
    """Hash values of one stream (0 actions, 1 starts) of every environment, on int64 tensors."""

    def __init__(self, seed, stream, n, device):
        salt = _mix((_mix(seed ^ 0x9E3779B1) + stream) & M32)
        self.k0 = _mix(torch.arange(n, device=device, dtype=torch.int64) ^ salt)
        self.k1 = _mix((self.k0 + 0x9E3779B1) & M32)

    def at(self, counter, who=slice(None)):
        h = self.k0[who] ^ (counter & M32)
        h = ((h ^ (h >> 16)) * 0x6A09E667 + self.k1[who]) & M32
        h = ((h ^ (h >> 15)) * 0xBB67AE85) & M32
        return h ^ (h >> 16)

    def start(self, t, who=slice(None)):
        return torch.stack([((self.at(4 * t + j, who) >> 8).double() * 2.0**-24 - 0.5) * float(np.float32(0.1)) for j in range(4)])


def _step64(z, push):
    x, xd, th, thd = z
    f32 = lambda v: float(np.float32(v))  # noqa: E731  the constants are float32 numbers
    force = torch.where(push, 10.0, -10.0).double()
    s, c = torch.sin(th), torch.cos(th)
    temp = (force + f32(0.05) * thd * thd * s) / f32(1.1)
    thacc = (f32(9.8) * s - c * temp) / (0.5 * (f32(4 / 3) - f32(0.1) * c * c / f32(1.1)))
    xacc = temp - f32(0.05) * thacc * c / f32(1.1)
    tau = f32(0.02)
    new = torch.stack([x + tau * xd, xd + tau * xacc, th + tau * thd, thd + tau * thacc])
    return new, (new[0].abs() > f32(2.4)) | (new[2].abs() > f32(12 * 2 * math.pi / 360))


def _layer(v, w, b, rows):
    return [sum((w[r * len(v) + i] * v[i] for i in range(len(v))), b[r]) for r in range(rows)]


def _push64(case, w, z):
    if case["policy"] == "per_env":
        l0, l1 = (sum((w[4 * r + i] * z[i] for i in range(4)), w[8 + r]) for r in (0, 1))
    else:
        w = [float(v) for v in w]
        v, sizes = list(z), {"linear": [4], "mlp16": [4, 16], "mlp32": [4, 32], "mlp64": [4, 64], "deep": [4, 16, 16]}[case["policy"]]
        at = 0
        for k, size in enumerate(sizes):
            rows = sizes[k + 1] if k + 1 < len(sizes) else 2
            v = _layer(v, w[at:at + rows * size], w[at + rows * size:at + rows * size + rows], rows)
            at += rows * size + rows
            if k + 1 < len(sizes):
                v = [torch.tanh(u) for u in v]
        l0, l1 = v
    return l1 > l0


def _packed(mask):
    n = mask.numel()
    m = torch.zeros(_words(n) * 32, dtype=torch.int64, device=mask.device)
    m[:n] = mask
    v = (m.reshape(-1, 32) << torch.arange(32, device=mask.device)).sum(1)
    return torch.where(v >= 2**31, v - 2**32, v).to(torch.int32)


def exact(case, seed):
    n, T = case["n"], case.get("T", 1)
    if "policy" in case and n * T * _cost(case["policy"]) * (3 if case["outputs"] == "full" else 1) > 5e11:
        return None
    # the inputs are the ones of prepare(), so they are made where it makes them
    d = _data(case, seed, DEVICE)
    act, res = _Stream(d["seed"], 0, n, DEVICE), _Stream(d["seed"], 1, n, DEVICE)
    z = d["planes"].double() if "planes" in d else res.start(0)
    limit = case.get("limit", 0)
    carried = d["ep_len"].to(torch.int64) if "ep_len" in d else torch.zeros(n, dtype=torch.int64, device=DEVICE)
    length = carried.clone()
    ret = torch.zeros(n, dtype=torch.float64, device=DEVICE)
    count = torch.zeros(n, dtype=torch.int32, device=DEVICE)
    lane = torch.arange(32, device=DEVICE)
    rows = {"done_bits": [], "action_bits": [], "trajectory": []}
    want = OUTPUTS[case["outputs"]] if "outputs" in case else ()
    for k in range(T):
        t = d["t0"] + k
        if "action" in d:
            push = d["action"] != 0
        elif "bits" in d:
            push = (((d["bits"][k].to(torch.int64) & M32).unsqueeze(1) >> lane) & 1).reshape(-1)[:n] != 0
        elif case.get("policy", "random") == "random":
            push = (act.at(t) >> 31) != 0
        else:
            push = _push64(case, d["weights"].double() if case["policy"] == "per_env" else d["weights"], z)
        z, done = _step64(z, push)
        length += 1
        if limit:
            done = done | (length >= limit)
        who = done.nonzero().squeeze(1)
        z[:, who] = d["starts"][k][:, who].double() if "starts" in d else res.start(t + 1, who)
        ret[who] += length[who].double()
        count[who] += 1
        length[who] = 0
        if "done_bits" in want:
            rows["done_bits"].append(_packed(done))
        if "action_bits" in want:
            rows["action_bits"].append(_packed(push))
        if "trajectory" in want:
            rows["trajectory"].append(z.clone())
    ones = torch.ones(n, dtype=torch.float64, device=DEVICE)
    if case["kind"] in ("step", "loop", "host"):
        if case["kind"] == "step" and case["aligned"]:
            z = torch.cat([z, torch.zeros(4, -n % 4, dtype=z.dtype, device=DEVICE)], 1)
        out = (z, ones, done.to(torch.uint8))
        return (*out, length.to(torch.int32)) if limit else out
    r = {"ep_return_sum": ret, "ep_count": count, "totals": torch.stack([ret.sum().long(), count.sum().long()])}
    for key in want:
        r[key] = ones.expand(T, n) if key == "reward_stream" else torch.stack(rows[key])
    if case["kind"] == "rollout":
        return {**r, "final_state": z}
    return {**r, "planes": z, "ep_len": length.to(torch.int32)}
