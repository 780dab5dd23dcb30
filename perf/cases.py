"""What is timed of this library: rollout steps, buffer fills, GAE with minibatch gathers, and whole TrainPPO calls.

A case names a kind of call, the frames and the network it runs on, and the sizes of the rollout.  The kinds are the
parts of Algorithm 2 as a user's program makes them through `Learner` and the buffer calls:

  act     one rollout step of all envs: observation into the buffer, actions <- pi(obs), outcome into the buffer
          (a recurrent policy acts through `Learner.act`, which carries its state, and resets it where an env is done)
  fill    D <- D U {...} for a whole horizon of device arrays
  buffer  GAE, advantage normalisation and every minibatch gather of one epoch, without a network
  train   one TrainPPO call: GAE, then gather -> forward -> loss -> backward -> Adam for every minibatch
"""
import math

import torch

from paper_2509_16434_b200 import binding as ppo
from paper_2509_16434_b200 import synth
from paper_2509_16434_b200.learner import Learner


def _texts(seq):
    return "-".join(str(v) for v in seq)


def _numbers(text):
    return tuple(int(v) for v in text.split("-"))


def _case(kind, w, microbatch=4096):
    return {"kind": kind, "N": w.N, "T": w.T, "H": w.H, "W": w.W, "conv_c": _texts(w.conv_c), "conv_k": _texts(w.conv_k),
            "fc": _texts(w.fc), "epochs": w.epochs, "minibatches": w.minibatches, "done_rate": w.done_rate, "P": w.P, "A": w.A,
            "norm": w.norm, "embed": w.embed, "n_lstm": w.n_lstm, "lstm_h": w.lstm_h, "microbatch": microbatch}


def _workload(case):
    return synth.Workload("case", case["N"], case["T"], case["H"], case["W"], _numbers(case["conv_c"]), _numbers(case["conv_k"]),
                          _numbers(case["fc"]), case["epochs"], case["minibatches"], case["done_rate"], case["P"], case["A"],
                          norm=case["norm"], embed=case["embed"], n_lstm=case["n_lstm"], lstm_h=case["lstm_h"])


# frames, channel counts and joint/action counts that are no round numbers: 90 x 122 pixels, 6000 samples, 7 actions
_ODD = synth.Workload("odd", 300, 20, 90, 122, (16, 32, 96), (5, 3, 3), (200, 120), 1, 3, P=24, A=7)


def listed():
    W = synth.WORKLOADS
    named = [
        # the paper's recurrent policy on a handful of envs (evaluation, the deployed gripper): latency of one decision
        ("act_policy_16", _case("act", W["paper_policy"].scaled(16))),
        # the same policy driving a simulator GPU's envs
        ("act_policy_512", _case("act", W["paper_policy"].scaled(512))),
        # feed-forward policy, the rollout step bench.py times beside its main line
        ("act_cfg2_1024", _case("act", W["cfg2"])),
        # the rollout of a simulator that hands over whole device arrays
        ("fill_cfg2", _case("fill", W["cfg2"])),
        # frames whose byte count is no multiple of 16, a horizon that is no power of two
        ("buffer_odd", _case("buffer", _ODD.scaled(1005))),
        # the bandwidth stress configuration, 4096 envs x 32 steps
        ("buffer_4k", _case("buffer", W["cfg5_4k"])),
        # smallest configuration: 4 minibatches of 1024 rows of 64 x 64, where launches and host time count
        ("train_cfg1", _case("train", W["cfg1"])),
        # ragged sizes, micro-batches that do not divide the minibatch of 2000 rows
        ("train_odd", _case("train", _ODD, 1024)),
        # ordinary size: 4 minibatches of 4096 rows of 160 x 120
        ("train_cfg2", _case("train", W["cfg2"])),
        # the largest network and frames at an eighth of the envs and one epoch: the same 4096-row micro-batches
        ("train_cfg4", _case("train", W["cfg4"].scaled(1024, epochs=1, minibatches=4))),
        # the paper's depth CNN (layer normalisation, 32-d embedding), and its whole recurrent policy on sequences
        ("train_paper_cnn", _case("train", W["paper_cnn"])),
        ("train_paper_policy", _case("train", W["paper_policy"])),
    ]
    return [dict(c, name=n) for n, c in named]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same ranges: families of networks on frames from 48 x 64 to 240 x 320, 16 to 4096 envs."""
    kind = rng.choice(["act", "act", "fill", "buffer", "train", "train", "train", "train"])
    family = rng.choice(["plain", "plain", "norm", "recurrent"])
    H = _log_int(rng, 48, 240)
    W = 2 * int(round(H * rng.uniform(1.2, 1.4) / 2))
    if family == "plain":
        depth = rng.choice([3, 4, 5])
        conv_c = [rng.choice([16, 32]), rng.choice([32, 48, 64]), rng.choice([64, 96, 128]), rng.choice([128, 192, 256]), 256][:depth]
        conv_k = [rng.choice([3, 5])] + [3] * (depth - 1)
        embed, P = 0, rng.choice([16, 24, 32, 40])
    else:
        conv_c, conv_k, embed, P = [16, 32, 64, 128], [3, 3, 3, 3], 32, 32
    fc = [rng.choice([120, 200, 256, 384, 512]) for _ in range(rng.choice([1, 2, 3]))]
    lstm = (rng.choice([1, 2]), rng.choice([256, 512, 1024])) if family == "recurrent" else (0, 0)
    T = rng.choice([8, 12, 16, 16, 20, 24, 32])
    minibatches = rng.choice([2, 3, 4])
    N = _log_int(rng, 16, 2048) if kind == "act" else _log_int(rng, 64, 4096)
    N = max(minibatches, N // minibatches * minibatches)
    w = synth.Workload("drawn", N, T, H, W, conv_c, conv_k, fc, 1, minibatches, rng.choice([0.0, 0.005, 0.01, 0.05]), P, rng.randint(4, 14),
                       norm=family != "plain", embed=embed, n_lstm=lstm[0], lstm_h=lstm[1])
    most = max((work(c) for c in listed() if c["kind"] == kind), key=lambda v: v["flops"] + 100 * v["bytes"])
    case = _case(kind, w, rng.choice([1024, 2048, 4096]))
    while case["N"] > minibatches and any(work(case)[k] > most[k] for k in most):
        case["N"] = max(minibatches, case["N"] * 4 // 5 // minibatches * minibatches)
    return case


def _make_learner(w, case, device, seed):
    L = Learner(w, case["microbatch"], device)
    shapes, gammas = synth.param_shapes(w)
    offsets = [o for o, _ in L.model.tensors()]
    L.model.load(synth.init_params(L.model.arena, offsets, shapes, seed, ones=gammas))
    return L


def prepare(case, seed):
    device = "cuda"
    w = _workload(case)
    kind = case["kind"]
    one_step = kind == "act"
    r = synth.rollout_torch(w.scaled(w.N, T=1) if one_step else w, device, seed)
    state = {"kind": kind, "w": w, "roll": r}
    if kind == "act":
        state["L"] = L = _make_learner(w.scaled(w.N, T=2, minibatches=1), case, device, seed)
        if L.recurrent:
            L.reset_rollout_state(w.N)
        return state
    action = r["eps"]
    logp = r["logp_jitter"] - 0.5 * (w.A * math.log(2 * math.pi) + (action * action).sum(-1))
    if kind == "train":  # actions and old log-probs of the policy itself, on the frames it saw
        state["L"] = L = _make_learner(w, case, device, seed)
        if not L.recurrent:
            mean = torch.cat([L.act(r["depth"][t], r["proprio"][t], r["eps"][t])[0] for t in range(w.T)])
            action = mean.view(w.T, w.N, w.A)
        L.write_rollout(r, action, logp)
        state["last_value"] = r["last_value"]
        del state["roll"]
        return state
    desc = ppo.buffer_desc(w.N, w.T, w.H, w.W, w.P, w.A)
    state["buffer"] = ppo.Buffer(desc, device)
    state["action"], state["logp"] = action, logp
    if kind == "buffer":
        for t in range(w.T):
            ppo.ppo_buffer_write_step(state["buffer"], t, r["depth"][t], r["proprio"][t], action[t], logp[t], r["value"][t],
                                      r["reward"][t], r["done"][t])
        state["mbs"] = [ppo.MinibatchArrays(desc, w.B, device) for _ in range(w.minibatches)]
        state["stats"] = torch.zeros(2, device=device)
        state["last_value"] = r["last_value"]
        del state["roll"]
    return state


def _fields(buf, *which):
    return [buf.field(f) for f in which]


def _run_act(state):
    L, r, w = state["L"], state["roll"], state["w"]
    depth, proprio, eps = r["depth"][0], r["proprio"][0], r["eps"][0]
    if L.recurrent:
        out = L.act(depth, proprio, eps)
        L.reset_rollout_state(w.N, r["done"][0])
        return list(out) + [L.roll_h, L.roll_c]
    L.act_into_buffer(0, depth, proprio, eps)
    ppo.ppo_buffer_write_outcome(L.buffer, 0, r["reward"][0], r["done"][0])
    return [f[0] for f in _fields(L.buffer, ppo.FIELD_DEPTH, ppo.FIELD_PROPRIO, ppo.FIELD_ACTION, ppo.FIELD_LOGP, ppo.FIELD_VALUE,
                                  ppo.FIELD_REWARD, ppo.FIELD_DONE)]


def _run_fill(state):
    buf, r = state["buffer"], state["roll"]
    for t in range(state["w"].T):
        ppo.ppo_buffer_write_step(buf, t, r["depth"][t], r["proprio"][t], state["action"][t], state["logp"][t], r["value"][t],
                                  r["reward"][t], r["done"][t])
    return _fields(buf, ppo.FIELD_DEPTH, ppo.FIELD_PROPRIO, ppo.FIELD_ACTION, ppo.FIELD_LOGP, ppo.FIELD_VALUE, ppo.FIELD_REWARD,
                   ppo.FIELD_DONE)


def _run_buffer(state):
    buf, w = state["buffer"], state["w"]
    ppo.ppo_compute_gae(buf, state["last_value"], w.gamma, w.lam, True, state["stats"])
    for k, mb in enumerate(state["mbs"]):
        ppo.ppo_shuffle_gather_minibatch(buf, 1, 0, k, w.minibatches, mb)
    out = [state["stats"]] + _fields(buf, ppo.FIELD_ADV, ppo.FIELD_RET)
    for mb in state["mbs"]:
        out += [mb.depth, mb.proprio, mb.action, mb.logp_old, mb.value_old, mb.adv, mb.ret, mb.index]
    return out


def _run_train(state):
    L = state["L"]
    L.train(state["last_value"], seed=1)
    m = L.model
    return [m.master, m.shadow, m.grad, m.adam_m, m.adam_v, L.loss, L.stats] + _fields(L.buffer, ppo.FIELD_ADV, ppo.FIELD_RET)


_RUN = {"act": _run_act, "fill": _run_fill, "buffer": _run_buffer, "train": _run_train}


def run(state):
    return _RUN[state["kind"]](state)


def _macs(w):
    """Multiply-adds of one sample's forward pass: (first convolution, everything else), and the number of weights."""
    first = rest = params = 0
    cin, h, wd = 1, w.H, w.W
    for l, (c, k) in enumerate(zip(w.conv_c, w.conv_k)):
        h, wd = (h + 2 * (k // 2) - k) // 2 + 1, (wd + 2 * (k // 2) - k) // 2 + 1
        n = c * k * k * cin
        first, rest = (first + n * h * wd, rest) if l == 0 else (first, rest + n * h * wd)
        params += n + c
        cin = c
    mats = []
    i = cin + w.P
    if w.embed:
        mats.append((w.embed, h * wd * cin))
        i = w.embed + w.P
    for _ in range(w.n_lstm):
        mats.append((4 * w.lstm_h, i + w.lstm_h))
        i = w.lstm_h
    for o in w.fc:
        mats.append((o, i))
        i = o
    mats.append((w.A + 1, i))
    rest += sum(o * i for o, i in mats)
    params += sum(o * i + o for o, i in mats)
    return first, rest, params


def work(case):
    w = _workload(case)
    first, rest, params = _macs(w)
    obs = 2 * w.H * w.W + 4 * w.P            # a frame and its proprioception
    record = obs + 4 * w.A + 16              # one gathered row: log-prob, value, advantage and return beside the action
    gae = 21 * w.M                           # reward, value, done read; advantage, return written; one normalising write
    kind = case["kind"]
    if kind == "act":
        state = 16 * w.n_lstm * w.lstm_h     # h and c in and out
        into = 0 if w.n_lstm else obs + 10   # the observation and outcome copied into the buffer
        return {"bytes": w.N * (obs + into + 8 * w.A + 8 + state) + 2 * params, "flops": 2 * w.N * (first + rest)}
    if kind == "fill":
        return {"bytes": 2 * w.M * (record - 3), "flops": 0}
    if kind == "buffer":
        return {"bytes": gae + w.M * (2 * record + 4), "flops": 10 * w.M}
    # every sample once per epoch, and the parameters with their moments once per minibatch; the backward pass costs
    # twice the forward one, less the input gradient of the first convolution
    return {"bytes": gae + w.epochs * (w.M * record + 30 * params * w.minibatches), "flops": w.epochs * w.M * (4 * first + 6 * rest)}


def tolerance(case):
    if case["kind"] == "fill":
        return "exact"
    if case["kind"] == "buffer":  # fp32 scan; the gathered rows are copies
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 1e-2}  # bf16 operands, fp32 sums; for train also through the Adam steps of one call
