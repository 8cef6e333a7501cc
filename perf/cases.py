"""Performance cases: what programs that use this library have it do, through the public entry points of the binding.

A policy server loads a base model and a drafter once and then samples action chunks for new observations: one
environment at a time in a control loop, a batch of parallel environments, or a queue of requests worked through a
fixed number of slots.  A case names one of the workload shapes of `paper_2512_15773_b200.inputs`, how many
environments a call serves and how it drafts; the observations and the noise of a state follow from its seed, the
weights are those of the policy and stay.  Weights are seeded random numbers of the documented distribution (there are
no trained checkpoints); deep transformers repeat two seeded blocks, which leaves sizes and value ranges as they are.
"""
import functools

import numpy as np
import torch

from paper_2512_15773_b200 import binding, inputs

SAMPLE, HOST, QUEUE = "sample", "host", "queue"


def _case(name, workload, batch, K, drafter="network", call=SAMPLE, requests=0, schedule=False):
    """One case.  batch: environments of a call, or slots of a queue; K: drafted steps per round, 0: every reverse
    step by the base model alone; schedule: K and the acceptance width of each round from the seeded Markov chain."""
    c = dict(workload=workload, batch=batch, K=K, drafter=drafter, call=call, requests=requests or batch, schedule=schedule)
    return dict(c, name=name) if name else c


def listed():
    return [
        # fp32 MLP policy: the smallest call there is, a chain of tiny launches
        _case("toy_mlp_b1", "toy_mlp", 1, 4),
        # one robot: observation and chunk in host memory, the time of the call is the control latency
        _case("pusht_b1_host", "pusht_xfmr", 1, 8, call=HOST),
        # evaluation of the same policy over a handful of parallel environments, short windows
        _case("pusht_b24", "pusht_xfmr", 24, 4),
        # conv-UNet policy on visual features: one robot, and a batch of simulators
        _case("robomimic_b1", "robomimic_unet", 1, 8),
        _case("robomimic_b32", "robomimic_unet", 32, 8),
        # the same batch without a drafter network (base output of the round's start reused), an odd batch
        _case("robomimic_b21_frozen", "robomimic_unet", 21, 8, drafter="frozen"),
        # batched serving, K and acceptance width scheduled per round: a small, and the full batch
        _case("serving_b32", "serving_xfmr", 32, 10, schedule=True),
        _case("serving_b256", "serving_xfmr", 256, 10, schedule=True),
        # continuous batching: requests queue for slots, a finished slot takes the next one
        _case("serving_queue_n600", "serving_xfmr", 150, 10, call=QUEUE, requests=600, schedule=True),
        # plain DDPM sampling with the base model alone
        _case("serving_b96_vanilla", "serving_xfmr", 96, 0),
        # VLA-scale action expert with 256 context tokens: a few robots, and a fleet
        _case("vla_b3", "vla_dit", 3, 16),
        _case("vla_b64", "vla_dit", 64, 16),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(lo * (hi / lo) ** rng.random())))


def draw(rng):
    """Another call of the same kinds; batch sizes spread over the logarithm of each workload's range."""
    kind = rng.choice(("toy_mlp", "pusht_xfmr", "robomimic_unet", "serving_xfmr", "serving_xfmr", "vla_dit"))
    drafter = rng.choice(("network", "network", "frozen"))
    if kind == "toy_mlp":
        return _case(None, kind, _log_int(rng, 1, 64), rng.randint(2, 6))
    if kind == "pusht_xfmr":
        return _case(None, kind, _log_int(rng, 1, 64), rng.randint(2, 8), call=rng.choice((SAMPLE, HOST)))
    if kind == "robomimic_unet":
        return _case(None, kind, _log_int(rng, 1, 32), rng.randint(0, 8), drafter)
    if kind == "vla_dit":
        return _case(None, kind, _log_int(rng, 1, 48), rng.randint(4, 16), drafter)
    batch = _log_int(rng, 1, 256)
    if rng.random() < 0.3:
        return _case(None, kind, batch, 10, call=QUEUE, requests=batch * 2 + rng.randint(0, batch), schedule=True)
    if rng.random() < 0.3:
        return _case(None, kind, batch, rng.randint(0, 8), drafter)
    return _case(None, kind, batch, 10, schedule=True)


def _net(wl, which, seed):
    n = wl[which]
    if n["arch"] not in ("xfmr", "dit") or n["layers"] <= 2:
        return inputs.make_net(seed, wl, which)
    p = inputs.make_net(seed, dict(wl, **{which: dict(n, layers=2)}), which)
    p["layers"] = [p["layers"][i % 2] for i in range(n["layers"])]
    return p


@functools.lru_cache(maxsize=8)
def _weights(workload, which):
    wl = inputs.WORKLOADS[workload]
    return binding.pack_weights(_net(wl, which, 1 if which == "base" else 2))


@functools.lru_cache(maxsize=2)
def _policy(workload, batch, K, drafter, schedule):
    """The handle of a policy server: loaded once, used for every call."""
    wl = inputs.WORKLOADS[workload]
    draft = dict(arch="frozen") if drafter == "frozen" else wl["draft"]
    cfg = binding.make_config(wl["H"], wl["A"], wl["To"], wl["Do"], wl["base"], draft, T=wl["T"], max_B=batch, max_K=max(K, 1),
                              precision=wl["precision"])
    policy = binding.Sampler(cfg)
    policy.load_weights(binding.BASE, _weights(workload, "base"))
    if drafter != "frozen":
        policy.load_weights(binding.DRAFT, _weights(workload, "draft"))
    if schedule:
        Ks, scales = inputs.markov_schedule(0, 512)
        policy.set_schedule(Ks, [binding.AcceptT(0, 1.0, s, 1) for s in scales])
    return policy


def prepare(case, seed):
    wl = inputs.WORKLOADS[case["workload"]]
    n = case["requests"]
    host = case["call"] == HOST
    g = torch.Generator(device="cuda").manual_seed(seed)
    obs = torch.randn(n, wl["To"], wl["Do"], generator=g, device="cuda")
    out = torch.zeros(n, wl["H"], wl["A"], device="cuda")
    if host:
        obs, out = (t.cpu().pin_memory().numpy() for t in (obs, out))
    return dict(case=case, seed=seed, obs=obs, out=out, accept=binding.AcceptT(0, 1.0, 1.0, 1),
                policy=_policy(case["workload"], case["batch"], case["K"], case["drafter"], case["schedule"]))


def run(state):
    c, policy, out = state["case"], state["policy"], state["out"]
    if c["call"] == HOST:
        policy.sample_chunk_host(state["obs"], c["batch"], c["K"], state["accept"], state["seed"], out)
    elif c["call"] == QUEUE:
        policy.serve(state["obs"], c["requests"], c["batch"], c["K"], state["accept"], state["seed"], out)
    else:
        policy.sample_chunk(state["obs"], c["batch"], c["K"], state["accept"], state["seed"], out)
    return out


def _forward_flops(wl, net):
    """Multiply-adds times two of one forward on one latent: what the layers need at least (the query and output
    projections of the decoder's short cross-attention can be applied to its memory tokens and are not counted)."""
    H, D, d = wl["H"], wl["H"] * wl["A"], net.get("d", 0)
    if net["arch"] == "mlp":
        dims = [D + 32 + wl["To"] * wl["Do"]] + [net["width"]] * net["layers"] + [D]
        return 2 * sum(a * b for a, b in zip(dims, dims[1:]))
    if net["arch"] == "xfmr":
        return 2 * H * (net["layers"] * (12 * d * d + H * d) + 2 * wl["A"] * d)
    if net["arch"] == "dit":
        return 2 * H * (net["layers"] * (14 * d * d + 2 * H * d + 2 * wl["To"] * d) + 2 * wl["A"] * d)
    if net["arch"] == "unet":
        levels, total = net["layers"], 2 * H * wl["A"] * d + 5 * H * d * d
        order = [lv for lv in range(levels) for _ in (0, 1)] + [levels - 1] * 2 + [lv for lv in range(levels - 2, -1, -1) for _ in (0, 1)]
        for (cin, cout), lv in zip(inputs.unet_block_channels(d, levels), order):
            total += (H >> lv) * (5 * cin * cout + 5 * cout * cout + (cin * cout if cin != cout else 0))
        return 2 * total
    return 0


def work(case):
    """Every reverse step of every chunk takes one base evaluation, and a drafter evaluation where it was drafted:
    K of K + 1 steps at best (5.5 drafted steps per round on average under the schedule).  Weights are read once."""
    wl = inputs.WORKLOADS[case["workload"]]
    K = 5.5 if case["schedule"] else case["K"]
    flops = _forward_flops(wl, wl["base"])
    size = 4 if wl["precision"] == 0 else 2
    nbytes = size * _weights(case["workload"], "base").size
    if case["drafter"] == "frozen":
        flops *= 1 + (1 / (K + 1) if K else 0)
    elif K:
        flops += K / (K + 1) * _forward_flops(wl, wl["draft"])
        nbytes += size * _weights(case["workload"], "draft").size
    chunk = wl["H"] * wl["A"] + wl["To"] * wl["Do"]
    once = sum(4 * wl["To"] * n["d"] * n["d"] * n["layers"] for n in (wl["base"], wl["draft"])
               if n["arch"] == "dit" and not (n is wl["draft"] and case["drafter"] == "frozen"))      # context keys and values
    return dict(bytes=nbytes + 4 * case["requests"] * chunk, flops=case["requests"] * (wl["T"] * flops + once))


def tolerance(case):
    """A chunk moves by 1e-4 of its norm when the sums of a bf16 forward change their order (fp32: 1e-6), four times the
    largest seen is stated where no decision is taken.  Where drafts are accepted or rejected, such a change also turns
    decisions that sit on their threshold: in 1 % of the chunks with a drafter network, in 7 % with the base output
    reused (their test statistic is close to zero), and a chunk that took one differently moves by up to 4.5 % of its
    norm at 32 latent values, 1 / sqrt(values) of that beyond."""
    wl = inputs.WORKLOADS[case["workload"]]
    if wl["precision"] == 0:
        return {"rel": 1e-4, "max": 1e-2}
    if case["K"] == 0:
        return {"rel": 1.2e-3, "max": 1e-2}
    turned = (0.07 if case["drafter"] == "frozen" else 0.013) * case["requests"]
    one = 0.045 * (32 / (wl["H"] * wl["A"])) ** 0.5
    return {"rel": min(0.03, 4 * one * (max(turned, 1.0) / case["requests"]) ** 0.5), "max": 0.9}
