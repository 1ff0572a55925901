"""Performance cases of the NetMax round simulator: what its users have it do, through the Python binding.

Five kinds of work cover the framework:
  rounds   synchronous rounds on a context that lives on the GPU (netmax_round), then the telemetry and the replicas
           they produced; with "refresh", the links have changed and the policy is generated again first;
  async    the paper's own process, one worker per global step on simulated clocks (netmax_async_steps), then the loss;
  host     a whole step through host buffers: replicas and centres in, rounds, replicas out (netmax_round_from_host);
  policy   the communication policy for new link speeds (Algorithm 3), installed in a context (netmax_set_policy);
  draws    peer draws alone, the sampler stress (netmax_sample_peers).

Sizes are those of `paper_2009_05766_b200.workloads` (ResNet18- and VGG19-sized vectors, the small and the sampling
configurations) and the ranges around them that the tests cover.
"""
import math

import numpy as np
import torch

from paper_2009_05766_b200 import binding, workloads

RESNET18 = workloads.config(2).d      # 11,173,962 parameters
VGG19 = workloads.config(3).d         # 20,000,000

# the largest work of one pass that draw() may give (workers x parameters, and that times rounds or steps)
MAX_ELEMENTS = 64 * RESNET18
MAX_UPDATES = 10 * MAX_ELEMENTS


def rounds_case(M, d, rounds, storage="f32", objective=1, pull_weight=0.0, refresh=False):
    return {"kind": "rounds", "M": M, "d": d, "rounds": rounds, "storage": storage, "objective": objective,
            "pull_weight": pull_weight, "refresh": refresh}


def listed():
    c1, c2, c3, c4, c5 = (workloads.config(k) for k in range(1, 6))
    return [
        # the smallest call: a program that looks at every round of a four-worker toy problem (launches and latency)
        dict(rounds_case(c1.M, c1.d, 1), name="toy_one_round"),
        # the same problem run to its end in one call
        dict(rounds_case(c1.M, c1.d, c1.rounds), name="toy_500_rounds"),
        # the headline: ResNet18-sized vectors on 8 workers, twenty rounds between looks at the loss
        dict(rounds_case(c2.M, RESNET18, 20), name="resnet18_8"),
        # the same with bfloat16 replicas
        dict(rounds_case(c2.M, RESNET18, 20, storage="bf16"), name="resnet18_8_bf16"),
        # VGG19-sized vectors on 16 workers in a dynamic network: links change every twenty rounds, policy generated again
        dict(rounds_case(c3.M, VGG19, c3.policy_period, refresh=True), name="vgg19_16_refresh"),
        # the largest state: 64 ResNet18-sized replicas
        dict(rounds_case(c4.M, RESNET18, 10), name="resnet18_64"),
        # very many workers with short vectors
        dict(rounds_case(c5.M, c5.d, 1000), name="sampling_4096"),
        # an in-between size with nothing round about it
        dict(rounds_case(93, 200_003, 25, storage="bf16"), name="ragged_93_bf16"),
        # the asynchronous timeline on ResNet18-sized vectors
        {"kind": "async", "M": c2.M, "d": RESNET18, "steps": 128, "storage": "f32", "name": "async_resnet18_8"},
        # one round per step through pinned host buffers (replicas held by the caller's own trainer)
        {"kind": "host", "M": c2.M, "d": RESNET18, "rounds": 1, "storage": "f32", "name": "host_resnet18_8"},
        # Algorithm 3 for the largest network
        {"kind": "policy", "M": c5.M, "K": c5.K, "name": "policy_4096"},
        # peer draws alone for the largest network
        {"kind": "draws", "M": c5.M, "rounds": 1024, "name": "draws_4096"},
    ]


def _log(rng, lo, hi):
    """A whole number from [lo, hi], uniform over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choices(["rounds", "async", "host", "policy", "draws"], weights=[11, 2, 2, 3, 2])[0]
    if kind == "rounds":
        refresh = rng.random() < 0.15
        M = _log(rng, 2, 64 if refresh else 4096)
        d = max(1, _log(rng, max(1 << 13, 2 * M), MAX_ELEMENTS) // M)
        rounds = _log(rng, 1, max(1, min(1000, MAX_UPDATES // (M * d))))
        return rounds_case(M, d, rounds, storage="bf16" if rng.random() < 0.25 else "f32",
                           objective=0 if rng.random() < 0.1 else 1, pull_weight=0.5 if not refresh and rng.random() < 0.15 else 0.0,
                           refresh=refresh)
    if kind == "async":     # the paper's 4 to 16 workers and some more
        M = _log(rng, 2, 64)
        d = _log(rng, 1 << 13, 8 * RESNET18) // M
        return {"kind": "async", "M": M, "d": d, "steps": _log(rng, 16, max(16, min(2000, 128 * RESNET18 // d))),
                "storage": "bf16" if rng.random() < 0.25 else "f32"}
    if kind == "host":
        M = _log(rng, 2, 64)
        return {"kind": "host", "M": M, "d": _log(rng, 1 << 16, 8 * RESNET18) // M, "rounds": _log(rng, 1, 8),
                "storage": "bf16" if rng.random() < 0.25 else "f32"}
    if kind == "policy":
        M = _log(rng, 4, 4096)
        return {"kind": "policy", "M": M, "K": 20 if M <= 64 else 8}
    M = _log(rng, 4, 4096)
    return {"kind": "draws", "M": M, "rounds": _log(rng, 16, min(4096, (1 << 22) // M))}


def _link_speeds(M, seed):
    """Heterogeneous symmetric links, log-uniform over 1 to 100 Gbps."""
    rng = np.random.default_rng([seed, 3])
    s = np.exp(rng.uniform(0.0, math.log(100.0), (M, M)))
    s = np.triu(s, 1)
    return s + s.T


def prepare(case, seed):
    kind, M = case["kind"], case["M"]
    d = case.get("d", 1024)
    storage = case.get("storage", "f32")
    speeds = _link_speeds(M, seed)
    # a policy that prefers fast links and never starves slow ones
    P = 0.5 * speeds / speeds.sum(axis=1, keepdims=True) + 0.5 / (M - 1)
    np.fill_diagonal(P, 0.0)
    P /= P.sum(axis=1, keepdims=True)
    ring = 1024
    long_vectors = d > 100_000
    std, sigma, lr = (0.01, 0.01, 0.1) if long_vectors else (1.0, 0.1, 0.05)
    size = binding.Netmax.workspace_size(M, d, ring, storage)
    workspace = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
    base = (workspace.data_ptr() + 255) // 256 * 256
    K = case.get("K", 20)
    sim = binding.Netmax(M=M, d=d, lr=lr, link_speed_gbps=speeds, prob=P, sigma=sigma, x0_std=std, c_std=std,
                         objective=case.get("objective", 1), seed=seed, trace_rounds=ring, policy_K=K, policy_R=K,
                         pull_weight=case.get("pull_weight", 0.0), storage=storage, workspace=base, workspace_bytes=size)
    state = {"case": case, "sim": sim, "workspace": workspace}
    if kind == "policy" or case.get("refresh"):
        state["new_links"] = _link_speeds(M, seed + 1_000_003)
    if kind == "async":
        sim.async_begin(None, beta=0.9)
    if kind == "host":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        state["x"], state["c"] = (torch.empty((M, d), dtype=torch.float32, pin_memory=True) for _ in range(2))
        for t in (state["x"], state["c"]):
            t.copy_(torch.randn((M, d), generator=gen, device="cuda").mul_(std))
        state["out"] = torch.empty((M, d), dtype=torch.float32, pin_memory=True)
    if kind == "draws":
        state["peers"] = torch.empty((case["rounds"], M), dtype=torch.int32, device="cuda")
        state["first"] = 0
    return state


def _replicas_on_device(state):
    """The current replicas as a tensor over the context's own memory."""
    case, sim, workspace = state["case"], state["sim"], state["workspace"]
    ptr, ld = sim.replicas_device()
    dtype, width = (torch.bfloat16, 2) if case["storage"] == "bf16" else (torch.float32, 4)
    at = ptr - workspace.data_ptr()
    rows = workspace[at: at + case["M"] * ld * width].view(dtype).view(case["M"], ld)
    return rows[:, : case["d"]]


def run(state):
    case, sim = state["case"], state["sim"]
    kind = case["kind"]
    if kind == "rounds":
        out = {}
        if case["refresh"]:
            sim.set_policy(link_speed_gbps=state["new_links"])
            out["P"], out["rho"] = sim.get_policy()
        sim.round(case["rounds"])
        first = sim.rounds_done - case["rounds"]
        out["consensus"], out["loss"] = sim.telemetry(first, case["rounds"])
        if case["M"] * case["d"] <= 1 << 20:    # small problems are looked at on the host
            out["peers"] = sim.peer_trace(first, case["rounds"])
            out["x"] = sim.read_replicas()
        else:
            out["x"] = _replicas_on_device(state)
        return out
    if kind == "async":
        sim.async_steps(case["steps"])
        now, done = sim.async_time()
        worker, peer, _, finish = sim.async_trace(done - case["steps"], case["steps"])
        consensus, loss = sim.measure()
        return {"now": now, "worker": worker, "peer": peer, "finish": finish, "consensus": consensus, "loss": loss,
                "x": _replicas_on_device(state)}
    if kind == "host":
        sim.round_from_host(state["x"].data_ptr(), state["c"].data_ptr(), case["rounds"], state["out"].data_ptr())
        return state["out"]
    if kind == "policy":
        sim.set_policy(link_speed_gbps=state["new_links"])
        P, rho = sim.get_policy()
        return {"P": P, "rho": rho}
    sim.sample_peers(state["first"], case["rounds"], state["peers"].data_ptr())
    state["first"] += case["rounds"]
    return state["peers"]


# floating-point operations of one element's update: noise 4, Eq. 15 and Eq. 16 8, telemetry 6
UPDATE_FLOPS = 18


def work(case):
    kind, M = case["kind"], case["M"]
    if kind == "draws":     # every threshold row read once, every draw written once
        return {"bytes": 4 * M * M + 4 * M * case["rounds"], "flops": 0}
    if kind == "policy":    # speeds in, P out; per grid point a row solve and a few products with Y
        return {"bytes": 16 * M * M, "flops": 100 * case["K"] ** 2 * M * M}
    d, width = case["d"], 2 if case["storage"] == "bf16" else 4
    if kind == "async":     # all replicas and centres in, the replicas out; one replica updated per step; then the loss
        return {"bytes": 3 * width * M * d, "flops": (UPDATE_FLOPS - 6) * case["steps"] * d + 6 * M * d}
    if kind == "host":      # fp32 over the host link, whatever the storage
        return {"bytes": 12 * M * d, "flops": UPDATE_FLOPS * case["rounds"] * M * d}
    refresh = 16 * M * M if case["refresh"] else 0
    return {"bytes": 3 * width * M * d + refresh, "flops": UPDATE_FLOPS * case["rounds"] * M * d}


def tolerance(case):
    if case["kind"] == "draws":
        return "exact"
    if case["kind"] == "policy":    # fp64 throughout, iterations settled to 1e-13 and better
        return {"rel": 1e-7}
    if case["storage"] == "bf16":   # an fp32 value next to a rounding boundary may land on the neighbouring bfloat16 code
        return {"rel": 1e-3, "max": 0.02}
    return {"rel": 2e-5}            # fp32 arithmetic on fp32 state; telemetry sums of fp32 partial sums
