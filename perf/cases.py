"""The work that a user of this library has it do, as cases that can be timed and compared.

Three kinds of work: the loss + gradient call for a discrete-action policy (`categorical`) and for a diagonal-Gaussian
one (`gaussian`), the learner's iteration around it (`learner`: ring, first-traversal append, loss, push), and the
ring's own data movement (`replay`: push, draw with gather, minibatches by index).  Sizes come from
`impact_inputs.CONFIGS`, from the tests and from the benchmark's sweep (timesteps from 80 to 4 M, trajectories from one
step to thousands, 1 to 512 actions); inputs follow the recipe of `impact_inputs`, drawn on the device.

How the calls are made is part of a case:
  direct    impact_loss_fwd_bwd with tensors, arguments checked and marshalled on every call
  prepared  prepare_loss_fwd_bwd once, the call re-issued on every pass (a learner loop over fixed buffers)
  graph     prepared calls over several train batches, captured once into a CUDA graph and replayed
"""
from __future__ import annotations

import math

import torch

import paper_1912_00167_b200 as ip
from paper_1912_00167_b200 import binding

FIELDS = ("actions", "rewards", "discounts", "worker_logp", "target_logits")
INPUTS = ("learner_logits", "target_logits", "worker_logp", "actions", "rewards", "discounts", "values",
          "bootstrap_values")
GAUSS_INPUTS = ("learner_mean", "learner_logstd", "target_mean", "target_logstd", "worker_logp", "actions", "rewards",
                "discounts", "values", "bootstrap_values")

# The hyper-parameter sets in use.  `default`: the named configurations (no KL term).  `kl`: the paper's other tables
# (a KL coefficient, rho = 2 in the target-worker clipping, lambda = 0.995, truncation above 1).  `ppo` and `impala`:
# the two baselines that run through the same call.
HYPER = {
    "default": dict(clip_eps=0.4),
    "kl": dict(clip_eps=0.4, kl_coef=1.0, rho_tw=2.0, lam=0.995, rho_bar=1.5, c_bar=1.2),
    "ppo": dict(clip_eps=0.2, is_source=binding.IS_NONE, ratio_mode=binding.RATIO_R2, lam=0.95),
    "impala": dict(objective=binding.OBJECTIVE_VTRACE_PG),
}
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


def listed():
    return [
        # the smallest named configuration, called as a first program would: latency and argument checks are all
        _cat("step tiny", 4, 20, 6, how="direct"),
        # the Atari-shaped configuration: worker batches arrive in pinned host memory, every batch is traversed twice
        dict(name="learner atari", kind="learner", how="direct", B=32, T=50, A=18, N=16, K=2, iterations=1),
        # the large-batch configuration with the ring's bookkeeping on the device: sixteen iterations in one CUDA graph
        dict(name="learner graph", kind="learner", how="graph", B=1024, T=128, A=18, N=32, K=4, iterations=16),
        # the benchmark's loss call on the large-batch configuration, eight train batches to a CUDA graph
        _cat("step large batch", 1024, 128, 18, how="graph", sets=8),
        # a million steps with bf16 storage, short Atari fragments, B that leaves a ragged last tile
        _cat("million steps bf16", 20972, 50, 18, dtype="bf16", grads="bf16"),
        # the largest point of the sweep for a small action set
        _cat("four million steps", 209716, 20, 6),
        # nine actions with every switch and output in use: KL term, value targets and advantages returned
        _cat("kl and targets", 2500, 100, 9, hyper="kl", extras=True),
        # an action set that is none of the Atari ones
        _cat("seven actions", 5243, 50, 7),
        # a wide action set
        _cat("wide actions", 4096, 128, 64),
        # few, very long fragments
        _cat("long fragments", 16, 4096, 18, extras=True),
        # continuous control (the Humanoid-shaped configuration)
        dict(name="continuous", kind="gaussian", how="prepared", B=512, T=128, D=17, hyper="default", extras=False),
        # minibatches out of the ring: a fresh batch pushed, one drawn into the learner's buffers, trajectories
        # shuffled by index; bf16 logits and fragments of 50 steps make rows that are no multiple of 16 bytes
        dict(name="replay minibatches", kind="replay", B=20972, T=50, A=18, dtype="bf16", N=2),
    ]


def _cat(name, B, T, A, how="prepared", dtype="f32", grads="f32", hyper="default", extras=False, sets=1):
    return dict(name=name, kind="categorical", how=how, B=B, T=T, A=A, dtype=dtype, grads=grads, hyper=hyper,
                extras=extras, sets=sets)


_MOST_BYTES = 400e6  # of a drawn case: what the largest listed ones move


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["categorical"] * 6 + ["gaussian"] * 2 + ["learner", "replay"])
    if kind == "learner":
        how = rng.choice(["direct", "graph"])
        T = _log_int(rng, 5, 128)
        steps = _log_int(rng, 80, 4000 if how == "direct" else 131072)
        K = rng.randint(1, 4)
        return dict(kind=kind, how=how, B=max(1, steps // T), T=T, A=rng.choice([4, 6, 9, 18]), N=rng.randint(4, 16),
                    K=K, iterations=1 if how == "direct" else rng.randint(4, 16))
    hyper = rng.choice(["default", "default", "default", "kl", "ppo", "impala"])
    T = _log_int(rng, 1, 4096) if rng.random() < 0.5 else rng.choice([20, 50, 100, 128])
    if kind == "gaussian":
        D = rng.choice([3, 6, 17]) if rng.random() < 0.6 else _log_int(rng, 1, 64)
        case = dict(kind=kind, how="prepared", D=D, hyper=hyper, extras=rng.random() < 0.3)
        per_step = 4 * (7 * D + 6)
    else:
        A = rng.choice([4, 6, 9, 18, 18, 64]) if rng.random() < 0.6 else _log_int(rng, 2, 512)
        dtype = rng.choice(["f32", "f32", "bf16"])
        if kind == "replay":
            case = dict(kind=kind, A=min(A, 64), dtype=dtype, N=rng.randint(2, 4))
            per_step = 200 if A <= 18 else 1000
        else:
            case = dict(kind=kind, how=rng.choice(["direct", "prepared", "prepared"]), A=A, dtype=dtype,
                        grads=rng.choice(["f32", dtype]), hyper=hyper, extras=rng.random() < 0.3, sets=1)
            per_step = 12 * A + 24
    steps = _log_int(rng, 80, max(80, int(min(4.2e6, 0.9 * _MOST_BYTES / per_step))))
    case.update(B=max(1, steps // T), T=T)
    return case


# ---- inputs -----------------------------------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _near_the_clip(l_theta, l_target, worker_logp, coef):
    """Steps whose likelihood ratio lies so close to a clip bound that two correct fp32 programs could decide
    differently; the generators below move them off the bound."""
    if coef.ratio_mode == binding.RATIO_R2:
        base = worker_logp.double()
    else:
        base = torch.maximum(l_target, worker_logp.double() - math.log(coef.rho_tw))
    ratio = torch.exp(l_theta - base)
    near = torch.zeros_like(ratio, dtype=torch.bool)
    for bound in (1.0 - coef.clip_eps, 1.0 + coef.clip_eps):
        near |= (ratio / bound - 1.0).abs() < 1e-4
    return near


def _rewards_and_values(g, B, T, sparse, p_done):
    u = torch.rand(B, T, device="cuda", generator=g)
    if sparse:
        rewards = torch.where(u < 0.05, torch.where(u < 0.025, -1.0, 1.0), 0.0)
    else:
        rewards = torch.randn(B, T, device="cuda", generator=g)
    done = torch.rand(B, T, device="cuda", generator=g) < p_done
    return dict(rewards=rewards.float(), discounts=torch.where(done, 0.0, 0.99).float(),
                values=torch.randn(B, T, device="cuda", generator=g),
                bootstrap_values=torch.randn(B, device="cuda", generator=g))


def _categorical_inputs(g, B, T, A, dtype, coef):
    learner = torch.randn(B, T, A, device="cuda", generator=g)
    target = learner + 0.1 * torch.randn(B, T, A, device="cuda", generator=g)
    worker = learner + 0.5 * torch.randn(B, T, A, device="cuda", generator=g)
    logp = torch.log_softmax(worker, -1)
    race = torch.empty_like(worker).exponential_(generator=g).log_()
    actions = (logp - race).argmax(-1, keepdim=True)  # a draw from the worker's policy
    d = dict(learner_logits=learner.to(dtype), target_logits=target.to(dtype),
             worker_logp=logp.gather(-1, actions).squeeze(-1).contiguous(), actions=actions.squeeze(-1).int())
    d.update(_rewards_and_values(g, B, T, True, 0.005))
    learner, target = d["learner_logits"], d["target_logits"]
    l_theta, l_target = (torch.log_softmax(z.double(), -1).gather(-1, actions).squeeze(-1) for z in (learner, target))
    near = _near_the_clip(l_theta, l_target, d["worker_logp"], coef).unsqueeze(-1)
    taken = learner.gather(-1, actions)
    learner.scatter_(-1, actions, torch.where(near, taken + 0.0625, taken).to(dtype))
    return d


def _gaussian_logp(actions, mean, logstd):
    z = (actions.double() - mean.double()) / logstd.double().exp()
    return (-0.5 * z * z - logstd.double() - 0.5 * math.log(2 * math.pi)).sum(-1)


def _gaussian_inputs(g, B, T, D, coef):
    mean = torch.randn(B, T, D, device="cuda", generator=g)
    logstd = -torch.rand(B, T, D, device="cuda", generator=g)
    t_mean = mean + 0.05 * torch.randn(B, T, D, device="cuda", generator=g)
    w_mean = mean + 0.3 * torch.randn(B, T, D, device="cuda", generator=g)
    noise = torch.randn(B, T, D, device="cuda", generator=g)
    actions = w_mean + logstd.exp() * noise
    worker_logp = _gaussian_logp(actions, w_mean, logstd).float()
    l_theta, l_target = _gaussian_logp(actions, mean, logstd), _gaussian_logp(actions, t_mean, logstd)
    mean[..., 0] += 0.0625 * _near_the_clip(l_theta, l_target, worker_logp, coef)
    d = dict(learner_mean=mean, learner_logstd=logstd, target_mean=t_mean, target_logstd=logstd.clone(),
             worker_logp=worker_logp, actions=actions)
    d.update(_rewards_and_values(g, B, T, False, 0.001))
    return d


def _outputs(B, T, grads, extras):
    out = dict(loss_terms=torch.zeros(8, device="cuda"), dvalues=torch.empty(B, T, device="cuda"))
    for name, (width, dtype) in grads.items():
        out[name] = torch.empty(B, T, width, device="cuda", dtype=dtype)
    if extras:
        out["vtarget"] = torch.empty(B, T, device="cuda")
        out["advantage"] = torch.empty(B, T, device="cuda")
    return out


# ---- states and passes ------------------------------------------------------------------------------------------
def prepare(case, seed):
    return {"categorical": _prepare_categorical, "gaussian": _prepare_gaussian, "learner": _prepare_learner,
            "replay": _prepare_replay}[case["kind"]](case, _generator(seed), seed)


def run(state):
    return state["pass"](state)


def _prepare_categorical(case, g, seed):
    B, T, A = case["B"], case["T"], case["A"]
    coef = ip.Coefficients(**HYPER[case["hyper"]])
    workspace = ip.new_workspace(B, T)
    sets = []
    for _ in range(case["sets"]):
        t = _categorical_inputs(g, B, T, A, DTYPES[case["dtype"]], coef)
        sets.append((tuple(t[n] for n in INPUTS),
                     _outputs(B, T, {"dlogits": (A, DTYPES[case["grads"]])}, case["extras"])))
    state = dict(sets=sets, coef=coef, workspace=workspace, out=[o for _, o in sets])
    if case["how"] == "direct":
        state["pass"] = _loss_direct
        return state
    calls = [ip.prepare_loss_fwd_bwd(*t, coef, workspace=workspace, **o) for t, o in sets]
    return _issue(state, calls, case["how"])


def _prepare_gaussian(case, g, seed):
    B, T, D = case["B"], case["T"], case["D"]
    coef = ip.Coefficients(**dict(HYPER[case["hyper"]], clip_eps=0.2, ent_coef=0.0))
    workspace = ip.new_workspace(B, T)
    t = _gaussian_inputs(g, B, T, D, coef)
    out = _outputs(B, T, {"dmean": (D, torch.float32), "dlogstd": (D, torch.float32)}, case["extras"])
    call = ip.prepare_loss_fwd_bwd_gaussian(*(t[n] for n in GAUSS_INPUTS), coef, workspace=workspace, **out)
    return _issue(dict(out=out), [call], case["how"])


def _issue(state, calls, how):
    state["calls"] = calls
    state["pass"] = _loss_prepared
    if how == "graph":
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            for call in calls:
                call()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            for call in calls:
                call()
        state["graph"] = graph
        state["pass"] = _replay
    return state


def _loss_direct(state):
    for tensors, out in state["sets"]:
        ip.impact_loss_fwd_bwd(*tensors, state["coef"], workspace=state["workspace"], **out)
    return state["out"]


def _loss_prepared(state):
    for call in state["calls"]:
        call()
    return state["out"]


def _replay(state):
    state["graph"].replay()
    return state["out"]


def _prepare_learner(case, g, seed):
    B, T, A, N, K = case["B"], case["T"], case["A"], case["N"], case["K"]
    coef = ip.Coefficients(**HYPER["default"])
    batches = [_categorical_inputs(g, B, T, A, torch.float32, coef) for _ in range(4)]
    nbytes = [batches[0][n].numel() * batches[0][n].element_size() for n in FIELDS]
    storage = torch.zeros(ip.ImpactBuffer.storage_bytes(N, nbytes), dtype=torch.uint8, device="cuda")
    ring = ip.ImpactBuffer(N, K, nbytes, seed=int(seed), storage=storage)
    state = dict(case=case, coef=coef, batches=batches, ring=ring, workspace=ip.new_workspace(B, T))
    if case["how"] == "direct":
        # worker batches as they arrive from the workers' hosts, without the target network's output
        state["host"] = [[b[n].cpu().pin_memory() for n in FIELDS[:4]] + [None] for b in batches]
        state["batch_in"], state["pushed"] = {}, 0
        state["out"] = _outputs(B, T, {"dlogits": (A, torch.float32)}, False)
        for _ in range(N):
            _push_from_host(state)
        state["pass"] = _learner_iteration
        return state
    # bookkeeping on the device: push if a slot is free, draw, loss on the drawn batch, all in one graph
    table = torch.tensor([[b[n].data_ptr() for n in FIELDS[:4]] + [0, b["target_logits"].data_ptr()] for b in batches],
                         dtype=torch.int64, device="cuda")
    record = ip.new_loss_inputs_record()
    t = batches[0]
    step = ring.prepare_device_step({n: f for f, n in enumerate(FIELDS)}, t["learner_logits"], t["values"],
                                    t["bootstrap_values"], push_sources=table, record=record)
    outs = [_outputs(B, T, {"dlogits": (A, torch.float32)}, False) for _ in range(4)]
    terms = [torch.zeros(8, device="cuda") for _ in range(case["iterations"])]
    calls = []
    for i in range(case["iterations"]):
        out = dict(outs[i % len(outs)], loss_terms=terms[i])
        calls += [step, ip.prepare_loss_fwd_bwd_from_record(record, B, T, A, torch.float32, coef,
                                                            workspace=state["workspace"], **out)]
    ring.device_begin()
    for _ in range(-(-2 * N // case["iterations"])):  # every slot live, the draws in their steady state
        for call in calls:
            call()
    for o in outs:
        del o["loss_terms"]
    state["out"] = dict(terms=terms, grads=outs[:case["iterations"]], ring=storage.view(torch.int32))
    return _issue(state, calls, "graph")


def _push_from_host(state):
    i = state["pushed"] % len(state["host"])
    slot = state["ring"].push(state["host"][i])
    state["batch_in"][slot] = i
    state["pushed"] += 1


def _learner_iteration(state):
    case, ring = state["case"], state["ring"]
    B, T, A = case["B"], case["T"], case["A"]
    slot, k = ring.sample()
    b = state["batches"][state["batch_in"][slot]]
    actions = ring.slot_view(slot, 0, torch.int32, (B, T))
    rewards = ring.slot_view(slot, 1, torch.float32, (B, T))
    discounts = ring.slot_view(slot, 2, torch.float32, (B, T))
    worker_logp = ring.slot_view(slot, 3, torch.float32, (B, T))
    kept = ring.slot_view(slot, 4, torch.float32, (B, T, A))
    target, copy = (b["target_logits"], kept) if k == 0 else (kept, None)  # first traversal: the append
    ip.impact_loss_fwd_bwd(b["learner_logits"], target, worker_logp, actions, rewards, discounts, b["values"],
                           b["bootstrap_values"], state["coef"], workspace=state["workspace"],
                           target_logits_copy=copy, **state["out"])
    if k == case["K"] - 1:
        _push_from_host(state)
    return state["out"]


def _prepare_replay(case, g, seed):
    B, T, A = case["B"], case["T"], case["A"]
    t = _categorical_inputs(g, B, T, A, DTYPES[case["dtype"]], ip.Coefficients())
    nbytes = [t[n].numel() * t[n].element_size() for n in FIELDS]
    storage = torch.zeros(ip.ImpactBuffer.storage_bytes(case["N"], nbytes), dtype=torch.uint8, device="cuda")
    ring = ip.ImpactBuffer(case["N"], 1, nbytes, seed=int(seed), storage=storage)
    fields = [t[n] for n in FIELDS]
    drawn = [torch.empty_like(x) for x in fields]
    # what a minibatch is made of: the drawn fields and the learner network's outputs, trajectory by trajectory
    sources = drawn + [t["learner_logits"], t["values"], t["bootstrap_values"]]
    order = torch.randperm(B, device="cuda", generator=g).int()
    return {"pass": _replay_pass, "ring": ring, "fields": fields, "drawn": drawn, "sources": sources, "order": order,
            "minibatch": [torch.empty_like(x) for x in sources]}


def _replay_pass(state):
    ring = state["ring"]
    ring.push(state["fields"])
    ring.sample(gather_dst=state["drawn"])
    for src, dst in zip(state["sources"], state["minibatch"]):
        ip.impact_gather_rows(src, state["order"], dst)
    return state["drawn"] + state["minibatch"]


# ---- what a pass cannot do without ------------------------------------------------------------------------------
def _categorical_bytes(M, B, A, in_bytes, out_bytes, extras):
    return M * (2 * A * in_bytes + 20 + A * out_bytes + 4 + (8 if extras else 0)) + 4 * B + 32


def work(case):
    B, T = case["B"], case["T"]
    M = B * T
    size = {"f32": 4, "bf16": 2}
    if case["kind"] == "categorical":
        A, n = case["A"], case["sets"]
        kl = 6 * A if case["hyper"] == "kl" else 0
        return {"bytes": n * _categorical_bytes(M, B, A, size[case["dtype"]], size[case["grads"]], case["extras"]),
                "flops": n * M * (17 * A + kl + 60)}
    if case["kind"] == "gaussian":
        D = case["D"]
        return {"bytes": M * (7 * 4 * D + 20 + (8 if case["extras"] else 0)) + 4 * B + 32, "flops": M * (24 * D + 60)}
    if case["kind"] == "learner":
        # a batch pushed per K iterations and its target logits kept at the first traversal, beside the loss itself
        A, n, K = case["A"], case["iterations"], case["K"]
        moved = 2 * 16 * M + 4 * A * M
        return {"bytes": n * (_categorical_bytes(M, B, A, 4, 4, False) + moved / K), "flops": n * M * (17 * A + 60)}
    row = case["A"] * size[case["dtype"]]
    slot, minibatch = M * (16 + row), M * (20 + 2 * row) + 4 * B
    return {"bytes": 2 * (slot + slot + minibatch) + 4 * B, "flops": 0}


def tolerance(case):
    """Against the fp64 oracle the listed cases and some fifty drawn ones are off by at most 1e-6 (2-norm) and 6e-5
    (largest difference) with fp32 gradients, by 1.7e-3 and 3.9e-3 where gradients are rounded to bf16; four times
    that is allowed between two programs."""
    if case["kind"] == "replay":
        return "exact"
    if case.get("grads") == "bf16":
        return {"rel": 7e-3, "max": 1.6e-2}
    return {"rel": 4e-6, "max": 2.5e-4}
