"""The work that users of preference-packed attention have it do, as measurable cases.

A case is a dict of plain values.  `kind` names the call sequence:

  step    one training pass of the attention path on device tensors: forward handing the backward
          its scratch, then backward; with `replan` the step also builds the plan of its batch
  score   forward only with the plan in hand (scoring with a frozen reference policy)
  around  the steps on either side of attention: position ids and rotary embedding on Q / K
          before it, the preference loss with its gradient behind it
  rows    the data side: groups sorted and packed into rows, rows dealt out to ranks
  host    one whole pass from and to page-locked host buffers

Packed structures (`shape`) are the workload recipes of paper_2602_24082_b200/workloads.py or
drawn here from the same kinds of length distributions; `layout` seeds the lengths, so a case
always means the same structure while the tensors follow the caller's seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2602_24082_b200 import binding as B
from paper_2602_24082_b200 import workloads as W


# ---------------------------------------------------------------------------- structures

def _rows_of(case):
    """[[(prompt, (responses, ...)), ...], ...] of a case."""
    shape, rng = case["shape"], np.random.Generator(np.random.PCG64(case["layout"]))
    if shape == "recipe0":
        return W.config0().rows
    if shape == "recipe1":
        return W.config1(case["layout"]).rows
    if shape == "recipe2":
        return W.config2(case["layout"]).rows
    if shape == "recipe3":
        return W.config3(case["layout"]).rows
    if shape == "recipe4":
        return W.config4(case["layout"]).rows
    # "drawn": groups of about `mean` tokens, `n` responses each, prompt : mean response = `rho`,
    # until `tokens` are reached; `per_row` groups follow each other in one row
    groups, left = [], case["tokens"]
    n, rho = case["n"], case["rho"]
    while left > 0:
        total = int(min(16384, max(n + 1, round(case["mean"] * math.exp(0.5 * rng.standard_normal())))))
        total = max(n + 1, min(total, left))
        rs = [max(1, int(round(total / (rho + n) * rng.uniform(0.5, 1.5)))) for _ in range(n)]
        while sum(rs) >= total:
            rs[int(np.argmax(rs))] -= 1
        groups.append((total - sum(rs), tuple(rs)))
        left -= total
    k = case["per_row"]
    return [groups[i:i + k] for i in range(0, len(groups), k)]


def _workload(case):
    return W.Workload(case["kind"], _rows_of(case), case["hq"], case["hkv"], case["d"], seed=case["layout"])


def _low_variance_ranges(case):
    """Image-token prefixes of the multi-response recipe: their Q, K, V rows have variance 0.5."""
    return W.config2(case["layout"]).low_var_ranges if case["shape"] == "recipe2" else []


def _group_lengths(case):
    rng = np.random.Generator(np.random.PCG64(case["layout"]))
    P, off, R = [], [0], []
    for _ in range(case["groups"]):
        n = int(rng.integers(1, 6))
        P.append(int(np.clip(round(768 * math.exp(0.8 * rng.standard_normal())), 1, 8192)))
        R += [int(rng.integers(16, 1537)) for _ in range(n)]
        off.append(len(R))
    return np.asarray(P, np.int32), np.asarray(off, np.int32), np.asarray(R, np.int32)


# ---------------------------------------------------------------------------- the cases

def _step(name, shape, hq, hkv, d, layout, **more):
    return dict({"name": name, "kind": "step", "shape": shape, "hq": hq, "hkv": hkv, "d": d,
                 "layout": layout, "replan": True, "deterministic": False}, **more)


def listed():
    drawn = dict(tokens=12000, mean=1800, n=2, rho=2, per_row=1)
    return [
        # the smallest call: one short sample, one head; latency and launches
        _step("tiny_step", "recipe0", 1, 1, 64, 0),
        # pairwise preference data on an 8B-class shape, one group per row: the ordinary step
        _step("pairs_step", "recipe1", 32, 8, 128, 1),
        # long prompt with an image-like prefix, four ranked responses, seven heads per KV head
        _step("ranking_step", "recipe2", 28, 4, 128, 2),
        # batch packing on top of preference packing, 72B-class shape
        _step("packed_rows_step", "recipe3", 64, 8, 128, 3),
        # two length-sorted rows of 32768 tokens: the largest step; its plan serves every layer
        _step("long_rows_step", "recipe4", 32, 8, 128, 2, replan=False),
        # head_dim 64, 1B-class shape; a layer of a model whose plan is already there
        _step("head64_step", "drawn", 32, 8, 64, 11, replan=False, **dict(drawn, tokens=16384)),
        # head_dim 96, no grouped heads
        _step("head96_step", "drawn", 16, 16, 96, 12, replan=False, **dict(drawn, n=3, mean=2600)),
        # bit-reproducible gradients, for runs that have to repeat exactly
        _step("deterministic_step", "recipe1", 32, 8, 128, 5, deterministic=True),
        # scoring with the frozen reference policy: forward only over long rows
        {"name": "score_long", "kind": "score", "shape": "recipe4", "hq": 32, "hkv": 8, "d": 128, "layout": 1},
        # rotary embedding before and preference loss behind the attention of long rows
        {"name": "around_long", "kind": "around", "shape": "recipe4", "hq": 32, "hkv": 8, "d": 128,
         "layout": 3},
        # one global batch of samples sorted, packed and dealt out to eight ranks
        {"name": "row_builder", "kind": "rows", "groups": 4096, "capacity": 16384, "ranks": 8, "layout": 7},
        # the ordinary step for a caller whose tensors live on the host
        {"name": "pairs_from_host", "kind": "host", "shape": "recipe1", "hq": 32, "hkv": 8, "d": 128,
         "layout": 1},
    ]


def draw(rng):
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    kind = rng.choice(["step"] * 8 + ["score"] * 2 + ["around", "rows", "host"])
    layout = rng.randrange(1 << 30)
    if kind == "rows":
        return {"kind": kind, "groups": log(17, 8192), "capacity": log(16384, 65536),
                "ranks": rng.choice([1, 3, 8, 64]), "layout": layout}
    d = rng.choice([64, 96, 128, 128, 128])
    hkv = rng.choice([1, 2, 4, 8])
    hq = hkv * rng.choice([1, 2, 4, 7, 8])
    tokens = log(200, 40000)
    if kind == "host":
        tokens = min(tokens, 10000)
    tokens = min(tokens, 32 * 40000 // max(32, hq))   # never more than the largest listed step
    case = {"kind": kind, "shape": "drawn", "hq": hq, "hkv": hkv, "d": d, "layout": layout,
            "tokens": tokens, "mean": log(100, 8000), "n": rng.choice([1, 2, 2, 3, 4, 8]),
            "rho": rng.choice([0.5, 1, 2, 4, 16]), "per_row": rng.choice([1, 1, 3, 8])}
    if kind == "step":
        case.update(replan=rng.random() < 0.5, deterministic=rng.random() < 0.2)
    return case


# ---------------------------------------------------------------------------- preparation

def prepare(case, seed):
    dev = torch.device("cuda:0")
    if case["kind"] == "rows":
        # another seed brings the batch in another order, as a shuffling loader does
        P, off, R = _group_lengths(case)
        perm = np.random.Generator(np.random.PCG64(seed)).permutation(len(P))
        R = np.concatenate([R[off[g]:off[g + 1]] for g in perm])
        off = np.concatenate([[0], np.cumsum(np.diff(off)[perm])]).astype(np.int32)
        P = np.ascontiguousarray(P[perm])
        return {"case": case, "P": torch.from_numpy(P).to(dev), "off": torch.from_numpy(off).to(dev),
                "R": torch.from_numpy(R).to(dev)}
    w = _workload(case)
    T, Hq, Hkv, D = w.total_tokens, w.num_q_heads, w.num_kv_heads, w.head_dim
    gen = torch.Generator(device=dev).manual_seed(seed)
    rand = lambda *shape: torch.randn(*shape, generator=gen, device=dev, dtype=torch.float32)
    st = {"case": case, "scale": w.softmax_scale, "q": rand(T, Hq, D).bfloat16(), "k": rand(T, Hkv, D).bfloat16()}
    kind = case["kind"]
    if kind == "around":
        st["plan"] = B.plan_for(w)
        # log-probabilities of sampled tokens: mostly likely ones, a tail of unlikely ones
        st["logp"] = -1.5 * torch.empty(T, device=dev).exponential_(generator=gen)
        st["ref"] = st["logp"] + 0.1 * rand(T)
        return st
    st["v"] = rand(T, Hkv, D).bfloat16()
    for lo, hi in _low_variance_ranges(case):
        for name in ("q", "k", "v"):
            st[name][lo:hi] *= math.sqrt(0.5)
    if kind == "score":
        st["plan"] = B.plan_for(w)
        return st
    st["do"] = rand(T, Hq, D).bfloat16()
    if kind == "host":
        for name in ("q", "k", "v", "do"):
            st[name] = st[name].cpu().pin_memory()
        st["call"] = B.HostStep(w)
        return st
    # a training program keeps the plan workspace and the backward scratch from step to step
    desc = w.descriptors()
    problem, _ = B.make_problem(desc, Hq, Hkv, D, T)
    plan_bytes, _, scratch_bytes = B.pp_plan_workspace_bytes(problem)
    st["desc"], st["tokens"] = desc, T
    st["workspace"] = torch.empty(plan_bytes, dtype=torch.uint8, device=dev)
    st["scratch"] = torch.empty(scratch_bytes, dtype=torch.uint8, device=dev)
    if not case["replan"]:
        st["plan"] = _plan(st)
    return st


def _plan(st):
    c = st["case"]
    plan = B.pp_build_plan(st["desc"], c["hq"], c["hkv"], c["d"], st["tokens"], workspace=st["workspace"])
    plan._bwd_scratch = st["scratch"]
    return plan


# ---------------------------------------------------------------------------- one pass

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "step":
        plan = _plan(st) if case["replan"] else st["plan"]
        o, lse = B.pp_attn_fwd(plan, st["q"], st["k"], st["v"], st["scale"], for_backward=True)
        dq, dk, dv = B.pp_attn_bwd(plan, st["q"], st["k"], st["v"], o, lse, st["do"], st["scale"],
                                   deterministic=case["deterministic"])
        return {"o": o, "lse": lse, "dq": dq, "dk": dk, "dv": dv}
    if kind == "score":
        o, lse = B.pp_attn_fwd(st["plan"], st["q"], st["k"], st["v"], st["scale"])
        return {"o": o, "lse": lse}
    if kind == "around":
        pos = B.pp_position_ids(st["plan"])
        q, k = B.pp_rope_qk(st["plan"], st["q"], st["k"])
        logp, reward, loss, grad = B.pp_preference_loss(st["plan"], st["logp"], st["ref"], 0.1)
        return {"pos": pos, "q": q, "k": k, "logp": logp, "reward": reward, "loss": loss, "grad": grad}
    if kind == "rows":
        out = B.pp_build_rows(st["P"], st["off"], st["R"], case["capacity"])
        order, rank_of_row, rank_cost = B.pp_assign_rows(out["row_cost"], case["ranks"])
        out = {k: v for k, v in out.items() if k != "status"}
        return dict(out, assign_order=order, rank_of_row=rank_of_row, rank_cost=rank_cost)
    o, lse, dq, dk, dv = st["call"](st["q"], st["k"], st["v"], st["do"])
    return {"o": o, "lse": lse, "dq": dq, "dk": dk, "dv": dv}


def work(case):
    """Bytes and operations one pass cannot do without (each input read once, each output written
    once; the visible query-key pairs only)."""
    if case["kind"] == "rows":
        P, off, R = _group_lengths(case)
        return {"bytes": 4 * (2 * (2 * len(P) + 1 + len(R)) + 2 * len(P)), "flops": 0}
    w = _workload(case)
    T, Hq, Hkv, D = w.total_tokens, w.num_q_heads, w.num_kv_heads, w.head_dim
    qb, kb, lse = 2 * T * Hq * D, 2 * T * Hkv * D, 4 * T * Hq
    fwd, bwd = w.useful_flops()
    if case["kind"] == "around":
        # rotation: read and write Q, K; ids; loss: two arrays read, the gradient written
        return {"bytes": 2 * (qb + kb) + 4 * T + 12 * T, "flops": 3 * T * (Hq + Hkv) * D}
    if case["kind"] == "score":
        return {"bytes": 2 * qb + 2 * kb + lse, "flops": fwd}
    # Q, K, V, dO in; O, LSE, dQ, dK, dV out
    return {"bytes": 4 * qb + 4 * kb + lse, "flops": fwd + bwd}


def tolerance(case):
    """bf16 results from fp32 sums, P and dS rounded to bf16 before their second products:
    measured against fp64, O is off by 1.9 - 2.1e-3 and the gradients by 2.3 - 3.2e-3 (relative
    2-norm); the rotation rounds once to bf16 (1.7e-3).  About four times that is allowed."""
    if case["kind"] == "rows":
        return "exact"
    if case["kind"] == "around":
        return {"rel": 5e-3}
    return {"rel": 1e-2}
