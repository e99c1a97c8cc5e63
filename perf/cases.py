"""Performance cases of the cross-layer MoE step: what a serving program has the library do.

A case names a model shape, a set of micro-batches and the way the library is called:

* ``step``  - one `eb_step` with the inputs already on the device (a layer step inside a serving loop);
* ``calls`` - the five calls one by one, the aggregation adding the residual (a loop that does something of its
  own between the calls);
* ``host``  - one `eb_step_host` from pinned host buffers to pinned host buffers;
* ``run``   - Algorithm 1 over all layers with `driver.run_full`, steps replayed from CUDA graphs if ``graphs``;
* ``trace`` - Algorithm 1 with routing and scheduling only, `driver.run_load_trace` (what the sweeps run).

The shapes are those of `synth.workload` and of the sweep (`synth.workload_c5`), from one token per micro-batch to
prompts of a thousand, plus ragged micro-batches and sizes that are multiples of 8 and of nothing larger.  Layer
counts are cut where the full model would not fit a card three times; a step touches the same matrices either way.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2608_07964_b200 import binding as B
from paper_2608_07964_b200 import driver, synth

# model shapes: layers, routed experts, top-k, shared experts, hidden, intermediate, virtual devices, expert table, skew
TINY = dict(L=4, E=8, K=2, S=0, H=256, I=512, D=4, mapping="contiguous", zipf=1.0)
DECODE = dict(L=24, E=60, K=4, S=4, H=2048, I=1408, D=8, mapping="mod", zipf=1.2)
FINE = dict(L=26, E=64, K=6, S=2, H=2048, I=1408, D=8, mapping="contiguous", zipf=0.8)
SWEEP = dict(L=8, E=64, K=6, S=0, H=2048, I=1408, D=8, mapping="contiguous", zipf=1.0)
LARGE = dict(L=8, E=8, K=2, S=0, H=4096, I=14336, D=8, mapping="contiguous", zipf=1.0)
ODD = dict(L=5, E=31, K=3, S=1, H=1000, I=712, D=5, mapping="mod", zipf=0.6)


def case(mode, shape, N, T, **more):
    """N micro-batches of T tokens each (about T when `ragged`), staggered over the layers unless `same_layer`."""
    c = dict(shape, mode=mode, N=N, T=T, ragged=False, same_layer=False, renorm=1, policy=B.POLICY_MAXUTIL, graphs=False)
    c.update(more)
    return c


def listed():
    return [
        # the smallest model end to end, all weights resident in L2: launches and latency
        dict(case("step", TINY, 4, 64), name="tiny_step"),
        # interactive decoding: one token in each of four micro-batches
        dict(case("step", DECODE, 4, 1), name="decode_one_token"),
        # batched decoding of a model with shared experts
        dict(case("step", DECODE, 8, 32), name="decode"),
        # the same from and to host memory, one step at a time
        dict(case("host", DECODE, 8, 32), name="decode_host"),
        # requests of unequal length, stage by stage, residual added, full-softmax gate weights, the linear policy
        dict(case("calls", SWEEP, 7, 77, ragged=True, renorm=0, policy=B.POLICY_CUMUTIL), name="ragged_calls"),
        # a model whose sizes are multiples of 8 only and whose devices hold unequal numbers of experts
        dict(case("step", ODD, 5, 93, ragged=True, policy=B.POLICY_DIFFPEAK), name="odd_sizes"),
        # fine-grained experts, micro-batches spread over the layers (the steady state of Algorithm 1)
        dict(case("step", FINE, 16, 512), name="fine_grained"),
        # the same model on its first step, all micro-batches at one layer (prefill; several hundred rows per expert)
        dict(case("step", FINE, 16, 512, L=4, same_layer=True), name="fine_prefill"),
        # large experts, prefill-sized micro-batches: the largest case
        dict(case("step", LARGE, 8, 1024), name="large_experts"),
        # large experts, decoding
        dict(case("step", LARGE, 8, 16), name="large_decode"),
        # Algorithm 1 over a whole model, steps replayed from graphs
        dict(case("run", SWEEP, 4, 128, graphs=True), name="whole_run"),
        # a scheduling study: routing and scheduling of 16 micro-batches, the expert pass left out
        dict(case("trace", SWEEP, 16, 128), name="load_trace"),
    ]


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    mode = rng.choice(["step", "step", "step", "step", "step", "calls", "host", "run", "trace"])
    more = dict(ragged=rng.random() < 0.5, same_layer=rng.random() < 0.25, renorm=rng.choice([1, 1, 0]),
                policy=rng.choice([B.POLICY_MAXUTIL, B.POLICY_MAXUTIL, B.POLICY_CUMUTIL, B.POLICY_DIFFPEAK, B.POLICY_ALL]),
                zipf=round(rng.uniform(0.0, 1.5), 2))
    if mode == "run":
        return case(mode, SWEEP, rng.randint(2, 4), log_int(rng, 1, 48), L=rng.randint(3, 6), graphs=rng.random() < 0.5, **more)
    if mode == "trace":
        return case(mode, SWEEP, rng.randint(2, 16), log_int(rng, 1, 256), L=rng.randint(3, 8), **more)
    shape = rng.choice([TINY, DECODE, DECODE, FINE, FINE, SWEEP, LARGE, ODD])
    if shape is LARGE:
        return case(mode, shape, rng.randint(2, 7), log_int(rng, 1, 700), **more)
    if shape is ODD:
        more.update(E=rng.randint(9, 47), K=rng.randint(1, 6), S=rng.randint(0, 3), D=rng.randint(2, 8),
                    H=8 * rng.randint(40, 250), I=8 * rng.randint(30, 180))
    return case(mode, shape, rng.randint(2, 16), log_int(rng, 1, 700), **more)


def tokens_of(c):
    """Tokens of every micro-batch: T each, or spread from about T/2 to 3T/2."""
    n, t = c["N"], c["T"]
    return [max(1, t // 2 + ((5 * j + 3) % n) * t // n) for j in range(n)] if c["ragged"] else [t] * n


def layers_of(c):
    return [0] * c["N"] if c["same_layer"] else [j * c["L"] // c["N"] for j in range(c["N"])]


def offsets(tokens):
    return [0] + np.cumsum(tokens).tolist()


def workload_of(c, seed=synth.BASE_SEED):
    return synth.Workload(name="case", L=c["L"], E=c["E"], K=c["K"], S=c["S"], H=c["H"], I=c["I"], D=c["D"],
                          mapping=c["mapping"], N=c["N"], T=c["T"], zipf_s=c["zipf"], renorm_topk=c["renorm"], seed=seed)


def weights(shape, gen):
    w = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
    return w.normal_(0.0, 0.02, generator=gen)


def prepare(c, seed):
    wl = workload_of(c, seed)
    tokens, layers, mode = tokens_of(c), layers_of(c), c["mode"]
    tok_off = offsets(tokens)
    T = tok_off[-1]
    bias = synth.zipf_bias(wl)
    step = B.from_workload(wl, max_tokens=T)
    step.out.zero_()
    s = SimpleNamespace(mode=mode, step=step, wl=wl, tok_off=tok_off, T=T, policy=c["policy"])
    if mode != "trace":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        n = wl.E + wl.S
        step.bind_weights(weights((wl.L, n, wl.I, wl.H), gen), weights((wl.L, n, wl.I, wl.H), gen),
                          weights((wl.L, n, wl.H, wl.I), gen))
    if mode in ("run", "trace"):
        table = [[synth.logits_for(wl, j, l, "cuda", bias, T=t) for l in range(wl.L)] for j, t in enumerate(tokens)]
        s.logits_of = lambda j, l: table[j][l]
    else:
        logits = torch.cat([synth.logits_for(wl, j, layers[j], "cuda", bias, T=t) for j, t in enumerate(tokens)])
    if mode != "trace":
        x = torch.cat([synth.hidden_for(wl, j, layers[j], "cuda", T=t) for j, t in enumerate(tokens)])
    if mode == "run":
        # blocks without normalisation layers: small hidden states keep the chain in range
        s.x0 = x * 0.05
        s.graphs = driver.StepGraphs(step, tok_off) if c["graphs"] else None
    elif mode == "host":
        s.h_logits, s.h_x = logits.cpu().pin_memory(), x.cpu().pin_memory()
        s.h_out = torch.zeros(T, wl.H, dtype=torch.bfloat16).pin_memory()
    elif mode != "trace":
        step.logits[:T].copy_(logits)
        step.x[:T].copy_(x)
    if mode in ("step", "calls", "host"):
        s.batch = B.Batch(tok_off, layers)
    return s


def record(steps, wl):
    """Run set, utilisation and joint load of every step, in a table of the longest run's length (one step per
    micro-batch and layer)."""
    t = np.zeros((wl.N * wl.L, 3 + wl.D), dtype=np.int64)
    for i, st in enumerate(steps):
        t[i] = [st["run_mask"], st["util_num"], st["util_den"]] + st["joint_load"]
    return t


def run(s):
    step, m, policy = s.step, s.wl.m, s.policy
    if s.mode == "step":
        step.eb_step(s.batch, m, policy)
    elif s.mode == "calls":
        step.eb_route(s.batch)
        step.eb_schedule(s.batch, m, policy)
        step.eb_permute(s.batch)
        step.eb_expert_ffn_grouped()
        step.eb_combine(s.batch, residual=step.x)
    elif s.mode == "host":
        res = step.eb_step_host(s.batch, m, s.h_logits, s.h_x, s.h_out, policy)
        return dict(out=s.h_out, run_mask=res["run_mask"], defer_mask=res["defer_mask"], util_num=res["util_num"],
                    util_den=res["util_den"])
    else:
        loop = (step, s.tok_off, s.wl.L, m, policy, s.logits_of)
        if s.mode == "run":
            r = driver.run_full(*loop, s.x0, graphs=s.graphs)
            return dict(x=r["x"], steps=record(r["steps"], s.wl))
        return dict(steps=record(driver.run_load_trace(*loop), s.wl))
    return dict(out=step.out, topk_idx=step.topk_idx, topk_w=step.topk_w, pos=step.pos, mb_load=step.mb_load,
                mb_cnt=step.mb_cnt, sched=step.sched, step_meta=step.step_meta)


def experts_hit(wl, bias, j, layer, tokens):
    """Routed experts that `tokens` tokens of micro-batch j touch at a layer."""
    z = synth.logits_for(wl, j, layer, "cpu", bias, T=tokens)
    return set(z.topk(wl.K, dim=1).indices.unique().tolist())


def work(c):
    """Every matrix that has rows is read once, every token's input is read and its output written once.  A step runs
    the fewest micro-batches its schedule may choose (all of them under the lock-step policy)."""
    wl, tokens, layers = workload_of(c), tokens_of(c), layers_of(c)
    bias = synth.zipf_bias(wl)
    route = sum(tokens) * (wl.E * 4 + wl.K * 8)
    if c["mode"] == "trace":
        return dict(bytes=float(wl.L * route), flops=float(wl.L * sum(tokens) * wl.E))
    n_run = wl.N if c["policy"] == B.POLICY_ALL else min(wl.m, wl.N)
    if c["mode"] == "run":
        places = [(j, l) for j in range(wl.N) for l in range(wl.L)]
        route *= wl.L
    else:
        places = [(j, layers[j]) for j in range(n_run)]
    hit = {}
    for j, l in places:
        hit.setdefault(l, set()).update(experts_hit(wl, bias, j, l, tokens[j]))
    mats = sum(len(v) + wl.S for v in hit.values())
    ran = sum(tokens[j] for j, _ in places)
    mat = 3 * wl.H * wl.I
    return dict(bytes=float(mats * mat * 2 + ran * wl.H * 4 + route), flops=float(2 * ran * (wl.K + wl.S) * mat))


def tolerance(c):
    """Scheduling is whole numbers.  The expert pass multiplies bf16 with 32-bit sums and rounds its intermediate, its rows
    and the aggregated sum to bf16: against 64-bit sums with no rounding in between the listed steps are off by 1.7e-3 to
    2.9e-3 (2-norm), single values by up to 1.6e-2, a whole run by 4.7e-3 and 2.3e-2.  Four times that."""
    if c["mode"] == "trace":
        return "exact"
    return dict(rel=1.15e-2, max=7e-2)
