"""Performance cases of the FEPLB MoE layer: what programs that use the library have it do.

A case names one layer geometry, one batch size and the calls a program makes per micro-batch:

  forward   ``Context.moe_forward`` on device-resident inputs: inference (decode with a few tokens,
            prefill with thousands) and the forward half of training
  host      ``Context.moe_forward_host``: the same with inputs and result in pinned host memory
  train     ``moe_forward`` with the pre-activations saved, then ``moe_backward`` with weight
            gradients, either accumulated over micro-batches or, with ``update``, written by the
            first micro-batch after an optimizer step, which also refreshes the transposed weights
  permute   router and data movement only (``route_topk``, ``route_hist``, ``dispatch``, ``combine``),
            for programs that bring an expert backend of their own

Sizes follow the named workloads of ``paper_2604_19654_b200.workloads`` (cfg1 .. cfg4 and the scaling
sweep), their decode-sized counterparts, and generic odd sizes.  Inputs are drawn like there:
activations and weights N(0, 0.02^2) in bf16, expert popularity Zipf, Dirichlet (redrawn per
micro-batch) or three hot experts of one rank, K distinct experts per token by Gumbel top-k, gates =
softmax of the selected logits.
"""
import math

import numpy as np
import torch

from paper_2604_19654_b200 import feplb as F

# Layer geometries: the named workloads, and one with nothing round about it (f not a multiple of
# 128, d not of 256, 60 experts, 5 ranks).
TINY = dict(d=128, f=64, E=8, K=2, R=2, dyn=2, max_num_dyn=2, tau=4, routing="zipf", alpha=1.2)
MID = dict(d=2048, f=768, E=64, K=6, R=4, dyn=4, max_num_dyn=8, tau=64, routing="dirichlet", alpha=0.3)
SKEW = dict(MID, routing="hot3", alpha=0.35, split=1)
RAGGED = dict(d=1920, f=704, E=60, K=4, R=5, dyn=4, max_num_dyn=8, tau=16, routing="dirichlet", alpha=0.5)
GLM = dict(d=6144, f=2048, E=128, K=8, R=8, dyn=4, max_num_dyn=8, tau=64, routing="dirichlet", alpha=0.2)
GLM32 = dict(GLM, E=32, R=4)          # the same expert shapes with as many experts as one training GPU holds


def _case(name, kind, T, layer, **more):
    c = dict(name=name, kind=kind, T=T, split=0, plan=False, accumulate=False, update=False)
    c.update(layer)
    c.update(more)
    return c


def listed():
    return [
        # a unit-test-sized layer (cfg1): latency of the host path and of six short launches
        _case("forward tiny T=256", "forward", 256, TINY),
        # serving, decode: a few dozen tokens per step; every touched expert's weights are streamed
        _case("forward mid T=64", "forward", 64, MID),
        # serving, decode at the GLM-5-like layer
        _case("forward glm T=128", "forward", 128, GLM),
        # odd sizes: ragged tiles in every dimension
        _case("forward ragged T=1537", "forward", 1537, RAGGED),
        # the benchmarked micro-batch (cfg2): prefill / training forward
        _case("forward mid T=4096", "forward", 4096, MID),
        # extreme skew (cfg4) with hot experts cut, by a program that logs the plan
        _case("forward skew T=4096", "forward", 4096, SKEW, plan=True),
        # GLM-5-like layer (cfg3): its micro-batch, and the largest point of the scaling sweep
        _case("forward glm T=16384", "forward", 16384, GLM),
        _case("forward glm T=65536", "forward", 65536, dict(GLM, R=16)),
        # a serving front end that holds its batches in host memory
        _case("host mid T=4096", "host", 4096, MID),
        # training, gradients accumulated over micro-batches
        _case("train mid T=4096", "train", 4096, MID, accumulate=True),
        # training at the GLM-5-like expert shapes, one micro-batch per optimizer step
        _case("train glm32 T=4096", "train", 4096, GLM32, update=True),
        # data movement for another expert backend
        _case("permute glm T=8192", "permute", 8192, GLM),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any kind, sizes spread logarithmically over the ranges of the listed ones."""
    while True:
        kind = rng.choice(["forward"] * 6 + ["host", "train", "train", "permute"])
        E = rng.choice([8, 16, 24, 32, 48, 60, 64, 96, 128])
        R = rng.choice([r for r in (1, 2, 3, 4, 5, 6, 8, 12, 16) if E % r == 0 and E // r >= 4])
        d = 128 * _log_int(rng, 1, 48)
        f = 64 * _log_int(rng, 1, 32)
        K = rng.randint(1, 8)
        top = {"forward": 65536, "host": 8192, "train": 16384, "permute": 32768}[kind]
        T = _log_int(rng, 64 if kind == "train" else 1, top)
        routing, alpha = rng.choice([("dirichlet", 0.2), ("dirichlet", 0.3), ("dirichlet", 0.5), ("zipf", 1.2), ("hot3", 0.35)])
        if routing == "hot3" and K < 4:
            continue
        c = _case("", kind, T, dict(d=d, f=f, E=E, K=K, R=R, dyn=rng.choice([2, 4]), max_num_dyn=8,
                                    tau=rng.choice([4, 16, 64]), routing=routing, alpha=alpha),
                  split=int(rng.random() < 0.2), plan=rng.random() < 0.3)
        if kind == "train":
            c["accumulate"] = rng.random() < 0.5
            c["update"] = not c["accumulate"]
            if 24 * E * d * f > 10e9:
                continue
        rows = T * K + (E * 127 if kind == "train" else 0)
        if rows * (2 * d + f) * 2 * (2.5 if kind == "train" else 1) > 15e9:
            continue
        del c["name"]
        return c


# ------------------------------------------------------------------------------------------ inputs

class State:
    pass


def _popularity(c, rng):
    E = c["E"]
    if c["routing"] == "dirichlet":
        p = np.maximum(rng.dirichlet(np.full(E, c["alpha"])), 1e-30)
    elif c["routing"] == "zipf":
        p = np.empty(E)
        p[rng.permutation(E)] = (np.arange(E) + 1.0) ** -c["alpha"]
    else:
        # three experts of one rank, each chosen by a share alpha * K / 3 of the tokens: an expert of weight w
        # is among a token's K with probability about 1 - exp(-w t), with t such that the shares add up to K
        share = min(0.9, c["alpha"] * c["K"] / 3.0)
        p = np.ones(E)
        hot = rng.integers(c["R"]) * (E // c["R"]) + rng.choice(E // c["R"], 3, replace=False)
        p[hot] = math.log(1.0 - share) / math.log(1.0 - min(0.95, (c["K"] - 3 * share) / (E - 3)))
    return p / p.sum()


def prepare(case, seed):
    c, s = case, State()
    T, d, f, E, K = (c[k] for k in ("T", "d", "f", "E", "K"))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    normal = lambda *shape: torch.empty(*shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.02, generator=gen)   # noqa: E731
    s.case = c
    s.cfg = F.make_config(T, K, E, c["R"], d, f, dyn=c["dyn"], max_num_dyn=c["max_num_dyn"], tau=c["tau"], split=c["split"],
                          row_align=128 if c["kind"] == "train" else 1)
    s.ctx = F.Context(s.cfg)
    s.x = normal(T, d)
    p = torch.from_numpy(_popularity(c, np.random.default_rng(seed))).float().cuda()
    u = torch.rand(T, E, generator=gen, device="cuda").clamp_(1e-20, 1.0 - 1e-7)
    s.logits = p.log() - (-u.log()).log()
    if c["kind"] == "permute":
        S = T * K
        s.ids = torch.empty(T, K, dtype=torch.int32, device="cuda")
        s.gates = torch.empty(T, K, dtype=torch.float32, device="cuda")
        s.counts = torch.empty(E, dtype=torch.int32, device="cuda")
        s.load = torch.empty(c["R"], dtype=torch.int32, device="cuda")
        s.x_perm = torch.empty(S, d, dtype=torch.bfloat16, device="cuda")
        s.s2r = torch.empty(T, K, dtype=torch.int32, device="cuda")
        s.r2t = torch.empty(S, dtype=torch.int32, device="cuda")
        s.y = normal(S, d)                      # what the program's experts made of the rows
        s.out = torch.empty(T, d, dtype=torch.bfloat16, device="cuda")
        return s
    top, ids = s.logits.topk(K, dim=1)
    s.ids, s.gates = ids.int(), torch.softmax(top, dim=1)
    s.logits = None
    s.w1, s.w3, s.w2 = normal(E, f, d), normal(E, f, d), normal(E, d, f)
    s.buf = F.Buffers(s.cfg)
    if c["kind"] == "host":
        s.host = [t.cpu().pin_memory() for t in (s.x, s.ids, s.gates)]
        s.out_host = torch.empty(T, d, dtype=torch.bfloat16).pin_memory()
    if c["kind"] == "train":
        s.bwd = F.BackwardBuffers(s.cfg)
        s.ctx.set_preact_buffer(s.bwd.ab)
        s.w1t, s.w3t, s.w2t = (torch.empty(E, *shape, dtype=torch.bfloat16, device="cuda") for shape in ((d, f), (d, f), (f, d)))
        s.ctx.transpose_weights(s.w1, s.w3, s.w2, s.w1t, s.w3t, s.w2t)
        s.dw = [torch.zeros(E, *shape, dtype=torch.float32, device="cuda") for shape in ((f, d), (f, d), (d, f))]
        s.d_out = normal(T, d)
    return s


def run(state):
    s, c = state, state.case
    if c["kind"] == "permute":
        s.ctx.route_topk(s.logits, s.ids, s.gates)
        s.ctx.route_hist(s.ids, s.counts, s.load)
        s.ctx.dispatch(s.x, s.ids, s.counts, s.x_perm, s.s2r, s.r2t)
        s.ctx.combine(s.y, s.s2r, s.gates, s.out)
        return dict(ids=s.ids, gates=s.gates, counts=s.counts, load=s.load, x_perm=s.x_perm, s2r=s.s2r, r2t=s.r2t, out=s.out)
    b = s.buf
    if c["kind"] == "host":
        s.ctx.moe_forward_host(*s.host, s.x, s.ids, s.gates, s.w1, s.w3, s.w2, b, s.out_host)
        return dict(out=s.out_host, counts=b.counts, load=b.rank_load)
    if c["update"]:
        s.ctx.transpose_weights(s.w1, s.w3, s.w2, s.w1t, s.w3t, s.w2t)
    p = s.ctx.moe_forward(s.x, s.ids, s.gates, s.w1, s.w3, s.w2, b, want_plan=c["plan"])
    got = dict(out=b.out, counts=b.counts, load=b.rank_load, s2r=b.slot_to_row)
    if p is not None:
        got.update(before=p.load_before, after=p.load_after)
    if c["kind"] == "train":
        s.ctx.moe_backward(s.d_out, s.gates, s.w1t, s.w3t, s.w2t, b, s.bwd, *s.dw, accumulate=c["accumulate"])
        got.update(d_x=s.bwd.d_x, d_gates=s.bwd.d_gates, dw1=s.dw[0], dw3=s.dw[1], dw2=s.dw[2])
    return got


# ------------------------------------------------------------------------------------------ bounds

def _touched(c):
    """Experts that receive rows, on average over micro-batches (slots taken as independent draws)."""
    E, S, a = c["E"], c["T"] * c["K"], c["alpha"]
    if c["routing"] == "dirichlet":
        miss = math.exp(math.lgamma(a * E) - math.lgamma(a * (E - 1)) + math.lgamma(a * (E - 1) + S) - math.lgamma(a * E + S))
    else:
        miss = (1.0 - 1.0 / E) ** S
    return E * (1.0 - miss)


def work(case):
    c = case
    T, d, f, E, K = (c[k] for k in ("T", "d", "f", "E", "K"))
    S, ffn, n = T * K, 6.0 * c["T"] * c["K"] * d * f, _touched(c)
    if c["kind"] == "permute":
        # logits in; ids, gates and row indices out; x and y in; the permuted rows and the result out
        return {"bytes": 4.0 * T * E + 16.0 * S + 4.0 * T * d + 4.0 * S * d, "flops": 0.0}
    weights = 6.0 * d * f
    if c["kind"] == "train":
        # weights in both layouts, fp32 gradients out (and in, when accumulating), x, out, d_out, d_x
        grads = 24.0 * d * f * n if c["accumulate"] else 12.0 * d * f * E
        refresh = 2 * weights * E if c["update"] else 0.0
        return {"bytes": 2 * weights * n + grads + refresh + 8.0 * T * d + 16.0 * S, "flops": 3.0 * ffn}
    return {"bytes": weights * n + 4.0 * T * d + 12.0 * S, "flops": ffn}


def tolerance(case):
    """About four times the distance of the results from the same layer in 64-bit arithmetic without intermediate
    rounding: 2.9e-3 for the forward result (h, y and out are rounded to bf16), 3.8e-3 for the worst gradient,
    1.7e-3 where only the combined rows are rounded."""
    return {"rel": {"permute": 6e-3, "train": 1.5e-2}.get(case["kind"], 1.1e-2)}
