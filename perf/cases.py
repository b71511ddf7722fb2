"""What the framework is timed on: the calls of its public API over the sizes they are used at.

A pass is one layer of one prefill step (or the part of it a caller asks for) on device buffers
that the caller keeps: the library allocates nothing per call, so a program holds a context, the
frozen router, a budget and its output buffers, and hands in new hidden states every time.

The inputs follow the recipes of ``paper_2608_14205_b200/inputs.py`` (router columns with a Zipf
popularity, unit-variance hidden states, task clusters for the sigmoid gates, a residual drift of
fixed relative norm), drawn on the GPU.  One thing is added: a token whose choice of experts hangs
on less than the rounding error of the router product is drawn again.  Two correct products that
add in a different order may order such a token's experts differently, and one moved assignment
shifts every later position of the dispatch index; without those tokens all whole-number outputs
are the same for every correct implementation.
"""
import dataclasses
import math

import torch

from paper_2608_14205_b200 import binding as B
from paper_2608_14205_b200 import inputs as I
from paper_2608_14205_b200 import serving as S

SOFTMAX, SIGMOID = I.GATE_SOFTMAX_TOPK, I.GATE_SIGMOID_GROUP_TOPK

# Shapes of the gates that the sizes below are taken at: the repository's own workloads, and one
# sigmoid gate without groups.  d hidden size, E experts, k per token, R expert-parallel ranks.
TINY = dict(d=1024, E=8, k=2, R=4, gate=SOFTMAX, n_group=1, topk_group=1, renorm=1, route_scale=1.0, rho=0.1,
            clusters=0, zipf_s=1.0, max_swaps=2, expert_bytes=0, window_ns=0)
MIXTRAL = dict(TINY, d=4096, R=8, zipf_s=1.2, max_swaps=1)
QWEN3 = dict(d=2048, E=128, k=8, R=8, gate=SOFTMAX, n_group=1, topk_group=1, renorm=1, route_scale=1.0, rho=0.15,
             clusters=0, zipf_s=1.0, max_swaps=6, expert_bytes=9 * 2**20, window_ns=0)
DSV3 = dict(d=7168, E=256, k=8, R=32, gate=SIGMOID, n_group=8, topk_group=4, renorm=1, route_scale=1.0, rho=0.1,
            clusters=3, zipf_s=1.1, max_swaps=128, expert_bytes=44_040_192, window_ns=500_000)
ONE_GROUP = dict(d=2048, E=64, k=6, R=8, gate=SIGMOID, n_group=1, topk_group=1, renorm=1, route_scale=2.5, rho=0.1,
                 clusters=3, zipf_s=1.0, max_swaps=4, expert_bytes=17 * 2**20, window_ns=500_000)

# The largest listed product of tokens, hidden size and passes over the hidden states.
LARGEST = 131072 * 2048 * 2


def listed():
    return [
        # fb_layer_step: both router passes, the plan and the dispatch index of one layer.
        # The smallest configuration: launches and latency.
        dict(TINY, name="layer tiny 512", call="layer", T=512),
        # A step with a handful of tokens (short prompts, a nearly drained batch).
        dict(QWEN3, name="layer qwen3 40", call="layer", T=40),
        # A gate of few experts, a medium prefill.
        dict(MIXTRAL, name="layer mixtral 4096", call="layer", T=4096),
        # An ordinary prefill step of a 128-expert softmax gate.
        dict(QWEN3, name="layer qwen3 8192", call="layer", T=8192),
        # The same model at the paper's batch, 16 sequences of 8K tokens: the largest call.
        dict(QWEN3, name="layer qwen3 131072", call="layer", T=131072),
        # A short, ragged prefill of the group-limited sigmoid gate.
        dict(DSV3, name="layer dsv3 1733", call="layer", T=1733),
        # The headline configuration.
        dict(DSV3, name="layer dsv3 16384", call="layer", T=16384),
        # A sigmoid gate without groups, ragged.
        dict(ONE_GROUP, name="layer sigmoid64 5003", call="layer", T=5003),
        # fb_predict_and_plan: the part that runs ahead of the layer, beside the attention before it.
        dict(DSV3, name="plan dsv3 16384", call="plan", T=16384),
        # One of 8 token shards of the headline batch: the separate device calls around the two
        # collectives (which need more than one GPU and are left out).
        dict(DSV3, name="shard dsv3 2048", call="shard", T=2048, world=8, rank=3),
        # A serving loop that also evaluates the quality of its predictions.
        dict(QWEN3, name="serve qwen3 8192", call="serve", T=8192),
        # fb_apply_swaps: the weights of a plan's experts trade places (five swaps of 44 MB experts).
        dict(name="exchange 5 x 44 MB", call="exchange", E=16, swaps=5, expert_bytes=44_040_192),
    ]


def _log_uniform(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    call = rng.choice(["layer", "layer", "layer", "plan", "plan", "shard", "serve", "exchange"])
    if call == "exchange":
        expert_bytes = 16 * _log_uniform(rng, 2**16, 44_040_192 // 16)       # 1 MB .. 44 MB
        return dict(call=call, E=16, swaps=rng.randint(1, 6), expert_bytes=expert_bytes)
    gate = rng.choice([
        TINY, MIXTRAL, QWEN3, QWEN3, DSV3, DSV3, ONE_GROUP,
        dict(QWEN3, E=64, k=rng.choice([4, 6, 8]), R=rng.choice([4, 8, 16])),
        dict(QWEN3, E=60, k=4, R=4, renorm=0),                                # weights without renormalisation
        dict(DSV3, d=4096, E=160, k=6, R=8, topk_group=3, route_scale=16.0),  # 20 experts per group
        dict(DSV3, R=64, rho=0.2, max_swaps=5),                               # long-prefill sweep: 4 experts per rank
    ])
    d = rng.choice([gate["d"], gate["d"], gate["d"], 8 * rng.randint(128, 896)])
    passes = 1 if call == "plan" else 2
    most = LARGEST // (passes * d) if call != "serve" else LARGEST // (4 * d)
    most = min(most, (1 << 21) // gate["k"])                                  # the planner's range of counts
    case = dict(gate, call=call, d=d, T=_log_uniform(rng, 1, min(most, 131072)))
    if call == "shard":
        world = rng.choice([2, 4, 8])
        case.update(world=world, rank=rng.randrange(world))
        case["T"] = max(1, case["T"] // world)
    return case


# ------------------------------------------------------------------ inputs

def _workload(case):
    return I.Workload("case", T=case["T"], d=case["d"], E=case["E"], k=case["k"], R=case["R"], layers=1,
                      gate=case["gate"], n_group=case["n_group"], topk_group=case["topk_group"],
                      renorm=case["renorm"], route_scale=case["route_scale"], rho=case["rho"],
                      skew="clusters" if case["clusters"] else "zipf", zipf_s=case["zipf_s"],
                      n_clusters=case["clusters"], max_swaps=case["max_swaps"])


def _undecided(x, W, select_bias, case):
    """Which rows' experts, or their order, hang on a difference that rounding may turn round.

    The fp32 sums of two implementations differ by up to about 1e-4 in a logit at the largest
    hidden size; the margins are twice that for logits, a quarter of it for sigmoid scores (the
    slope of a sigmoid is at most 1/4), twice the latter for sums of two scores."""
    E, k = case["E"], case["k"]
    bad = torch.empty(x.shape[0], dtype=torch.bool, device=x.device)
    for lo in range(0, x.shape[0], 16384):
        z = x[lo:lo + 16384].float() @ W.float().t()
        if case["gate"] == SOFTMAX:
            keys, margin = z, 2e-4
            eligible, b = E, torch.zeros(z.shape[0], dtype=torch.bool, device=x.device)
        else:
            keys, margin = torch.sigmoid(z) + select_bias, 5e-5
            G, kept = case["n_group"], case["topk_group"]
            grouped = keys.view(-1, G, E // G)
            score = grouped.topk(min(2, E // G), dim=2).values.sum(dim=2)
            ranked = score.sort(dim=1, descending=True)
            b = ranked.values[:, kept - 1] - ranked.values[:, kept] < 2 * margin if kept < G else \
                torch.zeros(z.shape[0], dtype=torch.bool, device=x.device)
            dropped = torch.ones_like(score, dtype=torch.bool).scatter_(1, ranked.indices[:, :kept], False)
            keys = grouped.masked_fill(dropped[:, :, None], -1e9).view(-1, E)
            eligible = kept * (E // G)
        top = keys.topk(min(k + 1, eligible), dim=1).values
        if top.shape[1] > 1:
            b = b | ((top[:, :-1] - top[:, 1:]).amin(dim=1) < margin)
        bad[lo:lo + 16384] = b
    return bad


def _hidden_states(case, wl, W, select_bias, g):
    """h_prev and H of one layer: unit noise around the sequence's cluster mean, then the drift."""
    T, d, dev = case["T"], case["d"], W.device
    mean = torch.zeros(1, d, device=dev)
    if case["clusters"]:
        Wf = W.float()
        offsets = torch.stack([_zipf_offsets(case, g, dev) for _ in range(case["clusters"])])
        mean = (offsets / (Wf * Wf).sum(dim=1).clamp_min(1e-12)) @ Wf
    n_seq = min(wl.n_sequences, T)
    of_seq = torch.randint(0, mean.shape[0], (n_seq,), generator=g, device=dev)
    cluster = of_seq[(torch.arange(T, device=dev) * n_seq) // T]
    h_prev = torch.empty(T, d, dtype=torch.bfloat16, device=dev)
    H = torch.empty_like(h_prev)
    todo = torch.arange(T, device=dev)
    for _ in range(12):
        for part in todo.split(16384):
            h = (torch.randn(part.numel(), d, generator=g, device=dev) + mean[cluster[part]]).to(torch.bfloat16)
            u = torch.randn(part.numel(), d, generator=g, device=dev)
            drift = case["rho"] * h.float().norm(dim=1, keepdim=True) / u.norm(dim=1, keepdim=True)
            h_prev[part], H[part] = h, (h.float() + u * drift).to(torch.bfloat16)
        x, y = (h_prev, H) if todo.numel() == T else (h_prev[todo], H[todo])
        todo = todo[_undecided(x, W, select_bias, case) | _undecided(y, W, select_bias, case)]
        if todo.numel() == 0:
            break
    return h_prev, H


def _zipf_offsets(case, g, dev):
    rank = torch.randperm(case["E"], generator=g, device=dev) + 1
    lw = -case["zipf_s"] * torch.log(rank.float())
    return 0.5 * (lw - lw.mean())


@dataclasses.dataclass
class State:
    case: dict
    router: object = None
    budget: object = None
    ctx: object = None
    loop: object = None
    h_prev: object = None
    H: object = None
    pi: object = None
    out: object = None
    counts_all: object = None
    weights: object = None


def prepare(case, seed):
    dev = torch.device("cuda", 0)
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    i32 = lambda n: torch.zeros(max(1, n), dtype=torch.int32, device=dev)   # noqa: E731
    if case["call"] == "exchange":
        E, n = case["E"], case["swaps"]
        s = State(case)
        s.weights = torch.randint(-2**15, 2**15, (E, case["expert_bytes"] // 2), generator=g, device=dev,
                                  dtype=torch.int16)
        s.pi = torch.randperm(E, generator=g, device=dev).to(torch.int32)
        pairs = torch.randperm(E, generator=g, device=dev)[:2 * n].view(n, 2).to(torch.int32)
        s.out = dict(swaps=torch.cat([s.pi[pairs.long()] // 2, pairs], dim=1).contiguous(), n_swaps=i32(1) + n)
        return s
    wl = _workload(case)
    T, E, k, R = case["T"], case["E"], case["k"], case["R"]
    W = I.make_router(wl, 0, int(seed)).to(dev)
    select_bias = 0.02 * torch.randn(E, generator=g, device=dev) if case["gate"] == SIGMOID else None
    s = State(case, router=B.make_router(W, None, select_bias))
    s.h_prev, s.H = _hidden_states(case, wl, W, select_bias, g)
    window = dict(global_ns=case["window_ns"], rank_ns=case["window_ns"], link_ns=case["window_ns"],
                  alpha_ns=(2000, 2000), fs_per_byte=(1111, 1111)) if case["window_ns"] else {}
    s.budget = S.make_budget_for(wl, T, expert_bytes=case["expert_bytes"], **window)
    if case["call"] == "serve":
        s.loop = S.ServingLoop(wl, T)
        return s
    s.ctx = B.Context(T, case["d"], E, k, R, case["gate"], case["n_group"], case["topk_group"], case["renorm"],
                      case["route_scale"])
    s.pi = torch.arange(E, dtype=torch.int32, device=dev)
    s.out = dict(counts=i32(E), pi_out=i32(E), swaps=i32(4 * max(1, min(case["max_swaps"], E // 2))).view(-1, 4),
                 n_swaps=i32(1), load_before=i32(R), load_after=i32(R))
    if case["call"] != "plan":
        s.out.update(ids=i32(T * k), w=torch.zeros(T * k, device=dev), slot_offsets=i32(E + 1),
                     rank_offsets=i32(R + 1), perm=i32(T * k), inv_perm=i32(T * k), rank_load=i32(R))
    if case["call"] == "shard":
        s.out["local_offsets"] = i32(E + 1)
        # what the other ranks' shards send: counts of the same size as this shard's
        s.counts_all = torch.randint(0, 2 * T * k // E + 2, (case["world"], E), generator=g, device=dev,
                                     dtype=torch.int32)
    return s


# ------------------------------------------------------------------ one pass

def run(s):
    case, o = s.case, s.out
    if case["call"] == "exchange":
        B.fb_apply_swaps(s.weights, case["expert_bytes"], case["E"], s.pi, o["swaps"], o["n_swaps"], case["swaps"])
        return s.weights
    T = case["T"]
    if case["call"] == "layer":
        s.ctx.fb_layer_step(s.router, s.h_prev, s.H, T, s.pi, s.budget, 0, o["counts"], o["pi_out"], o["swaps"],
                            o["n_swaps"], o["load_before"], o["load_after"], o["ids"], o["w"], o["slot_offsets"],
                            o["rank_offsets"], o["perm"], o["inv_perm"], o["rank_load"])
    elif case["call"] == "plan":
        s.ctx.fb_predict_and_plan(s.router, s.h_prev, T, s.pi, s.budget, 0, o["counts"], o["pi_out"], o["swaps"],
                                  o["n_swaps"], o["load_before"], o["load_after"])
    elif case["call"] == "shard":
        s.ctx.fb_predict_load(s.router, s.h_prev, T, o["counts"])
        s.ctx.fb_plan_swaps(o["counts"], s.pi, s.budget, 0, o["pi_out"], o["swaps"], o["n_swaps"], o["load_before"],
                            o["load_after"])
        s.ctx.fb_route_dispatch(s.router, s.H, T, o["pi_out"], o["ids"], o["w"], o["local_offsets"],
                                o["rank_offsets"], o["perm"], o["inv_perm"], o["rank_load"])
        s.ctx.fb_dispatch_slot_counts(o["local_offsets"], s.counts_all[case["rank"]])
        s.ctx.fb_dispatch_globalize(T, case["world"], case["rank"], s.counts_all, o["local_offsets"], o["ids"],
                                    o["pi_out"], o["inv_perm"], o["slot_offsets"], o["rank_offsets"], o["rank_load"])
    else:
        r = s.loop.layer_step(0, s.router, s.h_prev, s.H, s.budget, quality=True)
        quality = [r[m] for m in ("cos_hidden", "cos_logits", "hit_rate")]
        return dict(r["out"], pi_new=r["pi_new"], quality=quality)
    return o


def work(case):
    """Each pass reads its hidden states and the router once and writes its outputs once."""
    if case["call"] == "exchange":
        return dict(bytes=4 * case["swaps"] * case["expert_bytes"], flops=0)
    T, d, E, k = case["T"], case["d"], case["E"], case["k"]
    if case["call"] == "plan":
        return dict(bytes=2 * T * d + 2 * E * d + 8 * E, flops=2 * T * d * E)
    # ids, weights, perm and inv_perm: 16 bytes per assignment; both passes share the router's weights
    total = dict(bytes=2 * (2 * T * d) + 2 * E * d + 16 * T * k + 8 * E, flops=2 * (2 * T * d * E))
    if case["call"] == "shard":
        total["bytes"] += 4 * case["world"] * E
    return total


def tolerance(case):
    """Whole numbers are the same for every correct implementation (see _undecided).  The routing
    weights and the quality metrics follow from fp32 sums of exact products: with the sums in another
    order they move by up to 9.1e-7 (2-norm) and 8.3e-6 (largest, over the rms), against sums in fp64
    by up to 9.1e-7 and 1.9e-5."""
    if case["call"] in ("exchange", "plan"):
        return "exact"
    return {"rel": 4e-6, "max": 8e-5, "differ": 0.0}
