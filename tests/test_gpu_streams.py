"""Calls of one context on two streams.

A prediction call may run beside a routing call of the same context (the prediction of the next layer under the work of
this one).  They share no scratch, so each must give the bits it gives alone, however the two overlap.
"""
import pytest
import torch

from paper_2608_14205_b200 import binding as B
from paper_2608_14205_b200 import inputs as I
from tests import parity_util as P

pytestmark = pytest.mark.gpu


# few SM pairs per call, so that both calls' blocks are resident together: whole tiles, shared tiles, several tiles per pair
@pytest.mark.parametrize("name,T,pair_limit", [("tiny", 512, 0), ("qwen3", 200, 0), ("qwen3", 4000, 32), ("dsv3", 700, 12),
                                               ("qwen3", 2000, 2), ("dsv3", 700, 1)])
@pytest.mark.parametrize("routing", ["route", "layer"])
@pytest.mark.parametrize("prediction", ["predict", "plan"])
def test_prediction_and_routing_calls_of_one_context_overlap(name, T, pair_limit, routing, prediction):
    reps, wl = 150, I.WORKLOADS[name]
    layers = [I.make_layer(wl, l, 0, T=T) for l in range(2)]
    ctx = P.make_context(wl, T)
    ctx.fb_set_pair_limit(pair_limit)
    dev = torch.device("cuda", ctx.device)
    sb = layers[0].select_bias.to(dev) if layers[0].select_bias is not None else None
    router = B.make_router(layers[0].W.to(dev), None, sb)
    pi = layers[0].expert_to_slot.to(dev)
    budget = B.make_budget(**P.budget_kwargs(wl, T))
    x = [(li.h_prev.to(dev), li.H.to(dev)) for li in layers]
    i32 = lambda n: torch.full((max(1, n),), -3, dtype=torch.int32, device=dev)

    def pred_out():
        return dict(counts=i32(wl.E), pi_out=i32(wl.E), swaps=i32(4 * (wl.E // 2)).zero_(), n=i32(1), lb=i32(wl.R), la=i32(wl.R))

    def route_out():
        return dict(pred_out(), so=i32(wl.E + 1), ro=i32(wl.R + 1), rl=i32(wl.R))

    big = dict(ids=i32(T * wl.k), w=torch.zeros(T * wl.k, device=dev), perm=i32(T * wl.k), inv=i32(T * wl.k))

    def predict(i, o):
        if prediction == "plan":
            ctx.fb_predict_and_plan(router, x[i][0], T, pi, budget, 0, o["counts"], o["pi_out"], o["swaps"], o["n"], o["lb"], o["la"])
        else:
            ctx.fb_predict_load(router, x[i][0], T, o["counts"])

    def route(i, o):
        if routing == "layer":
            ctx.fb_layer_step(router, x[i][0], x[i][1], T, pi, budget, 0, o["counts"], o["pi_out"], o["swaps"], o["n"], o["lb"],
                              o["la"], big["ids"], big["w"], o["so"], o["ro"], big["perm"], big["inv"], o["rl"])
        else:
            ctx.fb_route_dispatch(router, x[i][1], T, pi, big["ids"], big["w"], o["so"], o["ro"], big["perm"], big["inv"], o["rl"])

    want = []
    for i in range(2):
        a, b = pred_out(), route_out()
        predict(i, a)
        torch.cuda.synchronize(dev)
        route(i, b)
        torch.cuda.synchronize(dev)
        want.append((a, b, {key: v.clone() for key, v in big.items()}))
    got = [(pred_out(), route_out()) for _ in range(reps)]
    side, main = torch.cuda.Stream(device=dev), torch.cuda.Stream(device=dev)
    torch.cuda.synchronize(dev)
    for j, (a, b) in enumerate(got):
        # two predictions and two routings of one context stay in order, each kind on a stream of its own
        with torch.cuda.stream(side):
            predict(j % 2, a)
        with torch.cuda.stream(main):
            route((j // 3) % 2, b)
    torch.cuda.synchronize(dev)
    assert ctx.fb_device_status() == 0
    for j, (a, b) in enumerate(got):
        for key, v in a.items():
            assert torch.equal(v, want[j % 2][0][key]), (j, "prediction", key)
        for key, v in b.items():
            assert torch.equal(v, want[(j // 3) % 2][1][key]), (j, "routing", key)
    for key, v in big.items():
        assert torch.equal(v, want[((reps - 1) // 3) % 2][2][key]), key
    ctx.close()


# The planner behind a router kernel neither runs on the SMs of another stream's kernel (its one warp got an issue slot in 30 there:
# planning took 50 to 70 us instead of 2) nor waits behind that kernel's blocks for the first SM that the router kernel leaves
# (600 us).  20 us leave room for the planner's launch.
@pytest.mark.parametrize("name,T,pairs", [("qwen3", 8192, 32), ("qwen3", 2000, 8), ("tiny", 512, 2)])
@pytest.mark.parametrize("other", ["on the other SMs", "right behind", "right behind, in waves"])
def test_planning_is_not_held_up_by_another_kernel(name, T, pairs, other):
    wl = I.WORKLOADS[name]
    li = I.make_layer(wl, 0, 0, T=T)
    ctx = P.make_context(wl, T)
    ctx.fb_set_pair_limit(pairs if other == "on the other SMs" else 0)
    dev = torch.device("cuda", ctx.device)
    router = B.make_router(li.W.to(dev), None, None)
    x, pi = li.h_prev.to(dev), li.expert_to_slot.to(dev)
    budget = B.make_budget(**P.budget_kwargs(wl, T))
    i32 = lambda n: torch.zeros(max(1, n), dtype=torch.int32, device=dev)
    o = (i32(wl.E), i32(wl.E), i32(4 * (wl.E // 2)), i32(1), i32(wl.R), i32(wl.R))
    n_sm = torch.cuda.get_device_properties(dev).multi_processor_count
    sink = torch.zeros(1024 * 1024, device=dev)
    main, side, gate = (torch.cuda.Stream(device=dev) for _ in range(3))

    def beside(call):
        times = []
        for _ in range(15):
            a, b, go = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True), torch.cuda.Event()
            with torch.cuda.stream(gate):
                torch.cuda._sleep(200000)                                      # until the host has queued the rest
                go.record()
            side.wait_event(go)
            main.wait_event(go)
            with torch.cuda.stream(side):
                if other == "on the other SMs":
                    torch.cuda._sleep(50000)                                   # until that kernel has its SMs
                a.record()
                call()
                b.record()
            with torch.cuda.stream(main):
                if other == "on the other SMs":
                    B.fb_standin_attention(sink, n_sm - 2 * pairs, 3000)       # some 400 us
                else:
                    torch.cuda._sleep(4000)                                    # 2 us
                    B.fb_standin_attention(sink, *((n_sm, 3000) if other == "right behind" else (1024, 400)))
            torch.cuda.synchronize(dev)
            times.append(a.elapsed_time(b) * 1e3)
        return min(times)                   # (now and then the other kernel has taken the SMs first)

    predict = beside(lambda: ctx.fb_predict_load(router, x, T, o[0]))
    plan = beside(lambda: ctx.fb_predict_and_plan(router, x, T, pi, budget, 0, *o))
    assert ctx.fb_device_status() == 0
    assert plan < predict + 20.0, (predict, plan)
    ctx.close()
