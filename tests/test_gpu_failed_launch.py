"""A call one of whose launches fails reports it and leaves nothing behind: the context's next calls give what they gave before.

The failure is made on the host (fb_fail_launch: the launch is not made).
"""
import pytest
import torch

from paper_2608_14205_b200 import binding as B
from paper_2608_14205_b200 import inputs as I
from tests import parity_util as P

pytestmark = pytest.mark.gpu


class _Calls:
    def __init__(self, name, T, pair_limit, bud):
        self.wl, self.T = I.WORKLOADS[name], T
        li = I.make_layer(self.wl, 0, 0, T=T)
        self.ctx = P.make_context(self.wl, T)
        self.ctx.fb_set_pair_limit(pair_limit)
        self.dev = torch.device("cuda", self.ctx.device)
        to = lambda t: t.to(self.dev) if t is not None else None
        self.router = B.make_router(to(li.W), to(li.logit_bias), to(li.select_bias))
        self.x, self.H, self.pi = to(li.h_prev), to(li.H), to(li.expert_to_slot)
        self.budget = B.make_budget(**P.budget_kwargs(self.wl, T, **bud))

    def run(self, call):
        wl, T, ctx = self.wl, self.T, self.ctx
        i32 = lambda n: torch.full((max(1, n),), -3, dtype=torch.int32, device=self.dev)
        plan = [i32(wl.E), i32(wl.E), i32(4 * (wl.E // 2)).zero_(), i32(1), i32(wl.R), i32(wl.R)]
        route = [i32(T * wl.k), torch.zeros(T * wl.k, device=self.dev), i32(wl.E + 1), i32(wl.R + 1), i32(T * wl.k),
                 i32(T * wl.k), i32(wl.R)]
        if call == "predict":
            ctx.fb_predict_load(self.router, self.x, T, plan[0])
        elif call == "plan":
            ctx.fb_predict_and_plan(self.router, self.x, T, self.pi, self.budget, 0, *plan)
        elif call == "route":
            ctx.fb_route_dispatch(self.router, self.H, T, self.pi, *route)
        else:
            ctx.fb_layer_step(self.router, self.x, self.H, T, self.pi, self.budget, 0, *plan, *route)
        assert ctx.fb_device_status() == 0
        return plan + route


# the plan made with the index, by the general planner between router and index, beside a persistent pass; an index over runs of tiles
@pytest.mark.parametrize("name,T,pair_limit,bud", [("qwen3", 700, 0, {}), ("qwen3", 700, 0, dict(mode=B.FB_PLAN_SWEEP)),
                                                   ("dsv3", 700, 0, dict(mode=B.FB_PLAN_WIDE, frontier_width=2)), ("qwen3", 1500, 2, {}),
                                                   ("qwen3", 1500, 2, dict(mode=B.FB_PLAN_SWEEP)), ("qwen3", 19000, 0, {})])
def test_a_failed_launch_leaves_nothing_behind(name, T, pair_limit, bud):
    c = _Calls(name, T, pair_limit, bud)
    want, launches = {}, {}
    for call in ("predict", "plan", "route", "layer"):
        before = c.ctx.fb_launch_count()
        want[call] = c.run(call)
        launches[call] = c.ctx.fb_launch_count() - before
    assert launches["route"] == 2 and launches["layer"] == (3 if bud else 2)
    for failing in want:
        for nth in range(1, launches[failing] + 1):
            c.ctx.fb_fail_launch(nth)
            with pytest.raises(B.FbError) as failed:
                c.run(failing)
            assert failed.value.status == B.FB_ERR_CUDA
            for call, outputs in want.items():
                for i, (a, b) in enumerate(zip(c.run(call), outputs)):
                    assert torch.equal(a, b), (failing, nth, call, i)
    c.ctx.close()


def test_a_failure_that_was_taken_back_or_refused_does_not_come():
    c = _Calls("tiny", 100, 0, {})
    with pytest.raises(B.FbError):
        c.ctx.fb_fail_launch(-1)
    c.run("layer")
    c.ctx.fb_fail_launch(1)
    c.ctx.fb_fail_launch(0)
    c.run("layer")
    c.ctx.close()
