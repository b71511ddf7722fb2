"""GPU parity: every entry point of the C-ABI library against the CPU oracle on the
same seeded inputs (see tests/parity_util.py for the comparison rules)."""
import dataclasses

import numpy as np
import pytest
import torch

from oracle import freebalance_oracle as O
from paper_2608_14205_b200 import binding as B
from paper_2608_14205_b200 import inputs as I
from tests import parity_util as P

pytestmark = pytest.mark.gpu


def _run(wl, T, layer=0, seed=0, with_logit_bias=False, placement=None, want_logits=True, sample=None,
         pair_limit=0, **bud):
    li = I.make_layer(wl, layer, seed, T=T, with_logit_bias=with_logit_bias)
    ctx = P.make_context(wl, max(T, 1))
    bkw = P.budget_kwargs(wl, max(T, 1), **bud)
    gpu = P.run_gpu_layer(ctx, wl, li, bkw, want_logits=want_logits, placement=placement, pair_limit=pair_limit)
    gpu["persistent_launches"] = ctx.fb_persistent_launch_count()
    rep = P.compare_layer(wl, li, bkw, gpu, placement=placement, sample_rows=sample)
    ctx.close()
    return rep, gpu


# ------------------------------------------------------------------ the paper-shaped configs, reduced T
@pytest.mark.parametrize("name,T,layer", [
    ("tiny", 512, 0), ("tiny", 512, 1), ("tiny", 500, 0), ("tiny", 1, 0), ("tiny", 129, 1),
    ("mixtral", 300, 0), ("mixtral", 1000, 3),
    ("qwen3", 1000, 0), ("qwen3", 2500, 7),
    ("dsv3", 777, 0), ("dsv3", 1500, 11),
    ("sweep32k", 900, 0),
])
def test_config_shapes_small(name, T, layer):
    rep, gpu = _run(I.WORKLOADS[name], T, layer)
    assert rep["n_swaps"] <= I.WORKLOADS[name].max_swaps


def test_mixtral_one_expert_per_rank_never_swaps():
    rep, gpu = _run(I.WORKLOADS["mixtral"], 640)
    assert rep["n_swaps"] == 0 and gpu["pi_out"] == list(range(8))


def test_dsv3_cost_model_admits_five_swaps():
    rep, gpu = _run(I.WORKLOADS["dsv3"], 2048)
    assert rep["n_swaps"] == 5
    assert rep["pred_max_over_mean_after"] < rep["pred_max_over_mean_before"]


def test_empty_batch():
    wl = I.WORKLOADS["tiny"]
    rep, gpu = _run(wl, 0)
    assert gpu["counts"].sum() == 0 and rep["n_swaps"] == 0 and gpu["slot_offsets"].tolist() == [0] * 9


# ------------------------------------------------------------------ gating / shape edge cases
def _wl(**kw):
    base = dict(name="edge", T=300, d=256, E=16, k=2, R=4, layers=1, max_swaps=4, skew="zipf", zipf_s=1.0)
    base.update(kw)
    return I.Workload(**base)


@pytest.mark.parametrize("kw", [
    dict(k=1), dict(E=8, k=8, R=2), dict(E=24, k=3, R=3), dict(E=40, k=4, R=5, d=1000), dict(E=200, k=8, R=8, d=8),
    dict(d=72), dict(E=256, k=8, R=64, d=512), dict(E=64, k=6, R=8, d=2048),
    dict(gate=1, n_group=16, topk_group=3, k=3),                  # groups of one expert
    dict(gate=1, n_group=4, topk_group=2, k=8, E=16),              # k = all eligible experts
    dict(gate=1, n_group=1, topk_group=1, k=2),                    # one group: plain sigmoid top-k
    dict(gate=1, n_group=8, topk_group=8, k=5, E=64, R=8),         # every group kept
    dict(gate=1, n_group=32, topk_group=8, k=8, E=256, R=32, d=512),
    dict(gate=1, n_group=2, topk_group=1, k=3, E=24, R=4, route_scale=2.5),
    dict(renorm=0), dict(gate=1, n_group=4, topk_group=2, k=2, renorm=0, route_scale=2.5),
])
def test_edge_shapes(kw):
    _run(_wl(**kw), 300, with_logit_bias=True)


@pytest.mark.parametrize("kw,T", [
    (dict(E=192, k=6, R=8, d=1600), 700),                                    # 7 stages
    (dict(E=192, k=6, R=8, d=1600), 100),
    (dict(E=224, k=8, R=7, d=1096), 450),                                    # 7 stages
    (dict(gate=1, n_group=6, topk_group=3, k=6, E=192, R=6, d=1600), 700),   # ranking selection, 7 stages
])
def test_widths_whose_operand_ring_has_an_odd_number_of_stages(kw, T):
    # At these widths as many stages as fit is an odd number.  (One MMA issuer there; odd rings that two
    # issuers share: test_pipeline_depth_does_not_change_results, and gates of 113 to 128 experts with
    # several tiles per pair, five stages, in test_row_selection_of_restricted_gates_at_every_lane_layout.)
    _run(_wl(**kw), T, with_logit_bias=True)
    _run(_wl(**kw), T, layer=1)


def test_select_bias_large_enough_to_change_the_selection():
    wl = _wl(gate=1, n_group=4, topk_group=2, k=2)
    li = I.make_layer(wl, 0, 0, T=200)
    li.select_bias = torch.zeros(wl.E)
    li.select_bias[13] = 4.0                       # expert 13 now wins everywhere, its group is kept
    ctx = P.make_context(wl, 200)
    bkw = P.budget_kwargs(wl, 200)
    gpu = P.run_gpu_layer(ctx, wl, li, bkw)
    P.compare_layer(wl, li, bkw, gpu)
    assert (gpu["ids"][:, 0] == 13).all() and gpu["counts"][13] == 200
    assert (gpu["w"] < 1.0).all()                  # weights use the unbiased score


def test_exact_ties_go_to_the_lowest_ids():
    wl = _wl(E=16, k=3)
    li = I.make_layer(wl, 0, 0, T=150)
    li.W = torch.zeros_like(li.W)                  # all logits equal
    ctx = P.make_context(wl, 150)
    bkw = P.budget_kwargs(wl, 150)
    gpu = P.run_gpu_layer(ctx, wl, li, bkw)
    assert (gpu["ids"] == np.array([0, 1, 2])).all()
    assert gpu["counts"].tolist() == [150, 150, 150] + [0] * 13
    assert np.allclose(gpu["w"], 1 / 3, atol=1e-6)
    wl2 = _wl(gate=1, n_group=4, topk_group=2, k=3)
    li2 = I.make_layer(wl2, 0, 0, T=150)
    li2.W = torch.zeros_like(li2.W)
    li2.select_bias = torch.zeros(wl2.E)
    gpu2 = P.run_gpu_layer(P.make_context(wl2, 150), wl2, li2, P.budget_kwargs(wl2, 150))
    assert (gpu2["ids"] == np.array([0, 1, 2])).all()


# ------------------------------------------------------------------ planner variants through the kernel
@pytest.mark.parametrize("bud", [
    dict(tau_tokens=10**6), dict(max_swaps=0), dict(global_ns=0), dict(gamma_num=0, gamma_den=1),
    dict(gamma_num=3, gamma_den=0),
    dict(ranks_per_node=2, alpha_ns=(100, 900), fs_per_byte=(2000, 9000), expert_bytes=100_000,
         global_ns=3000, rank_ns=2500, link_ns=1500, max_swaps=8),
    dict(alpha_ns=(50, 50), fs_per_byte=(10**6, 10**6), global_ns=900, max_swaps=8,
         expert_bytes_table=[(7 * e * e + 13) % 400 + 1 for e in range(32)]),
])
def test_planner_budget_variants(bud):
    wl = _wl(E=32, k=4, R=4, max_swaps=8)
    _run(wl, 400, placement=I.random_placement(32, seed=5), **bud)


@pytest.mark.parametrize("seed", range(12))
def test_plan_swaps_alone_on_random_counts(seed):
    rng = np.random.default_rng(seed)
    R = int(rng.choice([2, 4, 8, 16, 32, 64]))
    m = int(rng.choice([1, 2, 4, 8, 16]))
    E = R * m
    if E > 256:
        m = 256 // R
        E = R * m
    counts = I.random_counts(E, int(rng.integers(0, 200_000)), seed, zipf_s=float(rng.choice([0.5, 1.0, 1.5])))
    pi = I.random_placement(E, seed)
    bkw = dict(max_swaps=int(rng.integers(0, E // 2 + 1)), gamma_num=int(rng.choice([0, 1, 5])),
               gamma_den=int(rng.choice([1, 64, 100_000])), tau_tokens=int(rng.choice([0, 0, 50])),
               alpha_ns=(int(rng.integers(0, 500)), int(rng.integers(0, 5000))),
               fs_per_byte=(int(rng.integers(0, 3000)), int(rng.integers(0, 20000))),
               expert_bytes=int(rng.integers(0, 10**7)), ranks_per_node=int(rng.choice([0, 2, 8])),
               global_ns=[O.U64_OFF, 10**5, 10**6][int(rng.integers(0, 3))],
               rank_ns=[O.U64_OFF, 10**5][int(rng.integers(0, 2))],
               link_ns=[O.U64_OFF, 5 * 10**4][int(rng.integers(0, 2))])
    ctx = B.Context(128, 64, E, 1, R)
    dev = torch.device("cuda")
    ms = max(1, bkw["max_swaps"])
    out_pi = torch.zeros(E, dtype=torch.int32, device=dev)
    swaps = torch.zeros(4 * ms, dtype=torch.int32, device=dev)
    n = torch.zeros(1, dtype=torch.int32, device=dev)
    lb = torch.zeros(R, dtype=torch.int32, device=dev)
    la = torch.zeros(R, dtype=torch.int32, device=dev)
    ctx.fb_plan_swaps(counts.to(torch.int32).to(dev), pi.to(dev), B.make_budget(**bkw), seed, out_pi, swaps, n, lb, la)
    assert ctx.fb_device_status() == 0
    want = O.plan_swaps(counts.tolist(), pi.tolist(), R, O.Budget(**bkw), layer_id=seed)
    got_swaps = [tuple(r) for r in swaps.cpu().numpy().reshape(-1, 4)[:int(n.item())].tolist()]
    assert (got_swaps, out_pi.cpu().tolist(), lb.cpu().tolist(), la.cpu().tolist()) == want


@pytest.mark.parametrize("seed", range(24))
def test_planner_variants_random_plans_exact(seed):
    """The one-pass sweep, the widened frontier and per-expert sizes run the general planner loop:
    exact agreement with the oracle's variant."""
    rng = np.random.default_rng(500 + seed)
    R = int(rng.choice([2, 3, 4, 8, 16, 64]))
    m = int(rng.choice([1, 2, 4, 8, 32]))
    E = R * m
    if E > 256:
        m = 256 // R
        E = R * m
    counts = I.random_counts(E, int(rng.integers(0, 200_000)), seed, zipf_s=float(rng.choice([0.5, 1.0, 1.5])))
    pi = I.random_placement(E, seed)
    mode = [B.FB_PLAN_SWEEP, B.FB_PLAN_WIDE, B.FB_PLAN_LOOP][seed % 3]
    bkw = dict(max_swaps=int(rng.integers(1, E // 2 + 1)) if E >= 2 else 0, gamma_num=int(rng.choice([0, 1, 5])),
               gamma_den=int(rng.choice([1, 64, 100_000])), tau_tokens=int(rng.choice([0, 0, 50])),
               alpha_ns=(int(rng.integers(0, 500)), int(rng.integers(0, 5000))),
               fs_per_byte=(int(rng.integers(0, 3000)), int(rng.integers(0, 20000))),
               expert_bytes=int(rng.integers(0, 10**7)), ranks_per_node=int(rng.choice([0, 2, 8])),
               global_ns=[O.U64_OFF, 10**5, 10**6][int(rng.integers(0, 3))],
               rank_ns=[O.U64_OFF, 10**5][int(rng.integers(0, 2))],
               link_ns=[O.U64_OFF, 5 * 10**4][int(rng.integers(0, 2))],
               mode=mode, frontier_width=int(rng.integers(1, 5)))
    table = None
    if mode == B.FB_PLAN_LOOP or seed % 4 == 0:                  # the loop mode reaches this path through a size table
        table = torch.as_tensor(rng.integers(1, 10**6, size=E), dtype=torch.int64)
    ctx = B.Context(128, 64, E, 1, R)
    dev = torch.device("cuda")
    ms = max(1, bkw["max_swaps"])
    out_pi = torch.zeros(E, dtype=torch.int32, device=dev)
    swaps = torch.zeros(4 * ms, dtype=torch.int32, device=dev)
    n = torch.zeros(1, dtype=torch.int32, device=dev)
    lb = torch.zeros(R, dtype=torch.int32, device=dev)
    la = torch.zeros(R, dtype=torch.int32, device=dev)
    gbud = B.make_budget(expert_bytes_table=None if table is None else table.to(dev), **bkw)
    ctx.fb_plan_swaps(counts.to(torch.int32).to(dev), pi.to(dev), gbud, seed, out_pi, swaps, n, lb, la)
    assert ctx.fb_device_status() == 0
    obud = O.Budget(expert_bytes_table=None if table is None else tuple(int(x) for x in table), **bkw)
    want = O.plan(counts.tolist(), pi.tolist(), R, obud, layer_id=seed)
    got_swaps = [tuple(r) for r in swaps.cpu().numpy().reshape(-1, 4)[:int(n.item())].tolist()]
    assert (got_swaps, out_pi.cpu().tolist(), lb.cpu().tolist(), la.cpu().tolist()) == want
    ctx.close()


def test_planner_variant_worked_examples_on_gpu(golden):
    for name, mode in [("planner_sweep_overshoots.json", B.FB_PLAN_SWEEP), ("planner_wide_frontier.json", B.FB_PLAN_WIDE)]:
        gd = golden(name)
        E, R = gd["E"], gd["R"]
        ctx = B.Context(128, 64, E, 1, R)
        dev = torch.device("cuda")
        t = lambda x: torch.tensor(x, dtype=torch.int32, device=dev)
        out_pi, swaps, n, lb, la = t([0] * E), t([0] * 16), t([0]), t([0] * R), t([0] * R)
        bud = B.make_budget(max_swaps=min(gd["max_swaps"], E // 2), gamma_num=gd["gamma_num"], gamma_den=gd["gamma_den"],
                            mode=mode, frontier_width=gd.get("frontier_width", 1))
        ctx.fb_plan_swaps(t(gd["counts"]), t(gd["expert_to_slot"]), bud, 0, out_pi, swaps, n, lb, la)
        assert ctx.fb_device_status() == 0
        k = int(n.item())
        assert swaps.cpu().numpy().reshape(-1, 4)[:k].tolist() == gd["swaps"]
        assert out_pi.cpu().tolist() == gd["expert_to_slot_out"]
        assert lb.cpu().tolist() == gd["load_before"] and la.cpu().tolist() == gd["load_after"]
        ctx.close()


def test_planner_worked_examples_on_gpu(golden):
    for name in ["planner_two_swaps_one_tie.json", "planner_tie_then_stop.json"]:
        gd = golden(name)
        E, R = gd["E"], gd["R"]
        ctx = B.Context(128, 64, E, 1, R)
        dev = torch.device("cuda")
        t = lambda x: torch.tensor(x, dtype=torch.int32, device=dev)
        out_pi, swaps, n, lb, la = t([0] * E), t([0] * 12), t([0]), t([0] * R), t([0] * R)
        bud = B.make_budget(max_swaps=min(gd["max_swaps"], E // 2), gamma_num=gd["gamma_num"], gamma_den=gd["gamma_den"])
        ctx.fb_plan_swaps(t(gd["counts"]), t(gd["expert_to_slot"]), bud, 0, out_pi, swaps, n, lb, la)
        assert ctx.fb_device_status() == 0
        k = int(n.item())
        assert swaps.cpu().numpy().reshape(-1, 4)[:k].tolist() == gd["swaps"]
        assert out_pi.cpu().tolist() == gd["expert_to_slot_out"]
        assert lb.cpu().tolist() == gd["load_before"] and la.cpu().tolist() == gd["load_after"]


# ------------------------------------------------------------------ errors and repeatability
def test_device_detected_errors_and_recovery():
    wl = I.WORKLOADS["tiny"]
    li = I.make_layer(wl, 0, 0, T=256)
    ctx = P.make_context(wl, 256)
    bkw = P.budget_kwargs(wl, 256)
    bad = torch.tensor([0, 1, 2, 3, 4, 5, 6, 6], dtype=torch.int32)          # slot 6 twice
    gpu = P.run_gpu_layer(ctx, wl, li, bkw, placement=bad)
    assert gpu["status"] == B.FB_ERR_BAD_PLACEMENT
    assert gpu["swaps"] == [] and gpu["fused"]["swaps"] == []
    out_of_range = torch.tensor([0, 1, 2, 3, 4, 5, 6, 99], dtype=torch.int32)
    assert P.run_gpu_layer(ctx, wl, li, bkw, placement=out_of_range)["status"] == B.FB_ERR_BAD_PLACEMENT
    # the context stays usable and the scratch histogram was left clean
    gpu = P.run_gpu_layer(ctx, wl, li, bkw)
    P.compare_layer(wl, li, bkw, gpu)
    # counts beyond the planner's range
    dev = torch.device("cuda")
    big = torch.full((8,), 2**20, dtype=torch.int32, device=dev)
    z = lambda n: torch.zeros(n, dtype=torch.int32, device=dev)
    ctx.fb_plan_swaps(big, li.expert_to_slot.to(dev), B.make_budget(max_swaps=2), 0, z(8), z(8), z(1), z(4), z(4))
    assert ctx.fb_device_status() == B.FB_ERR_RANGE
    assert ctx.fb_device_status() == 0


def test_host_detected_errors():
    wl = I.WORKLOADS["tiny"]
    ctx = P.make_context(wl, 128)
    dev = torch.device("cuda")
    li = I.make_layer(wl, 0, 0, T=256)
    router = B.make_router(li.W.to(dev))
    counts = torch.zeros(8, dtype=torch.int32, device=dev)
    with pytest.raises(B.FbError) as e:
        ctx.fb_predict_load(router, li.h_prev.to(dev), 256, counts)            # T > T_max
    assert e.value.status == B.FB_ERR_UNSUPPORTED_SHAPE
    with pytest.raises(B.FbError) as e:
        ctx.fb_predict_load(router, None, 64, counts)
    assert e.value.status == B.FB_ERR_INVALID_ARG
    with pytest.raises(B.FbError) as e:
        ctx.fb_predict_load(router, li.h_prev.to(dev), -1, counts)
    assert e.value.status == B.FB_ERR_INVALID_ARG
    z = lambda n: torch.zeros(n, dtype=torch.int32, device=dev)
    with pytest.raises(B.FbError) as e:                                        # max_swaps > E/2
        ctx.fb_plan_swaps(counts, z(8), B.make_budget(max_swaps=5), 0, z(8), z(20), z(1), z(4), z(4))
    assert e.value.status == B.FB_ERR_INVALID_ARG
    with pytest.raises(B.FbError) as e:                                        # gamma out of range
        ctx.fb_plan_swaps(counts, z(8), B.make_budget(max_swaps=1, gamma_num=2**21), 0, z(8), z(4), z(1), z(4), z(4))
    assert e.value.status == B.FB_ERR_INVALID_ARG
    with pytest.raises(B.FbError):
        B.Context(128, 64, 300, 2, 4)


def test_repeated_calls_are_bit_identical():
    wl = I.WORKLOADS["qwen3"]
    li = I.make_layer(wl, 2, 0, T=1111)
    ctx = P.make_context(wl, 1111)
    bkw = P.budget_kwargs(wl, 1111)
    a = P.run_gpu_layer(ctx, wl, li, bkw, want_logits=False)
    b = P.run_gpu_layer(ctx, wl, li, bkw, want_logits=False)
    for key in ("counts", "ids_early", "ids", "perm", "inv_perm", "slot_offsets", "rank_load"):
        assert np.array_equal(a[key], b[key]), key
    assert a["swaps"] == b["swaps"] and a["fused"]["swaps"] == b["fused"]["swaps"]
    assert np.array_equal(a["w"], b["w"])


def test_host_buffer_entry_point_matches_device_entry_points():
    wl = I.WORKLOADS["qwen3"]
    T = 700
    li = I.make_layer(wl, 1, 0, T=T)
    ctx = P.make_context(wl, T)
    bkw = P.budget_kwargs(wl, T)
    gpu = P.run_gpu_layer(ctx, wl, li, bkw, want_logits=False)
    dev = torch.device("cuda")
    router = B.make_router(li.W.to(dev))
    E, R, k = wl.E, wl.R, wl.k
    pin = lambda t: t.contiguous().pin_memory()
    i32 = lambda n: torch.zeros(n, dtype=torch.int32).pin_memory()
    outs = dict(counts=i32(E), expert_to_slot_out=i32(E), swaps=i32(4 * bkw["max_swaps"]), n_swaps=i32(1),
                load_before=i32(R), load_after=i32(R), topk_ids=i32(T * k),
                topk_w=torch.zeros(T * k).pin_memory(), slot_offsets=i32(E + 1), rank_offsets=i32(R + 1),
                perm=i32(T * k), inv_perm=i32(T * k), rank_load=i32(R))
    ctx.fb_layer_step_host(router, pin(li.h_prev), pin(li.H), T, pin(li.expert_to_slot), B.make_budget(**bkw), 0,
                           **outs)
    assert ctx.fb_device_status() == 0
    # the host-buffer call is fb_layer_step plus copies: bit for bit the device-buffer call's results
    ly = gpu["layer"]
    assert outs["counts"].tolist() == ly["counts"].tolist()
    n = int(outs["n_swaps"].item())
    assert [tuple(r) for r in outs["swaps"].numpy().reshape(-1, 4)[:n].tolist()] == ly["swaps"]
    assert outs["expert_to_slot_out"].tolist() == ly["pi_out"]
    assert np.array_equal(outs["topk_ids"].numpy().reshape(T, k), ly["ids"])
    assert np.array_equal(outs["perm"].numpy(), ly["perm"]) and np.array_equal(outs["inv_perm"].numpy(), ly["inv_perm"])
    assert outs["rank_load"].tolist() == ly["rank_load"].tolist()
    assert np.allclose(outs["topk_w"].numpy().reshape(T, k), ly["w"], atol=0, rtol=0)


# ------------------------------------------------------------------ full size, the benchmark's launch configuration
def test_dsv3_full_size_every_output():
    wl = I.WORKLOADS["dsv3"]
    rep, gpu = _run(wl, wl.T, layer=0, want_logits=False)
    assert rep["n_swaps"] == 5
    assert rep["real_max_over_mean_after"] < rep["real_max_over_mean_before"]
    # near-tie bookkeeping at both thresholds (shown with pytest -s / -rP)
    for name in ("early", "final"):
        print(f"dsv3 full size, {name} pass: " + ", ".join(
            f"{key}={rep[f'{name}_{key}']}" for key in (
                "flagged", "mismatch_flagged", "mismatch_unflagged", "tight_eps", "flagged_tight",
                "mismatch_flagged_tight", "mismatch_unflagged_tight")))
        # the tight threshold exempts a few percent of the tokens at most
        assert rep[f"{name}_flagged_tight"] <= 0.05 * wl.T


@pytest.mark.parametrize("name", ["sweep32k", "sweep64k", "qwen3_b16"])     # qwen3_b16: 16 x 8K tokens, 131072 rows
def test_long_prefill_sweep_sampled(name):
    wl = I.WORKLOADS[name]
    rows = np.random.default_rng(0).choice(wl.T, size=2048, replace=False)
    rows.sort()
    rep, gpu = _run(wl, wl.T, layer=0, want_logits=False, sample=rows)
    assert rep["n_swaps"] <= wl.max_swaps


@pytest.mark.parametrize("name", ["mixtral", "qwen3"])
def test_mid_configs_full_size(name):
    wl = I.WORKLOADS[name]
    _run(wl, wl.T, layer=0, want_logits=False)


# ------------------------------------------------------------------ more layers, drifts and budgets
@pytest.mark.parametrize("layer", [19, 38, 57])
def test_dsv3_spread_layers(layer):
    rep, gpu = _run(I.WORKLOADS["dsv3"], 4096, layer=layer, want_logits=False)
    assert rep["n_swaps"] <= 5


@pytest.mark.parametrize("rho,cap", [(0.05, 0), (0.2, 2), (0.4, 10)])
def test_sweep_shape_drift_and_budget(rho, cap):
    wl = dataclasses.replace(I.WORKLOADS["sweep32k"], rho=rho, max_swaps=cap)
    rep, gpu = _run(wl, 3000, layer=1, want_logits=False)
    assert rep["n_swaps"] <= cap
    if cap == 0:
        assert gpu["pi_out"] == list(range(wl.E))          # empty plan keeps the placement


def test_planner_is_identical_on_every_replay():
    # every rank replays the planner on the same counts: R runs must give one plan
    wl = I.WORKLOADS["dsv3"]
    counts = I.random_counts(wl.E, 100_000, seed=11, zipf_s=1.1).to(torch.int32)
    ctx = B.Context(128, 64, wl.E, 1, wl.R)
    dev = torch.device("cuda")
    bud = B.make_budget(**P.budget_kwargs(wl, 12_500))
    seen = set()
    for _ in range(wl.R):
        z = lambda n: torch.zeros(n, dtype=torch.int32, device=dev)
        out_pi, swaps, n, lb, la = z(wl.E), z(4 * 128), z(1), z(wl.R), z(wl.R)
        ctx.fb_plan_swaps(counts.to(dev), torch.arange(wl.E, dtype=torch.int32, device=dev), bud, 3, out_pi, swaps, n,
                          lb, la)
        seen.add((tuple(out_pi.cpu().tolist()), tuple(swaps.cpu().tolist()[:4 * int(n.item())]), tuple(la.cpu().tolist())))
    assert len(seen) == 1


@pytest.mark.parametrize("name", ["qwen3", "dsv3"])
def test_all_equal_keys_take_the_overflow_path(name):
    # all logits equal: every key reaches the selection bound, the short candidate list
    # overflows and the plain scan must still pick the lowest ids (lowest groups first)
    wl = I.WORKLOADS[name]
    T = 300
    li = I.make_layer(wl, 0, 0, T=T)
    li.W = torch.zeros_like(li.W)
    if li.select_bias is not None:
        li.select_bias = torch.zeros(wl.E)
    ctx = P.make_context(wl, T)
    bkw = P.budget_kwargs(wl, T)
    gpu = P.run_gpu_layer(ctx, wl, li, bkw)
    assert gpu["status"] == 0
    assert (gpu["ids"] == np.arange(wl.k)).all() and (gpu["ids_early"] == np.arange(wl.k)).all()
    assert gpu["counts"].tolist() == [T] * wl.k + [0] * (wl.E - wl.k)
    P.compare_layer(wl, li, bkw, gpu)


@pytest.mark.parametrize("seed", range(16))
def test_random_shapes(seed):
    rng = np.random.default_rng(1000 + seed)
    gate = int(rng.integers(0, 2))
    if gate:
        n_group = int(rng.choice([1, 2, 4, 8]))
        gs = int(rng.choice([1, 2, 4, 8, 16, 32]))
        E = n_group * gs
        if E > 256 or E < 2:
            E, n_group, gs = 64, 8, 8
        topk_group = int(rng.integers(1, min(n_group, 8) + 1))
        k = int(rng.integers(1, min(8, topk_group * gs) + 1))
    else:
        E = int(rng.choice([2, 8, 24, 32, 64, 96, 128, 160, 256]))
        n_group = topk_group = 1
        k = int(rng.integers(1, min(8, E) + 1))
    divisors = [r for r in (1, 2, 4, 8, 16, 32, 64) if E % r == 0]
    R = int(rng.choice(divisors))
    d = int(rng.choice([8, 64, 200, 512, 1096]))
    T = int(rng.choice([1, 77, 128, 129, 300, 640]))
    wl = I.Workload(name="fuzz", T=T, d=d, E=E, k=k, R=R, layers=1, gate=gate, n_group=n_group,
                    topk_group=topk_group, renorm=int(rng.integers(0, 2)), route_scale=float(rng.choice([1.0, 2.5])),
                    rho=0.2, skew="zipf", zipf_s=1.0, max_swaps=int(rng.integers(0, E // 2 + 1)))
    _run(wl, T, layer=seed, with_logit_bias=bool(rng.integers(0, 2)))


@pytest.mark.parametrize("E,R", [(160, 8), (256, 8), (256, 4), (256, 2), (198, 6), (66, 2), (17, 1)])
@pytest.mark.parametrize("bud", [dict(), dict(gamma_num=0), dict(ranks_per_node=2, alpha_ns=(100, 900), fs_per_byte=(2000, 9000),
                                                                  expert_bytes=100_000, global_ns=6000, rank_ns=3000, link_ns=2500)])
def test_planner_with_many_experts_per_rank(E, R, bud):
    # more than 16 experts per rank, in the separate call and in the layer step (whole numbers: exact)
    _run(_wl(E=E, k=4, R=R, d=64, max_swaps=12), 700, placement=I.random_placement(E, seed=R), **bud)


@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17])
@pytest.mark.parametrize("gamma_num,most", [(1, 4), (0, 4), (1, 2**21)])
def test_planner_at_the_edges_of_its_lane_layouts(m, gamma_num, most):
    # whole numbers: exact.  Counts below 4 make nearly every choice a tie; the largest add up to the planner's range.
    R, rng = 8, np.random.default_rng(m)
    E, ms = R * m, max(1, min(R * m // 2, 20))
    counts = rng.integers(0, max(4, most // E), E)
    if most > 4:
        counts[rng.integers(0, E)] += most - int(counts.sum())
    pi = I.random_placement(E, m)
    bkw = dict(max_swaps=ms, gamma_num=gamma_num, gamma_den=7)
    ctx = B.Context(128, 64, E, 1, R)
    dev = torch.device("cuda")
    z = lambda n: torch.zeros(n, dtype=torch.int32, device=dev)
    out_pi, swaps, n, lb, la = z(E), z(4 * ms), z(1), z(R), z(R)
    ctx.fb_plan_swaps(torch.tensor(counts, dtype=torch.int32, device=dev), pi.to(dev), B.make_budget(**bkw), 0, out_pi, swaps,
                      n, lb, la)
    assert ctx.fb_device_status() == 0
    want = O.plan_swaps(counts.tolist(), pi.tolist(), R, O.Budget(**bkw), layer_id=0)
    got = [tuple(r) for r in swaps.cpu().numpy().reshape(-1, 4)[:int(n.item())].tolist()]
    assert (got, out_pi.cpu().tolist(), lb.cpu().tolist(), la.cpu().tolist()) == want


@pytest.mark.parametrize("name,T", [("qwen3", 700), ("dsv3", 1500), ("qwen3", 19000)])
def test_a_refused_placement_leaves_nothing_behind_for_the_next_call(name, T):
    # the sums that the router kernel hands to the dispatch index are put back to zero whatever comes of the index
    wl = I.WORKLOADS[name]
    li = I.make_layer(wl, 0, 0, T=T)
    ctx, bkw = P.make_context(wl, T), P.budget_kwargs(wl, T)
    assert P.run_gpu_layer(ctx, wl, li, bkw, placement=torch.zeros(wl.E, dtype=torch.int32))["status"] == B.FB_ERR_BAD_PLACEMENT
    gpu = P.run_gpu_layer(ctx, wl, li, bkw)
    P.compare_layer(wl, li, bkw, gpu, sample_rows=np.arange(0, T, 37))


# ------------------------------------------------------------------ persistent router kernel (several tiles per block pair)
@pytest.mark.parametrize("name,T,limit,d,lb", [
    ("dsv3", 777, 1, None, False), ("dsv3", 1500, 2, None, False), ("dsv3", 2049, 3, None, True),
    ("dsv3", 1000, 1, 448, False),      # 7 k-blocks: the two issuers' shares differ in length
    ("dsv3", 600, 1, 64, True),         # a single k-block: only one accumulator is written
    ("qwen3", 1000, 1, None, False), ("qwen3", 2500, 2, None, True), ("sweep32k", 900, 1, None, False),
])
def test_persistent_kernel_small(name, T, limit, d, lb):
    wl = I.WORKLOADS[name]
    if d is not None:
        wl = dataclasses.replace(wl, d=d)
    rep, gpu = _run(wl, T, layer=1, with_logit_bias=lb, want_logits=False, pair_limit=limit)
    # predict, predict+plan, route+dispatch and the one-call layer step all took that kernel
    assert gpu["persistent_launches"] == 4


@pytest.mark.parametrize("name", ["qwen3", "dsv3"])
def test_persistent_kernel_overflow_path(name):
    wl = I.WORKLOADS[name]
    T = 700
    li = I.make_layer(wl, 0, 0, T=T)
    li.W = torch.zeros_like(li.W)
    li.W[:, 0] = 0.02                     # rows differ in their common logit only: all keys of a row stay equal
    if li.select_bias is not None:
        li.select_bias = torch.zeros(wl.E)
    ctx = P.make_context(wl, T)
    bkw = P.budget_kwargs(wl, T)
    gpu = P.run_gpu_layer(ctx, wl, li, bkw, want_logits=False, pair_limit=1)
    assert ctx.fb_persistent_launch_count() == 4
    assert (gpu["ids"] == np.arange(wl.k)).all() and (gpu["ids_early"] == np.arange(wl.k)).all()
    P.compare_layer(wl, li, bkw, gpu)
    ctx.close()


def test_persistent_kernel_mixed_rows_overflow_and_not():
    # half of the rows have all keys equal (overflow path), the others are ordinary
    wl = I.WORKLOADS["dsv3"]
    T = 900
    li = I.make_layer(wl, 2, 0, T=T)
    li.h_prev[::2] = 0
    li.H[::2] = 0
    li.select_bias = torch.zeros(wl.E)
    ctx = P.make_context(wl, T)
    bkw = P.budget_kwargs(wl, T)
    gpu = P.run_gpu_layer(ctx, wl, li, bkw, want_logits=False, pair_limit=2)
    assert ctx.fb_persistent_launch_count() == 4
    assert (gpu["ids"][::2] == np.arange(wl.k)).all()
    P.compare_layer(wl, li, bkw, gpu)
    ctx.close()


def test_pair_limit_does_not_change_results():
    # The persistent kernel and the one-tile kernel add their fp32 products in the same order, so
    # a pair limit (which selects between them) changes no bit of any output - as long as the
    # k-range split, which regroups the sums, is off.
    wl = I.WORKLOADS["dsv3"]
    T = 3000
    li = I.make_layer(wl, 5, 0, T=T)
    ctx = P.make_context(wl, T)
    ctx.fb_set_split(0)
    bkw = P.budget_kwargs(wl, T)
    ref = P.run_gpu_layer(ctx, wl, li, bkw, want_logits=False)
    assert ctx.fb_persistent_launch_count() == 0
    for limit in (1, 5, 11):
        got = P.run_gpu_layer(ctx, wl, li, bkw, want_logits=False, pair_limit=limit)
        for key in ("counts", "ids_early", "ids", "w", "perm", "inv_perm", "slot_offsets", "rank_load"):
            assert np.array_equal(ref[key], got[key]), (limit, key)
        assert ref["swaps"] == got["swaps"] and ref["layer"]["swaps"] == got["layer"]["swaps"]
        assert np.array_equal(ref["layer"]["ids"], got["layer"]["ids"]) and np.array_equal(ref["layer"]["w"], got["layer"]["w"])
    assert ctx.fb_persistent_launch_count() == 12
    ctx.close()


@pytest.mark.parametrize("name,T,split,d", [("dsv3", 3000, 0, None), ("qwen3", 2500, 0, None), ("dsv3", 1100, 1, None),
                                             ("dsv3", 1300, 0, 2112), ("qwen3", 1300, 0, 2112)])
def test_pipeline_depth_does_not_change_results(name, T, split, d):
    # Short operand rings, and rings with an odd number of stages (where two MMA issuers work, at up to
    # 128 columns, a stage then alternates between them and they keep each other informed of their
    # progress): same bits as the full depth, through the one-tile kernel, tiles shared by several pairs
    # and the persistent kernel.  With three
    # stages an issuer that took a stale phase of a "full" barrier for its own would read operands
    # that have not arrived.  d = 2112 gives an odd number of k-blocks: in the persistent kernel the
    # issuer that owns a ring position then changes from tile to tile.
    wl = I.WORKLOADS[name]
    if d is not None:
        wl = dataclasses.replace(wl, d=d)
    li = I.make_layer(wl, 3, 0, T=T)
    ctx = P.make_context(wl, T)
    ctx.fb_set_split(split)
    bkw = P.budget_kwargs(wl, T)
    ref = {lim: P.run_gpu_layer(ctx, wl, li, bkw, want_logits=False, pair_limit=lim) for lim in (0, 3)}
    for stages in (3, 2, 5):
        ctx.fb_set_stage_limit(stages)
        for lim in (0, 3):
            for _ in range(3):
                got = P.run_gpu_layer(ctx, wl, li, bkw, want_logits=False, pair_limit=lim)
                assert got["status"] == 0
                for key in ("counts", "ids_early", "ids", "w", "perm", "inv_perm", "slot_offsets", "rank_load"):
                    assert np.array_equal(ref[lim][key], got[key]), (stages, lim, key)
                assert ref[lim]["swaps"] == got["swaps"] and ref[lim]["layer"]["swaps"] == got["layer"]["swaps"]
                assert np.array_equal(ref[lim]["layer"]["ids"], got["layer"]["ids"])
    ctx.fb_set_stage_limit(0)
    with pytest.raises(Exception):
        ctx.fb_set_stage_limit(1)
    ctx.close()


@pytest.mark.parametrize("name,T,d", [("qwen3", 8192, None), ("mixtral", 4096, None), ("dsv3", 4096, None),
                                       ("qwen3", 1000, None), ("dsv3", 2049, 2112), ("mixtral", 300, 2048)])
def test_k_range_split_on_and_off_agree_with_the_oracle(name, T, d):
    # Where two to eight times as many SM pairs as tile pairs fit, that many share a tile's k-range;
    # both settings must satisfy the oracle, and the counts may differ between them only in
    # near-tie tokens.
    wl = I.WORKLOADS[name]
    if d is not None:
        wl = dataclasses.replace(wl, d=d)
    li = I.make_layer(wl, 2, 0, T=T)
    bkw = P.budget_kwargs(wl, T)
    sample = None if T <= 2500 else np.sort(np.random.default_rng(1).choice(T, size=1500, replace=False))
    counts = {}
    for mode in (1, 0):
        ctx = P.make_context(wl, T)
        ctx.fb_set_split(mode)
        gpu = P.run_gpu_layer(ctx, wl, li, bkw, want_logits=sample is None)
        rep = P.compare_layer(wl, li, bkw, gpu, sample_rows=sample)
        counts[mode] = gpu["counts"]
        ctx.close()
    assert int(np.abs(counts[0] - counts[1]).sum()) <= 2 * wl.k * max(1, T // 200)
    for bias in (0, 5):                                   # accepted, without effect: still the oracle's results
        ctx = P.make_context(wl, T)
        ctx.fb_set_split(1, bias)
        gpu = P.run_gpu_layer(ctx, wl, li, bkw, want_logits=False)
        P.compare_layer(wl, li, bkw, gpu, sample_rows=sample)
        ctx.close()


def test_router_launch_events_and_pair_queries():
    wl = I.WORKLOADS["dsv3"]
    T = 1024
    li = I.make_layer(wl, 0, 0, T=T)
    ctx = P.make_context(wl, T)
    assert 1 <= ctx.fb_max_pairs() <= 74                 # one block pair per two SMs at most
    dev = torch.device("cuda", ctx.device)
    router = B.make_router(li.W.to(dev), None, li.select_bias.to(dev))
    counts = torch.zeros(wl.E, dtype=torch.int32, device=dev)
    before, after = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    x = li.h_prev.to(dev)
    ctx.fb_predict_load(router, x, T, counts)            # warm-up
    ctx.fb_time_next_router_launch(before, after)
    ctx.fb_predict_load(router, x, T, counts)
    ctx.fb_predict_load(router, x, T, counts)            # not timed: the request was for one launch
    torch.cuda.synchronize(dev)
    us = before.elapsed_time(after) * 1e3
    assert 1.0 < us < 500.0, us
    assert int(counts.sum().item()) == T * wl.k
    ctx.close()
    tiny = P.make_context(I.WORKLOADS["tiny"], 512)
    assert tiny.fb_max_pairs() == 0                      # E = 8: the persistent kernel does not apply
    with pytest.raises(Exception):
        tiny.fb_set_pair_limit(-1)
    tiny.close()


def test_main_loop_floor_launches_leave_no_trace():
    # The measurement launches (operands loaded only / loaded and multiplied, nothing after the main
    # loop) write no output, take no ticket and leave the context ready for the next normal call.
    for name, T in (("dsv3", 1500), ("tiny", 300), ("qwen3", 700)):
        wl = I.WORKLOADS[name]
        li = I.make_layer(wl, 1, 0, T=T)
        ctx = P.make_context(wl, T)
        dev = torch.device("cuda", ctx.device)
        sb = li.select_bias.to(dev) if li.select_bias is not None else None
        router = B.make_router(li.W.to(dev), None, sb)
        x = li.h_prev.to(dev)
        counts, ref = (torch.full((wl.E,), -7, dtype=torch.int32, device=dev) for _ in range(2))
        ctx.fb_predict_load(router, x, T, ref)
        launches = ctx.fb_launch_count()
        for what in (1, 2, 2, 1):
            ctx.fb_router_floor(router, x, T, what)
        torch.cuda.synchronize(dev)
        assert ctx.fb_device_status() == 0
        assert ctx.fb_launch_count() == launches + 4
        ctx.fb_predict_load(router, x, T, counts)
        torch.cuda.synchronize(dev)
        assert torch.equal(counts, ref) and int(counts.sum().item()) == T * wl.k
        with pytest.raises(Exception):
            ctx.fb_router_floor(router, x, T, 3)
        ctx.close()


def test_two_contexts_on_two_streams_do_not_interfere():
    # each context owns its scratch: calls of different contexts may overlap on the device
    wl = I.WORKLOADS["dsv3"]
    T = 1500
    dev = torch.device("cuda")
    layers = [I.make_layer(wl, l, 0, T=T) for l in (0, 1)]
    ctxs = [P.make_context(wl, T) for _ in layers]
    streams = [torch.cuda.Stream() for _ in layers]
    budget = B.make_budget(**P.budget_kwargs(wl, T))
    i32 = lambda n: torch.zeros(n, dtype=torch.int32, device=dev)

    def buffers():
        return dict(counts=i32(wl.E), pi_out=i32(wl.E), swaps=i32(4 * 128), n=i32(1), lb=i32(wl.R), la=i32(wl.R),
                    ids=i32(T * wl.k), w=torch.zeros(T * wl.k, device=dev), so=i32(wl.E + 1), ro=i32(wl.R + 1),
                    perm=i32(T * wl.k), inv=i32(T * wl.k), rl=i32(wl.R))

    def call(ctx, li_dev, o, stream):
        ctx.fb_layer_step(li_dev["router"], li_dev["h"], li_dev["H"], T, li_dev["pi"], budget, 0, o["counts"],
                          o["pi_out"], o["swaps"], o["n"], o["lb"], o["la"], o["ids"], o["w"], o["so"], o["ro"],
                          o["perm"], o["inv"], o["rl"], stream=stream)

    devs = [dict(router=B.make_router(li.W.to(dev), None, li.select_bias.to(dev)), h=li.h_prev.to(dev),
                 H=li.H.to(dev), pi=li.expert_to_slot.to(dev)) for li in layers]
    serial = [buffers() for _ in layers]
    for ctx, d, o in zip(ctxs, devs, serial):
        call(ctx, d, o, None)
        torch.cuda.synchronize()
    overlapped = [buffers() for _ in layers]
    torch.cuda.synchronize()
    for rep in range(5):
        for ctx, d, o, st in zip(ctxs, devs, overlapped, streams):
            call(ctx, d, o, st)
    torch.cuda.synchronize()
    for a, b in zip(serial, overlapped):
        for key in a:
            assert torch.equal(a[key], b[key]), key
    assert all(c.fb_device_status() == 0 for c in ctxs)
    for c in ctxs:
        c.close()


@pytest.mark.parametrize("kw,T,limit", [
    # narrow gates: four accumulator sets' worth of columns fit, so tiles alternate between two sets
    (dict(E=128, k=6, R=16, gate=1, n_group=4, topk_group=3, d=704), 1500, 1),
    (dict(E=64, k=4, R=8, gate=1, n_group=2, topk_group=2, d=448), 2049, 2),
    (dict(E=64, k=4, R=8, gate=0, d=1024), 1300, 1),
    (dict(E=32, k=2, R=4, gate=0, d=64), 1100, 1),
    (dict(E=256, k=8, R=32, gate=0, d=512), 900, 1),          # eight chunks: the wide bound tables
])
def test_persistent_kernel_narrow_and_wide_gates(kw, T, limit):
    wl = _wl(**kw)
    rep, gpu = _run(wl, T, layer=2, want_logits=False, pair_limit=limit)
    assert gpu["persistent_launches"] == 4


def test_dispatch_index_with_several_tiles_per_block():
    # more tiles than SMs: every block of the dispatch-index kernel walks a run of six tiles, a batch
    # of four and one of two (the carried counts are exercised)
    wl = _wl(E=64, k=4, R=8, gate=0, d=64, max_swaps=6)
    T = 100_000
    rng = np.random.default_rng(0)
    sample = np.sort(rng.choice(T, size=512, replace=False))
    rep, gpu = _run(wl, T, want_logits=False, sample=sample)
    assert rep["early_mismatch_unflagged"] == 0 and rep["final_mismatch_unflagged"] == 0


@pytest.mark.parametrize("E,k,R,T", [
    (8, 2, 4, 128 * 148 + 1),       # one 16-expert unit per row of the histogram table; runs of two tiles, the last of one row
    (40, 3, 5, 128 * 149),          # three units: a count that does not divide a warp
    (160, 6, 8, 128 * 148 * 5 - 3), # ten units; runs of five tiles: a batch of four and a single tile
    (256, 8, 64, 128 * 148 * 4),    # sixteen units, full batches
    (96, 7, 6, 100), (256, 1, 8, 129),   # one tile per block
])
def test_dispatch_index_over_table_widths_and_runs_of_tiles(E, k, R, T):
    # whole numbers only: the index is checked entry by entry against the oracle's on the GPU's own ids
    wl = _wl(E=E, k=k, R=R, gate=0, d=64, max_swaps=3)
    sample = None if T <= 2500 else np.sort(np.random.default_rng(3).choice(T, size=200, replace=False))
    _run(wl, T, want_logits=False, sample=sample)


@pytest.mark.parametrize("kw", [
    dict(E=16, k=2, R=4),                                             # one column per lane
    dict(E=33, k=4, R=3, renorm=0),                                   # two, the last lane holds one; softmax denominator
    dict(E=100, k=6, R=4),                                            # four
    dict(E=200, k=8, R=8, renorm=0), dict(E=250, k=8, R=5),           # eight; the last lane's second vector is padding
    dict(gate=1, n_group=5, topk_group=2, k=7, E=250, R=5),           # sixteen; bound from the lanes, idle lanes
    dict(gate=1, n_group=8, topk_group=3, k=6, E=160, R=8),           # groups of 20 over four lanes: two vectors per lane
    dict(gate=1, n_group=32, topk_group=4, k=8, E=64, R=8),           # groups of two
    dict(gate=1, n_group=3, topk_group=3, k=5, E=96, R=6, route_scale=2.5),   # every group kept
    dict(E=128, k=8, R=8), dict(gate=1, n_group=8, topk_group=4, k=8, E=256, R=32),   # ranking gates, tiles shared by pairs
])
@pytest.mark.parametrize("T,limit", [
    (1, 0), (17, 0), (129, 0),          # one tile pair: eight block pairs share it; slices of 16 rows, the last partly or not filled
    (1300, 0), (4500, 0),               # four and two pairs per tile in the layer call, more in the separate ones
    (1300, 2),                          # several tiles per pair: staged a few rows at a time
])
def test_row_selection_over_gates_and_shared_tiles(kw, T, limit):
    # same tolerances as every parity test (bf16 products are exact, sums in fp32)
    _run(_wl(d=1024, **kw), T, layer=1, with_logit_bias=T in (17, 1300), want_logits=limit == 0, pair_limit=limit)


@pytest.mark.parametrize("kw", [
    # eight columns per lane in rows of at most 128 columns (groups of 20, 24, 36, 12, 40 over 4, 4, 8, 2, 8 lanes)
    dict(n_group=5, topk_group=3, k=7, E=100, R=5), dict(n_group=5, topk_group=2, k=8, E=120, R=5),
    dict(n_group=6, topk_group=3, k=6, E=120, R=8), dict(n_group=3, topk_group=1, k=8, E=108, R=6),
    dict(n_group=9, topk_group=4, k=8, E=108, R=9), dict(n_group=10, topk_group=2, k=3, E=120, R=8),
    dict(n_group=3, topk_group=2, k=5, E=120, R=8),
    # groups that are no whole vectors, word by word: 22 columns over 2 lanes, 19 over 4, 3 over 2, 5 over 2
    dict(n_group=9, topk_group=3, k=8, E=198, R=9), dict(n_group=6, topk_group=4, k=8, E=114, R=6),
    dict(n_group=16, topk_group=5, k=8, E=48, R=8), dict(n_group=16, topk_group=2, k=6, E=80, R=8),
])
@pytest.mark.parametrize("T,limit", [(129, 0), (700, 1)])        # tiles shared by eight pairs; three tile pairs on one pair
def test_row_selection_of_restricted_gates_at_every_lane_layout(kw, T, limit):
    _run(_wl(d=1024, gate=1, route_scale=2.5, **kw), T, layer=1, with_logit_bias=limit == 0, want_logits=limit == 0, pair_limit=limit)


@pytest.mark.parametrize("T", [100, 1300])
def test_row_selection_breaks_ties_and_survives_overfull_lists(T):
    # half of the rows have equal keys everywhere (more candidates than a row's list holds), in the others
    # experts 2 i and 2 i + 1 have equal weights: every choice is decided by the lower id
    for kw in (dict(E=100, k=5, R=4), dict(gate=1, n_group=10, topk_group=4, k=7, E=200, R=8), dict(E=12, k=5, R=3)):
        wl = _wl(d=512, **kw)
        li = I.make_layer(wl, 2, 0, T=T)
        li.W[1::2] = li.W[0::2]
        li.h_prev[::2] = 0
        li.H[::2] = 0
        if li.select_bias is not None:
            li.select_bias = torch.zeros(wl.E)
        ctx = P.make_context(wl, T)
        bkw = P.budget_kwargs(wl, T)
        gpu = P.run_gpu_layer(ctx, wl, li, bkw, want_logits=False)
        P.compare_layer(wl, li, bkw, gpu)
        assert (gpu["ids"][::2] == np.arange(wl.k)).all()
        even = gpu["ids"][1::2] % 2 == 0                     # an odd expert is chosen only right after its twin
        assert (even[:, 1:] | (gpu["ids"][1::2, 1:] == gpu["ids"][1::2, :-1] + 1)).all() and even[:, 0].all()
        ctx.close()


@pytest.mark.parametrize("kw", [dict(E=8, k=2, R=4), dict(E=64, k=6, R=8, gate=1), dict(E=64, k=8, R=8), dict(E=128, k=7, R=8),
                                dict(E=60, k=4, R=4, renorm=0)])
def test_few_keys_per_lane_break_ties_between_lanes(kw):
    # one, two and four columns per lane; experts e and e + E / 2 have equal weights and lie in different lanes, which the
    # branch-free rounds leave to the exact ones - in every third row only, the others have no ties
    T, wl = 190, _wl(d=256, **kw)
    li = I.make_layer(wl, 1, 0, T=T)
    half = wl.E // 2
    li.W[half:, :128] = li.W[:half, :128]
    li.h_prev[::3, 128:] = 0
    li.H[::3, 128:] = 0
    if li.select_bias is not None:
        li.select_bias = torch.zeros(wl.E)
    ctx = P.make_context(wl, T)
    bkw = P.budget_kwargs(wl, T)
    gpu = P.run_gpu_layer(ctx, wl, li, bkw, want_logits=False)
    P.compare_layer(wl, li, bkw, gpu)
    ids = gpu["ids"][::3]
    assert (ids[:, 0] < half).all()
    assert ((ids[:, 1:] < half) | (ids[:, 1:] == ids[:, :-1] + half)).all()
    ctx.close()


@pytest.mark.parametrize("E,kw", [
    (256, dict(gate=0, n_group=1, topk_group=1)), (200, dict(gate=0, n_group=1, topk_group=1)),      # eight columns per lane
    (256, dict(gate=1, n_group=8, topk_group=4)), (250, dict(gate=1, n_group=5, topk_group=2)),      # bound from the groups; sixteen
])
@pytest.mark.parametrize("distance", [1, 3, 9, 40])
def test_ties_at_the_last_rank_go_to_the_lowest_ids(E, kw, distance):
    # small integers: exact logits.  Experts come in runs of copies `distance` apart, so that for some k the k-th
    # and the (k + 1)-th key are equal, in the same lane, in neighbouring ones and far apart
    dev = torch.device("cuda")
    T, d = 300, 512                                              # two tile pairs shared by several SM pairs: a warp per row
    g = torch.Generator().manual_seed(E + distance)
    x, W = (torch.randint(-3, 4, s, generator=g).float() for s in ((T, d), (E, d)))
    e = torch.arange(E)
    for copies in (2, 3, 5):
        Wc = W[e - (e // distance) % copies * distance]
        z = (x.double() @ Wc.double().T).numpy()
        key = z if kw["gate"] == 0 else None
        router = B.make_router(Wc.to(torch.bfloat16).to(dev), None, None)
        for k in range(1, 9):
            ctx = B.Context(T, d, E, k, 2, kw["gate"], kw["n_group"], kw["topk_group"], 1, 1.0)
            counts, ids = torch.zeros(E, dtype=torch.int32, device=dev), torch.zeros(T * k, dtype=torch.int32, device=dev)
            ctx.fb_predict_load(router, x.to(torch.bfloat16).to(dev), T, counts, ids)
            assert ctx.fb_device_status() == 0
            got = ids.cpu().numpy().reshape(T, k)
            if key is not None:
                assert np.array_equal(got, np.argsort(-key, axis=1, kind="stable")[:, :k]), (copies, k)
            else:
                # an expert is chosen only if every copy of it with a lower id (in the same group) is
                gs = E // kw["n_group"]
                for t in range(T):
                    chosen = set(got[t].tolist())
                    assert len(chosen) == k
                    for c in chosen:
                        for lower in range(c - distance, c - distance * ((c // distance) % copies) - 1, -distance):
                            assert lower in chosen or lower // gs != c // gs, (copies, k, t)
            ctx.close()


@pytest.mark.parametrize("kw,d", [
    (dict(E=128, gate=0, n_group=1, topk_group=1, renorm=1), 256), (dict(E=256, gate=1, n_group=8, topk_group=4, renorm=1), 256),
    (dict(E=100, gate=0, n_group=1, topk_group=1, renorm=0), 256), (dict(E=200, gate=1, n_group=10, topk_group=3, renorm=1), 256),
])
@pytest.mark.parametrize("split,limit", [(1, 0), (0, 0), (0, 1)])    # shared tiles; one tile per pair; several per pair
def test_rows_without_numbers_stay_inside_and_leave_the_others_alone(kw, d, split, limit):
    # a NaN or an infinity in a token's hidden state: its experts are unspecified, but distinct and in range, the
    # index holds them, and every other token comes out as without it
    dev = torch.device("cuda")
    T, k, R, E = 700, 8, 4, kw["E"]
    g = torch.Generator().manual_seed(E)
    clean = torch.randn(T, d, generator=g).to(torch.bfloat16)
    W = torch.randn(E, d, generator=g).to(torch.bfloat16).to(dev)
    sb = (torch.rand(E, generator=g) - 0.5).to(dev) if kw["gate"] else None
    router = B.make_router(W, None, sb)
    odd_rows = torch.arange(3, T, 7)
    odd = clean.clone()
    odd[odd_rows, 5] = torch.tensor([float("nan"), float("inf"), float("-inf")]).repeat(len(odd_rows))[:len(odd_rows)].to(torch.bfloat16)
    odd[130:260] = float("nan")                                      # a whole tile and its neighbours' edges
    same = torch.ones(T, dtype=torch.bool)
    same[odd_rows] = False
    same[130:260] = False
    pi = torch.randperm(E, generator=g).to(torch.int32).to(dev)
    budget = B.make_budget(max_swaps=4, global_ns=O.U64_OFF, rank_ns=O.U64_OFF, link_ns=O.U64_OFF, tau_tokens=0, gamma_num=1,
                           gamma_den=64, alpha_ns=(1, 1), fs_per_byte=(1, 1), ranks_per_node=0, expert_bytes=16)
    ids, w = {}, {}
    for name, x in (("clean", clean), ("odd", odd)):
        ctx = B.Context(T, d, E, k, R, kw["gate"], kw["n_group"], kw["topk_group"], kw["renorm"], 1.0)
        ctx.fb_set_split(split)
        ctx.fb_set_pair_limit(limit)
        out = P.GuardedOutputs(dev)
        i32 = out.i32
        counts, early = i32(E), i32(T * k)
        ctx.fb_predict_load(router, x.to(dev), T, counts, early)
        l_counts, pi_out, swaps, n, lb, la = i32(E), i32(E), i32(16), i32(1), i32(R), i32(R)
        so, ro, rl, perm, inv, got, weights = i32(E + 1), i32(R + 1), i32(R), i32(T * k), i32(T * k), i32(T * k), out.f32(T * k)
        ctx.fb_layer_step(router, x.to(dev), x.to(dev).clone(), T, pi, budget, 0, l_counts, pi_out, swaps, n, lb, la, got, weights,
                          so, ro, perm, inv, rl)
        assert ctx.fb_device_status() == 0
        out.check()
        ids[name], w[name] = got.cpu().numpy().reshape(T, k), weights.cpu().view(T, k)
        assert ids[name].min() >= 0 and ids[name].max() < E
        assert (np.diff(np.sort(ids[name], axis=1), axis=1) > 0).all()
        assert counts.cpu().tolist() == O.expert_histogram(early.cpu().numpy().reshape(T, k), E).tolist()
        assert l_counts.cpu().tolist() == O.expert_histogram(ids[name], E).tolist()      # both passes saw the same rows
        want = O.dispatch_index(ids[name], pi_out.cpu().tolist(), R)
        for a, b in zip((so, ro, perm, inv, rl), want):
            assert a.cpu().tolist() == b.tolist()
        ctx.close()
    assert np.array_equal(ids["clean"][same], ids["odd"][same])
    assert torch.equal(w["clean"][same], w["odd"][same])


@pytest.mark.parametrize("E", [24, 100, 128, 256])
@pytest.mark.parametrize("split,limit", [(1, 0), (0, 0), (0, 1)])
def test_experts_masked_out_come_last_lowest_id_first(E, split, limit):
    # a logit bias of -inf leaves three experts: they come first, the masked ones follow in order of their ids
    dev = torch.device("cuda")
    T, k, d = 700, 6, 128
    g = torch.Generator().manual_seed(E)
    x, W = (torch.randint(-3, 4, s, generator=g).float() for s in ((T, d), (E, d)))
    bias = torch.full((E,), float("-inf"))
    bias[[1, E // 2, E - 1]] = 0.0
    z = (x.double() @ W.double().T + bias.double()).numpy()
    router = B.make_router(W.to(torch.bfloat16).to(dev), bias.to(dev), None)
    ctx = B.Context(T, d, E, k, 2)
    ctx.fb_set_split(split)
    ctx.fb_set_pair_limit(limit)
    counts, ids = torch.zeros(E, dtype=torch.int32, device=dev), torch.zeros(T * k, dtype=torch.int32, device=dev)
    ctx.fb_predict_load(router, x.to(torch.bfloat16).to(dev), T, counts, ids)
    assert ctx.fb_device_status() == 0
    got = ids.cpu().numpy().reshape(T, k)
    assert np.array_equal(got, np.argsort(-z, axis=1, kind="stable")[:, :k])
    assert counts.cpu().tolist() == O.expert_histogram(got, E).tolist()
    ctx.close()


@pytest.mark.parametrize("kw", [dict(E=128, gate=0, n_group=1, topk_group=1), dict(E=256, gate=1, n_group=8, topk_group=4)])
def test_logit_dumps_at_any_word(kw):
    # one tile per pair, a gate of the ranking kernel: it stores 16 bytes at a time, the dump need not start on 16
    dev = torch.device("cuda")
    T, d, k, R, E = 300, 512, 6, 4, kw["E"]
    g = torch.Generator().manual_seed(E)
    x, W = (torch.randn(*s, generator=g).to(torch.bfloat16).to(dev) for s in ((T, d), (E, d)))
    router = B.make_router(W, None, None)
    ctx = B.Context(T, d, E, k, R, kw["gate"], kw["n_group"], kw["topk_group"], 1, 1.0)
    ctx.fb_set_split(0)
    pi = torch.randperm(E, generator=g).to(torch.int32).to(dev)
    results = []
    for offset in (0, 1, 2, 3):
        i32 = lambda n: torch.full((n,), -7, dtype=torch.int32, device=dev)
        counts, early, ids, perm, inv, so, ro, rl = i32(E), i32(T * k), i32(T * k), i32(T * k), i32(T * k), i32(E + 1), i32(R + 1), i32(R)
        w, z, z_early = (torch.full((n + 8,), -7.0, device=dev) for n in (T * k, T * E, T * E))
        ctx.fb_predict_load(router, x, T, counts, early, z_early[offset:])
        ctx.fb_route_dispatch(router, x, T, pi, ids, w, so, ro, perm, inv, rl, z[offset:])
        assert ctx.fb_device_status() == 0
        for dump in (z, z_early):
            assert bool((dump[:offset] == -7).all()) and bool((dump[offset + T * E:] == -7).all())
        results.append((counts, early, ids, perm, inv, z[offset:offset + T * E], z_early[offset:offset + T * E]))
    for other in results[1:]:
        assert all(torch.equal(a, b) for a, b in zip(results[0], other))
    ctx.close()


@pytest.mark.parametrize("kw", [dict(E=128, gate=0, n_group=1, topk_group=1), dict(E=256, gate=1, n_group=8, topk_group=4)])
def test_pair_limit_holds_for_logit_dumps(kw):
    # a dump under a limit walks several tiles on the pairs it is given, as a call without one does; the results are those
    # of the unlimited call (small integers: exact sums), weights to a few ulp (their sum is formed in another order)
    dev = torch.device("cuda")
    T, d, k, R, E = 1300, 448, 6, 4, kw["E"]
    g = torch.Generator().manual_seed(E)
    x, W = (torch.randint(-2, 3, s, generator=g).to(torch.bfloat16).to(dev) for s in ((T, d), (E, d)))
    router = B.make_router(W, None, None)
    ctx = B.Context(T, d, E, k, R, kw["gate"], kw["n_group"], kw["topk_group"], 1, 1.0)
    pi = torch.randperm(E, generator=g).to(torch.int32).to(dev)
    budget = B.make_budget(max_swaps=4, gamma_num=1, gamma_den=64, alpha_ns=(1, 1), fs_per_byte=(1, 1), expert_bytes=16)
    results = []
    for limit in (0, 1, 2, 5):
        ctx.fb_set_pair_limit(limit)
        i32 = lambda n: torch.full((n,), -7, dtype=torch.int32, device=dev)
        counts, early, ids, perm, inv, so, ro, rl = i32(E), i32(T * k), i32(T * k), i32(T * k), i32(T * k), i32(E + 1), i32(R + 1), i32(R)
        l_counts, pi_out, swaps, n, lb, la = i32(E), i32(E), torch.zeros(16, dtype=torch.int32, device=dev), i32(1), i32(R), i32(R)
        w, z, z_early, zl, zl_early = (torch.full((m,), -7.0, device=dev) for m in (T * k, T * E, T * E, T * E, T * E))
        before = ctx.fb_persistent_launch_count()
        ctx.fb_predict_load(router, x, T, counts, early, z_early)
        ctx.fb_route_dispatch(router, x, T, pi, ids, w, so, ro, perm, inv, rl, z)
        first = (counts, early, ids.clone(), perm.clone(), inv.clone(), z, z_early)
        ctx.fb_layer_step_observed(router, x, x.flip(0).contiguous(), T, pi, budget, 0, l_counts, pi_out, swaps, n, lb, la, ids, w,
                                   so, ro, perm, inv, rl, early, zl_early, zl)
        assert ctx.fb_device_status() == 0
        assert ctx.fb_persistent_launch_count() - before == (3 if limit else 0)
        results.append((*first, l_counts, pi_out, swaps, n, lb, la, ids, so, ro, perm, inv, rl, early, zl_early, zl, w))
    for other in results[1:]:
        assert all(torch.equal(a, b) for a, b in zip(results[0][:-1], other[:-1]))
        assert torch.allclose(results[0][-1], other[-1], rtol=0, atol=1e-6)
    ctx.close()


@pytest.mark.parametrize("T,d,kw", [
    (1000, 2048, dict(E=128, gate=0, n_group=1, topk_group=1)),        # 4 pairs per tile in the layer call, 8 in the separate ones
    (1000, 2048, dict(E=256, gate=1, n_group=8, topk_group=4)), (4500, 1024, dict(E=60, gate=1, n_group=4, topk_group=2)),
])
def test_layer_call_and_separate_calls_on_ordinary_data(T, d, kw):
    # the split off: the same bits.  On: the order of the additions may differ, so logits agree to rounding and a token is
    # routed differently only where its k-th and (k+1)-th keys are closer than twice the difference seen (of the keys: a
    # sigmoid's slope is at most a quarter, its two approximations add 1e-6)
    dev = torch.device("cuda")
    E, k, R = kw["E"], 6, 4
    g = torch.Generator().manual_seed(T + E)
    x, H, W = (torch.randn(*s, generator=g).to(torch.bfloat16) for s in ((T, d), (T, d), (E, d)))
    W = (W.float() / d ** 0.5).to(torch.bfloat16)
    H[1::2] = H[0]                                                       # one token at every place of a tile
    xd, Hd, Wd = x.to(dev), H.to(dev), W.to(dev)
    router = B.make_router(Wd, None, None)
    budget = B.make_budget(max_swaps=4, gamma_num=1, gamma_den=64, alpha_ns=(1, 1), fs_per_byte=(1, 1), expert_bytes=16)
    pi = torch.randperm(E, generator=g).to(torch.int32).to(dev)
    exact = H.double() @ W.double().T
    ctx = B.Context(T, d, E, k, R, kw["gate"], kw["n_group"], kw["topk_group"], 1, 1.0)
    i32 = lambda n: torch.zeros(n, dtype=torch.int32, device=dev)
    for split in (0, 1):
        ctx.fb_set_split(split)
        a, b = ([i32(E), i32(E), i32(16), i32(1), i32(R), i32(R), i32(T * k), torch.zeros(T * k, device=dev), i32(E + 1), i32(R + 1),
                 i32(T * k), i32(T * k), i32(R)] for _ in range(2))
        z, zl = (torch.zeros(T * E, device=dev) for _ in range(2))
        ctx.fb_predict_and_plan(router, xd, T, pi, budget, 0, *a[:6])
        ctx.fb_route_dispatch(router, Hd, T, a[1], *a[6:])
        ctx.fb_layer_step(router, xd, Hd, T, pi, budget, 0, *b)
        ids, ids_l = a[6].cpu().numpy().reshape(T, k), b[6].cpu().numpy().reshape(T, k)
        c = [v.clone() for v in b]
        ctx.fb_route_dispatch(router, Hd, T, a[1], *c[6:], z)
        ctx.fb_layer_step_observed(router, xd, Hd, T, pi, budget, 0, *c, None, None, zl)
        assert ctx.fb_device_status() == 0
        z, zl = z.cpu().double().view(T, E), zl.cpu().double().view(T, E)
        # n additions of fp32 products that are exact: n 2^-23 of the sum of their sizes, whatever the order
        bound = d * 2.0 ** -23 * (H.double().abs() @ W.double().abs().T)
        assert bool(((z - exact).abs() <= bound).all()) and bool(((zl - exact).abs() <= bound).all())
        if split == 0:
            assert all(torch.equal(u, v) for u, v in zip(a, b))
            assert torch.equal(z, zl) and bool((z[1::2] == z[1]).all())
            continue
        diff = max(float((z - zl).abs().max()), float((z[1::2] - z[1]).abs().max()), float((zl[1::2] - z[1]).abs().max()))
        key_diff = diff if kw["gate"] == 0 else diff / 4 + 1e-6
        gate = O.Gate(E=E, k=k, gate=kw["gate"], n_group=kw["n_group"], topk_group=kw["topk_group"], renorm=1, route_scale=1.0)
        key_gap, group_gap = O.near_tie_margins(z.numpy(), gate, None)
        moved = (np.sort(ids, axis=1) != np.sort(ids_l, axis=1)).any(axis=1)
        assert not (moved & (key_gap > 2 * key_diff) & (group_gap > 4 * key_diff)).any()
    ctx.close()


@pytest.mark.parametrize("kw", [
    dict(E=96, k=5, R=6), dict(E=128, k=6, R=8, gate=1, n_group=4, topk_group=3),        # persistent kernel
    dict(E=60, k=4, R=5), dict(E=120, k=6, R=8, gate=1, n_group=6, topk_group=3),        # row-per-warp kernel
])
@pytest.mark.parametrize("d", [192, 448, 1088])          # 3, 7 and 17 k-blocks
def test_odd_numbers_of_k_blocks_with_several_tiles_per_pair(kw, d):
    # two MMA issuers, several tiles per pair: with an odd number of k-blocks their ring positions trade places from tile
    # to tile, whatever the number of stages; small integers, so every result is exact
    dev = torch.device("cuda")
    kw = dict(dict(gate=0, n_group=1, topk_group=1), **kw)
    T, E, k, R = 2700, kw["E"], kw["k"], kw["R"]
    g = torch.Generator().manual_seed(E + d)
    x, W = (torch.randint(-3, 4, s, generator=g).to(torch.bfloat16).to(dev) for s in ((T, d), (E, d)))
    router = B.make_router(W, None, None)
    ctx = B.Context(T, d, E, k, R, kw["gate"], kw["n_group"], kw["topk_group"], 1, 1.0)
    pi = torch.randperm(E, generator=g).to(torch.int32).to(dev)
    i32 = lambda n: torch.full((n,), -7, dtype=torch.int32, device=dev)
    results = []
    for limit, stages in ((0, 0), (1, 0), (3, 0), (1, 2), (2, 2), (1, 3), (2, 4)):
        ctx.fb_set_pair_limit(limit)
        ctx.fb_set_stage_limit(stages)
        for _ in range(3 if limit else 1):
            counts, early, ids, perm, inv, so, ro, rl = i32(E), i32(T * k), i32(T * k), i32(T * k), i32(T * k), i32(E + 1), i32(R + 1), i32(R)
            ctx.fb_predict_load(router, x, T, counts, early)
            ctx.fb_route_dispatch(router, x, T, pi, ids, torch.zeros(T * k, device=dev), so, ro, perm, inv, rl)
            assert ctx.fb_device_status() == 0, (limit, stages)
            results.append((counts, early, ids, perm, inv, so, ro, rl))
    for other in results[1:]:
        assert all(torch.equal(a, b) for a, b in zip(results[0], other))
    ctx.close()


@pytest.mark.parametrize("pieces", [2, 3, 4, 5, 6, 7, 8])
def test_any_number_of_pairs_per_tile_gives_the_unshared_results(pieces):
    # small integers: every order of the sums is exact.  Token counts around the edges of row slices and tiles
    dev = torch.device("cuda")
    for kw in (dict(E=100, k=5, R=4, gate=0, n_group=1, topk_group=1), dict(E=256, k=8, R=8, gate=1, n_group=8, topk_group=4)):
        E, k, R, d = kw["E"], kw["k"], kw["R"], 7168
        for T in (1, 43, 45, 128, 151, 256, 300, 900):
            g = torch.Generator().manual_seed(T + pieces)
            x, W = (torch.randint(-2, 3, s, generator=g).to(torch.bfloat16).to(dev) for s in ((T, d), (E, d)))
            sb = (torch.randint(0, 4, (E,), generator=g) / 8.0).to(dev) if kw["gate"] else None
            router = B.make_router(W, None, sb)
            ctx = B.Context(T, d, E, k, R, kw["gate"], kw["n_group"], kw["topk_group"], 1, 1.0)
            pi = torch.randperm(E, generator=g).to(torch.int32).to(dev)
            tile_pairs = (T + 255) // 256
            results = []
            for split in (1, 0):
                ctx.fb_set_split(split)
                ctx.fb_set_pair_limit(tile_pairs * pieces)
                i32 = lambda n: torch.full((n,), -7, dtype=torch.int32, device=dev)
                counts, early, ids, perm, inv = i32(E), i32(T * k), i32(T * k), i32(T * k), i32(T * k)
                so, ro, rl, w = i32(E + 1), i32(R + 1), i32(R), torch.full((T * k,), -7.0, device=dev)
                z = torch.full((T * E,), -7.0, device=dev)
                ctx.fb_predict_load(router, x, T, counts, early, z)
                ctx.fb_route_dispatch(router, x, T, pi, ids, w, so, ro, perm, inv, rl)
                assert ctx.fb_device_status() == 0
                results.append((counts, early, ids, perm, inv, so, ro, rl, z, w))
            for a, b in zip(results[0][:-1], results[1][:-1]):
                assert torch.equal(a, b), (kw, T)
            assert torch.allclose(results[0][-1], results[1][-1], rtol=0, atol=1e-6)    # weights <= 1: a few ulp
            ctx.close()


def test_contexts_of_different_shapes_alive_together():
    # Kernel attributes (the dynamic shared-memory ceiling) belong to the kernel, not to a context:
    # a large-shape context must keep working after a small-shape one was created, and the
    # other way round, with calls through both interleaved.
    names = ["dsv3", "tiny", "qwen3"]
    T = 700
    wls = [I.WORKLOADS[n] for n in names]
    ctxs = [P.make_context(wl, T) for wl in wls]              # created largest first ...
    lis = [I.make_layer(wl, 0, 0, T=T) for wl in wls]
    bkws = [P.budget_kwargs(wl, T) for wl in wls]
    for rep in range(2):
        for ctx, wl, li, bkw in zip(ctxs, wls, lis, bkws):    # ... and used alternately
            gpu = P.run_gpu_layer(ctx, wl, li, bkw, want_logits=False, pair_limit=rep)   # rep 1: persistent kernel
            P.compare_layer(wl, li, bkw, gpu)
    late = P.make_context(I.WORKLOADS["mixtral"], T)           # a fourth shape created afterwards
    for ctx, wl, li, bkw in list(zip(ctxs, wls, lis, bkws))[::-1]:
        gpu = P.run_gpu_layer(ctx, wl, li, bkw, want_logits=False)
        P.compare_layer(wl, li, bkw, gpu)
    for c in ctxs + [late]:
        c.close()
