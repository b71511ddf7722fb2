"""GPU parity of the multi-step serving loop and the quality metrics against the oracle."""
import numpy as np
import pytest
import torch

from oracle import freebalance_oracle as O
from paper_2608_14205_b200 import binding as B
from paper_2608_14205_b200 import inputs as I
from paper_2608_14205_b200 import serving as S
from tests.test_oracle_serving import _budget, _gate, bits

pytestmark = pytest.mark.gpu


def _oracle_trace(layers_cpu):
    for (s, l), li in layers_cpu.items():
        sb = li.select_bias.numpy().astype(np.float64) if li.select_bias is not None else None
        yield s, l, bits(li.h_prev), bits(li.H), bits(li.W), sb, None


@pytest.mark.parametrize("name,T,steps,layers,sys_drift,quality", [
    ("tiny", 300, 3, 2, 0.0, True), ("tiny", 300, 3, 2, 0.0, False),
    ("qwen3", 700, 3, 2, 0.25, True),
    ("dsv3", 640, 3, 2, 0.25, True), ("dsv3", 640, 3, 2, 0.5, False),
])
def test_serving_loop_matches_the_oracle(name, T, steps, layers, sys_drift, quality):
    wl = I.WORKLOADS[name]
    cpu = {(s, l): I.make_step_layer(wl, l, s, 0, T=T, sys_drift=sys_drift)
           for s in range(steps) for l in range(layers)}
    records, summary, placements = O.serving_loop(_oracle_trace(cpu), _gate(wl), wl.R, _budget(wl, T))
    loop = S.ServingLoop(wl, T)
    budget = S.make_budget_for(wl, T)
    dev = loop.dev
    for rec, ((s, l), li) in zip(records, cpu.items()):
        sb = li.select_bias.to(dev) if li.select_bias is not None else None
        router = B.make_router(li.W.to(dev), None, sb)
        r = loop.layer_step(l, router, li.h_prev.to(dev), li.H.to(dev), budget, quality=quality)
        torch.cuda.synchronize(dev)
        o = r["out"]
        assert loop.ctx.fb_device_status() == 0
        assert r["pi_old"].cpu().tolist() == rec["pi_old"], "placement carried over from the previous step"
        n = int(o["n_swaps"].item())
        swaps = [tuple(x) for x in o["swaps"].cpu().numpy().reshape(-1, 4)[:n].tolist()]
        assert o["counts"].cpu().tolist() == rec["counts"].tolist()
        assert swaps == rec["swaps"] and r["pi_new"].cpu().tolist() == rec["pi_new"]
        realized, before, after, vanilla = loop.realised_loads(r, budget)
        assert realized == rec["realized"].tolist()
        assert O.max_over_mean(before) == rec["real_before"] and O.max_over_mean(after) == rec["real_after"]
        assert O.max_over_mean(vanilla) == rec["real_vanilla"]
        if quality:
            assert r["hit_rate"] == rec["hit_rate"]
            assert r["cos_hidden"] == pytest.approx(rec["cos_hidden"], abs=1e-12)     # same bf16 inputs, fp64 sums
            assert r["cos_logits"] == pytest.approx(rec["cos_logits"], abs=1e-5)      # fp32 vs fp64 logits
    for l in range(layers):
        assert loop.placement_of(l).cpu().tolist() == placements[l]
    loop.close()


def test_metric_kernels_on_constructed_inputs():
    dev = torch.device("cuda")
    a = torch.tensor([[1.0, 0.0, 0.0], [0.0, 0.0, 0.0], [1.0, 1.0, 0.0], [2.0, 0.0, 0.0]], device=dev)
    b = torch.tensor([[0.0, 3.0, 0.0], [1.0, 2.0, 3.0], [1.0, 0.0, 0.0], [-5.0, 0.0, 0.0]], device=dev)
    rows = torch.zeros(4, dtype=torch.float64, device=dev)
    mean = torch.zeros(1, dtype=torch.float64, device=dev)
    B.fb_row_cosine_mean(a, b, rows, mean)
    assert rows.cpu().tolist() == pytest.approx([0.0, 0.0, 2 ** -0.5, -1.0], abs=1e-15)
    assert mean.item() == pytest.approx((2 ** -0.5 - 1.0) / 4, abs=1e-15)
    ab, bb = a.to(torch.bfloat16), b.to(torch.bfloat16)
    B.fb_row_cosine_mean(ab, bb, rows, mean)
    assert mean.item() == pytest.approx((2 ** -0.5 - 1.0) / 4, abs=1e-15)
    B.fb_row_cosine_mean(a[:0], b[:0], rows, mean)
    assert mean.item() == 0.0
    # ragged width, many rows: against the oracle's definition
    g = torch.Generator().manual_seed(5)
    x, y = torch.randn(1000, 77, generator=g), torch.randn(1000, 77, generator=g)
    rows = torch.zeros(1000, dtype=torch.float64, device=dev)
    B.fb_row_cosine_mean(x.to(dev), y.to(dev), rows, mean)
    assert mean.item() == pytest.approx(O.row_cosine_mean(x.numpy(), y.numpy()), abs=1e-13)

    ids_a = torch.tensor([[0, 1, 2], [3, 4, 5], [6, 7, 8]], dtype=torch.int32, device=dev)
    ids_b = torch.tensor([[2, 1, 0], [5, 9, 10], [11, 12, 13]], dtype=torch.int32, device=dev)
    hits = torch.zeros(1, dtype=torch.int32, device=dev)
    B.fb_topk_hits(ids_a, ids_b, 3, 3, hits)
    assert hits.item() == 4
    assert O.topk_hit_rate(ids_a.cpu().numpy(), ids_b.cpu().numpy()) == pytest.approx(4 / 9)
    B.fb_topk_hits(ids_a, ids_b, 0, 3, hits)
    assert hits.item() == 0
    with pytest.raises(B.FbError):
        B.fb_topk_hits(ids_a, ids_b, 3, 9, hits)


@pytest.mark.parametrize("n", [8, 248, 256, 1016, 1024, 1032, 2056, 77])
def test_bf16_row_cosines_at_the_edges_of_steps_and_of_the_value_range(n):
    # products are exact in double and n of them are added: n 2^-53 of |x| |y|, and twice that for the norms
    g = torch.Generator().manual_seed(n)
    dev = torch.device("cuda")
    x, y = (torch.randn(64, n, generator=g).to(torch.bfloat16) for _ in range(2))
    for r, scale in enumerate([2.0 ** -130, 2.0 ** -126, 2.0 ** 120, 0.0]):      # subnormals, large values, zeros
        x[r] = (x[r].float() * scale).to(torch.bfloat16)
        y[r + 2] = (y[r + 2].float() * scale).to(torch.bfloat16)
    x[8, n // 2], y[9, n - 1], x[10, 0], y[11, n // 3] = float("inf"), float("-inf"), float("nan"), float("nan")
    rows, mean = torch.zeros(64, dtype=torch.float64, device=dev), torch.zeros(1, dtype=torch.float64, device=dev)
    B.fb_row_cosine_mean(x.to(dev), y.to(dev), rows, mean)
    a, b = x.double(), y.double()
    dot, na, nb = (a * b).sum(1), (a * a).sum(1), (b * b).sum(1)
    want = torch.where((na > 0) & (nb > 0), dot / (na.sqrt() * nb.sqrt()), torch.zeros(()).double())
    assert torch.allclose(rows.cpu(), want, rtol=0.0, atol=4 * n * 2.0 ** -53, equal_nan=True)


def test_row_cosines_of_more_rows_than_one_grid_holds():
    # 2^32 + 6 rows of one element: 8.6 GB of them and 34 GB of row results
    rows_n = 2 ** 32 + 6
    if torch.cuda.mem_get_info()[0] < 60 * 2 ** 30:
        pytest.skip("needs 60 GB of device memory")
    dev = torch.device("cuda")
    a = torch.ones(rows_n, 1, dtype=torch.bfloat16, device=dev)
    b = torch.ones(rows_n, 1, dtype=torch.bfloat16, device=dev)
    edges = [0, 2 ** 31 - 1, 2 ** 31, 2 ** 32 - 1, 2 ** 32, 2 ** 32 + 5]
    for i in edges:
        b[i] = -2.0
    rows, mean = torch.zeros(rows_n, dtype=torch.float64, device=dev), torch.zeros(1, dtype=torch.float64, device=dev)
    B.fb_row_cosine_mean(a, b, rows, mean)
    assert [rows[i].item() for i in edges] == [-1.0] * len(edges)
    assert [rows[i + 1].item() for i in edges[1:-2]] == [-1.0 if i + 1 in edges else 1.0 for i in edges[1:-2]]
    assert mean.item() == (rows_n - 2 * len(edges)) / rows_n      # whole numbers below 2^53: exact sums


@pytest.mark.parametrize("T,d,E,k", [(1, 8, 5, 1), (37, 72, 100, 8), (1000, 20, 33, 3), (8200, 64, 8, 2)])
def test_combined_metrics_match_the_separate_calls(T, d, E, k):
    # row sums are formed alike; the means add them in another order: 1e-12 is far above 2^-53 sqrt(T)
    g = torch.Generator().manual_seed(T)
    dev = torch.device("cuda")
    h = torch.randn(T, d, generator=g).to(torch.bfloat16).to(dev)
    H = (h.float().cpu() + 0.3 * torch.randn(T, d, generator=g)).to(torch.bfloat16).to(dev)
    H[T // 2] = 0                                                # a row that is zero on one side contributes 0
    za, zb = (torch.randn(T, E, generator=g).to(dev) for _ in range(2))
    ia, ib = (torch.rand(T, E, generator=g).topk(k, dim=1).indices.to(torch.int32).to(dev).contiguous() for _ in range(2))
    rows, mean = torch.zeros(3 * T, dtype=torch.float64, device=dev), torch.zeros(1, dtype=torch.float64, device=dev)
    hits, out = torch.zeros(1, dtype=torch.int32, device=dev), torch.zeros(3, dtype=torch.float64, device=dev)
    B.fb_prediction_quality(h, H, za, zb, ia, ib, T, d, E, k, rows, out)
    got = out.tolist()
    B.fb_row_cosine_mean(h, H, rows, mean)
    assert abs(got[0] - mean.item()) < 1e-12
    B.fb_row_cosine_mean(za, zb, rows, mean)
    assert abs(got[1] - mean.item()) < 1e-12
    B.fb_topk_hits(ia, ib, T, k, hits)
    assert got[2] == hits.item()


@pytest.mark.parametrize("T,d,E,k,R,gate,n_group,topk_group,renorm", [
    (1, 64, 8, 2, 4, "softmax", 1, 1, 1), (300, 128, 128, 8, 8, "softmax", 1, 1, 1), (9217, 128, 128, 8, 8, "softmax", 1, 1, 1),
    (19001, 64, 128, 8, 8, "softmax", 1, 1, 1), (9300, 128, 256, 8, 64, "sigmoid", 8, 4, 1), (19001, 64, 100, 3, 10, "softmax", 1, 1, 0),
])
def test_observed_layer_step_matches_the_separate_calls(T, d, E, k, R, gate, n_group, topk_group, renorm):
    # small integers: every summation order of the router GEMM is exact, so all results agree bit for bit
    # (tiles shared by several pairs, one per pair, more than the GPU has pairs; planner in either kernel)
    g = torch.Generator().manual_seed(T)
    dev = torch.device("cuda")
    ints = lambda *s: torch.randint(-3, 4, s, generator=g).to(torch.bfloat16).to(dev)
    h, H, W = ints(T, d), ints(T, d), ints(E, d)
    code = I.GATE_SOFTMAX_TOPK if gate == "softmax" else I.GATE_SIGMOID_GROUP_TOPK
    sb = (0.125 * torch.randint(0, 3, (E,), generator=g)).float().to(dev) if gate == "sigmoid" else None
    router, ctx = B.make_router(W, None, sb), B.Context(T, d, E, k, R, code, n_group, topk_group, renorm, 1.0)
    budget = B.make_budget(max_swaps=min(16, E // 2))
    pi = torch.randperm(E, generator=g).to(torch.int32).to(dev)
    i32 = lambda n: torch.full((n,), -7, dtype=torch.int32, device=dev)
    f32 = lambda n: torch.full((n,), float("nan"), device=dev)
    bufs = lambda: [i32(E), i32(E), i32(4 * (E // 2)), i32(1), i32(R), i32(R), i32(T * k), f32(T * k), i32(E + 1), i32(R + 1),
                    i32(T * k), i32(T * k), i32(R)]
    want, got = bufs(), bufs()
    ids, ids_early, z, z_early, zs = i32(T * k), i32(T * k), f32(T * E), f32(T * E), f32(2 * T * E)
    ctx.fb_predict_load(router, h, T, i32(E), ids, zs[:T * E])
    ctx.fb_layer_step(router, h, H, T, pi, budget, 0, *want)
    other = bufs()
    ctx.fb_route_dispatch(router, H, T, want[1], *other[6:], zs[T * E:])
    ctx.fb_layer_step_observed(router, h, H, T, pi, budget, 0, *got, ids_early, z_early, z)
    assert ctx.fb_device_status() == 0
    assert torch.equal(ids_early, ids) and torch.equal(torch.cat([z_early, z]), zs)
    for a, b in zip(got, want):
        assert torch.equal(a.nan_to_num(), b.nan_to_num())
    ctx.close()
