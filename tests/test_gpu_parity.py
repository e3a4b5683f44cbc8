"""GPU parity: every stage of the CUDA path, called through the C ABI, against the CPU oracle on
the same seeded inputs.  Routing indices and dispatch contents bit-exact (rows inside an expert
compared after sorting by source id: arrival order is free, Section IV-B of the paper), routing
weights within 1e-5 relative, combined output within 1e-4 (fp32, element-wise with an rms floor) /
2e-2 (bf16, per-token normwise) of the oracle: see parity_helpers.assert_output_close."""
import ctypes
import itertools

import numpy as np
import pytest
import torch

import oracle
from paper_2605_05888_b200 import binding as B
from paper_2605_05888_b200 import inputs
import parity_helpers as Hh

pytestmark = pytest.mark.gpu
FP32, BF16 = inputs.FP32, inputs.BF16
MODES = [B.DISPATCH_SCAN, B.DISPATCH_ATOMIC_STATIC, B.DISPATCH_ATOMIC_PAGED, B.DISPATCH_ATOMIC_ORDERED]

SMALL = [
    inputs.C1,
    inputs.C1.with_(seed=1), inputs.C1.with_(seed=2),
    inputs.Workload("ragged_bf16", T=333, H=264, E=12, R=3, K=3, F=200, dtype=BF16),
    inputs.Workload("qwen_small", T=97, H=512, E=60, R=4, K=4, F=352, dtype=BF16),
    inputs.Workload("many_experts", T=300, H=256, E=256, R=32, K=8, F=128, dtype=BF16, zipf_s=1.0),
    inputs.Workload("k_equals_e", T=50, H=64, E=4, R=2, K=4, F=64, dtype=FP32),
    inputs.Workload("one_token", T=1, H=128, E=8, R=1, K=2, F=128, dtype=BF16),
    inputs.Workload("top1", T=130, H=128, E=16, R=4, K=1, F=136, dtype=BF16, zipf_s=1.2),
    # the limits of the entry points: K = 32 picks per token, with 64 and with 256 experts
    inputs.Workload("max_k", T=70, H=128, E=64, R=4, K=32, F=64, dtype=BF16),
    inputs.Workload("max_e_max_k", T=45, H=64, E=256, R=8, K=32, F=64, dtype=BF16, zipf_s=1.0),
]


def run_stages(w, mode, x, wr, bias, wg, wu, wd, ffn_kernel=0):
    plan = Hh.make_plan(w, mode, ffn_kernel=ffn_kernel)
    el = Hh.el_dtype(w)
    dx, dwr, dbias = Hh.to_dev(x), Hh.to_dev(wr), Hh.to_dev(bias)
    idx = torch.empty((w.T, w.K), dtype=torch.int32, device="cuda")
    tw = torch.empty((w.T, w.K), dtype=torch.float32, device="cuda")
    plan.moe_route(dx, dwr, dbias, idx, tw)
    rows = plan.P * 128
    recv = torch.zeros((rows, w.H), dtype=el, device="cuda")
    cnt = torch.empty(w.E, dtype=torch.int32, device="cuda")
    te = torch.empty(plan.P, dtype=torch.int32, device="cuda")
    src = torch.empty(rows, dtype=torch.int32, device="cuda")
    slot = torch.empty((w.T, w.K), dtype=torch.int32, device="cuda")
    plan.moe_dispatch(dx, idx, recv, cnt, te, src, slot)
    if w.identity_experts:
        out_rows = recv
    else:
        out_rows = torch.zeros((rows, w.H), dtype=el, device="cuda")
        plan.moe_expert_ffn(recv, te, Hh.to_dev(wg), Hh.to_dev(wu), Hh.to_dev(wd), out_rows)
    y = torch.empty((w.T, w.H), dtype=el, device="cuda")
    plan.moe_combine(out_rows, slot, tw, y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    return dict(plan=plan, idx=idx, tw=tw, recv=recv, cnt=cnt, te=te, src=src, slot=slot, out_rows=out_rows, y=y)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("w", SMALL, ids=lambda w: w.name + f"_s{w.seed}")
def test_stages_match_oracle(w, mode):
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    g = run_stages(w, mode, x, wr, bias, wg, wu, wd)
    Hh.check_route(g["idx"], g["tw"], ref["topk_idx"], ref["topk_w"])
    Hh.check_dispatch(w, g["plan"].P, x, ref["topk_idx"], ref, g["recv"], g["cnt"], g["te"], g["src"], g["slot"])
    # expert outputs row by row (canonical order) and the combined result
    slot = g["slot"].cpu().numpy()
    got_rows = Hh.to_host_f64(g["out_rows"])[slot.ravel()]
    ref_rows = ref["out_rows"][ref["slot_of"].ravel()]
    Hh.assert_output_close(got_rows, ref_rows, w.dtype, "expert outputs")
    Hh.assert_output_close(Hh.to_host_f64(g["y"]), ref["y"], w.dtype, "combined output")
    if w.dtype == BF16:   # and within a bf16 step of the restatement that rounds where the kernels store bf16
        stored = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd, bf16_storage=True)
        Hh.assert_close_to_bf16_storage(Hh.to_host_f64(g["y"]), stored, "combined output")


@pytest.mark.parametrize("w", [SMALL[3], SMALL[4], SMALL[5]], ids=lambda w: w.name)
def test_simt_ffn_matches_oracle_bf16(w):
    """The fp32-FMA expert kernel on bf16 data: the second device implementation of step 3."""
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    g = run_stages(w, B.DISPATCH_SCAN, x, wr, bias, wg, wu, wd, ffn_kernel=1)
    Hh.assert_output_close(Hh.to_host_f64(g["y"]), ref["y"], w.dtype)


@pytest.mark.parametrize("split", [1, 2])
@pytest.mark.parametrize("w", [SMALL[3], SMALL[4], SMALL[5], SMALL[7],
                               inputs.Workload("three_tiles", T=700, H=320, E=4, R=2, K=2, F=392, dtype=BF16)],
                         ids=lambda w: w.name)
@pytest.mark.parametrize("kernel", [0, 2])
def test_tensor_core_ffn_forms_match_oracle(w, split, kernel):
    """Both forms of the tensor-core expert kernel - one CTA per tile (0) and the cta_group::2 form (2: two
    tiles of an expert per MMA; experts with an odd number of tiles leave one CTA of the last pair without
    work) - each as one launch for both GEMMs (per-tile counters gate GEMM2) and as two launches."""
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED, ffn_kernel=kernel, ffn_split=split)
    y = torch.empty((w.T, w.H), dtype=Hh.el_dtype(w), device="cuda")
    plan.moe_layer(Hh.to_dev(x), Hh.to_dev(wr), Hh.to_dev(bias), Hh.to_dev(wg), Hh.to_dev(wu), Hh.to_dev(wd), y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    Hh.assert_output_close(Hh.to_host_f64(y), ref["y"], w.dtype)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("w", [inputs.C1, SMALL[3], SMALL[5], SMALL[9], SMALL[10], inputs.C5(512), inputs.C5(256, 1.2)],
                         ids=lambda w: w.name)
def test_fused_layer_matches_oracle(w, mode):
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    plan = Hh.make_plan(w, mode)
    y = torch.empty((w.T, w.H), dtype=Hh.el_dtype(w), device="cuda")
    plan.moe_layer(Hh.to_dev(x), Hh.to_dev(wr), Hh.to_dev(bias), Hh.to_dev(wg), Hh.to_dev(wu), Hh.to_dev(wd), y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    assert plan.moe_last_launch_count() >= 3
    Hh.check_route(plan.layer_tensor(0), plan.layer_tensor(1), ref["topk_idx"], ref["topk_w"])
    Hh.check_dispatch(w, plan.P, x, ref["topk_idx"], ref, plan.layer_tensor(2), plan.layer_tensor(3),
                      plan.layer_tensor(4), plan.layer_tensor(5), plan.layer_tensor(6))
    Hh.assert_output_close(Hh.to_host_f64(y), ref["y"], w.dtype)
    # host-buffer entry point gives the same bytes
    hx = torch.from_numpy(x.view(np.int16) if x.dtype == np.uint16 else x).pin_memory()
    hy = torch.empty_like(hx).pin_memory()
    plan.moe_layer_host(hx, Hh.to_dev(wr), Hh.to_dev(bias), Hh.to_dev(wg), Hh.to_dev(wu), Hh.to_dev(wd), hy)
    y_bits = Hh.to_host_bits(y)
    assert np.array_equal(hy.numpy().view(y_bits.dtype), y_bits)


def test_identity_experts_closed_form():
    """Identity experts make the layer return x * sum_k w (a property that holds at any size)."""
    w = inputs.C5(2048, 1.2)
    x, wr, bias, *_ = Hh.oracle_inputs(w, with_experts=False)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED)
    y = torch.empty((w.T, w.H), dtype=torch.bfloat16, device="cuda")
    dx = Hh.to_dev(x)
    plan.moe_layer(dx, Hh.to_dev(wr), Hh.to_dev(bias), None, None, None, y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    ws = plan.layer_tensor(1).double().sum(1, keepdim=True)
    ref = (dx.double() * ws).cpu().numpy()
    Hh.assert_output_close(Hh.to_host_f64(y), ref, w.dtype)


# ------------------------------------------------------------------ router edge cases
def test_router_tie_patterns_exhaustive():
    """H = 8 >= E and Wr = [I | 0] make the logits equal x[:, :E]; x runs over {-1,0,1}^E, every tie
    pattern of the top-K selection, K = 1..E."""
    for E in (2, 3, 5):
        grid = np.array(list(itertools.product([-1.0, 0.0, 1.0], repeat=E)), np.float32)
        T = grid.shape[0]
        x = np.zeros((T, 8), np.float32)
        x[:, :E] = grid
        wr = np.zeros((E, 8), np.float32)
        wr[np.arange(E), np.arange(E)] = 1.0
        for K in range(1, E + 1):
            w = inputs.Workload("ties", T=T, H=8, E=E, R=1, K=K, F=8, dtype=FP32)
            plan = Hh.make_plan(w, B.DISPATCH_SCAN)
            idx = torch.empty((T, K), dtype=torch.int32, device="cuda")
            tw = torch.empty((T, K), dtype=torch.float32, device="cuda")
            plan.moe_route(Hh.to_dev(x), Hh.to_dev(wr), None, idx, tw)
            ridx, rw, _ = oracle.route(x, wr, None, K, FP32)
            Hh.check_route(idx, tw, ridx, rw)


# every chain: up to 64 experts, and more of them with few tokens; the tensor-core filter, from one k-block per accumulator on
@pytest.mark.parametrize("E,T,H", [(60, 200, 512), (160, 200, 512), (160, 1100, 512), (256, 1030, 1032)])
@pytest.mark.parametrize("renorm", [0, 1])
def test_router_renormalize_and_bias(renorm, E, T, H):
    w = inputs.Workload("renorm", T=T, H=H, E=E, R=4, K=4, F=8, dtype=BF16, zipf_s=1.0, seed=3)
    x, wr, bias, *_ = Hh.oracle_inputs(w, with_experts=False)
    cfg = B.make_config(w.T, w.H, w.E, w.R, w.K, w.F, w.dtype, renormalize=renorm)
    plan = B.Plan(cfg)
    idx = torch.empty((w.T, w.K), dtype=torch.int32, device="cuda")
    tw = torch.empty((w.T, w.K), dtype=torch.float32, device="cuda")
    plan.moe_route(Hh.to_dev(x), Hh.to_dev(wr), Hh.to_dev(bias), idx, tw)
    ridx, rw, _ = oracle.route(x, wr, bias, w.K, w.dtype, renormalize=renorm)
    Hh.check_route(idx, tw, ridx, rw)


# Every router kernel: the chain kernel's lane layouts (E <= 8, 16, 32, 64 and several CTAs per block of tokens), each
# with a block boundary inside T and an h range that ends inside a chunk, in both dtypes; above 1024 tokens and 64 experts
# the filter and the register-tiled kernel, with every tile height it picks (4 to 8 tokens per thread follows from T on a
# 148-SM part: T <= 4736 -> 4, <= 5920 -> 5, <= 7104 -> 6, <= 8288 -> 7, <= 9472 -> 8) and E below and at 256; the filter
# with h ranges that use its four accumulators unevenly.
ROUTER_SHAPES = [
    # (T, H, E, K, dtype, zipf_s)
    (77, 264, 7, 2, BF16, 0.0), (1100, 520, 8, 3, BF16, 1.0), (45, 132, 5, 5, FP32, 0.0),
    (333, 1032, 16, 2, BF16, 0.0), (90, 260, 13, 4, FP32, 1.0),
    (70, 520, 32, 6, BF16, 0.0), (1500, 264, 24, 2, BF16, 1.0), (33, 68, 17, 3, FP32, 0.0),
    (130, 776, 60, 4, BF16, 0.0), (1030, 136, 64, 8, BF16, 1.0), (21, 132, 33, 2, FP32, 0.0),
    (200, 72, 65, 8, BF16, 0.0), (4000, 40, 256, 8, BF16, 1.0), (5000, 40, 200, 4, BF16, 0.0),
    (6500, 40, 256, 8, BF16, 1.0), (8000, 40, 129, 2, BF16, 0.0), (9000, 40, 256, 8, BF16, 1.0),
    (300, 36, 100, 5, FP32, 1.0), (5100, 20, 256, 3, FP32, 0.0),
    (1100, 1032, 200, 8, BF16, 1.0), (1300, 2120, 129, 4, BF16, 0.0), (1025, 264, 65, 6, BF16, 1.0),
]


@pytest.mark.parametrize("shape", ROUTER_SHAPES, ids=lambda s: f"T{s[0]}_H{s[1]}_E{s[2]}_K{s[3]}_d{s[4]}_z{s[5]}")
def test_router_every_kernel_shape(shape):
    T, H, E, K, dtype, zipf = shape
    w = inputs.Workload("router_shape", T=T, H=H, E=E, R=1, K=K, F=8, dtype=dtype, zipf_s=zipf, seed=11,
                        identity_experts=True)
    x, wr, bias, *_ = Hh.oracle_inputs(w, with_experts=False)
    ridx, rw, _ = oracle.route(x, wr, bias, K, dtype)
    for route_filter in ((0, -1) if (dtype == BF16 and E > 64) else (0,)):   # -1: every chain, also above 1024 tokens
        plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED, route_filter=route_filter)
        idx = torch.empty((T, K), dtype=torch.int32, device="cuda")
        tw = torch.empty((T, K), dtype=torch.float32, device="cuda")
        plan.moe_route(Hh.to_dev(x), Hh.to_dev(wr), Hh.to_dev(bias), idx, tw)
        torch.cuda.synchronize()
        Hh.check_route(idx, tw, ridx, rw)


# The chain kernel where its shapes end: expert counts at the edges of its lane grids and clusters (8 / 16 / 32 / 64 /
# 128 / 192 / 256), one token, token counts around its blocks, one, two and eight chains per thread, an h range shorter
# than a box and one that ends inside a box and inside a stage; and both sides of the switches to the filter (bf16) and to
# the register-tiled kernel (fp32).
CHAIN_SHAPES = [
    # (T, H, E, K, dtype)
    (1, 8, 8, 8, BF16), (1, 4, 1, 1, FP32), (17, 72, 9, 2, BF16), (5000, 72, 8, 2, BF16), (5000, 36, 16, 3, FP32),
    (3, 584, 33, 4, BF16), (1, 2056, 64, 8, BF16), (601, 584, 31, 5, BF16), (4700, 72, 61, 4, BF16), (4700, 36, 64, 4, FP32),
    (1, 584, 256, 8, BF16), (9, 292, 193, 32, FP32), (129, 136, 128, 6, BF16), (768, 136, 192, 8, BF16),
    (769, 136, 192, 8, BF16), (768, 68, 256, 8, FP32), (769, 68, 256, 8, FP32),
    (1024, 136, 256, 8, BF16), (1025, 136, 256, 8, BF16), (864, 4104, 193, 8, BF16), (865, 4104, 193, 8, BF16),
    (1024, 68, 65, 8, FP32), (1025, 68, 65, 8, FP32), (1024, 136, 65, 8, BF16), (1025, 136, 65, 8, BF16),
    # just past what one wave of CTAs holds (two waves of fewer tokens each)
    (985, 72, 160, 4, BF16), (890, 72, 224, 8, BF16), (7200, 40, 32, 2, BF16), (14300, 36, 12, 2, FP32),
]


@pytest.mark.parametrize("shape", CHAIN_SHAPES, ids=lambda s: f"T{s[0]}_H{s[1]}_E{s[2]}_K{s[3]}_d{s[4]}")
def test_router_chain_kernel_edges(shape):
    T, H, E, K, dtype = shape
    w = inputs.Workload("router_edges", T=T, H=H, E=E, R=1, K=K, F=8, dtype=dtype, zipf_s=1.0, seed=13, identity_experts=True)
    x, wr, bias, *_ = Hh.oracle_inputs(w, with_experts=False)
    ridx, rw, _ = oracle.route(x, wr, bias, K, dtype)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED)
    idx = torch.empty((T, K), dtype=torch.int32, device="cuda")
    tw = torch.empty((T, K), dtype=torch.float32, device="cuda")
    plan.moe_route(Hh.to_dev(x), Hh.to_dev(wr), Hh.to_dev(bias), idx, tw)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    Hh.check_route(idx, tw, ridx, rw)


# The fp32 expert kernel where its tiles end: both tile sizes (few and many blocks), experts with 1 to 300 rows (so that
# warps, half tiles and whole tiles are left out), widths that are no multiple of its column blocks and sums whose
# length is no multiple of its stages, TP shards, and tiles computed whole because no row counts are given.
FP32_FFN = [
    # (T, H, E, K, F, tp, zipf_s)
    (1, 4, 2, 1, 4, 1, 0.0), (40, 36, 4, 2, 68, 1, 1.2), (300, 132, 3, 2, 100, 1, 1.2), (1200, 260, 8, 2, 1284, 1, 1.2),
    (700, 516, 16, 3, 1028, 1, 1.0), (1300, 2052, 8, 2, 260, 1, 1.0), (900, 1284, 16, 2, 1284, 1, 1.0), (129, 100, 6, 2, 264, 2, 1.0),
    # blocks of 8 and of 16 rows (warps side by side), columns that end inside a warp's, TP shards of 68 columns
    (200, 260, 16, 2, 1028, 1, 1.2), (500, 1028, 12, 2, 516, 1, 1.0), (100, 260, 16, 2, 136, 2, 0.0), (64, 516, 16, 2, 260, 1, 0.0),
]


@pytest.mark.parametrize("case", FP32_FFN, ids=lambda c: f"T{c[0]}_H{c[1]}_E{c[2]}_K{c[3]}_F{c[4]}_tp{c[5]}")
def test_fp32_expert_kernel_edges(case):
    T, H, E, K, F, tp, zipf = case
    w = inputs.Workload("fp32_edges", T=T, H=H, E=E, R=1, K=K, F=F, dtype=FP32, zipf_s=zipf, seed=17)
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED, tp_shards=tp)
    y = torch.empty((T, H), dtype=torch.float32, device="cuda")
    args = [Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)]
    plan.moe_layer(*args, y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    Hh.assert_output_close(Hh.to_host_f64(y), ref["y"], FP32)
    # the same rows without the counters: every tile computed whole, the same bytes in the rows there are
    rows = torch.empty((plan.P * 128, H), dtype=torch.float32, device="cuda")
    plan.moe_expert_ffn(plan.layer_tensor(2), plan.layer_tensor(4), *args[3:], rows)
    torch.cuda.synchronize()
    used = plan.layer_tensor(6).flatten().long()
    assert torch.equal(rows[used], plan.layer_tensor(7)[used])


@pytest.mark.parametrize("case", [c for c in FP32_FFN if c[0] >= 8], ids=lambda c: f"T{c[0]}_H{c[1]}_E{c[2]}_K{c[3]}_F{c[4]}_tp{c[5]}")
def test_fp32_fma_kernel_edges(case):
    """The same with ffn_kernel 1: the FMAs where the tensor cores would take over, every register tile of theirs among them."""
    T, H, E, K, F, tp, zipf = case
    w = inputs.Workload("fp32_edges", T=T, H=H, E=E, R=1, K=K, F=F, dtype=FP32, zipf_s=zipf, seed=17)
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED, tp_shards=tp, ffn_kernel=1)
    y = torch.empty((T, H), dtype=torch.float32, device="cuda")
    args = [Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)]
    plan.moe_layer(*args, y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0) and plan.moe_last_launch_count() == 5
    Hh.assert_output_close(Hh.to_host_f64(y), ref["y"], FP32)
    # (1e-6: the bound of the tensor-core form's test, below, holds for sums that round every addition as well)
    assert np.linalg.norm(Hh.to_host_f64(y) - ref["y"]) <= 1e-6 * np.linalg.norm(ref["y"])


# A caller's own tables in fp32: more blocks than the grid has CTAs (each goes on to further blocks, a barrier set per block),
# tiles of 0 to 128 rows; counters that are complete, incomplete (tiles whole) and absent (whole).
@pytest.mark.parametrize("case", [(1, 8, 1024, 132, 260), (40, 4, 2048, 260, 1284), (900, 3, 2048, 516, 516)], ids=lambda c: f"T{c[0]}_E{c[1]}_cap{c[2]}")
def test_fp32_expert_kernel_more_blocks_than_ctas(case):
    T, E, cap, H, F = case
    w = inputs.Workload("fp32_blocks", T=T, H=H, E=E, R=1, K=1, F=F, dtype=FP32, seed=18)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_STATIC, capacity_rows=cap)
    g = torch.Generator(device="cuda").manual_seed(18)
    wg, wu, wd = (torch.empty(s, device="cuda").normal_(0.0, 0.05, generator=g) for s in ((E, F, H), (E, F, H), (E, H, F)))
    recv = torch.empty((E * cap, H), device="cuda").normal_(generator=g)
    te = torch.arange(plan.P, dtype=torch.int32, device="cuda") // (cap // 128)
    te[1::5] = -1
    x = recv.double().view(E, cap, H)
    h = x @ wg.double().transpose(1, 2)
    want = ((h / (1 + torch.exp(-h)) * (x @ wu.double().transpose(1, 2))) @ wd.double().transpose(1, 2)).view(E * cap, H)
    rows_of = torch.randint(0, 129, (plan.P,), dtype=torch.int32, device="cuda", generator=g)
    owned = (te >= 0).repeat_interleave(128)
    stored = owned & (torch.arange(128, device="cuda").repeat(plan.P) < rows_of.repeat_interleave(128))
    for counts, done, rows in ((rows_of, T, stored), (rows_of, T - 1, owned), (None, None, owned)):
        out = torch.zeros_like(recv)
        rd = None if done is None else torch.full((1,), done, dtype=torch.int32, device="cuda")
        plan.moe_expert_ffn(recv, te, wg, wu, wd, out, counts, rd)
        torch.cuda.synchronize()
        assert plan.moe_last_status() == (0, 0)
        Hh.assert_output_close(Hh.to_host_f64(out[rows]), want[rows].cpu().numpy(), FP32)
        assert torch.count_nonzero(out[~rows]) == 0 or counts is not None     # (a block's rows that are not there hold anything)
        assert torch.count_nonzero(out[~owned]) == 0


# dtype fp32 on the tensor cores, where its items end: rows around 16, 32, 64 and 128 (one tile, two), H and F that end inside
# 64 gate columns, 128 columns, 32 and 64 k, sums of odd numbers of 32-k blocks and of fewer than 256 terms, TP shards.
# Per GEMM an element is off by at most n 2^-24 of sum |a b| (n additions; n <= K / 16 truncated ones and K / 32 rounded
# ones), in the 2-norm by about sqrt(K) times less: 1e-6 holds for K up to 2048 with room (seen: 3e-7).
SPLIT_FFN = [
    # (T, H, E, K, F, tp)
    (1, 68, 1, 1, 900, 1), (15, 68, 1, 1, 964, 1), (16, 100, 1, 1, 1028, 1), (17, 36, 2, 2, 932, 1), (33, 128, 1, 1, 960, 1), (65, 260, 2, 2, 900, 1),
    (127, 96, 1, 1, 2052, 1), (128, 516, 2, 1, 996, 1), (129, 260, 2, 2, 1284, 1), (300, 1028, 4, 2, 132, 1), (700, 324, 3, 3, 1088, 1),
    (400, 260, 2, 2, 1000, 2),
]


@pytest.mark.parametrize("case", SPLIT_FFN, ids=lambda c: f"T{c[0]}_H{c[1]}_E{c[2]}_K{c[3]}_F{c[4]}_tp{c[5]}")
def test_fp32_on_tensor_cores_edges(case):
    T, H, E, K, F, tp = case
    w = inputs.Workload("fp32_split", T=T, H=H, E=E, R=1, K=K, F=F, dtype=FP32, seed=23)
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)["y"]
    args = [Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)]
    errs = []
    for kernel in (0, 1):     # split, and the fp32 FMAs
        plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED, tp_shards=tp, ffn_kernel=kernel)
        y = torch.empty((T, H), dtype=torch.float32, device="cuda")
        for _ in range(2):    # the counters are back where they were
            plan.moe_layer(*args, y)
        torch.cuda.synchronize()
        assert plan.moe_last_status() == (0, 0)
        d = Hh.to_host_f64(y) - ref
        errs.append(np.linalg.norm(d) / np.linalg.norm(ref))
    assert errs[0] <= 1e-6 and errs[0] <= 1.05 * errs[1], errs


@pytest.mark.parametrize("mode", [B.DISPATCH_SCAN, B.DISPATCH_ATOMIC_STATIC, B.DISPATCH_ATOMIC_PAGED, B.DISPATCH_ATOMIC_ORDERED])
def test_fp32_on_tensor_cores_in_every_dispatch_mode(mode):
    """(Static regions too, where they are no larger than the batch can fill.)"""
    w = inputs.Workload("split_modes", T=256, H=132, E=2, R=1, K=1, F=1028, dtype=FP32, seed=29)
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    plan = Hh.make_plan(w, mode)
    assert B.moe_workspace_bytes(plan.cfg) > B.moe_workspace_bytes(Hh.make_plan(w, mode, ffn_kernel=1).cfg)
    y = torch.empty((w.T, w.H), dtype=torch.float32, device="cuda")
    plan.moe_layer(*[Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)], y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    assert np.linalg.norm(Hh.to_host_f64(y) - ref["y"]) <= 1e-6 * np.linalg.norm(ref["y"])


@pytest.mark.parametrize("rows", [1, 2, 15, 16, 17, 33, 127])
def test_fp32_on_tensor_cores_tiles_of_few_rows(rows):
    """A caller's own table: a full tile and one of few rows of the same expert, one of few rows alone."""
    T, H, E, F = 300, 100, 2, 932
    plan = B.Plan(B.make_config(T, H, E, 1, 1, F, FP32, dispatch_mode=B.DISPATCH_ATOMIC_PAGED))
    g = torch.Generator(device="cuda").manual_seed(rows)
    wg, wu, wd = (torch.empty(s, device="cuda").normal_(0.0, 0.05, generator=g) for s in ((E, F, H), (E, F, H), (E, H, F)))
    recv = torch.empty((plan.P * 128, H), device="cuda").normal_(generator=g)
    ints = lambda v: torch.tensor(v, dtype=torch.int32, device="cuda")
    te, count = ints([0, -1, 0, 1]), ints([128, 0, rows, rows])
    out = torch.zeros_like(recv)
    plan.moe_expert_ffn(recv, te, wg, wu, wd, out, count, ints([T]))
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    for tile in (0, 2, 3):
        e, n = int(te[tile]), int(count[tile])
        x = recv[tile * 128:tile * 128 + n].double()
        gate = x @ wg[e].double().T
        want = (gate * torch.sigmoid(gate) * (x @ wu[e].double().T)) @ wd[e].double().T
        assert (out[tile * 128:tile * 128 + n].double() - want).norm() <= 1e-6 * want.norm(), tile
    assert torch.count_nonzero(out[128:256]) == 0


# (x, Wg, Wu, Wd times powers of two): parts of numbers near the smallest exponents; rows of large numbers, whose parts are
# scaled the other way; an intermediate beyond what the parts of a row of ordinary x can hold.
@pytest.mark.parametrize("exps", [(0, 0, 0, 0), (0, 0, -120, 0), (0, 0, 0, -120), (-60, 0, 0, 0), (-112, 0, 115, 0), (0, -113, 0, 0), (40, -40, -40, 0), (60, 0, 0, -60),
                                  (60, 0, 0, 0), (0, 57, 57, -100), (33, 0, 0, -40)], ids=str)
def test_fp32_on_tensor_cores_over_the_range_of_exponents(exps):
    T, H, F = 48, 132, 932
    plan = B.Plan(B.make_config(T, H, 1, 1, 1, F, FP32, dispatch_mode=B.DISPATCH_ATOMIC_PAGED))
    g = torch.Generator(device="cuda").manual_seed(7)
    x, wg, wu, wd = (torch.empty(s, device="cuda").normal_(0.0, 1.0 if s[0] == T else 0.1, generator=g) * 2.0 ** e
                     for s, e in zip(((T, H), (1, F, H), (1, F, H), (1, H, F)), exps))
    recv = torch.zeros((plan.P * 128, H), device="cuda")
    recv[:T] = x
    if exps[0] == 33:
        recv[1:T] *= 2.0 ** -33              # one large row in a group of ordinary ones
    te = torch.full((plan.P,), -1, dtype=torch.int32, device="cuda")
    te[0] = 0
    out = torch.zeros_like(recv)
    plan.moe_expert_ffn(recv, te, wg, wu, wd, out, torch.tensor([T] + [0] * (plan.P - 1), dtype=torch.int32, device="cuda"),
                        torch.full((1,), T, dtype=torch.int32, device="cuda"))
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    gate = recv[:T].double() @ wg[0].double().T
    want = (gate * torch.sigmoid(gate) * (recv[:T].double() @ wu[0].double().T)) @ wd[0].double().T
    row = want.abs().amax(1, keepdim=True)
    assert (row < 3.4e38).all() and torch.isfinite(out[:T]).all()
    # 1e-6 per row as above; rows so small that fp32's own smallest steps show (2^-150 an element) by these besides
    assert (((out[:T].double() - want) / row).norm(dim=1) <= 1e-6 * (want / row).norm(dim=1) + 2.0 ** -150 / row[:, 0] * H ** 0.5).all()


def test_fp32_on_tensor_cores_infinities_and_nan():
    """What an infinity, a NaN, an overflow or a number that rounds up to bf16's infinity does to a row is what fp32 sums give."""
    T, H, F = 48, 72, 928
    plan = B.Plan(B.make_config(T, H, 1, 1, 1, F, FP32, dispatch_mode=B.DISPATCH_ATOMIC_PAGED))
    g = torch.Generator(device="cuda").manual_seed(5)
    wg, wu, wd = (torch.empty(s, device="cuda").normal_(0.0, 0.05, generator=g) for s in ((1, F, H), (1, F, H), (1, H, F)))
    x = torch.empty((T, H), device="cuda").normal_(generator=g)
    x[1, 3], x[2, 5], x[3, 7], x[4, 9] = float("inf"), float("-inf"), float("nan"), 3.4e38
    x[5] *= 1e38                 # sums that overflow or not
    x[6], x[7, ::2] = 0.0, 0.0
    wg[0, 10, 3], wd[0, 13, 14], wd[0, 17, 3], wd[0, 19, 4] = 0.0, float("nan"), 3.395e38, float("-inf")
    wg[0, 20:40] = wg[0, 20:40].bfloat16().float()      # (no middle and last parts: infinity times zero)
    recv = torch.zeros((plan.P * 128, H), device="cuda")
    recv[:T] = x
    te = torch.full((plan.P,), -1, dtype=torch.int32, device="cuda")
    te[0] = 0
    count, done = torch.tensor([T] + [0] * (plan.P - 1), dtype=torch.int32, device="cuda"), torch.full((1,), T, dtype=torch.int32, device="cuda")
    out = torch.zeros_like(recv)
    plan.moe_expert_ffn(recv, te, wg, wu, wd, out, count, done)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    def chain(a, b):             # one fp32 product and sum after the other
        s = np.zeros((a.shape[0], b.shape[0]), np.float32)
        for k in range(a.shape[1]):
            s = (a[:, k, None].astype(np.float64) * b[None, :, k].astype(np.float64) + s).astype(np.float32)
        return s
    with np.errstate(all="ignore"):
        xs, hg, hu, hd = (t.cpu().numpy() for t in (x, wg[0], wu[0], wd[0]))
        gate, up = chain(xs, hg), chain(xs, hu)
        want = chain((gate / (np.float32(1) + np.exp(-gate)) * up).astype(np.float32), hd)
    got = out[:T].cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(np.isposinf(got), np.isposinf(want)) and np.array_equal(np.isneginf(got), np.isneginf(want))
    assert np.isnan(want).any() and np.isinf(want).any() and np.isfinite(want).sum() > T * H // 2
    ok = np.isfinite(want)
    got, want = np.where(ok, got, 0).astype(np.float64), np.where(ok, want, 0).astype(np.float64)
    usual = np.delete(want, 3, axis=1)     # (column 3 is 1e37 times the others)
    scale = np.sqrt(np.mean(usual ** 2, axis=1, keepdims=True))
    assert (np.abs(got - want) <= 1e-4 * np.maximum(np.abs(want), scale)).all()


def _fp32_experts(T, H, E, K, F, spoil=None, **kw):
    plan = B.Plan(B.make_config(T, H, E, 1, K, F, FP32, dispatch_mode=B.DISPATCH_ATOMIC_PAGED, **kw))
    g = torch.Generator(device="cuda").manual_seed(11)
    normal = lambda *s, std=1.0: torch.empty(s, device="cuda").normal_(0.0, std, generator=g)
    a = dict(x=normal(T, H), wr=normal(E, H, std=0.02), wg=normal(E, F, H, std=0.02), wu=normal(E, F, H, std=0.02), wd=normal(E, H, F, std=0.02))
    if spoil is not None:
        spoil(a)
    y = torch.empty((T, H), device="cuda")

    def layer():
        plan.moe_layer(a["x"], a["wr"], None, a["wg"], a["wu"], a["wd"], y)
        return y
    return plan, a, layer


def _spoil(name, value, *at):
    def spoil(a):
        a[name][at] = value
    return spoil


def _times(name, factor, *at):
    def spoil(a):
        a[name][at] *= factor
    return spoil


NOT_FINITE = {"nan_row": _spoil("x", float("nan"), 17, 3), "inf_row": _spoil("x", float("-inf"), 17), "wg_inf": _spoil("wg", float("inf"), slice(None), 10, 3),
              "wg_nan": _spoil("wg", float("nan")), "wd_inf": _spoil("wd", float("inf"), 2, 10, 3), "large_row": _times("x", 1e37, 17),
              "all_nan": _spoil("x", float("nan")), "all_inf": _spoil("x", float("inf"))}


@pytest.mark.parametrize("what", NOT_FINITE)
def test_fp32_values_that_are_not_finite_take_no_longer_than_the_fmas(what):
    """(A tenth more is let pass as noise.)  And the same elements are NaN, infinite and finite as with the FMAs, which round elsewhere;
    tokens that nothing was done to keep their bytes."""
    shape = (1000, 1024, 16, 2, 2048)
    took, ys = [], []
    for kernel in (0, 1):
        plan, a, layer = _fp32_experts(*shape, spoil=NOT_FINITE[what], ffn_kernel=kernel)
        layer()
        best = 1e9
        for _ in range(3):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            ys.append(layer().clone())
            t1.record()
            torch.cuda.synchronize()
            best = min(best, t0.elapsed_time(t1))
        assert plan.moe_last_status() == (0, 0)
        took.append(best)
    assert took[0] <= 1.1 * took[1], took
    got, want = ys[0], ys[-1]
    assert torch.equal(got.isnan(), want.isnan()) and torch.equal(got.isposinf(), want.isposinf()) and torch.equal(got.isneginf(), want.isneginf())
    if what in ("nan_row", "inf_row", "large_row"):
        clean = _fp32_experts(*shape)[2]()
        others = torch.arange(shape[0], device="cuda") != 17
        assert torch.equal(got[others], clean[others]) and torch.isfinite(got[others]).all()


def test_fp32_plan_on_a_workspace_without_room_for_the_parts():
    """A workspace as large as the FMAs need is taken, and they are used; a byte less than they need is refused."""
    shape = (300, 260, 4, 2, 1028)
    plan, a, layer = _fp32_experts(*shape, ffn_kernel=1)
    want = layer().clone()
    cfg = B.make_config(*shape[:3], 1, *shape[3:], FP32, dispatch_mode=B.DISPATCH_ATOMIC_PAGED)
    full, lean = B.moe_workspace_bytes(cfg), B.moe_workspace_bytes(plan.cfg)
    assert full > lean
    room = torch.empty(full, dtype=torch.uint8, device="cuda")
    for nbytes, same in ((lean, True), (full - 1, True), (full, False)):
        small = B.Plan(cfg)
        small.close()
        room.fill_(0xff)
        small.handle, small.workspace = ctypes.c_void_p(), room
        assert B.lib().moe_plan_create(ctypes.byref(cfg), room.data_ptr(), nbytes, ctypes.byref(small.handle)) == 0
        y = torch.empty_like(want)
        small.moe_layer(a["x"], a["wr"], None, a["wg"], a["wu"], a["wd"], y)
        torch.cuda.synchronize()
        assert small.moe_last_status() == (0, 0) and torch.equal(y, want) == same
        assert (room[nbytes:] == 0xff).all()
    assert B.lib().moe_plan_create(ctypes.byref(cfg), room.data_ptr(), lean - 1, ctypes.byref(ctypes.c_void_p())) == -7


def test_fp32_experts_without_row_counts_on_a_pool_of_nan():
    """Rows that nobody wrote to hold NaN: the others are the bytes that a call with row counts gives."""
    plan, a, layer = _fp32_experts(700, 260, 6, 2, 1032)
    layer()
    w = inputs.Workload("nan_pool", T=700, H=260, E=6, R=1, K=2, F=1032, dtype=FP32)
    b = _dispatch_with_counters(w, plan, a["x"], plan.layer_tensor(0))
    used = b["slot"].flatten().long()
    pool = torch.full_like(b["recv"], float("nan"))
    pool[used] = b["recv"][used]
    outs = []
    for counts in ((), (b["tile_count"], b["rows_done"])):
        outs.append(torch.zeros_like(pool))
        plan.moe_expert_ffn(pool, b["te"], a["wg"], a["wu"], a["wd"], outs[-1], *counts)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    assert torch.equal(outs[0][used], outs[1][used]) and torch.isfinite(outs[0][used]).all()


# The CTA-pair expert kernel where its items end: an expert's rows around 16, 32, 128 (one tile), 129, 256 (a pair of
# tiles) and 257, all experts the same so that every count is met; in the paged layout (tiles of an expert apart) and
# the ordered one; H and F that end inside its 512- and 256-column blocks and inside a k-block; one and two launches.
@pytest.mark.parametrize("split", [1, 2])
@pytest.mark.parametrize("mode", [B.DISPATCH_ATOMIC_PAGED, B.DISPATCH_ATOMIC_ORDERED])
@pytest.mark.parametrize("rows", [1, 16, 17, 33, 112, 127, 128, 129, 145, 255, 256, 257, 300])
def test_pair_expert_kernel_row_counts(rows, mode, split):
    E, H, F = 3, (200, 776, 1032)[rows % 3], (72, 392, 520)[rows % 3]
    w = inputs.Workload("pair_rows", T=rows, H=H, E=E, R=1, K=E, F=F, dtype=BF16, seed=19)   # K = E: every expert gets every token
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    args = [Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)]
    ys = []
    for kernel in (2, 0):
        plan = Hh.make_plan(w, mode, ffn_kernel=kernel, ffn_split=split)
        for _ in range(2):      # twice: the second call meets the counters as the first one left them
            y = torch.empty((w.T, w.H), dtype=torch.bfloat16, device="cuda")
            plan.layer_tensor(2).fill_(float("nan"))   # rows that are not there must not reach the others
            plan.moe_layer(*args, y)
            torch.cuda.synchronize()
            assert plan.moe_last_status() == (0, 0)
        Hh.assert_output_close(Hh.to_host_f64(y), ref["y"], BF16)
        ys.append(y)
    assert torch.equal(ys[0], ys[1])     # the same sums in the same order: the same bytes as one CTA per tile


# Where the default takes the pair kernel: skewed experts (empty ones and ones of several tiles), TP shards, the push
# epilogue and a call without counters give the bytes of the one-CTA kernel (asked for with ffn_thin_tiles = -1).
@pytest.mark.parametrize("tp,combine", [(1, 0), (1, 1), (2, 0), (2, 1)])
def test_pair_expert_kernel_by_default(tp, combine):
    w = inputs.Workload("pair_default", T=900, H=1544, E=12, R=1, K=3, F=2064, dtype=BF16, zipf_s=1.2, seed=23)
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    args = [Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)]
    ys = []
    for thin in (0, -1):
        plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_ORDERED, tp_shards=tp, combine_mode=combine, ffn_thin_tiles=thin)
        y = torch.empty((w.T, w.H), dtype=torch.bfloat16, device="cuda")
        plan.moe_layer(*args, y)
        torch.cuda.synchronize()
        assert plan.moe_last_status() == (0, 0)
        ys.append(y)
        if combine == 0:
            rows = torch.empty((plan.P * 128, w.H), dtype=torch.bfloat16, device="cuda")
            plan.moe_expert_ffn(plan.layer_tensor(2), plan.layer_tensor(4), *args[3:], rows)
            torch.cuda.synchronize()
            used = plan.layer_tensor(6).flatten().long()
            assert torch.equal(rows[used], plan.layer_tensor(7)[used])
    assert torch.equal(ys[0], ys[1])


# H and F that end inside the 32 columns of an epilogue warp (at 8, 16 and 24 of them): some lanes of the warp store and
# others do not, several units of rows long, with and without the push epilogue.
@pytest.mark.parametrize("combine", [0, 1])
@pytest.mark.parametrize("extra", [8, 16, 24])
def test_pair_expert_kernel_columns_end_inside_a_warp(extra, combine):
    w = inputs.Workload("pair_cols", T=700, H=1536 + extra, E=4, R=1, K=2, F=1056 - extra, dtype=BF16, zipf_s=0.7, seed=24)
    args = [Hh.to_dev(a) for a in Hh.oracle_inputs(w)]
    ys = []
    for thin in (0, -1):        # pairs by default; one CTA per tile
        plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED, combine_mode=combine, ffn_thin_tiles=thin)
        y = torch.empty((w.T, w.H), dtype=torch.bfloat16, device="cuda")
        for i in (2, 7):
            plan.layer_tensor(i).fill_(float("nan"))
        plan.moe_layer(*args, y)
        torch.cuda.synchronize()
        assert plan.moe_last_status() == (0, 0)
        ys.append(y)
    assert torch.equal(ys[0], ys[1]) and bool(torch.isfinite(ys[0]).all())


def test_named_split_keeps_a_tokens_bytes_whatever_the_batch():
    """The tensor-core kernels add up each result in one order, in every form (narrow, M = 64, whole tiles, CTA pairs).  A plan
    that names ffn_split never takes the plain-FMA kernels for few tokens, so a token's bytes do not depend on its batch."""
    T, H, E, K, F = 300, 1536, 4, 2, 1024
    w = inputs.Workload("batch_bytes", T=T, H=H, E=E, R=1, K=K, F=F, dtype=BF16, seed=38)
    x, wr, _, wg, wu, wd = (Hh.to_dev(a) for a in Hh.oracle_inputs(w))
    for split in (1, 2):
        ys = {}
        for n in (1, 3, 5, 6, 16, 17, 70, 140, T):      # 300: more than a tile of rows per expert, CTA pairs
            plan = B.Plan(B.make_config(n, H, E, 1, K, F, BF16, ffn_split=split))
            ys[n] = torch.empty((n, H), dtype=torch.bfloat16, device="cuda")
            plan.moe_layer(x[:n], wr, None, wg, wu, wd, ys[n])
            assert plan.moe_last_status() == (0, 0)
        for n, y in ys.items():
            assert torch.equal(y, ys[T][:n]), (split, n)


# The refine kernel's numbering of the chains: token counts that give its CTAs 12 to 64 tokens (a whole wave on 148 SMs),
# with every token's candidates in ONE class of experts modulo eight (its bucket overflows into the others' free slots),
# with two classes, and with more candidates than a CTA has threads (every expert the same: all 256 are candidates).
@pytest.mark.parametrize("T", [1300, 3000, 5500, 8000, 9500])
@pytest.mark.parametrize("case", ["one_class", "two_classes", "all_equal"])
def test_router_filter_chain_numbering(T, case):
    H, E, K = 64, 256, 8
    w = inputs.Workload("numbering", T=T, H=H, E=E, R=1, K=K, F=8, dtype=BF16, seed=29, identity_experts=True)
    x, wr, _, *_ = Hh.oracle_inputs(w, with_experts=False)
    bias = np.zeros(E, np.float32)
    if case == "all_equal":
        wr[:] = wr[0]
    else:
        keep = (np.arange(E) % 8 == 3) if case == "one_class" else (np.arange(E) % 4 == 1)
        bias[~keep] = -50.0
    ridx, rw, _ = oracle.route(x, wr, bias, K, BF16)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED)
    idx = torch.empty((T, K), dtype=torch.int32, device="cuda")
    tw = torch.empty((T, K), dtype=torch.float32, device="cuda")
    plan.moe_route(Hh.to_dev(x), Hh.to_dev(wr), Hh.to_dev(bias), idx, tw)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    Hh.check_route(idx, tw, ridx, rw)


# The kernel for a handful of tokens: one to five tokens (an expert with one to five rows; six of this size go to the tensor cores),
# H and F that end inside a lane's vectors and a warp's columns, few and many experts (more tiles than the table's first
# 256 entries), TP shards, the push epilogue, and a call whose rows never become available.
FEW = [
    # (T, H, E, K, F, tp, combine)
    (1, 1032, 8, 2, 520, 1, 0), (2, 1288, 4, 4, 776, 1, 0), (3, 1024, 2, 2, 512, 1, 1), (4, 1544, 6, 3, 1056, 2, 0),
    (5, 1032, 5, 5, 520, 1, 1), (5, 1024, 256, 8, 512, 1, 0), (5, 1032, 128, 16, 1040, 2, 1), (6, 1032, 8, 2, 520, 1, 0), (1, 256, 8, 2, 256, 1, 0),
    (4, 264, 40, 6, 264, 1, 1), (3, 4096, 4, 2, 2064, 1, 0), (2, 2048, 24, 4, 2064, 1, 1), (1, 2048, 16, 16, 1040, 1, 0),
    # small layers of more tokens: experts of up to 32 rows (groups of eight), the largest of the range, one past it
    (32, 256, 4, 2, 264, 1, 0), (31, 264, 2, 2, 256, 1, 1), (9, 512, 16, 3, 528, 2, 0), (16, 512, 100, 4, 256, 1, 0), (33, 256, 4, 2, 256, 1, 0),
]


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("case", FEW, ids=lambda c: f"T{c[0]}_H{c[1]}_E{c[2]}_K{c[3]}_F{c[4]}_tp{c[5]}_push{c[6]}")
def test_few_tokens_kernel(case, mode):
    T, H, E, K, F, tp, combine = case
    w = inputs.Workload("few", T=T, H=H, E=E, R=1, K=K, F=F, dtype=BF16, zipf_s=1.2, seed=31)
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    plan = Hh.make_plan(w, mode, tp_shards=tp, combine_mode=combine)
    y = torch.empty((T, H), dtype=torch.bfloat16, device="cuda")
    plan.layer_tensor(2).fill_(float("nan"))     # rows that are not there must not reach the others
    plan.moe_layer(*[Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)], y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    Hh.assert_output_close(Hh.to_host_f64(y), ref["y"], BF16)


# Up to five tokens the layer resolves the addresses and combines inside the two expert kernels: the tables it leaves are
# a dispatch's, and the result is, byte for byte, that of the steps called one after the other.
@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("case", [c for c in FEW if c[0] not in (6, 33)], ids=lambda c: f"T{c[0]}_H{c[1]}_E{c[2]}_K{c[3]}_F{c[4]}_tp{c[5]}_push{c[6]}")
def test_few_tokens_layer_equals_its_steps(case, mode):
    T, H, E, K, F, tp, combine = case
    w = inputs.Workload("few", T=T, H=H, E=E, R=1, K=K, F=F, dtype=BF16, zipf_s=1.2, seed=32)
    x, wr, bias, wg, wu, wd = (Hh.to_dev(a) for a in Hh.oracle_inputs(w))
    plan = Hh.make_plan(w, mode, tp_shards=tp, combine_mode=combine)
    y, y2 = (torch.full((T, H), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    for i in range(9):
        if i not in (8, 9):
            plan.layer_tensor(i).zero_()
    plan.moe_layer(x, wr, bias, wg, wu, wd, y)
    down = 1 if T == 1 or min(T * K * tp, E * tp) * H * (F // tp) * 2 <= 64 << 20 else 2  # combined, or with a combine behind it
    assert plan.moe_last_launch_count() == (1 if E <= 64 else 2) + 1 + down
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    left = [plan.layer_tensor(i).clone() for i in range(8)]
    idx, tw, recv, cnt, te, src, slot, rows = left
    recv2, rows2 = torch.zeros_like(recv), torch.zeros_like(rows)
    cnt2, te2, src2, slot2 = (torch.empty_like(a) for a in (cnt, te, src, slot))
    tiles, done = torch.empty(plan.P, dtype=torch.int32, device="cuda"), torch.empty(1, dtype=torch.int32, device="cuda")
    plan.moe_dispatch(x, idx, recv2, cnt2, te2, src2, slot2, tiles, done)
    if combine:
        plan.moe_expert_ffn_push(recv2, te2, src2, wg, wu, wd, rows2, tiles, done)
        plan.moe_combine_staged(rows2, slot2, tw, y2)
    else:
        plan.moe_expert_ffn(recv2, te2, wg, wu, wd, rows2, tiles, done)
        plan.moe_combine(rows2, slot2, tw, y2)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    assert torch.equal(y, y2) and torch.equal(cnt, cnt2)
    flat, s, s2 = torch.arange(idx.numel(), device="cuda", dtype=torch.int32), slot.flatten().long(), slot2.flatten().long()
    assert torch.equal(src[s], flat) and int((src >= 0).sum()) == flat.numel()
    assert torch.equal(te[s // 128], idx.flatten()) and int((te >= 0).sum()) == int((cnt > 0).sum())
    assert torch.equal(recv[s], recv2[s2])
    assert torch.equal(rows, rows2) if combine else torch.equal(rows[s], rows2[s2])


def test_few_tokens_kernel_wait_runs_out_and_reports_it():
    w = inputs.Workload("few_wait", T=2, H=1024, E=4, R=1, K=2, F=512, dtype=BF16, seed=31)
    _, _, _, wg, wu, wd = Hh.oracle_inputs(w)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED, wait_limit_ns=1_000_000)
    rows = plan.P * 128
    recv, out = (torch.zeros((rows, w.H), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    te = torch.full((plan.P,), -1, dtype=torch.int32, device="cuda")
    te[0] = 1
    counts, done = torch.zeros(plan.P, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    plan.moe_expert_ffn(recv, te, Hh.to_dev(wg), Hh.to_dev(wu), Hh.to_dev(wd), out, counts, done)
    torch.cuda.synchronize()
    assert plan.moe_last_status()[0] == -6       # MOE_ERR_TIMEOUT; the context stays usable
    assert torch.count_nonzero(out) == 0


@pytest.mark.parametrize("T", [2, 6])
def test_layer_refuses_a_pool_beyond_the_work_list_whatever_the_batch(T):
    """More than 4608 tiles are outside what the bf16 expert kernels take: also for the few tokens that need no work list."""
    w = inputs.Workload("few_refused", T=T, H=256, E=8, R=1, K=2, F=256, dtype=BF16, seed=37)
    args = [Hh.to_dev(a) for a in Hh.oracle_inputs(w)]
    y = torch.empty((T, w.H), dtype=torch.bfloat16, device="cuda")
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_STATIC, capacity_rows=128 * 577)
    assert plan.P == 4616
    with pytest.raises(B.MoeError) as err:
        plan.moe_layer(*args, y)
    assert err.value.code == -3      # MOE_ERR_UNSUPPORTED
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_STATIC, capacity_rows=128 * 576)
    plan.moe_layer(*args, y)
    assert plan.moe_last_status() == (0, 0)


def test_few_tokens_kernel_expert_named_twice():
    """A caller's own routing may name an expert more than once for a token: more rows than tokens in a tile."""
    w = inputs.Workload("few_twice", T=3, H=520, E=4, R=1, K=4, F=264, dtype=BF16, seed=33)
    x, _, _, wg, wu, wd = Hh.oracle_inputs(w)
    idx = np.array([[2, 2, 2, 2], [2, 2, 2, 1], [2, 2, 2, 2]], np.int32)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED)
    rows = plan.P * 128
    recv, out = (torch.zeros((rows, w.H), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    cnt, te, src = (torch.empty(n, dtype=torch.int32, device="cuda") for n in (w.E, plan.P, rows))
    slot, tiles, done = (torch.empty(n, dtype=torch.int32, device="cuda") for n in ((w.T, w.K), (plan.P,), (1,)))
    plan.moe_dispatch(Hh.to_dev(x), Hh.to_dev(idx), recv, cnt, te, src, slot, tiles, done)
    dw = [Hh.to_dev(a) for a in (wg, wu, wd)]
    plan.moe_expert_ffn(recv, te, *dw, out, tiles, done)
    whole = torch.zeros_like(out)
    plan.moe_expert_ffn(recv, te, *dw, whole)     # without row counts: the tensor-core kernel, every tile whole
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0) and cnt.cpu().tolist() == [0, 1, 11, 0]
    used = slot.flatten().long()
    a, b = out[used].float(), whole[used].float()
    # both round an fp32 sum of F products to bf16 after an intermediate rounded to bf16: two units in the last place of the
    # largest output cover the order of additions
    assert float((a - b).abs().max()) <= 2 * 2.0 ** -8 * float(b.abs().max())


@pytest.mark.parametrize("push", [0, 1])
@pytest.mark.parametrize("case", [(1, 8, 2), (3, 5, 1), (1, 256, 1)], ids=lambda c: f"T{c[0]}_E{c[1]}_K{c[2]}")
def test_few_tokens_kernel_walks_every_owned_tile(case, push):
    """A caller's own table may name an owner for every tile of its static regions, also where no row is: more owned tiles
    than the batch has assignments, rows only in the last regions."""
    T, E, K = case
    w = inputs.Workload("few_owned", T=T, H=520, E=E, R=1, K=K, F=264, dtype=BF16, seed=34)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_STATIC)
    assert plan.P == E
    g = torch.Generator(device="cuda").manual_seed(34)
    wg, wu, wd = (torch.empty(s, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.05, generator=g)
                  for s in ((E, w.F, w.H), (E, w.F, w.H), (E, w.H, w.F)))
    recv = torch.empty((E * 128, w.H), dtype=torch.bfloat16, device="cuda").normal_(generator=g)
    te = torch.arange(E, dtype=torch.int32, device="cuda")
    counts, done = torch.zeros(E, dtype=torch.int32, device="cuda"), torch.full((1,), T * K, dtype=torch.int32, device="cuda")
    slots = [(E - 1) * 128 + i for i in range(T * K - T * K // 2)] + [(E - 2) * 128 + i for i in range(T * K // 2)]
    for s in slots:
        counts[s // 128] += 1
    src = torch.full((E * 128,), -1, dtype=torch.int32, device="cuda")
    src[slots] = torch.arange(T * K, dtype=torch.int32, device="cuda")
    whole = torch.zeros_like(recv)
    plan.moe_expert_ffn(recv, te, wg, wu, wd, whole)     # without row counts: the tensor-core kernel, every tile whole
    if push:
        out = torch.zeros((T * K, w.H), dtype=torch.bfloat16, device="cuda")
        plan.moe_expert_ffn_push(recv, te, src, wg, wu, wd, out, counts, done)
        got = out
    else:
        out = torch.zeros_like(recv)
        plan.moe_expert_ffn(recv, te, wg, wu, wd, out, counts, done)
        got = out[slots]
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    a, b = got.float(), whole[slots].float()
    # (the bound of test_few_tokens_kernel_expert_named_twice)
    assert float(b.abs().max()) > 0 and float((a - b).abs().max()) <= 2 * 2.0 ** -8 * float(b.abs().max())


def test_static_regions_of_more_rows_than_the_batch_keep_the_tensor_cores():
    """A decode-size plan may hold static regions that other callers fill (capacity_rows above the batch): whole tiles of
    rows belong on the tensor cores, with the same bytes as without row counts."""
    E, H, F, cap = 3, 520, 264, 256
    w = inputs.Workload("few_regions", T=1, H=H, E=E, R=1, K=1, F=F, dtype=BF16, seed=35)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_STATIC, capacity_rows=cap)
    g = torch.Generator(device="cuda").manual_seed(35)
    wg, wu, wd = (torch.empty(s, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.05, generator=g)
                  for s in ((E, F, H), (E, F, H), (E, H, F)))
    recv = torch.empty((E * cap, H), dtype=torch.bfloat16, device="cuda").normal_(generator=g)
    te = torch.arange(plan.P, dtype=torch.int32, device="cuda") // (cap // 128)
    counts, done = torch.full((plan.P,), 128, dtype=torch.int32, device="cuda"), torch.full((1,), E * cap, dtype=torch.int32, device="cuda")
    out, whole = torch.zeros_like(recv), torch.ones_like(recv)
    plan.moe_expert_ffn(recv, te, wg, wu, wd, out, counts, done)
    assert plan.moe_last_launch_count() == 1     # (the kernels for few tokens are two launches)
    plan.moe_expert_ffn(recv, te, wg, wu, wd, whole)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0) and torch.equal(out, whole)


# ------------------------------------------------------------------ dispatch edge cases
@pytest.mark.parametrize("mode", MODES)
def test_dispatch_all_tokens_to_one_expert_and_empty_experts(mode):
    w = inputs.Workload("skew", T=700, H=64, E=8, R=2, K=2, F=8, dtype=BF16)
    x = inputs.make_x(w)
    idx = np.zeros((w.T, w.K), np.int32)
    idx[:, 0], idx[:, 1] = 5, 2           # experts 5 and 2 get T rows each, the others none
    ref = oracle.dispatch(x, idx, w.E, w.R, w.dtype)
    plan = Hh.make_plan(w, mode)
    rows = plan.P * 128
    recv = torch.zeros((rows, w.H), dtype=torch.bfloat16, device="cuda")
    cnt = torch.empty(w.E, dtype=torch.int32, device="cuda")
    te = torch.empty(plan.P, dtype=torch.int32, device="cuda")
    src = torch.empty(rows, dtype=torch.int32, device="cuda")
    slot = torch.empty((w.T, w.K), dtype=torch.int32, device="cuda")
    plan.moe_dispatch(Hh.to_dev(x), Hh.to_dev(idx), recv, cnt, te, src, slot)
    assert plan.moe_last_status() == (0, 0)
    Hh.check_dispatch(w, plan.P, x, idx, ref, recv, cnt, te, src, slot)


def test_static_region_overflow_is_reported_not_silent():
    """Mode 1 with regions smaller than the load: the status word says overflow and names an expert,
    counts stay exact, dropped assignments get slot -1, nothing is written out of bounds."""
    w = inputs.Workload("overflow", T=600, H=64, E=4, R=1, K=1, F=8, dtype=BF16)
    x = inputs.make_x(w)
    idx = np.full((w.T, 1), 3, np.int32)
    cfg = B.make_config(w.T, w.H, w.E, w.R, w.K, w.F, w.dtype, dispatch_mode=B.DISPATCH_ATOMIC_STATIC,
                        capacity_rows=256)
    plan = B.Plan(cfg)
    rows = plan.P * 128
    guard = torch.full((rows + 128, w.H), 7.0, dtype=torch.bfloat16, device="cuda")
    cnt = torch.empty(w.E, dtype=torch.int32, device="cuda")
    te = torch.empty(plan.P, dtype=torch.int32, device="cuda")
    src = torch.empty(rows, dtype=torch.int32, device="cuda")
    slot = torch.empty((w.T, w.K), dtype=torch.int32, device="cuda")
    plan.moe_dispatch(Hh.to_dev(x), Hh.to_dev(idx), guard[:rows], cnt, te, src, slot)
    code, detail = plan.moe_last_status()
    assert code == -5 and detail == 3
    assert cnt.cpu().tolist() == [0, 0, 0, 600]
    s = slot.cpu().numpy().ravel()
    assert (s >= 0).sum() == 256 and (s == -1).sum() == 600 - 256
    assert torch.all(guard[rows:] == 7.0)


def test_bad_arguments_are_refused_on_the_host():
    cfg = B.make_config(16, 100, 8, 2, 2, 64, BF16)      # H*2 bytes not a multiple of 16
    with pytest.raises(B.MoeError) as ei:
        B.moe_workspace_bytes(cfg)
    assert ei.value.code == -2
    with pytest.raises(B.MoeError):
        B.moe_workspace_bytes(B.make_config(16, 128, 8, 3, 2, 64, BF16))   # E % R != 0
    with pytest.raises(B.MoeError):
        B.moe_workspace_bytes(B.make_config(16, 128, 8, 2, 9, 64, BF16))   # K > E


# ------------------------------------------------------------------ availability counters and the bounded wait
def _dispatch_with_counters(w, plan, dx, didx):
    rows = plan.P * 128
    b = dict(recv=torch.zeros((rows, w.H), dtype=Hh.el_dtype(w), device="cuda"),
             cnt=torch.empty(w.E, dtype=torch.int32, device="cuda"), te=torch.empty(plan.P, dtype=torch.int32, device="cuda"),
             src=torch.empty(rows, dtype=torch.int32, device="cuda"),
             slot=torch.empty((w.T, w.K), dtype=torch.int32, device="cuda"),
             tile_count=torch.full((plan.P,), 77, dtype=torch.int32, device="cuda"),
             rows_done=torch.full((1,), 77, dtype=torch.int32, device="cuda"))
    plan.moe_dispatch(dx, didx, b["recv"], b["cnt"], b["te"], b["src"], b["slot"], b["tile_count"], b["rows_done"])
    return b


@pytest.mark.parametrize("case", [(1, 8, 1, 1), (33, 8, 3, 1), (129, 16, 33, 32), (512, 8, 256, 8), (4096, 8, 256, 1), (4097, 8, 7, 1), (1365, 8, 5, 3)],
                         ids=lambda c: f"T{c[0]}_E{c[2]}_K{c[3]}")
def test_paged_dispatch_where_its_small_batches_end(case):
    """A caller's own ids, on buffers full of old values: every table entry of a dispatch that is one launch, up to 4096 ids and
    beyond; ids that are no expert; one expert with every row."""
    T, H, E, K = case
    w = inputs.Workload("small_dispatch", T=T, H=H, E=E, R=1, K=K, F=0, dtype=BF16, identity_experts=True)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED)
    g = torch.Generator(device="cuda").manual_seed(T)
    x = torch.empty((T, H), dtype=torch.bfloat16, device="cuda").normal_(generator=g)
    any_ids = torch.rand((T, E), device="cuda", generator=g).argsort(1)[:, :K].to(torch.int32).contiguous()
    one = torch.full((T, K), E - 1, dtype=torch.int32, device="cuda") if K == 1 else any_ids
    bad = any_ids.clone()
    bad[T // 2, 0] = E
    for ids in (any_ids, one, bad):
        old = lambda *s: torch.full(s, 12345, dtype=torch.int32, device="cuda")
        recv = torch.zeros((plan.P * 128, H), dtype=torch.bfloat16, device="cuda")
        count, te, src, slot, tc, done = old(E), old(plan.P), old(plan.P * 128), old(T, K), old(plan.P), old(1)
        for _ in range(2):
            plan.moe_dispatch(x, ids, recv, count, te, src, slot, tc, done)
        torch.cuda.synchronize()
        assert plan.moe_last_status() == ((0, 0) if ids is not bad else (-1, T // 2))
        flat, good = slot.flatten().long(), (ids.flatten() < E)
        assert (flat[~good] == -1).all() and done.item() == T * K
        want = torch.bincount(ids.flatten()[good].long(), minlength=E)
        assert torch.equal(count.long(), want)
        rows = flat[good]
        assert rows.unique().numel() == rows.numel() and torch.equal(te[rows // 128], ids.flatten()[good])
        source = torch.full((plan.P * 128,), -1, dtype=torch.int64, device="cuda")
        source[rows] = torch.arange(T * K, device="cuda")[good]
        assert torch.equal(src.long(), source)
        assert torch.equal(tc.long(), torch.bincount(rows // 128, minlength=plan.P))
        assert torch.equal(te >= 0, tc > 0) and torch.equal(torch.bincount(te[te >= 0].long(), minlength=E), (want + 127) // 128)
        assert torch.equal(recv[rows], x.repeat_interleave(K, 0)[good])


@pytest.mark.parametrize("case", [(1, 64, 1), (37, 64, 32), (511, 256, 8), (4096, 8, 1)], ids=lambda c: f"T{c[0]}_E{c[1]}_K{c[2]}")
def test_paged_dispatch_counters_seen_from_another_stream_follow_the_rows(case):
    """Whoever looks while a small dispatch runs: copies of rows_done, of the tiles' counters and of a piece of every row, in this
    order, on a second stream beside the dispatch (they wait for nothing).  Where the counters say so, the rows are there."""
    T, E, K = case
    H = 8192
    w = inputs.Workload("watched", T=T, H=H, E=E, R=1, K=K, F=0, dtype=BF16, identity_experts=True)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED)
    g = torch.Generator(device="cuda").manual_seed(T)
    x = torch.empty((T, H), dtype=torch.bfloat16, device="cuda").uniform_(1.0, 2.0, generator=g)
    ids = torch.rand((T, E), device="cuda", generator=g).argsort(1)[:, :K].to(torch.int32).contiguous()
    ints = lambda *n: torch.zeros(n, dtype=torch.int32, device="cuda")
    recv = torch.zeros((plan.P * 128, H), dtype=torch.bfloat16, device="cuda")
    count, te, src, slot, counters = ints(E), ints(plan.P), ints(plan.P * 128), ints(T, K), ints(plan.P + 1)
    looks = 40
    seen, rows = ints(looks, plan.P + 1), torch.zeros((looks, plan.P * 128, 8), dtype=torch.bfloat16, device="cuda")
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        for i in range(looks):
            seen[i, -1:].copy_(counters[-1:])
            seen[i, :-1].copy_(counters[:-1])
            rows[i].copy_(recv[:, -8:])
    early = late = 0
    for _ in range(20):
        recv.zero_()
        counters.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            graph.replay()
        plan.moe_dispatch(x, ids, recv, count, te, src, slot, counters[:plan.P], counters[plan.P:])
        torch.cuda.synchronize()
        assert plan.moe_last_status() == (0, 0) and counters[-1].item() == T * K
        flat, want = slot.flatten().long(), x[:, -8:].repeat_interleave(K, 0)
        there = (rows[:, flat] == want).all(2)                                   # [looks, T*K]
        tile_said = seen[:, :-1].gather(1, (flat // 128).expand(looks, -1)) >= 128
        said = tile_said | (seen[:, -1:] >= T * K)
        assert (there | ~said).all()
        assert ((seen[:, :-1] == counters[:-1]).all(1) | (seen[:, -1] < T * K)).all()
        early, late = early + (~said).any().item(), late + said.any().item()
    assert early and late


def test_paged_dispatch_replayed_from_a_graph():
    """The small dispatch's ticket is back at zero after every call: a captured call gives the same tables and counters each time."""
    w = inputs.Workload("graph_dispatch", T=300, H=264, E=12, R=1, K=4, F=0, dtype=BF16, identity_experts=True)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.empty((w.T, w.H), dtype=torch.bfloat16, device="cuda").normal_(generator=g)
    ids = torch.rand((w.T, w.E), device="cuda", generator=g).argsort(1)[:, :w.K].to(torch.int32).contiguous()
    b = _dispatch_with_counters(w, plan, x, ids)
    names = ("recv", "cnt", "te", "src", "slot", "tile_count", "rows_done")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan.moe_dispatch(x, ids, *(b[n] for n in names))
    for _ in range(3):
        for n in names:
            b[n].fill_(77)
        graph.replay()
        torch.cuda.synchronize()
        assert plan.moe_last_status() == (0, 0) and b["rows_done"].item() == w.T * w.K
        flat = b["slot"].flatten().long()
        assert torch.equal(b["tile_count"].long(), torch.bincount(flat // 128, minlength=plan.P))
        assert torch.equal(b["recv"][flat], x.repeat_interleave(w.K, 0)) and torch.equal(b["te"][flat // 128], ids.flatten())


@pytest.mark.parametrize("mode", MODES)
def test_dispatch_availability_counters_and_gated_consumer(mode):
    """Section IV-D in software: after dispatch every tile's status counter equals the rows stored in it
    and the global counter equals T*K; the tensor-core consumer gated on those counters gives the same
    result as the ungated one."""
    w = SMALL[3]
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    plan = Hh.make_plan(w, mode)
    dx = Hh.to_dev(x)
    b = _dispatch_with_counters(w, plan, dx, Hh.to_dev(ref["topk_idx"]))
    torch.cuda.synchronize()
    assert int(b["rows_done"][0]) == w.T * w.K
    per_tile = torch.bincount(b["slot"].flatten().long() // 128, minlength=plan.P).int()
    assert torch.equal(b["tile_count"], per_tile)
    out = torch.zeros_like(b["recv"])
    plan.moe_expert_ffn(b["recv"], b["te"], Hh.to_dev(wg), Hh.to_dev(wu), Hh.to_dev(wd), out, b["tile_count"], b["rows_done"])
    y = torch.empty((w.T, w.H), dtype=Hh.el_dtype(w), device="cuda")
    plan.moe_combine(out, b["slot"], Hh.to_dev(ref["topk_w"]), y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    Hh.assert_output_close(Hh.to_host_f64(y), ref["y"], w.dtype)


@pytest.mark.parametrize("mode", MODES)
def test_availability_trace_orders_the_events(mode):
    """With the trace on, every tile that holds 128 rows has a ready time between the dispatch start and
    the all-ready time, tiles with fewer rows have none, and the layer's result is unchanged."""
    w = inputs.Workload("trace", T=900, H=264, E=12, R=3, K=3, F=136, dtype=BF16, zipf_s=1.0, seed=9)
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    args = [Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)]
    plan = Hh.make_plan(w, mode)
    y0 = torch.empty((w.T, w.H), dtype=Hh.el_dtype(w), device="cuda")
    plan.moe_layer(*args, y0)
    plan.moe_availability_trace(True)
    y1 = torch.empty_like(y0)
    plan.moe_layer(*args, y1)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    tr = plan.layer_tensor(8).cpu().numpy()
    cnt = plan.layer_tensor(3).cpu().numpy()
    te = plan.layer_tensor(4).cpu().numpy()
    slot = plan.layer_tensor(6).cpu().numpy()
    per_tile = np.bincount(slot.ravel() // 128, minlength=plan.P)
    t0, t_all, ready = tr[0], tr[1], tr[2:]
    assert t0 > 0 and t_all >= t0
    full = per_tile == 128
    assert full.any() and (~full & (te >= 0)).any()
    assert (ready[full] >= t0).all() and (ready[full] <= t_all).all()
    assert (ready[~full] == 0).all()
    assert cnt.sum() == w.T * w.K
    assert torch.equal(y0, y1)
    plan.moe_availability_trace(False)


@pytest.mark.parametrize("kernel", [0, 2])
@pytest.mark.parametrize("split", [1, 2])
def test_expert_kernel_can_be_called_again_without_a_dispatch_in_between(split, kernel):
    """The expert kernel hands its items out through device counters and gates GEMM2 on per-tile GEMM1
    counters; it puts all of them back to zero itself.  Three calls in a row on one dispatch result (the
    counter-gated form, where no dispatch resets anything in between), each with DIFFERENT expert weights:
    a GEMM2 item that trusted the previous call's counters would read the previous call's intermediate,
    so every call is checked against the oracle for its own weights."""
    w = inputs.Workload("many_items", T=700, H=520, E=12, R=3, K=3, F=1032, dtype=BF16, seed=5)  # 288 items for 148 CTAs
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED, ffn_split=split, ffn_kernel=kernel)
    dx = Hh.to_dev(x)
    b = _dispatch_with_counters(w, plan, dx, Hh.to_dev(ref["topk_idx"]))
    outs = []
    for call in range(3):
        cwg, cwu, cwd = inputs.make_all_expert_weights(w.with_(seed=5 + 17 * call))
        out = torch.zeros_like(b["recv"])
        plan.moe_expert_ffn(b["recv"], b["te"], Hh.to_dev(cwg), Hh.to_dev(cwu), Hh.to_dev(cwd), out, b["tile_count"],
                            b["rows_done"])
        outs.append((out, cwg, cwu, cwd))
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    for out, cwg, cwu, cwd in outs:
        y = torch.empty((w.T, w.H), dtype=Hh.el_dtype(w), device="cuda")
        plan.moe_combine(out, b["slot"], Hh.to_dev(ref["topk_w"]), y)
        torch.cuda.synchronize()
        want = Hh.oracle_layer_for(w, x, wr, bias, cwg, cwu, cwd)
        Hh.assert_output_close(Hh.to_host_f64(y), want["y"], w.dtype)


@pytest.mark.parametrize("push", [0, 1])
@pytest.mark.parametrize("rows", [(5, 40, 64), (129, 190, 7), (128, 200, 256)], ids=lambda r: "_".join(map(str, r)))
def test_tensor_core_epilogue_lanes_that_do_not_store(rows, push):
    """The one-CTA kernel's three epilogues (narrow form, M = 64 form, whole tiles) where some lanes of a warp store and
    others do not: columns that end inside a warp's 32, rows without a source (push), the M = 64 form's unused lanes.  Every
    row against the same call without row counts (whole tiles only)."""
    E, H, F = len(rows), 328, 200
    w = inputs.Workload("epi_lanes", T=sum(rows), H=H, E=E, R=1, K=1, F=F, dtype=BF16, seed=36)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED)
    g = torch.Generator(device="cuda").manual_seed(36)
    W = [torch.empty(s, dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.05, generator=g) for s in ((E, F, H), (E, F, H), (E, H, F))]
    x = torch.empty((w.T, H), dtype=torch.bfloat16, device="cuda").normal_(generator=g)
    idx = torch.repeat_interleave(torch.arange(E, dtype=torch.int32), torch.tensor(rows)).reshape(-1, 1).cuda()
    b = _dispatch_with_counters(w, plan, x, idx)
    whole = torch.zeros_like(b["recv"])
    plan.moe_expert_ffn(b["recv"], b["te"], *W, whole)
    want = whole[b["slot"].flatten().long()]
    if push:
        got = torch.full((w.T, H), 7.0, dtype=torch.bfloat16, device="cuda")
        plan.moe_expert_ffn_push(b["recv"], b["te"], b["src"], *W, got, b["tile_count"], b["rows_done"])
    else:
        out = torch.full_like(whole, 7.0)
        plan.moe_expert_ffn(b["recv"], b["te"], *W, out, b["tile_count"], b["rows_done"])
        got = out[b["slot"].flatten().long()]
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0) and torch.equal(got, want)


@pytest.mark.parametrize("mode", MODES)
def test_expert_id_outside_the_range_is_reported_and_dropped(mode):
    """A caller-supplied topk_idx with an id that is no expert: the status word says bad argument and names
    the token, the assignment gets slot -1 and no row, every other assignment is dispatched as usual, and
    nothing outside the buffers is written (guard rows stay intact)."""
    w = inputs.Workload("bad_id", T=200, H=64, E=8, R=2, K=2, F=8, dtype=BF16)
    x = inputs.make_x(w)
    rng = np.random.default_rng(4)
    idx = np.stack([rng.permutation(w.E)[:w.K] for _ in range(w.T)]).astype(np.int32)
    idx[77, 1] = w.E + 5
    plan = Hh.make_plan(w, mode)
    rows = plan.P * 128
    guard = torch.full((rows + 128, w.H), 7.0, dtype=torch.bfloat16, device="cuda")
    cnt = torch.empty(w.E, dtype=torch.int32, device="cuda")
    te = torch.empty(plan.P, dtype=torch.int32, device="cuda")
    src = torch.empty(rows, dtype=torch.int32, device="cuda")
    slot = torch.empty((w.T, w.K), dtype=torch.int32, device="cuda")
    plan.moe_dispatch(Hh.to_dev(x), Hh.to_dev(idx), guard[:rows], cnt, te, src, slot)
    assert plan.moe_last_status() == (-1, 77)
    s = slot.cpu().numpy()
    assert s[77, 1] == -1 and (s.ravel() >= 0).sum() == w.T * w.K - 1
    good = idx.ravel() < w.E
    assert np.array_equal(cnt.cpu().numpy(), np.bincount(idx.ravel()[good], minlength=w.E))
    recv_h = Hh.to_host_bits(guard[:rows])
    flat = s.ravel()
    assert recv_h[flat[good]].tobytes() == np.repeat(x, w.K, axis=0)[good].tobytes()
    assert torch.all(guard[rows:] == 7.0)


@pytest.mark.parametrize("kernel", [0, 2])
def test_consumer_wait_runs_out_and_reports_it(kernel):
    """A flag that nothing sets: the consumer is given availability counters that stay at zero.  Its
    bounded wait (50 ms here) runs out, the kernel returns on its own, the status word says timeout
    and names the wait, and the same plan then runs a correct layer: nothing hangs, the context lives."""
    w = SMALL[3]
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED, ffn_kernel=kernel, wait_limit_ns=50_000_000)
    dx, dwg, dwu, dwd = Hh.to_dev(x), Hh.to_dev(wg), Hh.to_dev(wu), Hh.to_dev(wd)
    b = _dispatch_with_counters(w, plan, dx, Hh.to_dev(ref["topk_idx"]))
    never = torch.zeros(plan.P + 1, dtype=torch.int32, device="cuda")
    out = torch.zeros_like(b["recv"])
    t0 = torch.cuda.Event(enable_timing=True)
    t1 = torch.cuda.Event(enable_timing=True)
    t0.record()
    plan.moe_expert_ffn(b["recv"], b["te"], dwg, dwu, dwd, out, never[:plan.P], never[plan.P:])
    t1.record()
    code, detail = plan.moe_last_status()
    # MOE_ERR_TIMEOUT; the wait site is the producer's tile-availability wait (7) or, since every role's wait
    # has the same bound, the MMA (4) or epilogue (5) wait that starved behind it: the first to expire is kept
    assert code == -6 and detail in (7, 4, 5, 8), (code, detail)
    assert t0.elapsed_time(t1) < 2000.0
    y = torch.empty((w.T, w.H), dtype=Hh.el_dtype(w), device="cuda")
    plan.moe_layer(dx, Hh.to_dev(wr), Hh.to_dev(bias), dwg, dwu, dwd, y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    Hh.assert_output_close(Hh.to_host_f64(y), ref["y"], w.dtype)


@pytest.mark.parametrize("split", [1, 2])
@pytest.mark.parametrize("kernel", [0, 2])
def test_consumer_wait_runs_out_with_other_tiles_in_flight(kernel, split):
    """Some tiles are ready and computed while others never become so: the wait (20 ms) runs out with loads and MMAs of the
    ready tiles in flight.  The kernel lands them, reports the timeout and returns; the layer then gives its bytes again."""
    w = inputs.Workload("wait_busy", T=1000, H=1544, E=4, R=1, K=2, F=1040, dtype=BF16, zipf_s=0.7, seed=25)
    args = [Hh.to_dev(a) for a in Hh.oracle_inputs(w)]
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED, ffn_kernel=kernel, ffn_split=split, wait_limit_ns=20_000_000)
    y, y2 = (torch.empty((w.T, w.H), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    plan.moe_layer(*args, y)
    b = _dispatch_with_counters(w, plan, args[0], plan.layer_tensor(0))
    owned = (b["te"] >= 0).nonzero().flatten()
    for ready in (1, int(owned.numel()) // 2, int(owned.numel()) - 1):
        counts = torch.zeros_like(b["tile_count"])
        counts[owned[:ready]] = 128
        plan.moe_expert_ffn(b["recv"], b["te"], *args[3:], torch.zeros_like(b["recv"]), counts, torch.zeros_like(b["rows_done"]))
        assert plan.moe_last_status()[0] == -6       # MOE_ERR_TIMEOUT
        plan.moe_layer(*args, y2)
        assert plan.moe_last_status() == (0, 0) and torch.equal(y, y2)


@pytest.mark.parametrize("split", [1, 2])
@pytest.mark.parametrize("kernel", [0, 2])
def test_expert_kernel_with_a_tiny_wait_limit_reports_or_computes(kernel, split):
    """Limits shorter than a load, an MMA or an item take: any role may give up first, with what the others have issued still
    in flight.  Every call either reports the timeout or has computed its bytes, and the next plan's layer is untouched."""
    w = inputs.Workload("wait_tiny", T=1000, H=1544, E=4, R=1, K=2, F=1016, dtype=BF16, zipf_s=0.7, seed=26)   # (F below 1024: 0 is one CTA per tile)
    args = [Hh.to_dev(a) for a in Hh.oracle_inputs(w)]
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED, ffn_kernel=kernel, ffn_split=split)
    y, y2 = (torch.empty((w.T, w.H), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    plan.moe_layer(*args, y)
    b = _dispatch_with_counters(w, plan, args[0], plan.layer_tensor(0))
    want = torch.zeros_like(b["recv"])
    plan.moe_expert_ffn(b["recv"], b["te"], *args[3:], want, b["tile_count"], b["rows_done"])
    used = b["slot"].flatten().long()
    for limit in (1, 500, 2_000, 5_000, 20_000, 100_000):
        tiny = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED, ffn_kernel=kernel, ffn_split=split, wait_limit_ns=limit)
        out = torch.zeros_like(want)
        tiny.moe_expert_ffn(b["recv"], b["te"], *args[3:], out, b["tile_count"], b["rows_done"])
        code = tiny.moe_last_status()[0]
        assert code in (0, -6) and (code != 0 or torch.equal(out[used], want[used]))
        plan.moe_layer(*args, y2)
        assert plan.moe_last_status() == (0, 0) and torch.equal(y, y2)


def test_fp32_expert_kernel_with_a_tiny_wait_limit_reports_or_computes():
    """The same for dtype fp32 on the tensor cores: the limit bounds its waits (with 1 ns GEMM2's wait for the intermediate of
    another CTA runs out).  Every call either reports the timeout or has computed its bytes."""
    w = inputs.Workload("wait_fp32", T=1000, H=516, E=4, R=1, K=2, F=1028, dtype=FP32, zipf_s=0.7, seed=27)
    args = [Hh.to_dev(a) for a in Hh.oracle_inputs(w)]
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED)
    y, y2 = (torch.empty((w.T, w.H), dtype=torch.float32, device="cuda") for _ in range(2))
    plan.moe_layer(*args, y)
    b = _dispatch_with_counters(w, plan, args[0], plan.layer_tensor(0))
    want = torch.zeros_like(b["recv"])
    plan.moe_expert_ffn(b["recv"], b["te"], *args[3:], want, b["tile_count"], b["rows_done"])
    used = b["slot"].flatten().long()
    codes = []
    for limit in (1, 500, 2_000, 5_000, 20_000, 100_000):
        tiny = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED, wait_limit_ns=limit)
        out = torch.zeros_like(want)
        tiny.moe_expert_ffn(b["recv"], b["te"], *args[3:], out, b["tile_count"], b["rows_done"])
        codes.append(tiny.moe_last_status()[0])
        assert codes[-1] in (0, -6) and (codes[-1] != 0 or torch.equal(out[used], want[used]))
        plan.moe_layer(*args, y2)
        assert plan.moe_last_status() == (0, 0) and torch.equal(y, y2)
    assert codes[0] == -6


# ------------------------------------------------------------------ dispatch and experts in one launch
OVERLAP_CASES = [SMALL[3], SMALL[4], SMALL[5], SMALL[7],
                 inputs.Workload("three_tiles", T=700, H=320, E=4, R=2, K=2, F=392, dtype=BF16),
                 inputs.Workload("many_items", T=2100, H=520, E=12, R=3, K=3, F=1032, dtype=BF16, seed=5, zipf_s=1.0),
                 inputs.Workload("long_rows", T=260, H=9216, E=8, R=2, K=2, F=128, dtype=BF16),
                 inputs.Workload("max_k_overlapped", T=70, H=128, E=64, R=4, K=32, F=64, dtype=BF16)]   # rows of 18 KB: two chunks per row


@pytest.mark.parametrize("split", [1, 2])
@pytest.mark.parametrize("w", OVERLAP_CASES, ids=lambda w: w.name)
def test_overlapped_dispatch_and_experts_match_oracle(w, split):
    """Section IV-D end to end: the launch that computes the experts also dispatches (its first CTAs walk the
    tokens in ascending order and raise the tiles' status counters, the others start on a tile when its counter
    reaches the rows the tile will hold).  Routing, dispatch contents and output against the oracle; both as one
    launch for the two GEMMs and as two."""
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_ORDERED, overlap=1, ffn_split=split)
    y = torch.empty((w.T, w.H), dtype=Hh.el_dtype(w), device="cuda")
    args = [Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)]
    for _ in range(2):      # twice: the second call meets the counters as the first one left them
        # a row that a consumer read before its producer had stored it would show: the pool holds 1e30 everywhere
        plan.layer_tensor(2).fill_(1.0e30)
        plan.moe_layer(*args, y)
        torch.cuda.synchronize()
        assert plan.moe_last_status() == (0, 0)
        router = 2 if (w.dtype == BF16 and w.E > 64) else 1                     # many experts: chains + select, or filter + refine
        assert plan.moe_last_launch_count() == router + 1 + (2 if split == 1 else 1)   # router, expert launch(es) carrying the dispatch, combine
        Hh.check_route(plan.layer_tensor(0), plan.layer_tensor(1), ref["topk_idx"], ref["topk_w"])
        Hh.check_dispatch(w, plan.P, x, ref["topk_idx"], ref, plan.layer_tensor(2), plan.layer_tensor(3),
                          plan.layer_tensor(4), plan.layer_tensor(5), plan.layer_tensor(6))
        Hh.assert_output_close(Hh.to_host_f64(y), ref["y"], w.dtype)
    # the same bytes as the stream-ordered launches give
    plan2 = Hh.make_plan(w, B.DISPATCH_ATOMIC_ORDERED, ffn_split=split)
    y2 = torch.empty_like(y)
    plan2.moe_layer(*args, y2)
    torch.cuda.synchronize()
    assert torch.equal(y, y2)


def test_overlapped_consumer_wait_runs_out_and_reports_it():
    """The consumer's wait for a tile's status counter, in the overlapped launch, with a limit far below the time
    the producers need (1 microsecond): waits run out, the kernel returns by itself with MOE_ERR_TIMEOUT and a
    wait site, nothing hangs, and a plan with the normal limit then computes the right layer."""
    w = inputs.Workload("overlap_timeout", T=4096, H=2048, E=8, R=2, K=2, F=256, dtype=BF16)
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    args = [Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)]
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_ORDERED, overlap=1, wait_limit_ns=1000)
    y = torch.empty((w.T, w.H), dtype=torch.bfloat16, device="cuda")
    # The dispatch gives up half-way too (its own waits have the same limit) and leaves entries of slot_of and of
    # the source information unwritten: whatever they hold must not be used as a row number by the later stages.
    plan.layer_tensor(6).fill_(2 ** 31 - 1)
    plan.layer_tensor(5).fill_(2 ** 31 - 1)
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record()
    plan.moe_layer(*args, y)
    t1.record()
    code, detail = plan.moe_last_status()
    assert code == -6 and detail in (3, 4, 5, 7, 8), (code, detail)
    assert t0.elapsed_time(t1) < 2000.0
    good = Hh.make_plan(w, B.DISPATCH_ATOMIC_ORDERED, overlap=1)
    good.moe_layer(*args, y)
    torch.cuda.synchronize()
    assert good.moe_last_status() == (0, 0)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    Hh.assert_output_close(Hh.to_host_f64(y), ref["y"], w.dtype)


def test_overlapped_launch_starts_expert_work_before_the_dispatch_ends():
    """The timeline of one traced overlapped layer: full tiles appear throughout the dispatch (ascending token
    order: the first one early), and the first GEMM1 item begins to load before the last row has been stored."""
    w = inputs.Workload("overlap_trace", T=8192, H=2048, E=8, R=2, K=2, F=512, dtype=BF16)
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    args = [Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)]
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_ORDERED, overlap=1)
    y = torch.empty((w.T, w.H), dtype=torch.bfloat16, device="cuda")
    plan.moe_layer(*args, y)
    plan.moe_availability_trace(True)
    plan.layer_tensor(9).zero_()
    plan.moe_layer(*args, y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    tr = plan.layer_tensor(8).cpu().numpy()
    items = plan.layer_tensor(9).cpu().numpy()
    t0, t_all, ready = tr[0], tr[1], tr[2:]
    full = ready[ready > 0]
    assert full.size > 0 and t_all > t0
    first_tile = (full.min() - t0) / (t_all - t0)
    started = items[items[:, 0] > 0]
    gemm1 = started[(started[:, 2] & 1) == 0]
    assert gemm1[:, 0].min() < t_all, "no expert item began before the dispatch was over"
    assert first_tile < 0.5, f"first full tile only after {first_tile:.2f} of the dispatch"
    plan.moe_availability_trace(False)


# ------------------------------------------------------------------ push-style combine
PUSH_CASES = [SMALL[3], SMALL[4], SMALL[5], SMALL[7], SMALL[8],
              inputs.Workload("three_tiles", T=700, H=320, E=4, R=2, K=2, F=392, dtype=BF16),
              inputs.Workload("half_tiles", T=900, H=264, E=6, R=3, K=2, F=136, dtype=BF16, zipf_s=1.0, seed=2)]


@pytest.mark.parametrize("w", PUSH_CASES, ids=lambda w: w.name)
def test_push_combine_stages_match_oracle_and_the_gather_path(w):
    """Section IV-B, all-to-all combine: the expert kernel reads the source information of every row after its
    final GEMM and stores the result at the token's position t*K+k; the reduction then reads K consecutive rows.
    Through the C ABI (moe_expert_ffn_push, moe_combine_staged): every staged row is the expert output of its
    assignment, y matches the oracle, and y is the same bytes as the gather path's."""
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    g = run_stages(w, B.DISPATCH_ATOMIC_PAGED, x, wr, bias, wg, wu, wd)          # the gather path, for comparison
    plan = g["plan"]
    staged = torch.full((w.T * w.K, w.H), 7.0, dtype=torch.bfloat16, device="cuda")
    plan.moe_expert_ffn_push(g["recv"], g["te"], g["src"], Hh.to_dev(wg), Hh.to_dev(wu), Hh.to_dev(wd), staged)
    y = torch.empty((w.T, w.H), dtype=torch.bfloat16, device="cuda")
    plan.moe_combine_staged(staged, g["slot"], g["tw"], y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    slot = g["slot"].flatten().long()
    assert torch.equal(staged, g["out_rows"][slot]), "a staged row is not the expert output of its assignment"
    assert torch.equal(y, g["y"])
    Hh.assert_output_close(Hh.to_host_f64(y), ref["y"], w.dtype)


@pytest.mark.parametrize("overlap", [0, 1])
@pytest.mark.parametrize("mode", [B.DISPATCH_SCAN, B.DISPATCH_ATOMIC_PAGED, B.DISPATCH_ATOMIC_ORDERED])
@pytest.mark.parametrize("w", [SMALL[3], SMALL[4], SMALL[5]], ids=lambda w: w.name)
def test_layer_with_push_combine(w, mode, overlap):
    if overlap and mode != B.DISPATCH_ATOMIC_ORDERED:
        pytest.skip("the overlapped launch belongs to the ordered dispatch")
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    args = [Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)]
    plan = Hh.make_plan(w, mode, combine_mode=1, overlap=overlap)
    y = torch.empty((w.T, w.H), dtype=torch.bfloat16, device="cuda")
    plan.moe_layer(*args, y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    Hh.assert_output_close(Hh.to_host_f64(y), ref["y"], w.dtype)
    gather = Hh.make_plan(w, mode)
    y2 = torch.empty_like(y)
    gather.moe_layer(*args, y2)
    torch.cuda.synchronize()
    assert torch.equal(y, y2)


def test_push_combine_is_refused_where_it_is_not_built():
    with pytest.raises(B.MoeError) as ei:
        B.moe_workspace_bytes(B.make_config(64, 128, 8, 2, 2, 64, FP32, combine_mode=1))
    assert ei.value.code == -3


# ------------------------------------------------------------------ expert + tensor parallelism
TP_CASES = [(inputs.Workload("tp_bf16", T=333, H=264, E=12, R=3, K=3, F=400, dtype=BF16), 2),
            (inputs.Workload("tp_bf16_4", T=700, H=320, E=4, R=2, K=2, F=1024, dtype=BF16, zipf_s=1.0), 4),
            (inputs.Workload("tp_many", T=300, H=256, E=64, R=8, K=8, F=256, dtype=BF16, zipf_s=1.0), 4),
            (inputs.Workload("tp_filtered_router", T=260, H=512, E=128, R=8, K=4, F=256, dtype=BF16, zipf_s=1.0), 2),  # 128 experts, few tokens: every chain
            (inputs.Workload("tp_filter", T=1100, H=512, E=96, R=8, K=4, F=128, dtype=BF16, zipf_s=1.0), 2),  # the router's filter path
            (inputs.Workload("tp_fp32", T=130, H=128, E=8, R=2, K=2, F=192, dtype=FP32), 3)]


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("case", TP_CASES, ids=lambda c: f"{c[0].name}_S{c[1]}")
def test_tp_shards_layer_matches_oracle(case, mode):
    """Section VII: one receive region per TP shard, every row stored to each.  Routing (every pick listed once per
    shard), dispatch contents of the E*S regions and the output against the oracle's TP layer - which itself equals
    the plain layer - in every dispatch scheme; the output also agrees with the same plan without shards."""
    w, S = case
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd, tp_shards=S)
    args = [Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)]
    plan = Hh.make_plan(w, mode, tp_shards=S)
    assert plan.P == (w.T * w.K * S // 128 + w.E * S if mode != B.DISPATCH_ATOMIC_STATIC else plan.P)
    y = torch.empty((w.T, w.H), dtype=Hh.el_dtype(w), device="cuda")
    plan.moe_layer(*args, y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    Hh.check_route(plan.layer_tensor(0), plan.layer_tensor(1), ref["topk_idx"], ref["topk_w"])
    ws = w.with_(E=w.E * S, K=w.K * S)
    Hh.check_dispatch(ws, plan.P, x, ref["topk_idx"], ref, plan.layer_tensor(2), plan.layer_tensor(3),
                      plan.layer_tensor(4), plan.layer_tensor(5), plan.layer_tensor(6))
    Hh.assert_output_close(Hh.to_host_f64(y), ref["y"], w.dtype)
    plain = Hh.make_plan(w, mode)
    y2 = torch.empty_like(y)
    plain.moe_layer(*args, y2)
    torch.cuda.synchronize()
    Hh.assert_output_close(Hh.to_host_f64(y), Hh.to_host_f64(y2), w.dtype, "with and without TP shards")


def test_tp_shards_with_overlap_and_push_combine():
    w, S = TP_CASES[1]
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd, tp_shards=S)
    args = [Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)]
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_ORDERED, tp_shards=S, overlap=1, combine_mode=1)
    y = torch.empty((w.T, w.H), dtype=torch.bfloat16, device="cuda")
    plan.moe_layer(*args, y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    Hh.assert_output_close(Hh.to_host_f64(y), ref["y"], w.dtype)


def test_tp_shards_limits_are_refused_on_the_host():
    for cfg, code in [(B.make_config(64, 128, 8, 2, 2, 100, BF16, tp_shards=3), -1),     # F % S != 0
                      (B.make_config(64, 128, 128, 2, 2, 64, BF16, tp_shards=4), -3),    # E*S > 256
                      (B.make_config(64, 128, 64, 2, 16, 64, BF16, tp_shards=4), -3)]:   # K*S > 32
        with pytest.raises(B.MoeError) as ei:
            B.moe_workspace_bytes(cfg)
        assert ei.value.code == code


# ------------------------------------------------------------------ random small shapes
def _random_workloads(n, seed):
    rng = np.random.default_rng(seed)
    out = []
    for i in range(n):
        dtype = BF16 if rng.random() < 0.7 else FP32
        q = 8 if dtype == BF16 else 4                       # row pitch must be a multiple of 16 bytes
        E = int(rng.choice([1, 2, 3, 5, 8, 12, 24, 40, 64, 100, 256]))
        R = int(rng.choice([r for r in (1, 2, 3, 4, 5, 8) if E % r == 0]))
        K = int(rng.integers(1, min(E, 8) + 1))
        out.append(inputs.Workload(f"rand{i}", T=int(rng.integers(1, 400)), H=q * int(rng.integers(2, 40)), E=E, R=R,
                                   K=K, F=q * int(rng.integers(2, 40)), dtype=dtype,
                                   zipf_s=float(rng.choice([0.0, 1.0])), seed=int(rng.integers(0, 1000))))
    return out


@pytest.mark.parametrize("w", _random_workloads(24, 2024), ids=lambda w: f"{w.name}_T{w.T}_H{w.H}_E{w.E}_K{w.K}_F{w.F}_d{w.dtype}")
def test_random_small_layers_match_oracle(w):
    """Seeded random small shapes (ragged T, K = 1 ... 8, E from 1 to 256, odd H and F multiples, both
    dtypes, biased and unbiased routers), every dispatch scheme, whole layer against the oracle."""
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    ref = Hh.oracle_layer_for(w, x, wr, bias, wg, wu, wd)
    for mode in MODES:
        plan = Hh.make_plan(w, mode)
        y = torch.empty((w.T, w.H), dtype=Hh.el_dtype(w), device="cuda")
        plan.moe_layer(Hh.to_dev(x), Hh.to_dev(wr), Hh.to_dev(bias), Hh.to_dev(wg), Hh.to_dev(wu), Hh.to_dev(wd), y)
        torch.cuda.synchronize()
        assert plan.moe_last_status() == (0, 0)
        Hh.check_route(plan.layer_tensor(0), plan.layer_tensor(1), ref["topk_idx"], ref["topk_w"])
        Hh.check_dispatch(w, plan.P, x, ref["topk_idx"], ref, plan.layer_tensor(2), plan.layer_tensor(3),
                          plan.layer_tensor(4), plan.layer_tensor(5), plan.layer_tensor(6))
        Hh.assert_output_close(Hh.to_host_f64(y), ref["y"], w.dtype)


@pytest.mark.parametrize("w", [w for w in _random_workloads(24, 2024) if w.dtype == BF16][:10],
                         ids=lambda w: f"{w.name}_T{w.T}_H{w.H}_E{w.E}_K{w.K}_F{w.F}")
def test_random_small_layers_variants_agree_bit_for_bit(w):
    """The variants of the bf16 layer do the same arithmetic in the same order per output element - ordered
    dispatch with the dispatch inside the expert launch, push-style combine, both together - so on the same
    seeded random shapes their y must equal the plain ordered layer's y bit for bit (which the test above holds
    against the oracle)."""
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    args = [Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)]
    ys = []
    for kw in ({}, {"overlap": 1}, {"combine_mode": 1}, {"overlap": 1, "combine_mode": 1}):
        plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_ORDERED, **kw)
        y = torch.full((w.T, w.H), 7.0, dtype=torch.bfloat16, device="cuda")
        for _ in range(2):
            plan.moe_layer(*args, y)
        torch.cuda.synchronize()
        assert plan.moe_last_status() == (0, 0), kw
        ys.append(y)
    for kw, y in zip(("overlap", "push", "overlap + push"), ys[1:]):
        assert torch.equal(y, ys[0]), kw


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("dtype", [BF16, FP32])
def test_empty_batch_is_a_legal_call(mode, dtype):
    """T = 0: every entry point accepts it, launches nothing that could touch a row, reports no error."""
    w = inputs.Workload("empty", T=0, H=128, E=8, R=2, K=2, F=128, dtype=dtype)
    _, wr, bias, wg, wu, wd = Hh.oracle_inputs(w.with_(T=4))
    plan = Hh.make_plan(w, mode)
    el = Hh.el_dtype(w)
    x = torch.empty((0, w.H), dtype=el, device="cuda")
    y = torch.empty((0, w.H), dtype=el, device="cuda")
    idx = torch.empty((0, w.K), dtype=torch.int32, device="cuda")
    tw = torch.empty((0, w.K), dtype=torch.float32, device="cuda")
    dwr, dwg, dwu, dwd = (Hh.to_dev(a) for a in (wr, wg, wu, wd))
    plan.moe_route(x, dwr, None, idx, tw)
    rows = plan.P * 128
    recv = torch.full((rows, w.H), 3.0, dtype=el, device="cuda")
    cnt = torch.full((w.E,), 9, dtype=torch.int32, device="cuda")
    te = torch.full((plan.P,), 9, dtype=torch.int32, device="cuda")
    src = torch.full((rows,), 9, dtype=torch.int32, device="cuda")
    slot = torch.empty((0, w.K), dtype=torch.int32, device="cuda")
    plan.moe_dispatch(x, idx, recv, cnt, te, src, slot)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    assert cnt.eq(0).all() and te.eq(-1).all() and recv.eq(3.0).all()      # nobody owns a tile, no row was written
    out_rows = torch.full((rows, w.H), 5.0, dtype=el, device="cuda")
    plan.moe_expert_ffn(recv, te, dwg, dwu, dwd, out_rows)
    plan.moe_combine(out_rows, slot, tw, y)
    plan.moe_layer(x, dwr, None, dwg, dwu, dwd, y)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0)
    assert out_rows.eq(5.0).all()                                          # no tile, no expert work


@pytest.mark.parametrize("dtype", [BF16, FP32])
def test_combine_treats_a_slot_beyond_the_pool_as_absent(dtype):
    """slot_of entries at or beyond the pool's rows (what an abandoned dispatch can leave behind) add nothing
    and are never used as an address: y is the weighted sum over the valid slots only."""
    w = inputs.Workload("bad_slots", T=64, H=256, E=8, R=2, K=4, F=128, dtype=dtype)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED)
    rows = plan.P * 128
    g = torch.Generator(device="cuda").manual_seed(5)
    pool = torch.randn((rows, w.H), device="cuda", generator=g).to(Hh.el_dtype(w))
    slot = torch.randint(0, rows, (w.T, w.K), device="cuda", generator=g, dtype=torch.int32)
    slot[::3, 1] = rows               # first row past the pool
    slot[1::3, 2] = 2 ** 31 - 1       # as far out as an int goes
    slot[2::3, 0] = -1                # a dropped assignment
    tw = torch.rand((w.T, w.K), device="cuda", generator=g)
    y = torch.empty((w.T, w.H), dtype=Hh.el_dtype(w), device="cuda")
    plan.moe_combine(pool, slot, tw, y)
    torch.cuda.synchronize()
    valid = (slot >= 0) & (slot < rows)
    want = (pool.double()[slot.clamp(0, rows - 1).long()] * (tw.double() * valid).unsqueeze(-1)).sum(1)
    tol = 2.0 ** -7 if dtype == BF16 else 1e-5
    assert torch.allclose(y.double(), want, rtol=tol, atol=tol)


def test_pipelined_host_steps_match_single_steps():
    """moe_layer_host_submit / _wait with two steps in flight: five batches, each result identical to
    the same batch run alone through moe_layer (bit for bit: same kernels, same order)."""
    w = SMALL[3]
    _, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    dwr, dbias, dwg, dwu, dwd = (Hh.to_dev(a) for a in (wr, bias, wg, wu, wd))
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED)
    xs = [inputs.make_x(w.with_(seed=10 + i)) for i in range(5)]
    hx = [torch.from_numpy(x.view(np.int16)).pin_memory() for x in xs]
    hy = [torch.empty_like(h).pin_memory() for h in hx]
    tickets = []
    for i in range(5):
        tickets.append(plan.moe_layer_host_submit(hx[i], dwr, dbias, dwg, dwu, dwd, hy[i]))
        if i >= 1:
            plan.moe_layer_host_wait(tickets[i - 1])
    plan.moe_layer_host_wait(tickets[-1])
    assert tickets == list(range(5)) and plan.moe_last_status() == (0, 0)
    for i in range(5):
        y = torch.empty((w.T, w.H), dtype=torch.bfloat16, device="cuda")
        plan.moe_layer(Hh.to_dev(xs[i]), dwr, dbias, dwg, dwu, dwd, y)
        torch.cuda.synchronize()
        assert np.array_equal(hy[i].numpy().view(np.uint16), Hh.to_host_bits(y)), f"step {i}"


def test_layer_output_is_bit_identical_across_runs_and_dispatch_schemes():
    """Arrival order changes where a row sits, not what is computed for it: a row's GEMM result does not
    depend on its position in a tile and combine sums in ascending k, so y is the same bytes in every
    dispatch scheme and in every run, although the atomic schemes place rows in a different order each time."""
    w = SMALL[5]   # 256 experts, top-8, skewed
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    dev = [Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)]
    outs, orders = [], []
    for mode in MODES:
        plan = Hh.make_plan(w, mode)
        for _ in range(3):
            y = torch.empty((w.T, w.H), dtype=torch.bfloat16, device="cuda")
            plan.moe_layer(*dev, y)
            torch.cuda.synchronize()
            outs.append(Hh.to_host_bits(y).tobytes())
            orders.append(plan.layer_tensor(6).cpu().numpy().tobytes())
    assert len(set(outs)) == 1
    assert len(set(orders)) > 1     # the placements did differ (scan vs atomic at the least)


def test_overlapped_launch_many_runs_same_bytes():
    """Forty runs of the overlapped launch on a layer with hot and cold experts (several tiles per hot expert, the
    narrow form for the cold ones, two expert launches): every run must give the bytes of the stream-ordered layer,
    with the receive pool refilled with 1e30 before each run - a consumer that started a tile too early, or a
    counter left over from the run before, would change them."""
    w = inputs.Workload("overlap_soak", T=3000, H=1024, E=48, R=4, K=4, F=512, dtype=BF16, zipf_s=1.0, seed=9)
    x, wr, bias, wg, wu, wd = Hh.oracle_inputs(w)
    dev = [Hh.to_dev(a) for a in (x, wr, bias, wg, wu, wd)]
    base = Hh.make_plan(w, B.DISPATCH_ATOMIC_ORDERED, ffn_split=1)
    y0 = torch.empty((w.T, w.H), dtype=torch.bfloat16, device="cuda")
    base.moe_layer(*dev, y0)
    torch.cuda.synchronize()
    assert base.moe_last_status() == (0, 0)
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_ORDERED, overlap=1, ffn_split=1)
    y = torch.empty_like(y0)
    for i in range(40):
        plan.layer_tensor(2).fill_(1.0e30)
        y.fill_(3.0)
        plan.moe_layer(*dev, y)
        torch.cuda.synchronize()
        assert plan.moe_last_status() == (0, 0), i
        assert torch.equal(y, y0), i


# The router that fetches its candidates' rows one by one: odd token counts (a CTA of one), H that ends inside its 512-column
# steps and inside 64 columns, one and several slices of the approximate logits, one wave of CTAs and two, few and all experts.
DIRECT_SHAPES = [(160, 7168, 256, 8, 0.0), (593, 8184, 256, 8, 1.2), (591, 7176, 193, 3, 0.0), (1183, 5128, 129, 1, 1.0), (577, 8192, 68, 32, 0.0),
                 (301, 4104, 256, 16, 0.0)]


@pytest.mark.parametrize("shape", DIRECT_SHAPES, ids=lambda s: f"T{s[0]}_H{s[1]}_E{s[2]}_K{s[3]}_z{s[4]}")
def test_router_direct_kernel_edges(shape):
    T, H, E, K, zipf = shape
    w = inputs.Workload("direct", T=T, H=H, E=E, R=1, K=K, F=8, dtype=BF16, zipf_s=zipf, seed=31)
    x, (wr, bias) = inputs.make_x(w), inputs.make_router(w)
    ridx, rw, _ = oracle.route(x, wr, bias, K, BF16)
    plan, idx, tw = _route_only(w, x, wr, bias)
    assert plan.moe_last_status() == (0, 0)
    Hh.check_route(idx, tw, ridx, rw)


@pytest.mark.parametrize("tokens", [300, 900])
def test_router_on_a_workspace_without_room_for_the_slices(tokens):
    """One set of logits and the norms: the picks and the weights (the chains' at 300 tokens, the filter's at 900) all the same."""
    w = inputs.Workload("direct_lean", T=tokens, H=4608, E=256, R=1, K=8, F=8, dtype=BF16, seed=33, identity_experts=True)
    x, wr, bias, *_ = Hh.oracle_inputs(w, with_experts=False)
    ridx, rw, _ = oracle.route(x, wr, bias, w.K, BF16)
    plan, idx, tw = _route_only(w, x, wr, bias)
    full, chains = B.moe_workspace_bytes(plan.cfg), B.moe_workspace_bytes(B.make_config(w.T, w.H, w.E, 1, w.K, 0, BF16, identity_experts=1, route_filter=-1,
                                                                                        dispatch_mode=plan.cfg.dispatch_mode))
    lean = chains + (1024 if tokens > 864 else 0)
    assert lean < full and plan.moe_last_launch_count() == 2
    plan.close()
    plan.handle = ctypes.c_void_p()
    plan.workspace.fill_(0xff)
    base = (plan.workspace.data_ptr() + 255) // 256 * 256
    assert B.lib().moe_plan_create(ctypes.byref(plan.cfg), base, lean - 1, ctypes.byref(ctypes.c_void_p())) == -7
    assert B.lib().moe_plan_create(ctypes.byref(plan.cfg), base, lean, ctypes.byref(plan.handle)) == 0
    plan.moe_route(Hh.to_dev(x), Hh.to_dev(wr), Hh.to_dev(bias), idx, tw)
    torch.cuda.synchronize()
    assert plan.moe_last_status() == (0, 0) and plan.moe_last_launch_count() == 2
    Hh.check_route(idx, tw, ridx, rw)
    assert (plan.workspace[base - plan.workspace.data_ptr() + lean:] == 0xff).all()


def test_router_direct_kernel_degenerate_rows():
    """Rows of zeros (every expert a candidate), experts that are equal or an ulp apart, biases of minus infinity and of the
    lowest number, infinities and NaN in x and in Wr: the picks and their weights that every chain gives."""
    w = inputs.Workload("direct_wild", T=300, H=5120, E=256, R=1, K=8, F=8, dtype=BF16, seed=32)
    x, (wr, _) = inputs.make_x(w), inputs.make_router(w)
    x[::7] = 0
    wr[40:80] = wr[40]
    wr[90, 5] ^= 1
    wr[91] = wr[90]
    wr[91, 5] ^= 1
    bias = np.zeros(w.E, np.float32)
    bias[100:200], bias[200:230] = -np.inf, -np.finfo(np.float32).max
    ridx, rw, _ = oracle.route(x, wr, bias, w.K, BF16)
    plan, idx, tw = _route_only(w, x, wr, bias)
    assert plan.moe_last_status() == (0, 0)
    Hh.check_route(idx, tw, ridx, rw)
    inf, nan, big = (int(inputs.fp32_to_bf16_bits(np.full(1, v, np.float32))[0]) for v in (np.inf, np.nan, 3e38))
    xs = x.copy()
    xs[1, 3], xs[2, 4], xs[3, 5], xs[4, 6] = inf, inf ^ 0x8000, nan, big
    for case in range(3):
        ws = wr.copy()
        if case:
            ws[17, 9] = inf if case == 1 else nan
        plan, idx, tw = _route_only(w, xs, ws, bias)
        _, want_idx, want_w = _route_only(w, xs, ws, bias, route_filter=-1)
        assert plan.moe_last_status() == (0, 0)
        assert torch.equal(idx, want_idx)
        assert torch.allclose(tw, want_w, rtol=1e-5, atol=1e-7, equal_nan=True)


def _zero_tokens(step):
    def spoil(x, wr):
        x[::step] = 0
    return spoil


def _put(name, at, value):
    def spoil(x, wr):
        (x if name == "x" else wr)[at] = value
    return spoil


def _small_router(x, wr):
    wr.mul_(5e-4)


ROUTER_DATA = {"one_zero": _put("x", 7, 0), "zeros_12_percent": _zero_tokens(8), "all_zero": _zero_tokens(1), "one_nan": _put("x", (7, 100), float("nan")),
               "nans_12_percent": _put("x", slice(None, None, 8), float("nan")), "infs_12_percent": _put("x", (slice(None, None, 8), 3), float("-inf")),
               "one_nan_weight": _put("wr", (3, 5), float("nan")), "one_inf_weight": _put("wr", (3, 5), float("inf")), "zero_router": _put("wr", slice(None), 0), "small_router": _small_router}


@pytest.mark.parametrize("tokens", [256, 512])
@pytest.mark.parametrize("what", ROUTER_DATA)
def test_router_direct_kernel_takes_no_longer_than_every_chain(what, tokens):
    """Whatever padding or a new router's weights hold; and the chains' picks and weights.  (A twentieth more is let pass as noise.)"""
    H, E, K = 7168, 256, 8
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.empty((tokens, H), device="cuda").normal_(generator=g).bfloat16()
    wr = torch.empty((E, H), device="cuda").normal_(0.0, 0.02, generator=g).bfloat16()
    ROUTER_DATA[what](x, wr)
    got, took = [], []
    for route_filter in (0, -1):
        plan = B.Plan(B.make_config(tokens, H, E, 1, K, 0, BF16, dispatch_mode=B.DISPATCH_ATOMIC_PAGED, identity_experts=1, route_filter=route_filter))
        idx, tw = torch.empty((tokens, K), dtype=torch.int32, device="cuda"), torch.empty((tokens, K), device="cuda")
        best = 1e9
        for _ in range(6):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda._sleep(100000)      # (the launches are in the queue by the time the first one starts)
            t0.record()
            for _ in range(8):
                plan.moe_route(x, wr, None, idx, tw)
            t1.record()
            torch.cuda.synchronize()
            best = min(best, t0.elapsed_time(t1))
        assert plan.moe_last_status() == (0, 0)
        got.append((idx, tw))
        took.append(best)
    assert torch.equal(got[0][0], got[1][0]) and torch.allclose(got[0][1], got[1][1], rtol=1e-5, atol=1e-8, equal_nan=True)
    assert took[0] <= 1.05 * took[1], took


def test_router_direct_kernel_many_candidates():
    """More than 64 candidates in a CTA of two tokens, from one of them or both: infinities, ties and near ties across 70 to 256
    experts, beside tokens that have few; E below and above 128, an odd number of tokens, H that ends inside 64 columns."""
    for T, H, E in ((251, 7176, 256), (601, 8184, 136), (1001, 7168, 100)):
        w = inputs.Workload("many", T=T, H=H, E=E, R=1, K=8, F=8, dtype=BF16, seed=35)
        x, (wr, _) = inputs.make_x(w), inputs.make_router(w)
        inf = int(inputs.fp32_to_bf16_bits(np.full(1, np.inf, np.float32))[0])
        wr[10:80] = wr[10]
        wr[20:75, 3] ^= 1                                    # an ulp apart in one column
        bias = np.zeros(E, np.float32)
        bias[10:80] = 100.0                                  # those 70 are every token's best: ties are candidates of all
        for b in (bias, None):
            ridx, rw, _ = oracle.route(x, wr, b, w.K, BF16)
            plan, idx, tw = _route_only(w, x, wr, b)
            assert plan.moe_last_status() == (0, 0)
            Hh.check_route(idx, tw, ridx, rw)
        xs = x.copy()
        xs[::9, 5], xs[T - 1, 0] = inf, inf ^ 0x8000
        plan, idx, tw = _route_only(w, xs, wr, None)
        _, want_idx, want_w = _route_only(w, xs, wr, None, route_filter=-1)
        assert plan.moe_last_status() == (0, 0) and torch.equal(idx, want_idx)
        assert torch.allclose(tw, want_w, rtol=1e-5, atol=1e-7, equal_nan=True)


def _route_only(w, x, wr, bias, **kw):
    plan = Hh.make_plan(w, B.DISPATCH_ATOMIC_PAGED, **kw)
    idx = torch.empty((w.T, w.K), dtype=torch.int32, device="cuda")
    tw = torch.empty((w.T, w.K), dtype=torch.float32, device="cuda")
    plan.moe_route(Hh.to_dev(x), Hh.to_dev(wr), Hh.to_dev(bias), idx, tw)
    torch.cuda.synchronize()
    return plan, idx, tw


@pytest.mark.parametrize("T,H", [(150, 512), (1100, 512), (1030, 1032), (1100, 4104)])   # (150 tokens: every chain; then the filter)
@pytest.mark.parametrize("case", ["zero_rows", "equal_experts", "near_ties", "one_sign"])
def test_router_filter_degenerate_rows(case, T, H):
    """The tensor-core filter of the wide router where its candidate sets are as large as they get: tokens that are
    all zero (every logit equal: all 256 experts are candidates, the picks are experts 0..K-1), experts with identical
    weight rows (exact ties decided by index), logits a few ulps apart, and rows of one sign (every addition rounds the same
    way, and the magnitudes add up to what the error bound allows for).  Several k-blocks in each of its four accumulators."""
    w = inputs.Workload("filter_" + case, T=T, H=H, E=256, R=8, K=8, F=8, dtype=BF16, identity_experts=True, seed=4)
    x, wr, bias, *_ = Hh.oracle_inputs(w, with_experts=False)
    x, wr = x.copy(), wr.copy()
    if case == "zero_rows":
        x[::3] = 0
    elif case == "equal_experts":
        wr[1::2] = wr[0::2]                 # experts 2i and 2i+1 are the same row: every logit comes twice
    elif case == "one_sign":
        x, wr = x & 0x7FFF, wr & 0x7FFF
        x[::2] = inputs.fp32_to_bf16_bits(np.full(1, 1.0078125, np.float32))[0]      # (and half of the tokens constant)
    else:
        wr[:] = wr[0]                        # all experts alike ...
        wr[:, 0] = inputs.fp32_to_bf16_bits(np.linspace(-1e-2, 1e-2, w.E).astype(np.float32))   # ... but for one column
    plan, idx, tw = _route_only(w, x, wr, None)
    assert plan.moe_last_status() == (0, 0)      # (the error bound held on every candidate)
    ridx, rw, _ = oracle.route(x, wr, None, w.K, w.dtype)
    if case == "one_sign":
        # The ruled-out experts' approximate logits are in the denominator, and here a logit is the sum of all magnitudes (up
        # to 70, a unit in its last place is 8e-6): a weight may be off by as much, relatively, as two logits are, and they
        # are off by at most 0.16 of the bound eps (measured on such rows).
        fx, fw = ((a.astype(np.uint32) << 16).view(np.float32).astype(np.float64) for a in (x, wr))
        eps = (H / 2 + 68 * -(-H // 256) + 3) * 2.0 ** -23 * np.linalg.norm(fx, axis=1) * np.linalg.norm(fw, axis=1).max()
        assert np.array_equal(idx.cpu().numpy(), ridx)
        assert (np.abs(tw.cpu().numpy() - rw) <= rw * (1e-5 + 2 * 0.16 * eps[:, None]) + 1e-7).all()
    else:
        Hh.check_route(idx, tw, ridx, rw)
    # and the kernel that runs every chain (above 1024 tokens another one) gives the same
    plan2, idx2, tw2 = _route_only(w, x, wr, None, route_filter=-1)
    assert plan2.moe_last_status() == (0, 0)
    assert torch.equal(idx, idx2)


def test_router_filter_with_a_tiny_wait_limit_reports_or_routes():
    """Every wait of the two filter kernels is bounded.  With a limit of a nanosecond a wait either still finds its
    copy landed (a poll takes longer than that) or runs out: then the kernels give up by themselves and the status says
    so.  Never a hang, never a wrong pick without a status; a plan with the normal limit routes correctly afterwards."""
    w = inputs.Workload("filter_timeout", T=2048, H=2048, E=256, R=8, K=8, F=8, dtype=BF16, identity_experts=True)
    x, wr, bias, *_ = Hh.oracle_inputs(w, with_experts=False)
    ridx, rw, _ = oracle.route(x, wr, bias, w.K, w.dtype)
    plan, idx, tw = _route_only(w, x, wr, bias, wait_limit_ns=1)
    code, detail = plan.moe_last_status()
    if code == 0:
        Hh.check_route(idx, tw, ridx, rw)
    else:
        assert code == -6 and detail in (3, 4, 5), (code, detail)
    plan2, idx2, tw2 = _route_only(w, x, wr, bias)
    assert plan2.moe_last_status() == (0, 0)
    Hh.check_route(idx2, tw2, ridx, rw)


@pytest.mark.parametrize("ties", [0, 200])
def test_router_direct_kernel_with_a_tiny_wait_limit_reports_or_routes(ties):
    """The same for the kernel that fetches its candidates' rows, few of them and, with equal experts, all of Wr."""
    w = inputs.Workload("direct_timeout", T=300, H=5120, E=256, R=8, K=8, F=8, dtype=BF16, identity_experts=True)
    x, wr, bias, *_ = Hh.oracle_inputs(w, with_experts=False)
    wr[:ties] = wr[0]
    ridx, rw, _ = oracle.route(x, wr, bias, w.K, w.dtype)
    for limit in (1, 1_000, 20_000):
        plan, idx, tw = _route_only(w, x, wr, bias, wait_limit_ns=limit)
        code, detail = plan.moe_last_status()
        if code == 0:
            Hh.check_route(idx, tw, ridx, rw)
        else:
            assert code == -6 and detail in (3, 4, 5), (code, detail)
        plan2, idx2, tw2 = _route_only(w, x, wr, bias)
        assert plan2.moe_last_status() == (0, 0)
        Hh.check_route(idx2, tw2, ridx, rw)
