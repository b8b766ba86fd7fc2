"""Parity of the CUDA path (called through the C ABI) with the CPU oracle on the same seeded inputs.

Integers (top-k indices, counts, offsets, permutation) must match bit for bit.  Floats: relative
Frobenius error <= 1e-2 against the oracle's exact mode and max-abs error <= 2e-2 against its
declared-rounding mode (bf16 roundings at the tensors the interface declares bf16), per tensor.
"""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from paper_2607_01844_b200 import binding, synth
from parity_util import check_float, rel_fro

pytestmark = pytest.mark.gpu


def to_dev(host):
    return {k: (v.cuda() if torch.is_tensor(v) else v) for k, v in host.items()}


def np_bias(host):
    return None if host["bias"] is None else host["bias"].cpu().numpy()


def run(w, gemm_path=binding.GEMM_AUTO, host=None):
    host = host or synth.make_inputs(w, "cpu")
    inp = to_dev(host)
    ctx = binding.context_for(w, gemm_path=gemm_path)
    buf = binding.LayerBuffers(w)
    binding.forward(ctx, inp, buf)
    if w.backward:
        binding.backward(ctx, inp, buf)
    binding.mop_poll(ctx)
    torch.cuda.synchronize()
    return host, inp, ctx, buf


def check_integers(w, host, buf):
    xb = synth.bits(host["x"])
    idx, gate = oracle.route(xb, host["W_r"].numpy(), np_bias(host), w.k, w.score_fn, w.bias_mode)
    assert np.array_equal(buf.idx.cpu().numpy(), idx), "top-k indices"
    g = buf.gate.cpu().numpy()
    assert np.all(np.abs(g - gate) <= 1e-6 + 1e-5 * np.abs(gate)), "gates"
    counts, offsets, perm_row, row_src = oracle.permute(idx, w.E)
    assert np.array_equal(buf.counts.cpu().numpy(), counts), "counts"
    assert np.array_equal(buf.offsets.cpu().numpy(), offsets), "offsets"
    assert np.array_equal(buf.perm_row.cpu().numpy(), perm_row), "perm_row"
    assert np.array_equal(buf.row_src.cpu().numpy(), row_src), "row_src"
    Xp = synth.bits(buf.Xp)
    assert np.array_equal(Xp, xb[row_src // w.k]), "Xp rows"
    return idx, g


def check_layer(w, gemm_path):
    host, inp, ctx, buf = run(w, gemm_path)
    idx, gate = check_integers(w, host, buf)   # the float checks use the CUDA path's gates (<= 1e-5 apart)
    xb, Wg, Wu, Wd = (synth.bits(host[n]) for n in ("x", "W_gate", "W_up", "W_down"))
    case = f"{w.name}-T{w.T}d{w.d}E{w.E}k{w.k}f{w.f}-path{gemm_path}"
    Y_e = oracle.ffn_fwd(xb, idx, gate, Wg, Wu, Wd)
    Y_d = oracle.ffn_fwd(xb, idx, gate, Wg, Wu, Wd, declared=True)
    check_float("Y", buf.Y.float().cpu().numpy(), Y_e, Y_d, case)
    if w.backward:
        dYb = synth.bits(host["dY"])
        ex = np.arange(w.E, dtype=np.int32)
        dX_e, dg_e = oracle.ffn_bwd_tokens(xb, dYb, idx, gate, Wg, Wu, Wd)
        dX_d, dg_d = oracle.ffn_bwd_tokens(xb, dYb, idx, gate, Wg, Wu, Wd, declared=True)
        dW_e = oracle.ffn_bwd_experts(xb, dYb, idx, gate, Wg, Wu, Wd, ex)
        dW_d = oracle.ffn_bwd_experts(xb, dYb, idx, gate, Wg, Wu, Wd, ex, declared=True)
        check_float("dX", buf.dX.float().cpu().numpy(), dX_e, dX_d, case)
        check_float("dgate", buf.dgate.cpu().numpy(), dg_e, dg_d, case)
        for name, got, e, dd in zip(("dW_gate", "dW_up", "dW_down"), (buf.dW_gate, buf.dW_up, buf.dW_down), dW_e,
                                    dW_d):
            check_float(name, got.cpu().numpy(), e, dd, case)
    return ctx, buf


SMALL = [
    synth.WORKLOADS["c1_tiny"],
    synth.small("c1_tiny", backward=True),
    synth.small("c2_mid", T=300, d=192, E=12, k=3, f=320, backward=True, seed=11),          # ragged tiles
    synth.small("c3_trillion", T=200, d=256, E=40, k=8, f=128, backward=True, seed=12),     # sigmoid + bias
    synth.small("c3_trillion", T=130, d=64, E=33, k=1, f=64, bias_mode=2, backward=True, seed=13),
    synth.small("c1_tiny", T=64, d=128, E=4, k=4, f=64, backward=True, seed=14),            # k = E
    synth.small("c1_tiny", T=1, d=64, E=3, k=2, f=64, backward=True, seed=15),              # one token
    synth.small("c1_tiny", T=77, d=72, E=5, k=2, f=40, backward=True, seed=16),             # d, f multiples of 8 only
]


@pytest.mark.parametrize("w", SMALL, ids=lambda w: f"{w.name}-T{w.T}d{w.d}E{w.E}k{w.k}f{w.f}{'b' if w.backward else ''}")
@pytest.mark.parametrize("path", [binding.GEMM_SCALAR, binding.GEMM_AUTO, binding.GEMM_TENSOR_TN],
                         ids=["scalar", "auto", "tokens_on_n"])
def test_small_layers_match_oracle(w, path):
    if path == binding.GEMM_TENSOR_TN and (w.d % 64 or w.f % 64):
        with pytest.raises(binding.MopError) as e:      # a forced tensor-core schedule refuses odd shapes
            binding.context_for(w, gemm_path=path)
        assert e.value.code == 6
        return
    check_layer(w, path)


@pytest.mark.parametrize("path", [binding.GEMM_TENSOR_2CTA, binding.GEMM_TENSOR_MIXED, binding.GEMM_TENSOR_TN],
                         ids=["2cta", "mixed", "tokens_on_n"])
def test_two_cta_schedules_match_oracle_and_the_one_cta_kernel(path):
    w = synth.small("c2_mid", T=1500, d=256, E=6, k=2, f=320, backward=True, seed=21)   # 500 rows per expert
    _, buf = check_layer(w, path)
    _, _, _, ref = run(w, binding.GEMM_TENSOR_1CTA)
    for n in ("H", "Yp", "Y", "dX", "dW_gate", "dW_up", "dW_down"):   # same accumulation order
        assert torch.equal(getattr(buf, n), getattr(ref, n)), n
    # dgate is a sum over f whose partial sums are grouped by the kernel's tile shape
    assert torch.allclose(buf.dgate, ref.dgate, rtol=1e-4, atol=1e-4 * float(ref.dgate.abs().max()))


GATHER = [
    synth.small("c3_trillion", T=200, d=256, E=40, k=8, f=128, seed=41),      # 40 rows per expert: one ragged tile each
    synth.small("c2_mid", T=1500, d=256, E=6, k=2, f=320, seed=42),           # 500 rows per expert: two tiles
    synth.small("c4_skew", T=1024, d=192, E=16, k=4, f=192, seed=43),         # skewed counts, hot and empty experts
    synth.small("c1_tiny", T=3, d=64, E=5, k=1, f=64, seed=44),               # fewer rows than experts
]


@pytest.mark.parametrize("w", GATHER, ids=lambda w: f"{w.name}-T{w.T}d{w.d}E{w.E}k{w.k}f{w.f}")
def test_gathering_forward_matches_oracle_and_the_permuting_forward(w):
    host = synth.make_inputs(w, "cpu")
    inp = to_dev(host)
    ctx = binding.context_for(w, backward=False)
    buf = binding.LayerBuffers(w)
    buf.Xp.fill_(float("nan"))                       # the gathering form must not touch (or need) Xp
    binding.forward(ctx, inp, buf, gather=True)
    binding.mop_poll(ctx)
    torch.cuda.synchronize()
    assert torch.isnan(buf.Xp.float()).all()
    xb, Wg, Wu, Wd = (synth.bits(host[n]) for n in ("x", "W_gate", "W_up", "W_down"))
    idx, _ = oracle.route(xb, host["W_r"].numpy(), np_bias(host), w.k, w.score_fn, w.bias_mode)
    assert np.array_equal(buf.idx.cpu().numpy(), idx)
    gate = buf.gate.cpu().numpy()
    Y_e = oracle.ffn_fwd(xb, idx, gate, Wg, Wu, Wd)
    Y_d = oracle.ffn_fwd(xb, idx, gate, Wg, Wu, Wd, declared=True)
    check_float("Y", buf.Y.float().cpu().numpy(), Y_e, Y_d, f"gather-{w.name}-T{w.T}")
    _, _, _, ref = run(dataclasses.replace(w, backward=False), binding.GEMM_TENSOR_TN, host)
    for n in ("H", "Yp", "Y"):                       # same tiles, same accumulation order
        assert torch.equal(getattr(buf, n), getattr(ref, n)), n


def test_gathering_forward_refuses_the_scalar_path():
    w = synth.small("c1_tiny", T=77, d=72, E=5, k=2, f=40, seed=16)
    host, inp, ctx, buf = run(w)
    with pytest.raises(binding.MopError) as e:
        binding.forward(ctx, inp, buf, gather=True)
    assert e.value.code == 6


@pytest.mark.parametrize("T,d,E,k,f", [(40, 8, 3, 2, 8),            # narrower than one box
                                       (700, 264, 5, 2, 392),       # one vector past tiles of 256 and of 128
                                       (333, 200, 4, 1, 136),       # a weight tile whose second chunk is partly, or wholly, outside
                                       (90, 1000, 7, 3, 1416)],     # the last K block of every GEMM is partly filled
                         ids=lambda v: str(v))
def test_widths_that_are_multiples_of_8_only_run_on_the_tensor_cores(T, d, E, k, f):
    w = synth.small("c3_trillion", T=T, d=d, E=E, k=k, f=f, backward=True, seed=47)
    ctx, buf = check_layer(w, binding.GEMM_AUTO)
    binding.mop_profile_enable(ctx)
    host = synth.make_inputs(w, "cpu")
    inp = to_dev(host)
    binding.forward(ctx, inp, buf)
    binding.backward(ctx, inp, buf)
    names = binding.mop_profile_read(ctx)
    assert {"gemm_up_swiglu", "gemm_wgrad_down"} <= set(names) and not [n for n in names if n.startswith("scalar")]


@pytest.mark.parametrize("d,f", [(128, 192), (72, 136)], ids=lambda v: str(v))
@pytest.mark.parametrize("T,E,k,experts", [(16, 8, 8, 1),       # 128 rows of 16 tokens: one tile with a box of 64 rows
                                           (16, 6, 6, 2),       # 48 rows each
                                           (3, 32, 31, 1),      # 93 rows of 3 tokens
                                           (37, 5, 4, 1),       # 148 rows, the last ones of the box past the end
                                           (200, 4, 4, 1)],     # 800 rows: four tiles
                         ids=lambda v: str(v))
def test_experts_named_more_than_once_for_a_token(T, E, k, experts, d, f):
    """A caller's own indices: an expert may get more rows than there are tokens."""
    w = synth.small("c1_tiny", T=T, d=d, E=E, k=k, f=f, backward=True, seed=50)
    host = synth.make_inputs(w, "cpu")
    inp = to_dev(host)
    idx = np.random.default_rng(51).integers(0, experts, (T, k)).astype(np.int32) + E - experts
    gate = np.random.default_rng(52).uniform(0.1, 0.4, (T, k)).astype(np.float32)
    ctx, b = binding.context_for(w), binding.LayerBuffers(w)
    b.idx.copy_(torch.from_numpy(idx))
    b.gate.copy_(torch.from_numpy(gate))
    binding.mop_moe_permute(ctx, inp["x"], b.idx, b.counts, b.offsets, b.perm_row, b.row_src, b.Xp)
    binding.mop_moe_expert_ffn_fwd(ctx, b.Xp, b.offsets, b.row_src, b.gate, inp["W_gate"], inp["W_up"], inp["W_down"], b.G, b.U,
                                   b.H, b.Yp)
    binding.mop_moe_combine(ctx, b.Yp, b.perm_row, b.Y)
    binding.backward(ctx, inp, b)
    binding.mop_poll(ctx)
    for got, want in zip((b.counts, b.offsets, b.perm_row, b.row_src), oracle.permute(idx, E)):
        assert np.array_equal(got.cpu().numpy(), want)
    xb, Wg, Wu, Wd, dYb = (synth.bits(host[n]) for n in ("x", "W_gate", "W_up", "W_down", "dY"))
    case = f"repeated-T{T}d{d}E{E}k{k}f{f}"
    check_float("Y", b.Y.float().cpu().numpy(), oracle.ffn_fwd(xb, idx, gate, Wg, Wu, Wd),
                oracle.ffn_fwd(xb, idx, gate, Wg, Wu, Wd, declared=True), case)
    exact, declared = (oracle.ffn_bwd_tokens(xb, dYb, idx, gate, Wg, Wu, Wd, declared=v) for v in (False, True))
    check_float("dX", b.dX.float().cpu().numpy(), exact[0], declared[0], case)
    check_float("dgate", b.dgate.cpu().numpy(), exact[1], declared[1], case)
    ex = np.arange(E, dtype=np.int32)
    exact, declared = (oracle.ffn_bwd_experts(xb, dYb, idx, gate, Wg, Wu, Wd, ex, declared=v) for v in (False, True))
    for n, e, dd in zip(("dW_gate", "dW_up", "dW_down"), exact, declared):
        check_float(n, getattr(b, n).cpu().numpy(), e, dd, case)


@pytest.mark.parametrize("T,d,E,k,f", [(1500, 256, 3, 1, 320),      # 500 rows: a tile of 256 whose second CTA is half outside
                                       (1121, 200, 4, 2, 136),      # widths at every edge of a pair's halves, K tails of any length
                                       (1344, 64, 3, 1, 64),        # 448 rows, one tile, the second CTA wholly outside
                                       (1024, 192, 9, 2, 128),      # 228 rows: single CTAs that prefetch, short last expert
                                       (1350, 320, 40, 16, 64)],    # many tiles per pair: both accumulators and the stage ring wrap
                         ids=lambda v: str(v))
@pytest.mark.parametrize("accumulate", [False, True], ids=["write", "add"])
def test_weight_gradients_on_cta_pairs(T, d, E, k, f, accumulate):
    w = synth.small("c4_skew", T=T, d=d, E=E, k=k, f=f, backward=True, skew=E > 4, seed=49)
    assert w.M >= (224 if E == 9 else 448) * E
    host = synth.make_inputs(w, "cuda")
    out = []
    # SCALAR: no tensor core at all, other sums (odd widths); 1CTA: the same sums in the same order
    for path in (binding.GEMM_AUTO, binding.GEMM_SCALAR if d % 64 or f % 64 else binding.GEMM_TENSOR_1CTA):
        ctx = binding.context_for(w, gemm_path=path, dw_accumulate=accumulate)
        buf = binding.LayerBuffers(w)
        for g in (buf.dW_gate, buf.dW_up, buf.dW_down):
            g.fill_(0.5)
        binding.forward(ctx, host, buf)
        binding.backward(ctx, host, buf)
        binding.mop_poll(ctx)
        out.append(buf)
    for n in ("dW_gate", "dW_up", "dW_down"):
        a, b = getattr(out[0], n), getattr(out[1], n)
        if d % 64 or f % 64:    # fp32 sums in another order of bf16 intermediates that may flip their rounding
            assert rel_fro(a.cpu().numpy(), b.cpu().numpy()) < 1e-3
        else:
            assert torch.equal(a, b), n


@pytest.mark.parametrize("E,k,T,d,f", [(512, 8, 300, 64, 448),     # one K block per item, 27 items per cluster and more
                                       (400, 4, 500, 640, 512),    # 10 K blocks: items announced one ahead
                                       (160, 2, 700, 1600, 1088)],  # 25 K blocks: announced near the end of the one before
                         ids=lambda v: str(v))
def test_tokens_on_n_kernels_with_many_more_items_than_clusters(E, k, T, d, f):
    """Work items are handed out through rings of 16 entries: more than 16 items per cluster wrap them."""
    w = synth.small("c2_mid", T=T, d=d, E=E, k=k, f=f, backward=True, seed=46)
    host = synth.make_inputs(w, "cuda")
    _, _, _, buf = run(w, binding.GEMM_TENSOR_TN, host)
    assert int((buf.counts > 0).sum()) * -(-f // 128) > 17 * 74
    _, _, _, ref = run(w, binding.GEMM_TENSOR_1CTA, host)     # bit for bit the one-CTA kernel, which the cases above tie to the oracle
    for n in ("H", "Yp", "Y", "dX", "dW_gate", "dW_up", "dW_down"):
        assert torch.equal(getattr(buf, n), getattr(ref, n)), n


def test_tokens_on_n_kernels_with_three_token_tiles_and_half_filled_k_stages():
    """700 rows per expert (three token tiles of 240) with d = 320 and f = 192: K is 2.5 and 1.5 pipeline
    stages of 128, so the last stage of every GEMM is half zero fill; all four token-row GEMMs forced
    onto the tokens-on-N kernel, compared with the oracle and bit for bit with the one-CTA kernel."""
    w = synth.small("c2_mid", T=1400, d=320, E=4, k=2, f=192, backward=True, seed=45)
    _, buf = check_layer(w, binding.GEMM_TENSOR_TN)
    assert int(buf.counts.max()) > 512
    _, _, _, ref = run(w, binding.GEMM_TENSOR_1CTA)
    for n in ("H", "Yp", "Y", "dX", "dW_gate", "dW_up", "dW_down"):
        assert torch.equal(getattr(buf, n), getattr(ref, n)), n


def test_all_keys_equal_goes_to_lowest_ids_and_leaves_experts_empty():
    w = synth.small("c1_tiny", T=96, d=64, E=6, k=2, f=64, backward=True, seed=17)
    host = synth.make_inputs(w, "cpu")
    host["W_r"] = torch.zeros_like(host["W_r"])
    host, inp, ctx, buf = run(w, host=host)
    assert np.array_equal(buf.idx.cpu().numpy(), np.tile(np.arange(2, dtype=np.int32), (96, 1)))
    assert np.array_equal(buf.counts.cpu().numpy(), np.array([96, 96, 0, 0, 0, 0], np.int32))
    assert torch.all(buf.dW_gate[2:] == 0) and torch.all(buf.dW_down[2:] == 0)
    check_integers(w, host, buf)


def test_an_overflowing_expert_does_not_reach_its_neighbours_gradients():
    """Backward with non-finite upstream gradients for the tokens of ONE expert (k = 1, so a token has one
    expert): that expert's gradients are lost, every other expert's dW and every other token's dX and dgate
    keep the bits of the clean run.  The rows of an expert end inside a 16-row K group of the weight-gradient
    GEMMs for all but a few experts here, so the K tail of the expert before the poisoned one is exercised."""
    w = synth.small("c5_train", T=1500, d=128, E=7, k=1, f=192, backward=True, seed=41)
    host = synth.make_inputs(w, "cpu")
    inp = to_dev(host)
    for path in (binding.GEMM_AUTO, binding.GEMM_TENSOR_1CTA):
        ctx = binding.context_for(w, gemm_path=path)
        clean, bad = binding.LayerBuffers(w), binding.LayerBuffers(w)
        binding.forward(ctx, inp, clean)
        binding.backward(ctx, inp, clean)
        counts = clean.counts.cpu().numpy()
        e0 = int(np.argsort(counts)[len(counts) // 2])                    # an expert with rows, not the first one
        if e0 == 0:
            e0 = 1
        assert counts[e0] > 0 and counts[e0 - 1] % 16 != 0
        poisoned = dict(inp)
        dY = inp["dY"].clone()
        mine = (clean.idx[:, 0] == e0)
        dY[mine] = float("inf")
        dY[mine.nonzero()[::2, 0]] = float("nan")
        poisoned["dY"] = dY
        binding.forward(ctx, poisoned, bad)
        binding.backward(ctx, poisoned, bad)
        binding.mop_poll(ctx)
        others = torch.ones(w.E, dtype=torch.bool, device="cuda")
        others[e0] = False
        for name in ("dW_gate", "dW_up", "dW_down"):
            a, b = getattr(clean, name), getattr(bad, name)
            assert torch.equal(a[others], b[others]), f"{name} of the other experts (path {path})"
            assert not torch.isfinite(b[e0]).all(), f"{name} of the poisoned expert should be lost"
        assert torch.equal(clean.dX[~mine], bad.dX[~mine]) and torch.equal(clean.dgate[~mine], bad.dgate[~mine])


@pytest.mark.parametrize("T,d,E,k,f", [(50, 384, 2, 1, 72),       # boxes.  25 rows: two steps, the second partly filled; f ends inside a box
                                       (700, 256, 3, 2, 320),     # two tiles per expert, steps beyond every buffer
                                       (40, 128, 8, 2, 200),      # fewer rows than a tile's smallest box asks for
                                       (130, 2048, 1, 1, 136),    # one more row per expert than the line asks for at the longest K
                                       (128, 2048, 1, 1, 136),    # by warps: on the line
                                       (50, 2048, 2, 1, 72), (40, 512, 8, 2, 200),
                                       (600, 2056, 2, 2, 136)],   # longer K, three tiles per expert
                         ids=lambda v: str(v))
def test_swiglu_backward_by_warps_and_by_boxes(T, d, E, k, f):
    check_layer(synth.small("c3_trillion", T=T, d=d, E=E, k=k, f=f, backward=True, seed=T), binding.GEMM_AUTO)


@pytest.mark.parametrize("T,k,E", [(2048, 2, 24), (2049, 2, 24), (4096, 1, 1024), (1025, 4, 7), (4609, 1, 3),
                                   (49152, 2, 257), (98304, 1, 1024), (24576, 4, 5),          # one launch: its longest runs
                                   (49153, 2, 257), (98305, 1, 1024), (33000, 3, 3)])         # three kernels
def test_permutation_tables_and_rows_on_both_sides_of_the_single_launch_limit(T, k, E):
    """Up to 98304 assignments the permutation is one cluster launch, beyond that three kernels: tables and copied rows must be the
    oracle's on both sides of that limit, with few experts and with many."""
    gen = torch.Generator().manual_seed(T + E)
    idx = torch.rand((T, E), generator=gen).topk(k, 1).indices.to(torch.int32)
    counts, offsets, perm_row, row_src = oracle.permute(idx.numpy(), E)
    ctx = binding.Context(T, 64, E, k, 64)
    dev = {n: torch.empty(s, dtype=torch.int32, device="cuda") for n, s in
           (("counts", (E,)), ("offsets", (E + 1,)), ("perm_row", (T * k,)), ("row_src", (T * k,)))}
    x = torch.randn((T, 64)).to(torch.bfloat16).cuda()
    Xp = torch.empty((T * k, 64), dtype=torch.bfloat16, device="cuda")
    binding.mop_moe_permute(ctx, x, idx.cuda(), dev["counts"], dev["offsets"], dev["perm_row"], dev["row_src"], Xp)
    binding.mop_poll(ctx)
    assert np.array_equal(dev["counts"].cpu().numpy(), counts) and np.array_equal(dev["offsets"].cpu().numpy(), offsets)
    assert np.array_equal(dev["perm_row"].cpu().numpy(), perm_row) and np.array_equal(dev["row_src"].cpu().numpy(), row_src)
    assert torch.equal(Xp.cpu(), x.cpu()[torch.from_numpy(row_src // k).long()])


@pytest.mark.parametrize("T,k,E", [(1, 1, 1), (11, 3, 5), (512, 2, 33), (1025, 1, 1024), (341, 12, 40),   # 1, 1, 1, 2, 4 blocks
                                   (8192, 1, 2), (2731, 3, 257),                # eight: 32 assignments a warp, 64
                                   (32768, 3, 31), (32769, 3, 31)])             # the longest runs, the three kernels
def test_permutation_in_one_launch_with_indices_out_of_range(T, k, E):
    """Assignments whose index names no expert get row -1 and are counted nowhere; the others keep their order."""
    gen = torch.Generator().manual_seed(3 * T + E)
    idx = torch.randint(-1, E + 1, (T, k), generator=gen, dtype=torch.int32)
    flat = idx.numpy().reshape(-1)
    ok = (flat >= 0) & (flat < E)
    counts = np.bincount(flat[ok], minlength=E)
    order = np.flatnonzero(ok)[np.argsort(flat[ok], kind="stable")]
    perm_row = np.full(T * k, -1, dtype=np.int32)
    perm_row[order] = np.arange(order.size)
    ctx = binding.Context(T, 64, E, k, 64)
    dev = {n: torch.full((s,), -7, dtype=torch.int32, device="cuda") for n, s in
           (("counts", E), ("offsets", E + 1), ("perm_row", T * k), ("row_src", T * k))}
    binding.mop_moe_permute(ctx, None, idx.cuda(), dev["counts"], dev["offsets"], dev["perm_row"], dev["row_src"], None)
    got = {n: v.cpu().numpy() for n, v in dev.items()}
    assert np.array_equal(got["counts"], counts) and np.array_equal(got["offsets"], np.concatenate(([0], np.cumsum(counts))))
    assert np.array_equal(got["perm_row"], perm_row) and np.array_equal(got["row_src"][:order.size], order)
    assert (got["row_src"][order.size:] == -7).all()


@pytest.mark.parametrize("T,d,E,k", [(24576, 64, 40, 4), (24577, 64, 40, 4), (98400, 64, 7, 1)])
def test_forward_on_both_sides_of_the_single_launch_permutation(T, d, E, k):
    """The token tiles come from the permutation or from a block beside the row copy: the same bits as the separate calls'."""
    test_small_forward_in_one_call_equals_the_separate_calls(T, d, E, k, 0, 0)


@pytest.mark.parametrize("T,d,E,k,score,bias", [(1, 64, 256, 32, 1, 1), (7, 64, 3, 3, 0, 0), (9, 1032, 65, 4, 1, 2),     # one block, eight
                                                (256, 64, 129, 8, 1, 1), (255, 520, 64, 4, 0, 0), (128, 1024, 40, 4, 1, 1),
                                                (257, 64, 64, 4, 1, 1), (129, 1024, 40, 4, 0, 0), (60, 64, 257, 4, 1, 0)])   # in three
def test_small_forward_in_one_call_equals_the_separate_calls(T, d, E, k, score, bias):
    """Selection, permutation and row copy in one launch: the same bits as the separate entry points', on both sides of its limits."""
    w = synth.Workload("one", T, d, E, k, 64, score, bias, 0.01 if bias else 0.0, seed=T + E)
    inp = synth.make_inputs(w, "cuda")
    ctx = binding.context_for(w, route_path=binding.ROUTE_EXACT)
    one, sep = binding.LayerBuffers(w), binding.LayerBuffers(w)
    binding.forward(ctx, inp, one)
    binding.mop_moe_route(ctx, inp["x"], inp["W_r"], inp["bias"], sep.idx, sep.gate)
    binding.mop_moe_permute(ctx, inp["x"], sep.idx, sep.counts, sep.offsets, sep.perm_row, sep.row_src, sep.Xp)
    binding.mop_moe_expert_ffn_fwd(ctx, sep.Xp, sep.offsets, sep.row_src, sep.gate, inp["W_gate"], inp["W_up"], inp["W_down"],
                                   None, None, sep.H, sep.Yp)
    binding.mop_moe_combine(ctx, sep.Yp, sep.perm_row, sep.Y)
    binding.mop_poll(ctx)
    for name in ("idx", "gate", "counts", "offsets", "perm_row", "row_src", "Xp", "Y"):
        assert torch.equal(getattr(one, name), getattr(sep, name)), name
    x, W_r = synth.bits(inp["x"]), inp["W_r"].cpu().numpy()
    idx, gate = oracle.route(x, W_r, None if not bias else inp["bias"].cpu().numpy(), k, score, bias)
    assert np.array_equal(one.idx.cpu().numpy(), idx) and np.allclose(one.gate.cpu().numpy(), gate, rtol=1e-5, atol=1e-6)


@pytest.mark.parametrize("E,k", [(31, 5), (200, 8), (500, 3), (1024, 32)])
def test_selection_of_equal_signed_zero_and_infinite_logits(E, k):
    """x = 1 everywhere and one row of W_r: the logits are that row.  Ties go to the lower id, -0 equals +0, infinities keep their place."""
    d, T = 8, 5
    gen = torch.Generator().manual_seed(E)
    row = torch.randint(-2, 3, (E,), generator=gen).float()
    row[::3] = torch.where(torch.arange(0, E, 3) % 2 == 0, 0.0, -0.0)
    row[E // 2], row[E // 3] = float("inf"), float("-inf")
    W_r = torch.zeros((d, E))
    W_r[0] = row
    order = np.lexsort((np.arange(E), -row.numpy().astype(np.float64)))[:k]
    ctx = binding.Context(T, d, E, k, 64)
    x = torch.zeros((T, d), dtype=torch.bfloat16)
    x[:, 0] = 1.0
    idx = torch.empty((T, k), dtype=torch.int32, device="cuda")
    gate = torch.empty((T, k), dtype=torch.float32, device="cuda")
    binding.mop_moe_route(ctx, x.cuda(), W_r.cuda(), None, idx, gate)
    assert (idx.cpu().numpy() == order).all()


@pytest.mark.parametrize("E,k", [(33, 3), (65, 8), (128, 1), (257, 8), (513, 32), (1024, 2)])     # every number of keys a lane holds
@pytest.mark.parametrize("score,bias", [(0, 2), (1, 0), (1, 1), (1, 2)])
def test_selection_with_every_form_of_key_matches_oracle(E, k, score, bias):
    w = synth.Workload("keys", 70, 64, E, k, 64, score, bias, 0.05 if bias else 0.0, seed=E + score)
    inp = synth.make_inputs(w, "cuda")
    ctx = binding.context_for(w, route_path=binding.ROUTE_EXACT)
    idx = torch.empty((w.T, k), dtype=torch.int32, device="cuda")
    gate = torch.empty((w.T, k), dtype=torch.float32, device="cuda")
    b = inp["bias"] if not bias or inp["bias"] is not None else torch.randn(E, device="cuda") * 0.05
    binding.mop_moe_route(ctx, inp["x"], inp["W_r"], b, idx, gate)
    want, g = oracle.route(synth.bits(inp["x"]), inp["W_r"].cpu().numpy(), None if b is None else b.cpu().numpy(), k, score, bias)
    assert np.array_equal(idx.cpu().numpy(), want) and np.allclose(gate.cpu().numpy(), g, rtol=1e-5, atol=1e-6)


@pytest.mark.parametrize("T,d,k", [(1, 8, 1), (9, 72, 2), (3, 264, 32), (130, 1032, 9), (60, 520, 3),      # a thread per vector, 1, 2, 8, 8, 4 rows
                                   (3600, 256, 3), (3600, 264, 2), (900, 1032, 6),    # the same with larger blocks
                                   (3000, 520, 5), (2500, 760, 1),                    # the same beyond the line: short rows
                                   (2000, 768, 2), (1800, 1016, 5), (1500, 1032, 3),  # a warp per 2 KiB of a row: partly filled, twice
                                   (1480, 1024, 9), (1481, 1024, 9)])                 # the last size on one side of the line, whole pieces
def test_combine_sums_the_rows_in_order(T, d, k):
    """Bit for bit the fp32 sum in ascending j, rounded once; rows of -1 are left out."""
    gen = torch.Generator().manual_seed(T + d)
    Yp = torch.randn((T * k, d), generator=gen).to(torch.bfloat16).cuda()
    perm = torch.randperm(T * k, generator=gen).to(torch.int32).reshape(T, k)
    perm[torch.rand((T, k), generator=gen) < 0.1] = -1
    ctx = binding.Context(T, d, max(k, 4), k, 64)
    Y = torch.empty((T, d), dtype=torch.bfloat16, device="cuda")
    binding.mop_moe_combine(ctx, Yp, perm.cuda().reshape(-1), Y)
    acc = torch.zeros((T, d), device="cuda")
    for j in range(k):
        rows = perm[:, j].cuda().long()
        acc = torch.where(rows[:, None] >= 0, acc + Yp[rows.clamp(min=0)].float(), acc)
    assert torch.equal(Y, acc.to(torch.bfloat16))


def test_zero_tokens_is_a_no_op():
    w = synth.small("c1_tiny", T=0, d=64, E=4, k=2, f=64, backward=True)
    host, inp, ctx, buf = run(w)
    assert torch.all(buf.offsets == 0) and torch.all(buf.counts == 0)
    assert torch.all(buf.dW_gate == 0) and torch.all(buf.dW_up == 0) and torch.all(buf.dW_down == 0)


def test_results_are_bitwise_reproducible():
    w = synth.small("c2_mid", T=512, d=256, E=16, k=4, f=256, backward=True, seed=18)
    _, _, _, a = run(w)
    _, _, _, b = run(w)
    for n in ("idx", "gate", "perm_row", "Xp", "H", "Yp", "Y", "dX", "dgate", "dW_gate", "dW_up", "dW_down"):
        assert torch.equal(getattr(a, n), getattr(b, n)), n


def test_dw_accumulate_adds_into_existing_gradients():
    w = synth.small("c1_tiny", T=128, d=64, E=4, k=2, f=64, backward=True, seed=19)
    host = synth.make_inputs(w, "cpu")
    inp = to_dev(host)
    ctx = binding.context_for(w, dw_accumulate=True)
    buf = binding.LayerBuffers(w)
    for t in (buf.dW_gate, buf.dW_up, buf.dW_down):
        t.fill_(1.0)
    binding.forward(ctx, inp, buf)
    binding.backward(ctx, inp, buf)
    _, _, _, ref = run(w, host=host)
    for n in ("dW_gate", "dW_up", "dW_down"):
        assert torch.allclose(getattr(buf, n), getattr(ref, n) + 1.0, atol=1e-5), n


def test_bad_arguments_return_codes():
    w = synth.WORKLOADS["c1_tiny"]
    ctx = binding.context_for(w)
    buf = binding.LayerBuffers(w)
    with pytest.raises(binding.MopError) as e:
        binding.mop_moe_combine(ctx, None, buf.perm_row, buf.Y)
    assert e.value.code == 1
    with pytest.raises(binding.MopError) as e:
        binding.mop_moe_combine(ctx, buf.Yp.data_ptr() + 2, buf.perm_row, buf.Y)
    assert e.value.code == 3
    with pytest.raises(binding.MopError) as e:   # backward on a forward-only context
        binding.mop_moe_expert_ffn_bwd(ctx, *([buf.Yp] * 17))
    assert e.value.code == 6
    with pytest.raises(binding.MopError) as e:
        binding.Context(16, 64, 4, 5, 64)
    assert e.value.code == 1


LAYER_OUT = ("idx", "gate", "counts", "offsets", "perm_row", "row_src", "Xp", "G", "U", "H", "Yp", "Y")


@pytest.mark.parametrize("name", ("x", "W_r", "W_gate", "W_up", "W_down") + LAYER_OUT)
def test_forward_in_one_call_checks_every_argument_before_it_launches(name):
    w = synth.small("c1_tiny", T=24, d=64, E=4, k=2, f=64, backward=True, seed=31)
    inp = synth.make_inputs(w, "cuda")
    ctx, b = binding.context_for(w), binding.LayerBuffers(w)
    tensors = {**{n: inp[n] for n in ("x", "W_r", "W_gate", "W_up", "W_down")}, **{n: getattr(b, n) for n in LAYER_OUT}}
    for n in LAYER_OUT:
        tensors[n].fill_(7)

    def call(**changed):
        a = {**{n: t.data_ptr() for n, t in tensors.items()}, "bias": None, **changed}
        binding.mop_moe_layer_fwd(ctx, a["x"], a["W_r"], a["bias"], a["W_gate"], a["W_up"], a["W_down"], *(a[n] for n in LAYER_OUT))

    launched = ctx.launch_count
    for changed, code in (({name: None}, 1), ({name: tensors[name].data_ptr() + 4}, 3), ({"bias": inp["W_r"].data_ptr()}, 1)):
        with pytest.raises(binding.MopError) as e:
            call(**changed)
        assert e.value.code == code
    torch.cuda.synchronize()
    assert ctx.launch_count == launched
    for n in LAYER_OUT:
        assert bool((tensors[n] == 7).all()), n
    call(G=None, U=None)                       # no stash: accepted
    call()
    binding.mop_poll(ctx)


def test_the_step_can_be_captured_into_a_cuda_graph_and_replayed():
    """The device entry points allocate nothing and never synchronise, so a whole step captures."""
    w = synth.small("c2_mid", T=512, d=256, E=16, k=4, f=192, backward=True, seed=29)
    host, inp, ctx, ref = run(w)
    buf = binding.LayerBuffers(w)
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(graph, stream=side):
            binding.forward(ctx, inp, buf, side)
            binding.backward(ctx, inp, buf, side)
    torch.cuda.synchronize()
    for _ in range(2):                                  # replays are steps of their own
        for n in ("Y", "dX", "dgate", "dW_gate", "dW_up", "dW_down"):
            getattr(buf, n).zero_()
        graph.replay()
        torch.cuda.synchronize()
        for n in ("idx", "gate", "Y", "dX", "dgate", "dW_gate", "dW_up", "dW_down"):
            assert torch.equal(getattr(buf, n), getattr(ref, n)), n
    binding.mop_poll(ctx)


def test_largest_expert_count_and_routing_degree():
    """E = 1024 and k = 32 are the limits of the selection kernel; most experts get zero to four rows."""
    w = synth.small("c1_tiny", T=48, d=64, E=1024, k=32, f=64, backward=True, seed=27)
    _, buf = check_layer(w, binding.GEMM_AUTO)
    assert int((buf.counts == 0).sum()) > 0
    w2 = synth.small("c3_trillion", T=40, d=64, E=1024, k=32, f=64, seed=28)      # sigmoid + bias at the limits
    check_layer(w2, binding.GEMM_AUTO)


def test_shapes_beyond_the_limits_are_refused():
    for args, code in (((16, 64, 1025, 2, 64), 2), ((64, 64, 64, 33, 64), 2), ((16, 60, 4, 2, 64), 3),
                       ((16, 64, 4, 2, 36), 3), ((-1, 64, 4, 2, 64), 1), ((16, 64, 0, 1, 64), 1)):
        with pytest.raises(binding.MopError) as e:
            binding.Context(*args)
        assert e.value.code == code, args


def test_forward_host_entry_point_matches_device_path():
    w = synth.small("c2_mid", T=256, d=128, E=8, k=2, f=192, seed=20)
    host, inp, _, buf = run(w)
    ctx = binding.context_for(w, host_io=True)
    xh = host["x"].pin_memory()
    Yh = torch.empty_like(xh).pin_memory()
    idxh = torch.empty((w.T, w.k), dtype=torch.int32).pin_memory()
    gh = torch.empty((w.T, w.k), dtype=torch.float32).pin_memory()
    binding.mop_moe_forward_host(ctx, xh, inp["W_r"], inp["bias"], inp["W_gate"], inp["W_up"], inp["W_down"], Yh, idxh,
                                 gh)
    assert torch.equal(Yh, buf.Y.cpu()) and torch.equal(idxh, buf.idx.cpu()) and torch.equal(gh, buf.gate.cpu())


@pytest.mark.parametrize("T,host_io", [(40, 1), (40, 2), (400, 1), (400, 2)])     # routed in one launch, and by the separate calls
def test_host_entry_points_refuse_a_missing_router_or_bias(T, host_io):
    w = synth.small("c3_trillion", T=T, d=128, E=8, k=2, f=64, seed=20)
    inp = synth.make_inputs(w, "cuda")
    ctx = binding.context_for(w, host_io=host_io)
    xh = inp["x"].cpu().pin_memory()
    Yh = torch.empty_like(xh).pin_memory()
    call = binding.mop_moe_forward_host if host_io == 1 else binding.mop_moe_forward_host_async
    assert inp["bias"] is not None
    for W_r, bias in ((None, inp["bias"]), (inp["W_r"], None)):
        with pytest.raises(binding.MopError) as e:
            call(ctx, xh, W_r, bias, inp["W_gate"], inp["W_up"], inp["W_down"], Yh)
        assert e.value.code == 1
    call(ctx, xh, inp["W_r"], inp["bias"], inp["W_gate"], inp["W_up"], inp["W_down"], Yh)
    if host_io == 2:
        binding.mop_host_drain(ctx)
    buf = binding.LayerBuffers(w)
    binding.forward(binding.context_for(w), inp, buf)
    assert torch.equal(Yh, buf.Y.cpu())


@pytest.mark.parametrize("backward", [False, True], ids=["fwd", "train"])
def test_pipelined_host_steps_match_the_device_path_step_by_step(backward):
    """Five steps with different inputs in flight through the two slots; every step's results are its own."""
    w = synth.small("c2_mid", T=300, d=128, E=8, k=2, f=192, seed=23, backward=backward)
    steps = 5
    hosts = [synth.make_inputs(dataclasses.replace(w, seed=100 + i), "cpu") for i in range(steps)]
    weights = to_dev(hosts[0])                      # one set of weights, per-step activations
    ctx = binding.context_for(w, host_io=2)
    outs = []
    for h in hosts:
        o = {"x": h["x"].pin_memory(), "Y": torch.empty_like(h["x"]).pin_memory(),
             "idx": torch.empty((w.T, w.k), dtype=torch.int32).pin_memory(),
             "gate": torch.empty((w.T, w.k), dtype=torch.float32).pin_memory()}
        if backward:
            o["dY"] = h["dY"].pin_memory()
            o["dX"] = torch.empty_like(h["x"]).pin_memory()
            o["dgate"] = torch.empty((w.T, w.k), dtype=torch.float32).pin_memory()
        outs.append(o)
    dW = [torch.empty_like(weights[n], dtype=torch.float32) for n in ("W_gate", "W_up", "W_down")]
    for o in outs:
        if backward:
            binding.mop_moe_train_step_host_async(ctx, o["x"], o["dY"], weights["W_r"], weights["bias"],
                                                  weights["W_gate"], weights["W_up"], weights["W_down"], o["Y"],
                                                  o["dX"], o["dgate"], *dW)
        else:
            binding.mop_moe_forward_host_async(ctx, o["x"], weights["W_r"], weights["bias"], weights["W_gate"],
                                               weights["W_up"], weights["W_down"], o["Y"], o["idx"], o["gate"])
    binding.mop_host_drain(ctx)
    binding.mop_poll(ctx)
    ref_ctx = binding.context_for(w)
    for i, (h, o) in enumerate(zip(hosts, outs)):
        inp = dict(weights)
        inp["x"] = h["x"].cuda()
        if backward:
            inp["dY"] = h["dY"].cuda()
        buf = binding.LayerBuffers(w)
        binding.forward(ref_ctx, inp, buf)
        if backward:
            binding.backward(ref_ctx, inp, buf)
        torch.cuda.synchronize()
        assert torch.equal(o["Y"], buf.Y.cpu()), f"Y of step {i}"
        if backward:
            assert torch.equal(o["dX"], buf.dX.cpu()) and torch.equal(o["dgate"], buf.dgate.cpu()), f"step {i}"
        else:
            assert torch.equal(o["idx"], buf.idx.cpu()) and torch.equal(o["gate"], buf.gate.cpu()), f"step {i}"
    if backward:   # dW holds the last step's gradients
        for got, name in zip(dW, ("dW_gate", "dW_up", "dW_down")):
            assert torch.equal(got, getattr(buf, name)), name


def test_pipelined_host_entry_points_need_their_context_mode():
    w = synth.small("c1_tiny", T=8, d=64, E=4, k=2, f=64, seed=24)
    ctx = binding.context_for(w, host_io=True)
    with pytest.raises(binding.MopError) as e:
        binding.mop_host_drain(ctx)
    assert e.value.code == 6


ROUTER_BWD = [
    synth.small("c1_tiny", T=200, d=128, E=8, k=2, f=64, backward=True, seed=30),                       # softmax
    synth.small("c3_trillion", T=300, d=192, E=40, k=8, f=64, backward=True, seed=31),                  # sigmoid + post bias
    synth.small("c3_trillion", T=130, d=64, E=33, k=3, f=64, bias_mode=2, backward=True, seed=32),      # sigmoid, pre-logit bias
    synth.small("c2_mid", T=257, d=72, E=12, k=12, f=64, bias_mode=2, bias_std=0.1, backward=True, seed=33),  # softmax, k = E
]


@pytest.mark.parametrize("w", ROUTER_BWD, ids=lambda w: f"{w.name}-T{w.T}d{w.d}E{w.E}k{w.k}s{w.score_fn}b{w.bias_mode}")
def test_router_backward_matches_oracle(w):
    host = synth.make_inputs(w, "cpu")
    if w.bias_mode and host["bias"] is None:
        host["bias"] = torch.randn(w.E) * 0.1
    inp = to_dev(host)
    ctx = binding.context_for(w)
    buf = binding.LayerBuffers(w)
    logits = torch.empty((w.T, w.E), dtype=torch.float32, device="cuda")
    binding.mop_moe_route(ctx, inp["x"], inp["W_r"], inp["bias"], buf.idx, buf.gate, logits)
    binding.mop_moe_permute(ctx, inp["x"], buf.idx, buf.counts, buf.offsets, buf.perm_row, buf.row_src, buf.Xp)
    g = torch.Generator().manual_seed(w.seed)
    dgate = torch.randn((w.T, w.k), generator=g).cuda()
    dX0 = (torch.randn((w.T, w.d), generator=g) * 0.5).to(torch.bfloat16).cuda()
    dX = dX0.clone()
    dWr = torch.full((w.d, w.E), 7.0, device="cuda")
    dbias = torch.full((w.E,), 7.0, device="cuda")
    binding.mop_moe_route_bwd(ctx, logits, inp["bias"], buf.idx, buf.gate, dgate, buf.Xp, buf.offsets, buf.perm_row,
                              inp["W_r"], dWr, dbias, dX)
    torch.cuda.synchronize()
    bias = None if host["bias"] is None else host["bias"].numpy()
    idx = buf.idx.cpu().numpy()
    dz, dWr_ref, dXr_ref, db_ref = oracle.route_bwd(synth.bits(host["x"]), host["W_r"].numpy(), bias, w.k, w.score_fn,
                                                    w.bias_mode, idx, dgate.cpu().numpy())
    assert rel_fro(dWr.cpu().numpy(), dWr_ref) < 1e-5
    assert np.max(np.abs(dbias.cpu().numpy() - db_ref)) <= 1e-5 * max(1.0, np.abs(db_ref).max())
    # dX = bf16(dX_in + router part): one bf16 rounding of the sum
    want = dX0.float().cpu().numpy().astype(np.float64) + dXr_ref
    got = dX.float().cpu().numpy()
    assert np.max(np.abs(got - want)) <= 2.0 ** -8 * np.maximum(1.0, np.abs(want)).max()
    assert rel_fro(got, want) < 4e-3


@pytest.mark.parametrize("T,d,E,k", [(100, 328, 160, 4),      # 16 warps per block of dW_r, the last block of columns partly filled
                                     (150, 264, 300, 3),      # 8 warps, experts with fewer rows than warps
                                     (900, 264, 300, 7),      # 8 warps, up to 40 rows per expert: more than four per warp for some
                                     (1, 392, 4, 4), (33, 136, 3, 2), (5000, 264, 6, 2)],  # dX: fewer tokens than warps, half a piece, many rounds
                         ids=lambda v: str(v))
def test_router_backward_with_many_blocks_matches_oracle(T, d, E, k):
    test_router_backward_matches_oracle(synth.small("c3_trillion", T=T, d=d, E=E, k=k, f=64, bias_mode=2, backward=True, seed=34))


def test_backward_with_recomputation_equals_backward_with_stash():
    """Activation checkpointing: forward without the G, U stash, backward recomputes them from Xp."""
    w = synth.small("c2_mid", T=700, d=256, E=10, k=3, f=192, backward=True, seed=40)
    host, inp, _, ref = run(w)
    ctx = binding.Context(w.T, w.d, w.E, w.k, w.f, w.score_fn, w.bias_mode, 2)
    buf = binding.LayerBuffers(w)
    binding.mop_moe_route(ctx, inp["x"], inp["W_r"], inp["bias"], buf.idx, buf.gate)
    binding.mop_moe_permute(ctx, inp["x"], buf.idx, buf.counts, buf.offsets, buf.perm_row, buf.row_src, buf.Xp)
    binding.mop_moe_expert_ffn_fwd(ctx, buf.Xp, buf.offsets, buf.row_src, buf.gate, inp["W_gate"], inp["W_up"],
                                   inp["W_down"], None, None, buf.H, buf.Yp)
    binding.mop_moe_combine(ctx, buf.Yp, buf.perm_row, buf.Y)
    binding.mop_moe_expert_ffn_bwd(ctx, inp["dY"], buf.Xp, None, None, None, buf.offsets, buf.perm_row, buf.row_src,
                                   buf.gate, inp["W_gate"], inp["W_up"], inp["W_down"], buf.dX, buf.dW_gate, buf.dW_up,
                                   buf.dW_down, buf.dgate)
    binding.mop_poll(ctx)
    for n in ("Y", "dX", "dgate", "dW_gate", "dW_up", "dW_down"):
        assert torch.equal(getattr(buf, n), getattr(ref, n)), n
    plain = binding.context_for(w)                      # a context without the recompute buffers refuses
    with pytest.raises(binding.MopError) as e:
        binding.mop_moe_expert_ffn_bwd(plain, inp["dY"], buf.Xp, None, None, None, buf.offsets, buf.perm_row,
                                       buf.row_src, buf.gate, inp["W_gate"], inp["W_up"], inp["W_down"], buf.dX,
                                       buf.dW_gate, buf.dW_up, buf.dW_down, buf.dgate)
    assert e.value.code == 6


def test_random_small_shapes_match_oracle():
    """Seeded random shapes: E not a multiple of 32, k from 1 to E, d and f multiples of 8 (scalar
    kernels) or of 64 (tensor-core kernels), tokens that leave experts empty."""
    rng = np.random.default_rng(1234)
    for i in range(10):
        E = int(rng.integers(1, 70))
        k = int(rng.integers(1, min(E, 8) + 1))
        if i % 2:
            d, f = int(rng.integers(1, 5)) * 64, int(rng.integers(1, 5)) * 64
        else:
            d, f = int(rng.integers(2, 20)) * 8, int(rng.integers(2, 20)) * 8
        T = int(rng.integers(1, 400))
        mode = [(0, 0), (1, 1), (1, 2), (0, 2), (1, 0)][i % 5]
        w = synth.small("c1_tiny", T=T, d=d, E=E, k=k, f=f, score_fn=mode[0], bias_mode=mode[1], bias_std=0.05,
                        backward=True, seed=100 + i)
        check_layer(w, binding.GEMM_AUTO)


def test_a_wait_that_runs_out_is_reported_and_the_context_stays_usable():
    """Failure path without a fault: a device-side wait on a barrier that nothing completes gives up
    after its limit, records a code, the kernel returns; mop_poll reports MOP_ERR_TIMEOUT once, and
    the same context then runs the layer correctly."""
    w = synth.small("c1_tiny", backward=True)
    host = synth.make_inputs(w, "cpu")
    inp = to_dev(host)
    ctx = binding.context_for(w)
    buf = binding.LayerBuffers(w)
    binding.mop_selftest_wait_timeout(ctx, 20_000_000)          # about 10 ms of SM cycles
    with pytest.raises(binding.MopError) as e:
        binding.mop_poll(ctx)
    assert e.value.code == 7
    binding.mop_poll(ctx)                                        # the word was cleared
    binding.forward(ctx, inp, buf)
    binding.backward(ctx, inp, buf)
    binding.mop_poll(ctx)
    check_integers(w, host, buf)


@pytest.mark.parametrize("T,d,E", [(17, 72, 9), (16, 64, 8),          # one chain per thread, tile edges of 16 x 8
                                   (2001, 136, 33), (2001, 72, 62), (1984, 64, 64),       # 32 x 32 tiles, W rows at every alignment
                                   (4100, 136, 33), (4096, 64, 64), (8200, 64, 260),       # 64 x 32 tiles
                                   (9000, 200, 34), (12000, 72, 127)])                     # 64 x 64 tiles
def test_exact_scoring_shapes_give_the_contract_chains(T, d, E):
    w = synth.small("c2_mid", T=T, d=d, E=E, k=2, f=64, seed=48)
    inp = synth.make_inputs(w, "cuda")
    ctx = binding.context_for(w, route_path=binding.ROUTE_EXACT)
    buf = binding.LayerBuffers(w)
    z = torch.empty((T, E), dtype=torch.float32, device="cuda")
    binding.mop_moe_route(ctx, inp["x"], inp["W_r"], None, buf.idx, buf.gate, z)
    acc = torch.zeros((T, E), dtype=torch.float64, device="cuda")
    for i in range(d):     # one fp32 rounding per step: the product of a bf16 and an fp32 number and the sum are exact enough in fp64
        acc = (acc + inp["x"][:, i:i + 1].double() * inp["W_r"][i].double()).float().double()
    # (a sum that fp64 rounds onto an fp32 tie is the only way to differ: at most a handful of last bits)
    differ = z.double() != acc
    assert int(differ.sum()) <= 1e-6 * z.numel() + 1 and torch.allclose(z.double(), acc, rtol=1e-6, atol=1e-6)
    idx, _ = oracle.route(synth.bits(inp["x"][:300]), inp["W_r"].cpu().numpy(), None, 2, w.score_fn, w.bias_mode)
    assert np.array_equal(buf.idx[:300].cpu().numpy(), idx[:300])


@pytest.mark.parametrize("T,d,E", [(40, 1000, 9),                        # 16 x 8: the ring of stages around, the last one partly filled
                                   (1500, 776, 17), (4000, 8, 8),        # 32 x 8, and a single stage of 8 steps
                                   (1300, 520, 40), (1300, 456, 41),     # 32 x 32
                                   (4100, 392, 62), (8200, 328, 65),     # 64 x 32
                                   (9472, 328, 64), (9000, 456, 34),     # 64 x 64, two blocks on an SM
                                   (12000, 456, 127)])                   # 64 x 64, one
def test_exact_scoring_with_more_steps_than_its_ring_holds(T, d, E):
    test_exact_scoring_shapes_give_the_contract_chains(T, d, E)


FAST_ROUTE = [
    synth.small("c3_trillion", T=1000, d=512, E=256, k=8, f=64, seed=60),                  # sigmoid + post-score bias
    synth.small("c3_trillion", T=777, d=320, E=64, k=3, f=64, bias_mode=2, seed=61),        # sigmoid, bias before the score
    synth.small("c2_mid", T=900, d=256, E=128, k=6, f=64, seed=62),                         # softmax
    synth.small("c3_trillion", T=300, d=192, E=1024, k=32, f=64, seed=63),                  # the selection's limits
    synth.small("c2_mid", T=257, d=64, E=64, k=32, f=64, seed=64),                          # half of the experts picked
    synth.small("c3_trillion", T=130, d=7168, E=384, k=8, f=64, seed=65),                   # the long chains of configs 3-5
    synth.small("c3_trillion", T=600, d=448, E=64, k=4, f=64, seed=66),                     # one narrow tile of experts, K in halves
    synth.small("c3_trillion", T=520, d=512, E=320, k=8, f=64, seed=67),                    # a wide tile and 64 more experts
]


@pytest.mark.parametrize("w", FAST_ROUTE, ids=lambda w: f"{w.name}-T{w.T}d{w.d}E{w.E}k{w.k}s{w.score_fn}b{w.bias_mode}")
def test_tensor_core_scoring_gives_the_indices_of_the_exact_chains(w):
    """Logits from three bf16 pieces of W_r on the tensor cores, the contract's chain only where the order is in
    doubt: indices and their order equal the oracle's (and the exact path's) bit for bit, gates within tolerance,
    and the returned logits are the chain's value or within the documented bound of it."""
    host = synth.make_inputs(w, "cpu")
    inp = to_dev(host)
    out = {}
    for path in (binding.ROUTE_EXACT, binding.ROUTE_TENSOR):
        ctx = binding.context_for(w, route_path=path)
        idx = torch.empty((w.T, w.k), dtype=torch.int32, device="cuda")
        gate = torch.empty((w.T, w.k), dtype=torch.float32, device="cuda")
        logits = torch.empty((w.T, w.E), dtype=torch.float32, device="cuda")
        binding.mop_moe_route(ctx, inp["x"], inp["W_r"], inp["bias"], idx, gate, logits)
        binding.mop_poll(ctx)
        out[path] = (idx.cpu().numpy(), gate.cpu().numpy(), logits.cpu().numpy(), binding.mop_route_stats(ctx))
    xb = synth.bits(host["x"])
    ref_idx, ref_gate, ref_z, _ = oracle.route(xb, host["W_r"].numpy(), np_bias(host), w.k, w.score_fn, w.bias_mode,
                                               want_logits=True)
    for path, (idx, gate, z, stats) in out.items():
        assert np.array_equal(idx, ref_idx), f"indices, route path {path}"
        assert np.all(np.abs(gate - ref_gate) <= 1e-6 + 1e-5 * np.abs(ref_gate)), f"gates, route path {path}"
    assert np.array_equal(out[binding.ROUTE_EXACT][2], ref_z)                       # the chain, bit for bit
    assert out[binding.ROUTE_EXACT][3] == (0, 0, 0)
    # the approximate logits stay inside the bound the selection relies on (and far inside it)
    z = out[binding.ROUTE_TENSOR][2]
    xn = np.linalg.norm(oracle.bf16_bits_to_f64(xb), axis=1)
    wmax = np.linalg.norm(host["W_r"].numpy().astype(np.float64), axis=0).max()
    eps = 24.0 * 2.0 ** -24 * xn * wmax
    err = np.abs(z.astype(np.float64) - ref_z.astype(np.float64)).max(1)
    assert np.all(err <= eps), float((err / eps).max())
    tokens, chains, beyond = out[binding.ROUTE_TENSOR][3]
    print(f"{w.name} T={w.T} d={w.d} E={w.E}: logit error {err.max():.2e} = {float((err / eps).max()):.3f} of the bound; "
          f"{tokens} of {w.T} tokens re-evaluated, {chains} chains")
    assert 0 <= tokens <= w.T and chains >= tokens and beyond == 0
    assert float((err / eps).max()) < 0.5


@pytest.mark.parametrize("w", [
    synth.small("c4_skew", T=1501, d=64, E=64, k=4, f=64, skew=True, seed=71),              # one stage of the row, experts without pairs
    synth.small("c4_skew", T=1300, d=448, E=320, k=16, f=64, skew=True, seed=72),           # many experts with a few pairs past a tile
    synth.small("c2_mid", T=900, d=320, E=1024, k=8, f=64, seed=73),                        # softmax: picks' gates only, E at its largest
], ids=lambda w: f"T{w.T}d{w.d}E{w.E}k{w.k}s{w.score_fn}")
def test_tensor_core_scoring_with_most_tokens_in_doubt(w):
    """Enough listed tokens for the chains to be evaluated expert by expert (one long column of W_r widens the error bound
    of them all); every pair of a router without weights."""
    inp = synth.make_inputs(w, "cuda")
    inp["W_r"][:, 5] *= 64.0
    for Wr in (inp["W_r"], torch.zeros_like(inp["W_r"])):
        ctx = binding.context_for(w, route_path=binding.ROUTE_TENSOR)
        exact = binding.context_for(w, route_path=binding.ROUTE_EXACT)
        out = []
        for c in (ctx, exact):
            idx = torch.empty((w.T, w.k), dtype=torch.int32, device="cuda")
            gate = torch.empty((w.T, w.k), dtype=torch.float32, device="cuda")
            binding.mop_moe_route(c, inp["x"], Wr, inp["bias"], idx, gate)
            binding.mop_poll(c)
            out.append((idx, gate))
        assert torch.equal(out[0][0], out[1][0])
        assert torch.all((out[0][1] - out[1][1]).abs() <= 1e-6 + 1e-5 * out[1][1].abs())
        tokens, chains, beyond = binding.mop_route_stats(ctx)
        assert beyond == 0 and chains >= tokens
        if Wr is inp["W_r"]:
            assert tokens >= 6 * 148
        elif not w.bias_mode:
            assert (tokens, chains) == (w.T, w.T * w.E)


def test_tensor_core_scoring_can_be_captured_behind_other_work():
    """Side stream, emptied lists and dependent launches inside a graph, after a copy and a join of two streams."""
    w = synth.small("c3_trillion", T=1000, d=512, E=256, k=8, f=64, seed=75)
    inp = synth.make_inputs(w, "cuda")
    ctx = binding.context_for(w, route_path=binding.ROUTE_TENSOR)
    want, got = ((torch.empty((w.T, w.k), dtype=torch.int32, device="cuda"), torch.empty((w.T, w.k), device="cuda")) for _ in range(2))
    binding.mop_moe_route(ctx, inp["x"], inp["W_r"], inp["bias"], *want)
    torch.cuda.synchronize()
    x, W_r = torch.zeros_like(inp["x"]), torch.zeros_like(inp["W_r"])
    side, other, graph = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(graph, stream=side):
            other.wait_stream(side)
            with torch.cuda.stream(other):
                W_r.copy_(inp["W_r"])
            x.copy_(inp["x"])
            side.wait_stream(other)
            binding.mop_moe_route(ctx, x, W_r, inp["bias"], *got, stream=side)
    for _ in range(3):
        for t in (x, W_r, *got):
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    binding.mop_poll(ctx)


def test_tensor_core_scoring_with_equal_and_duplicate_keys():
    """W_r = 0 makes all keys of a token equal (every expert is re-evaluated and the lower ids win); two equal
    columns of W_r make one exact tie per token that only the chain can order."""
    w = synth.small("c2_mid", T=96, d=128, E=64, k=4, f=64, seed=66)
    host = synth.make_inputs(w, "cpu")
    for mode in ("zero", "duplicate"):
        Wr = torch.zeros_like(host["W_r"]) if mode == "zero" else host["W_r"].clone()
        if mode == "duplicate":
            Wr[:, 40] = Wr[:, 3]
        ctx = binding.context_for(w, route_path=binding.ROUTE_TENSOR)
        idx = torch.empty((w.T, w.k), dtype=torch.int32, device="cuda")
        gate = torch.empty((w.T, w.k), dtype=torch.float32, device="cuda")
        binding.mop_moe_route(ctx, host["x"].cuda(), Wr.cuda(), None, idx, gate)
        binding.mop_poll(ctx)
        ref_idx, ref_gate = oracle.route(synth.bits(host["x"]), Wr.numpy(), None, w.k, w.score_fn, w.bias_mode)
        assert np.array_equal(idx.cpu().numpy(), ref_idx), mode
        assert np.all(np.abs(gate.cpu().numpy() - ref_gate) <= 1e-6 + 1e-5 * np.abs(ref_gate)), mode
        if mode == "zero":
            assert binding.mop_route_stats(ctx) == (w.T, w.T * w.E, 0)


def test_tensor_core_scoring_refuses_shapes_it_cannot_take():
    with pytest.raises(binding.MopError) as e:
        binding.Context(64, 64, 40, 2, 64, route_path=binding.ROUTE_TENSOR)      # E not a multiple of 64
    assert e.value.code == 6
