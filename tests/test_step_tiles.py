"""The tile shapes of the sparse step's products, each reached by a step of its own.

The widths are chosen by estimated clocks, so a shape in a test runs what the rules give it and not what the test was written
for. Every case here states the tiles it is for; that the rules still give them is checked on the host through
sf_ffn_step_plan, and the step itself is checked on the GPU at sizes with several tiles to a CTA pair and with ragged last
tiles. Operands are small integers: every product, partial sum and stored gradient sum is an integer below 2^24 (asserted
from the inputs), so all outputs of a correct step are known exactly, up to one rounding to bf16."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_06183_b200 import binding, synth
from util import to_dev, bits, f32, Guarded

W2_FD, Y1 = binding.SF_FFN_W2_FD, binding.SF_FFN_SAVE_Y1

# (T, D, F, V, M, flags) -> what the plan has to say
CASES = {
    # y1 with the V:N:M selection of groups of eight in its epilogue: two accumulators, six tiles to a pair
    "vnm8_192_columns": ((2816, 256, 7296, 64, 8, 0), dict(y1_selects=1, y1_cols=192)),
    "vnm8_128_columns_v64": ((3968, 1280, 1408, 64, 8, 0), dict(y1_selects=1, y1_cols=128)),
    "vnm8_128_columns_v128": ((2688, 256, 2944, 128, 8, 0), dict(y1_selects=1, y1_cols=128)),
    # y1 with the row-wise choice of M = 4 in its epilogue, dy1 on the 2:4 mask, at 224 columns
    "act24_224_columns_v64": ((1920, 1408, 5504, 64, 4, W2_FD), dict(y1_selects=1, y1_cols=224, dy1_cols=224)),
    "act24_224_columns_v128": ((1920, 1408, 5504, 128, 4, 0), dict(y1_selects=1, y1_cols=224, dy1_cols=224)),
    # dy1 on the mask of a wide V:N:M group: 224 columns, 256 with the accumulators alternating, a run-time width
    "drelu_m16_224_columns": ((1024, 768, 9728, 64, 16, 0), dict(y1_selects=0, dy1_rows=256, dy1_cols=224)),
    "drelu_m16_256_columns": ((768, 1024, 15872, 128, 16, 0), dict(dy1_rows=256, dy1_cols=256)),
    "drelu_m16_160_columns": ((768, 512, 9728, 64, 16, W2_FD), dict(dy1_rows=256, dy1_cols=160)),
    "drelu_m32_224_columns": ((1024, 768, 10240, 128, 32, 0), dict(dy1_rows=256, dy1_cols=224)),
    "drelu_m32_256_columns": ((1024, 1024, 12288, 64, 32, W2_FD), dict(dy1_rows=256, dy1_cols=256)),
    # y3 and dX at 256 columns with the accumulators alternating, half-empty last row and column, four tiles to a pair
    "plain_256_columns": ((4224, 4224, 512, 64, 8, 0), dict(y3_rows=256, y3_cols=256)),
    # both weight gradients in one launch, CTA pairs that go from the first product's tiles to the second's
    "shared_gradients_256_columns": ((256, 640, 7040, 64, 8, 0), dict(weight_grad_launches=1, weight_grad_cols=256)),
    "shared_gradients_160_columns": ((256, 640, 6272, 64, 8, 0), dict(weight_grad_launches=1, weight_grad_cols=160)),
    "shared_gradients_256_columns_fd": ((256, 640, 7552, 64, 8, W2_FD), dict(weight_grad_launches=1, weight_grad_cols=256)),
    "shared_gradients_128_columns_fd": ((256, 640, 7040, 64, 8, W2_FD), dict(weight_grad_launches=1, weight_grad_cols=128)),
}


def _tiles(rows, cols, tile_rows, tile_cols):
    return -(-rows // tile_rows) * -(-cols // tile_cols)


@pytest.mark.parametrize("name", CASES)
def test_the_rules_give_each_case_the_tiles_it_is_for(name):
    (T, D, F, V, M, flags), want = CASES[name]
    plan = binding.sf_ffn_step_plan(binding.make_desc(T, D, F, V, M, flags=flags))
    assert {k: getattr(plan, k) for k in want} == want
    # several tiles to a CTA pair in the product that the case is for
    if "weight_grad_cols" in want:
        m2, n2 = (F, D) if flags & W2_FD else (D, F)
        first = _tiles(m2, n2, 256, plan.weight_grad_cols)
        tiles = first + _tiles(F, D, 256, plan.weight_grad_cols)
        assert first % plan.cta_pairs != 0 and first > plan.cta_pairs       # some pairs take tiles of both products
    elif name.startswith("plain"):
        tiles = _tiles(T, D, plan.y3_rows, plan.y3_cols)
        assert T % plan.y3_rows == 128 and D % plan.y3_cols == 128
    elif name.startswith("drelu"):
        tiles = _tiles(F, T, plan.dy1_rows, plan.dy1_cols)
    else:
        tiles = _tiles(F, T, plan.y1_rows, plan.y1_cols)
        assert F % plan.y1_rows == 128                                      # the last row of tiles is half empty
    assert tiles > 2 * plan.cta_pairs


def test_plan_of_a_step_on_the_host():
    """The plan follows the flags and refuses what the step refuses."""
    plan = lambda *a, **k: binding.sf_ffn_step_plan(binding.make_desc(*a, **k))
    assert plan(4096, 2048, 8192, 64, 8).y1_selects == 1
    assert plan(4096, 2048, 8192, 64, 8, flags=binding.SF_FFN_UNFUSED_ACT).y1_selects == 0
    assert plan(4096, 2048, 8192, 64, 8).weight_grad_launches == 1
    lean = plan(4096, 2048, 8192, 64, 8, flags=binding.SF_FFN_PACKED_GRAD_OPERANDS)
    assert (lean.weight_grad_launches, lean.weight_grad_cols) == (2, 0)
    assert plan(16384, 8192, 28672, 64, 8).dy1_rows == 512
    with pytest.raises(binding.SparseFFNError) as e:
        plan(1000, 256, 1024, 64, 8)
    assert e.value.status == binding.SF_ERR_SHAPE
    assert binding.lib().sf_ffn_step_plan(None, None) == binding.SF_ERR_NULL


# Whole steps, in one launch and in two: see gemm_dual_tn_pays
@pytest.mark.parametrize("T,D,F,launches", [(1920, 1408, 5504, 1),      # four rounds of tiles either way: the launch counts (170.3 us, 174.7)
                                            (4096, 1024, 2816, 1),      # slightly narrower tiles apart, worth less than a launch (151.1, 155.2)
                                            (10240, 1920, 1792, 1),     # (324.7, 326.4)
                                            (4096, 384, 28032, 2),      # narrower tiles apart, worth more (707, 708)
                                            (16256, 384, 28032, 2),     # (2413, 2390)
                                            (15744, 256, 11648, 2),     # (837, 834)
                                            (4096, 3072, 12288, 1),     # sixteen rounds either way (1.000)
                                            (16384, 1536, 23040, 1),    # fifteen rounds or sixteen, long ones (0.985 and 1.004)
                                            (16384, 2048, 28672, 2),    # twenty-five or twenty-six, longer (1.015)
                                            (8192, 4096, 16384, 2),     # as many rounds, long ones (1.004)
                                            (16384, 8192, 28672, 2)])   # (1.022)
def test_weight_gradients_share_a_launch_where_that_ends_sooner(T, D, F, launches):
    assert binding.sf_ffn_step_plan(binding.make_desc(T, D, F, 64, 8)).weight_grad_launches == launches


@pytest.mark.parametrize("T,F", [(2048, 28672), (4096, 4096), (8192, 2048)])
@pytest.mark.parametrize("D", [256, 512])
def test_short_reductions_with_many_tiles_keep_wide_tiles(T, F, D):
    """A tile costs its hand-overs however narrow it is: a product with two to four k-stages and enough tiles for every CTA
    pair must not be cut into 32- or 64-column ones (measured 1.2 to 1.6 times the time)."""
    plan = binding.sf_ffn_step_plan(binding.make_desc(T, D, F, 64, 8, flags=binding.SF_FFN_UNFUSED_ACT))
    assert plan.y1_rows == 512 or plan.y1_cols >= 128


@pytest.mark.parametrize("T,D", [(8192, 16384), (16384, 8192), (4096, 16640)])
@pytest.mark.parametrize("F", [256, 512, 768])
def test_short_reductions_beyond_the_l2_stay_on_256_row_tiles(T, D, F):
    """y3 and dX with two to six k-stages and an output larger than the L2 last as long as their writes, on 512-row tiles as on
    256-row ones, and the smaller tiles leave fewer pairs idle at the end; longer reductions go to 512-row tiles, smaller
    outputs by the clocks."""
    y3_rows = lambda *a: binding.sf_ffn_step_plan(binding.make_desc(*a, 64, 8)).y3_rows
    assert y3_rows(T, D, F) == 256
    assert y3_rows(T, D, 16 * F) == 512
    assert y3_rows(8192, 7296, F) == 512


def _integers(shape, limit, seed):
    return np.random.default_rng(seed).integers(-limit, limit + 1, size=shape).astype(np.float32)


def _step(X, W1, W2, dY, T, D, F, V, M, flags):
    desc = binding.make_desc(T, D, F, V, M, flags=flags)
    nctx, nws = binding.sf_ffn_workspace_size(desc)
    w2_fd = bool(flags & W2_FD)
    bufs = dict(context=Guarded(nctx, zero=True), workspace=Guarded(nws, zero=True), Y=Guarded((T, D), torch.bfloat16),
                dX=Guarded((T, D), torch.bfloat16), dW1=Guarded((F, D), torch.bfloat16),
                dW2=Guarded((F, D) if w2_fd else (D, F), torch.bfloat16))
    ctx, ws, Y, dX, dW1, dW2 = (b.t for b in bufs.values())
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda().to(torch.bfloat16)
    x, w1, w2, dy = dev(X), dev(W1), dev(W2.T if w2_fd else W2), dev(dY)
    binding.sf_sparse_ffn_fwd(desc, x, w1, w2, Y, ctx, ws)
    binding.sf_sparse_ffn_bwd(desc, dy, x, w1, w2, ctx, dX, dW1, dW2, ws)
    assert binding.sf_check_status(ws) == binding.SF_OK
    for name, b in bufs.items():
        b.check(name)
    G = F // M
    view = lambda buf, field: binding.sf_ctx_view(desc, buf, field)
    out = dict(vals=bits(view(ctx, binding.SF_CTX_Y2_VALS)).reshape(T, 2 * G),
               relu=bits(view(ctx, binding.SF_CTX_RELU_VALS)).reshape(T, 2 * G),
               meta=bits(view(ctx, binding.SF_CTX_META)).reshape(T, G // 4),
               colidx=view(ctx, binding.SF_CTX_COLIDX).cpu().numpy().reshape(T // V, G, 4),
               Y=f32(Y), dX=f32(dX), dW1=f32(dW1), dW2=f32(dW2).T if w2_fd else f32(dW2))
    if M == 8:
        m24 = bits(view(ctx, binding.SF_CTX_Y2_META24)).reshape(T, F // 16)
        out["y2_24"] = oracle.decompress24(bits(view(ctx, binding.SF_CTX_Y2_VALS24)).reshape(T, F // 2), m24)
        out["relu_24"] = oracle.decompress24(bits(view(ctx, binding.SF_CTX_RELU_VALS24)).reshape(T, F // 2), m24)
        dy1 = oracle.decompress24(bits(view(ws, binding.SF_CTX_DY1_VALS24)).reshape(T, F // 2), m24)
    else:
        dy1 = oracle.decompress_vnm(bits(view(ws, binding.SF_CTX_DY1_VALS)).reshape(T, 2 * G), out["meta"], out["colidx"], V=V, M=M)
    out["dy1"] = oracle.bf16_to_f32(dy1)
    if flags & Y1:
        out["y1"] = f32(view(ctx, binding.SF_CTX_Y1)).reshape(T, F)
    return out


def _exact_product(A, B, what):
    """A [m, k] B [k, n] in float64 on the GPU; no partial sum, in whatever order, may leave float32's integers."""
    a, b = (torch.from_numpy(np.ascontiguousarray(x)).cuda().double() for x in (A, B))
    assert float((a.abs() @ b.abs()).max()) < 2.0 ** 24, what
    return (a @ b).float().cpu().numpy()


def _round(x):
    return oracle.bf16_to_f32(synth.f32_to_bf16_bits(x)).reshape(x.shape)


@pytest.mark.gpu
@pytest.mark.parametrize("name", CASES)
def test_step_on_these_tiles_is_exact(name):
    (T, D, F, V, M, flags), _ = CASES[name]
    X, dY = _integers((T, D), 1, 1), _integers((T, D), 1, 2)
    W1, W2 = _integers((F, D), 2, 3), _integers((D, F), 2, 4)
    prune = lambda w: oracle.bf16_to_f32(oracle.prune24(synth.f32_to_bf16_bits(w).reshape(w.shape), 1, 0).dense)
    y1 = _round(_exact_product(X, prune(W1).T, "y1"))
    act = oracle.vnm_sparsify(synth.f32_to_bf16_bits(y1).reshape(y1.shape), V=V, M=M)
    y2, relu = oracle.bf16_to_f32(act.dense), np.where(act.mask, np.maximum(y1, 0), 0).astype(np.float32)
    dy2 = _exact_product(dY, prune(np.ascontiguousarray(W2.T)).T, "dy2")
    assert (2.0 * np.abs(dy2) * relu).max() < 2.0 ** 24
    dy1 = _round(2.0 * dy2 * relu)
    ref = dict(vals=act.vals, relu=act.relu_vals, meta=act.meta, colidx=act.colidx, dy1=dy1,
               Y=_round(_exact_product(y2, W2.T, "Y")), dX=_round(_exact_product(dy1, W1, "dX")),
               dW1=_round(_exact_product(dy1.T, X, "dW1")), dW2=_round(_exact_product(dY.T, y2, "dW2")))
    if M == 8:
        ref.update(y2_24=act.dense, relu_24=synth.f32_to_bf16_bits(relu).reshape(relu.shape))
    for f in (flags, flags | Y1):                       # without and with y1 kept: other buffers, the same step
        got = _step(X, W1, W2, dY, T, D, F, V, M, f)
        if f & Y1:
            assert np.array_equal(got.pop("y1"), y1)
        assert got.keys() == ref.keys()
        for k in ref:
            assert np.array_equal(got[k], ref[k]), k
    if M == 8:                                          # and the selection as a kernel of its own on a stored y1
        got = _step(X, W1, W2, dY, T, D, F, V, M, flags | binding.SF_FFN_UNFUSED_ACT)
        for k in ref:
            assert np.array_equal(got[k], ref[k]), ("two kernels", k)


# y1 with SquaredReLU and dy1 of the dense step write two results a tile through TMA at full width only. 522 tiles on 74 pairs are eight
# rounds of ten k-stages, so that no estimate takes a narrower one; the last row and the last column of tiles are half empty.
@pytest.mark.gpu
@pytest.mark.parametrize("flags", [0, W2_FD])
def test_dense_step_on_full_width_tiles_is_exact(flags):
    T, D, F = 2176, 640, 14720
    X, dY, W1, W2 = (_integers(shape, 1, seed) for seed, shape in enumerate([(T, D), (T, D), (F, D), (D, F)], 11))
    w2_fd = bool(flags & W2_FD)
    desc = binding.make_desc(T, D, F, 64, 8, flags=flags)
    nctx, nws = binding.sf_ffn_workspace_size(desc)
    bufs = dict(context=Guarded(nctx, zero=True), workspace=Guarded(nws, zero=True), Y=Guarded((T, D), torch.bfloat16),
                dX=Guarded((T, D), torch.bfloat16), dW1=Guarded((F, D), torch.bfloat16),
                dW2=Guarded((F, D) if w2_fd else (D, F), torch.bfloat16))
    ctx, ws, Y, dX, dW1, dW2 = (b.t for b in bufs.values())
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda().to(torch.bfloat16)
    x, w1, w2, dy = dev(X), dev(W1), dev(W2.T if w2_fd else W2), dev(dY)
    binding.sf_dense_ffn_fwd(desc, x, w1, w2, Y, ctx, ws)
    binding.sf_dense_ffn_bwd(desc, dy, x, w1, w2, ctx, dX, dW1, dW2, ws)
    assert binding.sf_check_status(ws) == binding.SF_OK
    for name, b in bufs.items():
        b.check(name)
    y1 = _round(_exact_product(X, W1.T, "y1"))
    relu = np.maximum(y1, 0)
    h = _round(relu * relu)
    dy1 = _round(2.0 * _exact_product(dY, W2, "dy2") * relu)
    n = T * F * 2
    assert np.array_equal(f32(ctx[:n].view(torch.bfloat16)).reshape(T, F), y1)
    assert np.array_equal(f32(ctx[n:2 * n].view(torch.bfloat16)).reshape(T, F), h)
    assert np.array_equal(f32(Y), _round(_exact_product(h, W2.T, "Y")))
    assert np.array_equal(f32(dX), _round(_exact_product(dy1, W1, "dX")))
    assert np.array_equal(f32(dW1), _round(_exact_product(dy1.T, X, "dW1")))
    assert np.array_equal(f32(dW2).T if w2_fd else f32(dW2), _round(_exact_product(dY.T, h, "dW2")))
