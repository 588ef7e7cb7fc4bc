"""Parity of the tensor-core products (dense, 2:4-sparse, Venom-gathered) with float64 products of
the oracle's masked matrices. Inputs to the sparse kernels are the ORACLE's packed operands, so a
metadata-layout or gather mistake in the kernel cannot hide behind the GPU's own packer."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_06183_b200 import binding, synth
from util import to_dev, bits, f32, rel_fro, assert_close_elementwise, Guarded

pytestmark = pytest.mark.gpu
TOL = 1e-2      # relative Frobenius error, bf16 outputs vs float64-accumulated reference


def _f64(b):
    return oracle.bf16_to_f32(b).astype(np.float64)


@pytest.mark.parametrize("a_k,b_k", [(True, True), (True, False), (False, True), (False, False)])
@pytest.mark.parametrize("M,N,K", [(128, 256, 64), (384, 512, 448), (256, 256, 128), (512, 768, 1024)])
def test_dense_gemm_layouts(a_k, b_k, M, N, K):
    A = synth.normal_bf16((M, K) if a_k else (K, M), 0, 1, seed=1, stream=M + K)
    B = synth.normal_bf16((N, K) if b_k else (K, N), 0, 1, seed=2, stream=N + K)
    C, ws = binding.sf_gemm_dense(to_dev(A), a_k, to_dev(B), b_k)
    assert binding.sf_check_status(ws) == binding.SF_OK
    Af = _f64(A) if a_k else _f64(A).T
    Bf = _f64(B) if b_k else _f64(B).T
    assert rel_fro(f32(C), Af @ Bf.T) < TOL
    assert_close_elementwise(f32(C), Af @ Bf.T, K, "dense product")


def test_dense_gemm_exact_small_integers():
    # integer data: every product and partial sum is exact, so the result must match exactly
    rng = np.random.default_rng(0)
    A = synth.f32_to_bf16_bits(rng.integers(-3, 4, size=(128, 128)).astype(np.float32))
    B = synth.f32_to_bf16_bits(rng.integers(-3, 4, size=(256, 128)).astype(np.float32))
    C, ws = binding.sf_gemm_dense(to_dev(A), True, to_dev(B), True)
    assert binding.sf_check_status(ws) == binding.SF_OK
    assert np.array_equal(f32(C), (_f64(A) @ _f64(B).T).astype(np.float32))


@pytest.mark.parametrize("Mr,Nc,K", [(128, 256, 128), (256, 512, 640), (384, 256, 1024), (1024, 768, 2048)])
def test_sparse24_gemm_against_oracle_packing(Mr, Nc, K):
    W = synth.prune_sweep_matrix(Mr, K, seed=Mr + K, tie_frac=0.1)
    W = synth.f32_to_bf16_bits(synth.bf16_bits_to_f32(W) * 50.0)       # O(1) magnitudes
    X = synth.normal_bf16((Nc, K), 0, 1, seed=3, stream=K)
    p = oracle.prune24(W, group_dim=1, mode=0)
    meta = torch.from_numpy(p.meta.view(np.int16)).cuda()
    Ct, ws = binding.sf_gemm_sparse24(to_dev(p.vals), meta, to_dev(X))
    assert binding.sf_check_status(ws) == binding.SF_OK
    ref = _f64(X) @ _f64(p.dense).T                                     # [Nc, Mr] = X W_s^T
    assert Ct.shape == (Nc, Mr)
    assert rel_fro(f32(Ct), ref) < TOL
    assert_close_elementwise(f32(Ct), ref, K, "2:4 product")


@pytest.mark.parametrize("b_k", [True, False])
@pytest.mark.parametrize("Mr,Nc,K", [(256, 256, 128), (512, 768, 1152)])
def test_sparse24_gemm_row_major_output(b_k, Mr, Nc, K):
    W = synth.prune_sweep_matrix(Mr, K, seed=Mr + K + 1, tie_frac=0.1)
    W = synth.f32_to_bf16_bits(synth.bf16_bits_to_f32(W) * 50.0)
    B = synth.normal_bf16((Nc, K) if b_k else (K, Nc), 0, 1, seed=4, stream=K)
    p = oracle.prune24(W, group_dim=1, mode=0)
    meta = torch.from_numpy(p.meta.view(np.int16)).cuda()
    C, ws = binding.sf_gemm_sparse24_rm(to_dev(p.vals), meta, to_dev(B), b_k)
    assert binding.sf_check_status(ws) == binding.SF_OK
    Bf = _f64(B) if b_k else _f64(B).T
    assert rel_fro(f32(C), _f64(p.dense) @ Bf.T) < TOL
    assert_close_elementwise(f32(C), _f64(p.dense) @ Bf.T, K, "2:4 product, row-major output")


@pytest.mark.parametrize("a_k,b_k", [(True, True), (False, False)])
@pytest.mark.parametrize("M,N,K", [(8320, 8192, 64),      # one k-stage: the epilogue is the tile's time; half-empty last row
                                   (4096, 16640, 512),
                                   (8320, 8192, 576)])    # nine: the ring of stages turns inside a tile
def test_dense_gemm_output_beyond_the_l2(a_k, b_k, M, N, K):
    # small integers: every partial sum is exact in float32, only the bf16 rounding of the result is left
    g = torch.Generator(device="cuda")
    g.manual_seed(K)
    ints = lambda *s: torch.randint(-3, 4, s, generator=g, device="cuda")
    A, B = ints(M, K), ints(N, K)
    dev = lambda t, kmajor: (t if kmajor else t.T).to(torch.bfloat16).contiguous()
    out = Guarded((M, N), torch.bfloat16)
    C, ws = binding.sf_gemm_dense(dev(A, a_k), a_k, dev(B, b_k), b_k, C_out=out.t)
    assert binding.sf_check_status(ws) == binding.SF_OK
    out.check("dense product")
    assert torch.equal(C, (A.double() @ B.double().T).to(torch.bfloat16))


@pytest.mark.parametrize("K", [768, 1088])         # nine rounds of 12 k-stages (the next launch is let in late) and of 17 (at the start)
def test_dense_gemm_read_by_the_next_launch(K):
    """Each product is the operand of the next launch, which is set up while it runs; three turns through one pair of buffers."""
    g = torch.Generator(device="cuda")
    g.manual_seed(K)
    ints = lambda *s: torch.randint(-1, 2, s, generator=g, device="cuda").to(torch.bfloat16)
    M, N = 2688, 14848
    C, D = (torch.empty(s, dtype=torch.bfloat16, device="cuda") for s in ((M, N), (M, 256)))
    ws = torch.zeros(binding.sf_gemm_workspace_size(M, K), dtype=torch.uint8, device="cuda")
    operands = [(ints(M, K), ints(N, K), ints(256, N)) for _ in range(3)]
    got = []
    for A, B, E in operands:
        binding.sf_gemm_dense(A, True, B, True, C_out=C, workspace=ws)
        binding.sf_gemm_dense(C, True, E, True, C_out=D, workspace=ws)
        got.append(D.clone())
    assert binding.sf_check_status(ws) == binding.SF_OK
    for (A, B, E), d in zip(operands, got):
        c = (A.double() @ B.double().T).to(torch.bfloat16)             # integers: exact in float32, one rounding to bf16
        assert float((c.double().abs() @ E.double().abs().T).max()) < 2.0 ** 24
        assert torch.equal(d, (c.double() @ E.double().T).to(torch.bfloat16))


def _integer_24_product(Mr, Nc, K, b_k, run):
    """Small integers: every partial sum is exact in float32, so only the bf16 rounding of the result is left."""
    rng = np.random.default_rng(Mr + Nc)
    W = rng.integers(-3, 4, size=(Mr, K)).astype(np.float32)
    B = rng.integers(-3, 4, size=(Nc, K)).astype(np.float32)
    p = oracle.prune24(synth.f32_to_bf16_bits(W), group_dim=1, mode=0)
    meta = torch.from_numpy(p.meta.view(np.int16)).cuda()
    C, ws = run(to_dev(p.vals), meta, to_dev(synth.f32_to_bf16_bits(B if b_k else np.ascontiguousarray(B.T))))
    assert binding.sf_check_status(ws) == binding.SF_OK
    return bits(C), synth.f32_to_bf16_bits(oracle.bf16_to_f32(p.dense) @ B.T)


# The stores of row-major products: half-empty last tiles, several tiles to a CTA pair, the shortest reduction. Exact on small integers,
# nothing written outside the result. Some of these sizes take narrow tiles, which store from registers (dense with
# K = 64, E4M3 dense, 2:4 512 x 1792); test_stores_on_the_tiles_named has the full-width ones by name.
@pytest.mark.parametrize("kind,Mr,Nc,K", [("dense", 2688, 4864, 64), ("dense", 5248, 2304, 320),
                                          ("sparse24", 256, 18944, 128), ("sparse24", 9728, 512, 256),
                                          ("sparse24", 6400, 4352, 128), ("sparse24", 512, 1792, 384),
                                          ("fp8", 4096, 4608, 256), ("fp8", 256, 18944, 512), ("fp8_dense", 2560, 4864, 128)])
def test_full_width_stores_stay_inside_the_result(kind, Mr, Nc, K):
    g = torch.Generator(device="cuda")
    g.manual_seed(Mr + K)
    ints = lambda *s: torch.randint(-3, 4, s, generator=g, device="cuda")
    A, B = ints(Mr, K), ints(Nc, K)
    out = Guarded((Mr, Nc), torch.bfloat16)
    bf = lambda t: t.to(torch.bfloat16)
    if kind == "dense":
        _, ws = binding.sf_gemm_dense(bf(A), True, bf(B), True, C_out=out.t)
    elif kind == "sparse24":
        vals, meta, A = binding.sf_prune24_compress(bf(A), 1, 0, want_dense=True)
        _, ws = binding.sf_gemm_sparse24_rm(vals, meta, bf(B), True, C_out=out.t)
    else:
        q = lambda t: binding.sf_fp8_quantize(bf(t), 1.0)
        if kind == "fp8":
            vals, meta, A = binding.sf_prune24_compress_fp8(bf(A), 0, 1.0, want_dense=True)
            A = A.view(torch.float8_e4m3fn)
            _, ws = binding.sf_gemm_fp8_sparse24(vals, meta, q(B), 1.0, C_out=out.t)
        else:
            _, ws = binding.sf_gemm_fp8_dense(q(A), q(B), 1.0, C_out=out.t)
    assert binding.sf_check_status(ws) == binding.SF_OK
    out.check(kind)
    assert torch.equal(out.t, bf(A.double() @ B.double().T))


def _tiles_24(Mr, Nc, K, transposed=False):
    """(rows, columns) of the tiles of a 2:4 product: y3 of a step is the row-major one, y1 the transposed one."""
    if transposed:
        plan = binding.sf_ffn_step_plan(binding.make_desc(Nc, K, Mr, 64, 8, flags=binding.SF_FFN_UNFUSED_ACT))
        return plan.y1_rows, plan.y1_cols
    plan = binding.sf_ffn_step_plan(binding.make_desc(Mr, Nc, K, 64, 8))
    return plan.y3_rows, plan.y3_cols


# The same on stated tiles. The dense products (E4M3 ones too) have seven rounds of tiles and more, of at least four k-stages: a narrower
# tile costs more per column and saves at most a seventh of the last round, so that no estimate takes one.
@pytest.mark.parametrize("kind,Mr,Nc,K,rows", [("dense", 2688, 14848, 256, 256),      # half-empty last row of tiles
                                               ("dense", 14976, 2304, 320, 256),
                                               ("fp8_dense", 2560, 14848, 512, 256),
                                               ("sparse24", 8448, 8192, 512, 256),    # overlapping accumulators, fourteen tiles to a pair
                                               ("sparse24", 256, 18944, 256, 256),    # one tile to a pair
                                               ("sparse24", 6400, 4352, 256, 512),    # last row half empty, narrow last column of 96
                                               ("sparse24", 9728, 512, 256, 512),
                                               ("sparse24", 3328, 4864, 256, 512),    # more narrow tiles than two per idle pair: round robin
                                               ("fp8", 4096, 4608, 512, 512), ("fp8", 8448, 8192, 1024, 256),
                                               ("fp8", 256, 18944, 512, 256),
                                               ("fp8", 6400, 4352, 256, None)])       # one k-stage (the plan starts at 256 in bf16)
def test_stores_on_the_tiles_named(kind, Mr, Nc, K, rows):
    if kind in ("sparse24", "fp8") and rows:      # E4M3: the rule and the width of a bf16 product with half the reduction
        assert _tiles_24(Mr, Nc, K if kind == "sparse24" else K // 2) == (rows, 224 if rows == 512 else 256)
    test_full_width_stores_stay_inside_the_result(kind, Mr, Nc, K)


@pytest.mark.parametrize("b_k", [True, False])
@pytest.mark.parametrize("Mr,Nc,K", [(8192, 8192, 512),    # 512-row tiles, a narrow last column of 128
                                     (8448, 4352, 512),    # the same, last tile row half empty, narrow column of 96
                                     (8192, 7168, 384),    # whole columns only
                                     (512, 256, 1024)])    # fewer tiles than CTA pairs
def test_sparse24_gemm_tile_shapes(b_k, Mr, Nc, K):
    got, ref = _integer_24_product(Mr, Nc, K, b_k, lambda v, m, b: binding.sf_gemm_sparse24_rm(v, m, b, b_k))
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("b_k", [True, False])
@pytest.mark.parametrize("Mr,Nc,K,rows", [(4352, 16640, 768, 256),   # beyond the L2, the longest reduction of that rule
                                          (8192, 8192, 256, 256),    # the smallest square beyond it
                                          (7680, 6400, 512, 512)])   # within it: a narrow last column of 128
def test_sparse24_gemm_short_reductions_about_the_l2(b_k, Mr, Nc, K, rows):
    assert binding.sf_ffn_step_plan(binding.make_desc(Mr, Nc, K, 64, 4)).y3_rows == rows     # y3 is this product
    got, ref = _integer_24_product(Mr, Nc, K, b_k, lambda v, m, b: binding.sf_gemm_sparse24_rm(v, m, b, b_k))
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("Mr,Nc,K", [(37632, 256, 128), (256, 7680, 128), (8576, 4864, 512)])    # 256-row tiles
def test_sparse24_gemm_tile_shapes_transposed_output(Mr, Nc, K):
    got, ref = _integer_24_product(Mr, Nc, K, True, binding.sf_gemm_sparse24)
    assert np.array_equal(got, np.ascontiguousarray(ref.T))


@pytest.mark.parametrize("Mr,Nc,K,tile", [(8576, 4864, 512, (256, 224)),     # half-empty last row, narrow last column of 160
                                          (256, 7680, 256, (256, 64)),       # one row of tiles
                                          (2688, 2304, 2048, (512, 224)),    # 512-row tiles: 128 rows in the last, column of 64
                                          (2944, 2560, 2048, (512, 224)),    # 384 rows in the last: its second half is half empty; 96
                                          (19072, 512, 2048, (512, 224))])   # two tiles to some pairs
def test_transposed_stores_on_the_tiles_named(Mr, Nc, K, tile):
    assert _tiles_24(Mr, Nc, K, transposed=True) == tile
    out = Guarded((Nc, Mr), torch.bfloat16)
    got, ref = _integer_24_product(Mr, Nc, K, True, lambda v, m, b: binding.sf_gemm_sparse24(v, m, b, Ct_out=out.t))
    out.check("transposed product")
    assert np.array_equal(got, np.ascontiguousarray(ref.T))


@pytest.mark.parametrize("Mr,Nc,K", [(4096, 8192, 512), (8192, 8192, 512)])    # set up while the metadata is converted, and after it
def test_sparse24_gemm_transposed_output_call_after_call(Mr, Nc, K):
    """Two operands in turn through one workspace: each product has to read the metadata that its own call converted."""
    rng = np.random.default_rng(K)
    B = rng.integers(-3, 4, size=(Nc, K)).astype(np.float32)
    packed = [oracle.prune24(synth.f32_to_bf16_bits(rng.integers(-3, 4, size=(Mr, K)).astype(np.float32)), group_dim=1, mode=0)
              for _ in range(2)]
    dev = [(to_dev(p.vals), torch.from_numpy(p.meta.view(np.int16)).cuda()) for p in packed]
    x = to_dev(synth.f32_to_bf16_bits(B))
    ws = torch.zeros(binding.sf_gemm_workspace_size(Mr, K), dtype=torch.uint8, device="cuda")
    outs = [torch.empty((Nc, Mr), dtype=torch.bfloat16, device="cuda") for _ in range(6)]
    for i, out in enumerate(outs):
        binding.sf_gemm_sparse24(*dev[i % 2], x, Ct_out=out, workspace=ws)
    assert binding.sf_check_status(ws) == binding.SF_OK
    # integers: exact in float32, one rounding to bf16
    refs = [synth.f32_to_bf16_bits(B @ oracle.bf16_to_f32(p.dense).T) for p in packed]
    for i, out in enumerate(outs):
        assert np.array_equal(bits(out), refs[i % 2])


def test_sparse24_gemm_one_hot_metadata_probe():
    """Each kept value is a distinct power of two in an otherwise zero row and B is an identity
    slice, so the output says which K position every stored value was multiplied with."""
    Mr, Nc, K = 128, 256, 128
    rng = np.random.default_rng(5)
    W = np.zeros((Mr, K), dtype=np.float32)
    for r in range(Mr):
        for g in range(K // 4):
            pos = sorted(rng.choice(4, size=2, replace=False))
            W[r, 4 * g + pos[0]] = 1.0 + (g % 7)
            W[r, 4 * g + pos[1]] = -(1.0 + (g % 5))
    Wb = synth.f32_to_bf16_bits(W)
    p = oracle.prune24(Wb, 1, 0)
    assert np.array_equal(p.dense, Wb)
    X = np.zeros((Nc, K), dtype=np.float32)
    X[np.arange(K), np.arange(K)] = 1.0                                  # first K rows: identity
    Ct, ws = binding.sf_gemm_sparse24(to_dev(p.vals), torch.from_numpy(p.meta.view(np.int16)).cuda(),
                                      to_dev(synth.f32_to_bf16_bits(X)))
    assert binding.sf_check_status(ws) == binding.SF_OK
    got = f32(Ct)                                                        # [Nc, Mr]; rows < K give W^T
    assert np.array_equal(got[:K].T, W)
    assert not got[K:].any()


@pytest.mark.parametrize("T,F,Nc,V,M", [(128, 256, 256, 128, 8), (256, 1024, 512, 128, 8), (256, 512, 256, 64, 8),
                                        (128, 1024, 256, 128, 16), (128, 512, 256, 64, 4),
                                        # Table 5's group widths: 93.75 % and 96.875 % sparse
                                        (256, 2048, 512, 128, 32), (256, 2048, 256, 64, 32),
                                        (256, 4096, 512, 128, 64), (128, 4096, 256, 64, 64), (384, 2048, 768, 128, 64)])
def test_venom_gemm_against_oracle_packing(T, F, Nc, V, M):
    P = synth.normal_bf16((T, F), 0.2, 1.0, seed=T + F + M)
    Bt = synth.normal_bf16((F, Nc), 0, 1, seed=7, stream=F)
    a = oracle.vnm_sparsify(P, V=V, M=M)
    meta = torch.from_numpy(a.meta.view(np.int16)).cuda()
    colidx = torch.from_numpy(a.colidx).cuda()
    out = Guarded((T, Nc), torch.bfloat16)
    C, ws = binding.sf_gemm_venom(to_dev(a.vals), meta, colidx, to_dev(Bt), V, M, C_out=out.t)
    assert binding.sf_check_status(ws) == binding.SF_OK
    out.check("Venom product output")
    ref = _f64(a.dense) @ _f64(Bt)
    assert rel_fro(f32(C), ref) < TOL
    assert_close_elementwise(f32(C), ref, 4 * F // M, "Venom product")


def test_gemm_shape_errors():
    A = torch.zeros((100, 64), dtype=torch.bfloat16, device="cuda")
    B = torch.zeros((256, 64), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(binding.SparseFFNError) as e:
        binding.sf_gemm_dense(A, True, B, True)
    assert e.value.status == binding.SF_ERR_SHAPE


def test_bounded_wait_runs_out_and_is_reported():
    """A wait on a barrier that nothing completes gives up after its clock budget, the kernel sets
    the status word and returns; the host reads SF_ERR_TIMEOUT once, then SF_OK again, and the
    context keeps working."""
    ws = torch.zeros((256,), dtype=torch.uint8, device="cuda")
    assert binding.sf_check_status(ws) == binding.SF_OK
    binding.sf_selftest_wait_expiry(ws, budget_clocks=1_000_000)
    assert binding.sf_check_status(ws) == binding.SF_ERR_TIMEOUT
    assert binding.sf_check_status(ws) == binding.SF_OK              # reported once, then cleared
    A = synth.normal_bf16((128, 64), 0, 1, seed=1)
    B = synth.normal_bf16((256, 64), 0, 1, seed=2)
    Cm, ws2 = binding.sf_gemm_dense(to_dev(A), True, to_dev(B), True)
    assert binding.sf_check_status(ws2) == binding.SF_OK
    assert rel_fro(f32(Cm), _f64(A) @ _f64(B).T) < TOL


@pytest.mark.parametrize("budget", [200_000, 1_000_000, 3_000_000])
def test_an_expired_wait_is_one_answer_for_the_warp(budget):
    """The self-test completes the barrier right after lane 0 has given up, so the other lanes of the warp see it complete;
    the status word is set only if all of them were told that the wait failed."""
    ws = torch.zeros((256,), dtype=torch.uint8, device="cuda")
    for _ in range(3):
        binding.sf_selftest_wait_expiry(ws, budget_clocks=budget)
        assert binding.sf_check_status(ws) == binding.SF_ERR_TIMEOUT
