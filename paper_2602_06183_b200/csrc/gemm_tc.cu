// Tensor-core products of the FFN step on sm_100a: tcgen05.mma with TMEM accumulators, operands
// staged in shared memory by TMA, warp-specialised roles.
//
//   mode DENSE     D[M,N] = A[M,K] B[N,K]^T                       (Eqs. 1-8; weight-gradient products)
//   mode SPARSE24  A is 2:4-compressed (values [M,K/2] + metadata) (Algorithm 1 line 4, Algorithm 2 line 2)
//   mode VENOM     A is V:N:M-compressed; B rows are gathered by the block's kept columns
//                  (Algorithm 1 line 7, Algorithm 2 line 5)
//
// CTA = 6 warps: warp 0 TMA producer, warp 1 MMA issuer (+ TMEM owner), warps 2-5 epilogue (each
// owns the 32 TMEM lanes of its quadrant). Tile 128 x 256, persistent over tiles (m fastest).
// Venom mode adds warps 6-17, which gather the kept rows of B into the 128B-swizzled MN-major
// layout the MMA reads: 8 warps issue TMA row gathers, 4 warps issue 16-byte cp.async copies.
// A stage holds A (16 KB dense, 8 KB compressed), B (32 KB) and, for sparse modes, one 2 KB metadata
// atom covering 128 rows x 128 logical K (copied smem -> TMEM by tcgen05.cp every second stage);
// 4 stages dense, 5 stages sparse.
// Dense mode double-buffers the 256-column accumulator so the epilogue of tile i overlaps the main
// loop of tile i+1; sparse modes keep one accumulator plus the metadata columns.
// Every mbarrier wait is bounded; on expiry the CTA raises a flag in the status word and leaves.
// The waits that carry no clock budget, and what ends each of them:
//   TMEM allocation (before griddepcontrol.wait, so possibly while the predecessor still runs): two CTAs of these kernels do
//     not fit one SM (kExclusiveSmem below), so the columns are free as soon as a CTA is placed; should another library's
//     kernel hold some, it gives them back when it ends, and it does not wait for this one: a kernel behind this one in the
//     stream is placed after every CTA here has triggered, which it does after its allocation
//   cluster barriers: set-up, which every CTA of a placed cluster reaches without waiting for anything but the above; teardown,
//     which every role reaches because its own waits are bounded
//   named barriers of a set of epilogue warps: entered by all four or by none (the vote behind the accumulator wait)
//   griddepcontrol.wait: the predecessor, whose CTAs are all placed by then (it triggers from each of them) and bounded likewise
#include "sf_common.cuh"
#include "tc_ptx.cuh"
#include "gemm_tc.cuh"
#include "sparse_fmt.cuh"

namespace sf {

namespace {

using namespace ptx;

constexpr int BM = 128, BN = 256;
constexpr int kMaxStages = 5;
constexpr int kBStageBytes = 32768, kMetaStageBytes = 2048;
// dense: A 16 KB + B 32 KB, 4 stages; sparse modes: A 8 KB (stored half) + B 32 KB + metadata 2 KB, 5 stages
__host__ __device__ constexpr int a_stage_bytes(bool sparse) { return sparse ? 8192 : 16384; }
__host__ __device__ constexpr int stage_bytes(bool sparse) {
  return a_stage_bytes(sparse) + kBStageBytes + (sparse ? kMetaStageBytes : 0);
}
__host__ __device__ constexpr int num_stages(bool sparse) { return sparse ? 5 : 4; }
constexpr int kEpiWarpBytes = 32 * 32 * 2;                                            // 32 x 32 bf16, or 16 token pairs x 32
constexpr int kEpiStageBytes = 4 * kEpiWarpBytes;                                     // 4 warps
__host__ __device__ constexpr int smem_bytes(bool sparse) {
  return 1024 /*align slack*/ + num_stages(sparse) * stage_bytes(sparse) + kEpiStageBytes + 256 /*barriers*/;
}
constexpr int kThreads = 192;                 // dense / 2:4 modes: producer, MMA, 4 epilogue warps
constexpr int kThreadsVenom = 576;            // + 8 TMA-gather warps and 4 cp.async-gather warps
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kMetaTmemCol = 256;

// More than half of an SM's 228 KB: a kernel that allocates all of TMEM takes this much, so that no two of its CTAs, nor one
// of the kernel before it, share an SM (the second would sit in its TMEM allocation until the first ends).
constexpr int kExclusiveSmem = 228 * 1024 / 2 + 1;
static_assert(smem_bytes(false) >= kExclusiveSmem && smem_bytes(true) >= kExclusiveSmem, "one CTA per SM");

struct SmemCtl {
  uint64_t full[kMaxStages];
  uint64_t empty[kMaxStages];
  uint64_t tmem_full[2];
  uint64_t tmem_empty[2];
  uint32_t tmem_base;
  int abort_flag;
};

// Tile raster: bands of kRasterM tile rows, m fastest inside a band. The tiles that run at the same
// time then form a near-square block (8 x ~9 for 74 CTA pairs), so a wave touches ~17 operand
// panels instead of ~65 and operands larger than the L2 are not re-read once per tile column.
constexpr int kRasterM = 8;
__device__ __forceinline__ void tile_coords(int tile, int num_m, int num_n, int& mt, int& nt) {
  const int per_band = kRasterM * num_n;
  const int band = tile / per_band, rem = tile - band * per_band;
  const int m_start = band * kRasterM;
  const int gm = min(kRasterM, num_m - m_start);
  nt = rem / gm;
  mt = m_start + (rem - nt * gm);
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  return float_to_bf16_bits(lo) | (float_to_bf16_bits(hi) << 16);
}


// Which epilogues run on two sets of four warps (one set per accumulator) on CTA pairs.
__host__ __device__ constexpr bool is_drelu_t(int epi) { return epi == EPI_DRELU24_T || epi == EPI_DRELUV_T; }
__host__ __device__ constexpr bool two_sets(int epi) { return epi == EPI_VNM8 || epi == EPI_ACT24_T || is_drelu_t(epi); }
// Dense products, and the row-major 2:4 products on tiles of full width: two sets share every tile, each takes half of its columns
// (dense, where the last tile's epilogue is exposed: 1024 x 256 x 1024 17.3 -> 14.3 us; 2:4, with the store through TMA, 2048 x
// 2048 x 2048 14.9 -> 13.8, 4096 x 2048 x 1024 16.5 -> 15.3, 8192 x 16384, K = 256 117 -> 85; narrow 2:4 tiles have too few columns
// for two: 1024 x 256 x 1024 7.72 us with one set and 7.86 with two).
__host__ __device__ constexpr bool split_sets(int mode, int epi, int expand, bool var) {
  return (mode == MODE_DENSE && epi != EPI_ROUTE && !expand) || (mode == MODE_SPARSE24 && epi == EPI_STORE && !var);
}

// This warp has read its part of an accumulator for the last time: hand it back to the MMA warp.
__device__ __forceinline__ void release_accumulator(int lane, uint64_t* tmem_empty_bar) {
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive_leader(tmem_empty_bar);
}

// A tile of accumulator columns (tokens) is transposed through shared memory as words of two neighbouring
// tokens, [token pair][32 features]. This thread takes the eight features at `sp` of one pair back as two
// rows of packed features: r0 = even token, r1 = odd token. Pairs alternate which 16-byte half they fetch
// first, so that each of the two loads of a quarter-warp touches every bank exactly once.
__device__ __forceinline__ void pair_rows(const uint32_t* sp, int lane, uint32_t (&r0)[4], uint32_t (&r1)[4]) {
  const int swap = (lane >> 2) & 1;
  const uint4 q0 = *reinterpret_cast<const uint4*>(sp + 4 * swap), q1 = *reinterpret_cast<const uint4*>(sp + 4 - 4 * swap);
  const uint4 qa = swap ? q1 : q0, qb = swap ? q0 : q1;
  r0[0] = __byte_perm(qa.x, qa.y, 0x5410); r0[1] = __byte_perm(qa.z, qa.w, 0x5410);
  r0[2] = __byte_perm(qb.x, qb.y, 0x5410); r0[3] = __byte_perm(qb.z, qb.w, 0x5410);
  r1[0] = __byte_perm(qa.x, qa.y, 0x7632); r1[1] = __byte_perm(qa.z, qa.w, 0x7632);
  r1[2] = __byte_perm(qb.x, qb.y, 0x7632); r1[3] = __byte_perm(qb.z, qb.w, 0x7632);
}

// Four lanes hold a row of 64 bytes each, as four 16-byte units in registers; afterwards lane k of the four holds unit k of all four
// rows, in the order of the rows. Two exchanges, each of the half that the other side needs.
__device__ __forceinline__ void quad_transpose(uint32_t (&x)[16], int lane) {
  const bool hi = lane & 2, odd = lane & 1;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t got = __shfl_xor_sync(0xFFFFFFFFu, hi ? x[j] : x[8 + j], 2);
    if (hi) x[j] = got; else x[8 + j] = got;
  }
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t got = __shfl_xor_sync(0xFFFFFFFFu, odd ? x[8 * h + j] : x[8 * h + 4 + j], 1);
      if (odd) x[8 * h + j] = got; else x[8 * h + 4 + j] = got;
    }
}

// ---- stores through TMA -----------------------------------------------------------------------------
// What bounded the plain store: an epilogue thread holds a row, so a 16-byte store of a warp went to 32 rows, 32 cycles of the
// load/store unit's data pipe each (counted: 33 wavefronts a store; 7200 clocks for the 256 x 224 outputs of an SM in a 512-row tile;
// 56 % of the pipe's peak at 8192 x 16384, K = 128, now 14.5 %, and every sector written to the L2 in two halves), on the chain from one
// main loop to the next and in the way of the MMAs' shared-memory reads. Here a warp puts 32 x 32 results into shared memory, 64 bytes a row, and one
// thread hands them to TMA. Same box, call after call: 2:4 row-major 8192 x 16384, K = 128 115 -> 67 us, K = 1024 215 -> 167,
// K = 4096 535 -> 503; E4M3 2:4 4096 x 16384 x 4096 170 -> 150; dense 8192 x 16384, K = 128 119 -> 79, 16384 x 8192, K = 512 168 -> 131.
// Four lanes exchanging their rows' units and storing 64 bytes of eight rows per instruction gave E4M3 152 and dense K = 512 168;
// reading a 512-row tile out into registers first and handing its accumulator back before storing (the stores then run beside
// the next main loop, which they slow) 151; an evict-first hint nothing.
// 32 x 32 chunk of a tile, rounded (w: this lane's row), through one of the warp's buffers to C; rows of 64 bytes, swizzled as
// the store's tensor map expects it (64-byte swizzle), so that a thread per row writes without bank conflicts.
template <int kBufs>
__device__ __forceinline__ void store_chunk(const CUtensorMap* tmapC, uint8_t* bufs, uint32_t& buf, const uint32_t* w, int col, int row,
                                            int lane) {
  if (lane == 0) bulk_wait_read<kBufs - 1>();                              // the chunk before (or the one before that) has left
  __syncwarp();
  uint8_t* b = bufs + buf * kEpiWarpBytes;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    *reinterpret_cast<uint4*>(b + lane * 64 + ((j ^ ((lane >> 1) & 3)) << 4)) = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
  fence_proxy_async_smem();
  __syncwarp();
  if (lane == 0) {
    tma_store_2d(tmapC, b, col, row);
    bulk_commit();
  }
  if (kBufs == 2) buf ^= 1u;
}

// ---- epilogue (shared by the one-CTA and the two-CTA kernels) ---------------------------------------
// One epilogue warp owns TMEM lanes [32q, 32q+32) of a 128 x 256 accumulator tile whose first row is
// m0 and first column n0; `taddr` is the TMEM address of (lane 32q, column 0) of that accumulator.
// kTileN: accumulator columns of the tile (a multiple of 32). Columns at or beyond n_limit (a ragged last
// tile, whole 32-column chunks only since N % 32 == 0) are not stored. `part` of `parts`: the share of the tile's
// columns that this warp takes.
// A thread holds one row. EPI_STORE stores from there (16 bytes of 32 rows per instruction), or 64 bytes of eight rows after an
// exchange among four lanes where the rows are scattered (kScatter: row_map); other tiles of full width go out through TMA instead
// (epi_store_tile). Narrow tiles (run-time width), where the latency of a chunk is what counts, keep the first: with the
// exchange the step at T 1024, D 256, F 1024 took 40.4 us instead of 40.0. The exchange in the routed step at T 8192, D 4096, F 16384 in
// four experts: 1277 -> 1257 us. The two-operand epilogues of the dense step move a chunk through shared memory, 64 contiguous bytes of
// eight rows per instruction: y1 + SquaredReLU at T 4096, D 2048, F 8192 129 -> 96 us.
// kEarly: the accumulator is handed back when the first chunk has been read; the second part starts with its last chunk, so that
// the columns at either end of the tile are the first to be read.
// kTma: the two-operand epilogues hand their chunks to TMA (T 10496, D 384, F 7424, the dense step 504 -> 488 us).
template <int kEpi, int kTileN = BN, bool kEarly = false, bool kScatter = false, bool kTma = false>
__device__ __forceinline__ void epi_tile(const GemmArgs& args, uint32_t taddr, int64_t m0, int64_t n0, int64_t n_limit,
                                         int q, int lane, uint8_t* my_stage, int part = 0, int parts = 1, bool second = false,
                                         uint64_t* tmem_empty_bar = nullptr, const CUtensorMap* tmapC = nullptr,
                                         const CUtensorMap* tmapC2 = nullptr, uint32_t* buf = nullptr) {
  if constexpr (kEpi == EPI_ROUTE) {
    const int64_t row = m0 + q * 32 + lane;                                // this thread's D row
    // the row is a token, the first route_E columns its logits
    uint32_t v[32];
    tmem_ld_32x32b_x32(taddr, v);
    tmem_ld_wait_on(v);
    const int E = args.route_E;
    int best = 0;
    float bestv = __uint_as_float(v[0]);
#pragma unroll
    for (int e = 1; e < 16; ++e) {
      const float x = __uint_as_float(v[e]);
      if (e < E && x > bestv) { bestv = x; best = e; }                     // strict: ties stay with the lower expert
    }
    args.route_expert[row] = best;
    if (args.route_logits) {
#pragma unroll
      for (int e = 0; e < 16; ++e)
        if (e < E) args.route_logits[row * E + e] = __uint_as_float(v[e]);
    }
    return;
  }
  // chunks of 32 columns (warp-uniform): this warp's part of the live ones
  const int live = (int)min((int64_t)(kTileN / 32), (n_limit - n0) >> 5);
  const int ch0 = live * part / parts, nch = live * (part + 1) / parts;
  if (ch0 >= nch) {
    if (kEarly) release_accumulator(lane, tmem_empty_bar);
    return;
  }
  // EPI_STORE: this thread's row (formed here: inside the chunk loop the step at T 1024, D 256, F 1024 takes 38.58 us instead of 38.42)
  const int64_t row = m0 + q * 32 + lane;
  uint16_t* const crow = reinterpret_cast<uint16_t*>(second ? args.C2 : args.C) + row * (second ? args.ldc2 : args.ldc);
  // kScatter: this thread stores 16-byte unit `lane & 3` of the four rows of its four lanes
  int rows4[4];
  uint16_t* const cq = reinterpret_cast<uint16_t*>(args.C) + (lane & 3) * 8;
  if (kScatter) {
    const int r = __ldg(args.row_map + row);
#pragma unroll
    for (int i = 0; i < 4; ++i) rows4[i] = __shfl_sync(0xFFFFFFFFu, r, (lane & 28) + i);
  }
  // EPI_SQRELU, EPI_DRELU: this thread moves 16-byte unit `u` of the rows `t8 + 8 i` of a chunk.
  const int t8 = lane >> 2, u = lane & 3;
  const int64_t out = m0 + q * 32 + t8;
  // 32 x 32 bf16 in shared memory, 64 bytes a row, the four units of a row XOR-ed with bits of the row: conflict-free
  // both for a thread per row and for four threads per row.
  auto unit = [&](int r, int k) { return reinterpret_cast<uint4*>(my_stage + r * 64 + ((k ^ ((r >> 1) & 3)) << 4)); };
  auto store_rows = [&](const uint32_t (&w)[16], void* C, int64_t ldc, int64_t col0) {
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 4; ++j) *unit(lane, j) = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 4; ++i)
      *reinterpret_cast<uint4*>(reinterpret_cast<uint16_t*>(C) + (out + 8 * i) * ldc + col0 + u * 8) = *unit(t8 + 8 * i, u);
  };
  uint4 a4[4];                                                             // EPI_DRELU: y1 of the next chunk
  auto fetch = [&](int ch) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      a4[i] = __ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const uint16_t*>(args.aux) + (out + 8 * i) * args.ldaux + n0 + ch * 32 + u * 8));
  };
  if (kEpi == EPI_DRELU) fetch(ch0);
  // `v` holds (once its load is complete) the chunk's accumulator columns; `next` starts the load of the chunk after
  auto at = [&](int i) { return kEarly && part == 1 ? nch - 1 - (i - ch0) : i; };
  auto chunk = [&](int i, uint32_t (&v)[32], uint32_t (&next)[32]) {
    const int ch = at(i);
    const int64_t col0 = n0 + ch * 32;
    uint32_t w[16];
    if (kEpi == EPI_DRELU) {                                               // y1 to a thread per row
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 4; ++i) *unit(t8 + 8 * i, u) = a4[i];
      __syncwarp();
      if (ch + 1 < nch) fetch(ch + 1);
    }
    tmem_ld_wait_on(v);
    if (kEarly && i == ch0) release_accumulator(lane, tmem_empty_bar);
    if (i + 1 < nch) tmem_ld_32x32b_x32(taddr + at(i + 1) * 32, next);
    if (kEpi == EPI_DRELU) {                                               // C = bf16(2 * acc * relu(aux))
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint4 a = *unit(lane, j);
        const uint32_t aw[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float r0 = fmaxf(bf16_bits_to_float(aw[e] & 0xFFFFu), 0.f);
          const float r1 = fmaxf(bf16_bits_to_float(aw[e] >> 16), 0.f);
          w[4 * j + e] = pack_bf16x2(__fmul_rn(__fmul_rn(2.f, __uint_as_float(v[8 * j + 2 * e])), r0),
                                     __fmul_rn(__fmul_rn(2.f, __uint_as_float(v[8 * j + 2 * e + 1])), r1));
        }
      }
    } else if (kEpi == EPI_STORE) {
      const float al = args.out_scale != 0.f ? args.out_scale : 1.f;        // x 1 is exact: bf16 products unchanged
#pragma unroll
      for (int j = 0; j < 16; ++j)
        w[j] = pack_bf16x2(__fmul_rn(__uint_as_float(v[2 * j]), al), __fmul_rn(__uint_as_float(v[2 * j + 1]), al));
    } else {
#pragma unroll
      for (int j = 0; j < 16; ++j) w[j] = pack_bf16x2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
    }
    if (kEpi == EPI_STORE) {
      if constexpr (kScatter) {
        quad_transpose(w, lane);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (rows4[i] >= 0)
            *reinterpret_cast<uint4*>(cq + rows4[i] * args.ldc + col0) = make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
      } else {
        uint4* c = reinterpret_cast<uint4*>(crow + col0);
#pragma unroll
        for (int j = 0; j < 4; ++j) c[j] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
      }
    } else if (kEpi != EPI_STORE_T) {
      // kTma: EPI_SQRELU has both buffers for its outputs, EPI_DRELU stages y1 in the first
      if constexpr (kTma && kEpi == EPI_SQRELU) store_chunk<2>(tmapC, my_stage, *buf, w, (int)col0, (int)m0 + q * 32, lane);
      else if constexpr (kTma) store_chunk<1>(tmapC, my_stage + kEpiWarpBytes, *buf, w, (int)col0, (int)m0 + q * 32, lane);
      else store_rows(w, args.C, args.ldc, col0);
      if (kEpi == EPI_SQRELU) {
#pragma unroll
        for (int j = 0; j < 16; ++j) w[j] = bf2_sq(bf2_relu(w[j]));
        if constexpr (kTma) store_chunk<2>(tmapC2, my_stage, *buf, w, (int)col0, (int)m0 + q * 32, lane);
        else store_rows(w, args.C2, args.ldc2, col0);
      }
    } else {
      // Transposed output: D row = feature (lane), D column = token. C is [N, M] row-major; through shared memory token by token
      // (32 16-bit stores, four 16-byte loads). With a short reduction a warp's walk from chunk to chunk is the tile's time, and this is
      // the shortest: 8192 x 16384, K = 128 74.6 us, by fragments and TMA (epi_store_t_tile) 108, by words of two tokens that are
      // taken apart again 96.5; 28672 x 2048, K = 128 38.1, 51.8 and 47.0; 4096 x 4096, K = 1024 24.9, 24.8 and 24.8.
      __syncwarp();
#pragma unroll
      for (int t = 0; t < 32; ++t)
        reinterpret_cast<uint16_t*>(unit(t, lane >> 3))[lane & 7] = (uint16_t)(w[t >> 1] >> (16 * (t & 1)));
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 4; ++i)
        *reinterpret_cast<uint4*>(reinterpret_cast<uint16_t*>(args.C) + (col0 + i * 8 + t8) * args.ldc + m0 + q * 32 + u * 8) = *unit(t8 + 8 * i, u);
    }
  };
  // two register buffers: the TMEM load of the next 32 columns is in flight while this chunk is converted
  uint32_t va[32], vb[32];
  tmem_ld_32x32b_x32(taddr + at(ch0) * 32, va);
  if constexpr (kEpi == EPI_STORE_T) {
    // Unrolled: with a short reduction this epilogue is the tile's time, and the staging of a chunk overlaps the stores of the
    // one before. 8192 x 16384, K = 128 73.5 us rolled, 71.5 unrolled; 4096 x 16384, K = 256 45.3 and 44.3.
#pragma unroll
    for (int i = 0; i < kTileN / 32; i += 2) {
      if (i >= nch) break;
      chunk(i, va, vb);
      if (i + 1 < kTileN / 32 && i + 1 < nch) chunk(i + 1, vb, va);
    }
    return;
  }
#pragma unroll 1
  for (int i = ch0; i < nch; i += 2) {
    chunk(i, va, vb);
    if (i + 1 < nch) chunk(i + 1, vb, va);
  }
}


// ---- plain and transposed stores of a whole tile -------------------------------------------------------
// kEarly: as in epi_tile.
template <int kTileN, int kBufs, bool kEarly>
__device__ __forceinline__ void epi_store_tile(const GemmArgs& args, const CUtensorMap* tmapC, uint32_t taddr, int64_t m0, int64_t n0,
                                               int64_t n_limit, int q, int lane, uint8_t* bufs, uint32_t& buf, int part, int parts,
                                               uint64_t* tmem_empty_bar) {
  const int live = (int)min((int64_t)(kTileN / 32), (n_limit - n0) >> 5);
  const int ch0 = live * part / parts, nch = live * (part + 1) / parts;
  if (ch0 >= nch) {
    if (kEarly) release_accumulator(lane, tmem_empty_bar);
    return;
  }
  const float al = args.out_scale != 0.f ? args.out_scale : 1.f;           // x 1 is exact: bf16 products unchanged
  const int row = (int)m0 + q * 32;
  auto pack = [&](float lo, float hi) { return pack_bf16x2(__fmul_rn(lo, al), __fmul_rn(hi, al)); };
  auto at = [&](int i) { return kEarly && part == 1 ? nch - 1 - (i - ch0) : i; };
  auto chunk = [&](int i, uint32_t (&v)[32], uint32_t (&next)[32]) {
    tmem_ld_wait_on(v);
    if (kEarly && i == ch0) release_accumulator(lane, tmem_empty_bar);
    if (i + 1 < nch) tmem_ld_32x32b_x32(taddr + at(i + 1) * 32, next);
    uint32_t w[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) w[j] = pack(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
    store_chunk<kBufs>(tmapC, bufs, buf, w, (int)n0 + at(i) * 32, row, lane);
  };
  uint32_t va[32], vb[32];
  tmem_ld_32x32b_x32(taddr + at(ch0) * 32, va);
#pragma unroll 1
  for (int i = ch0; i < nch; i += 2) {
    chunk(i, va, vb);
    if (i + 1 < nch) chunk(i + 1, vb, va);
  }
}

// The transposed store: D row = feature, D column = token, C is [tokens, features] row-major. The accumulator is read as the 8 x 8
// fragments that stmatrix transposes on its way to shared memory, [32 tokens][32 features], and leaves through TMA as above: the
// fewest passes over the shared memory that the main loop works on. For 512-row tiles; against words of two tokens staged by
// lane and taken apart again 16384 x 8192, K = 4096 502.9 -> 499.2 us, 4096 x 16384, K = 2048 140.4 -> 138.8.
template <int kTileN>
__device__ __forceinline__ void epi_store_t_tile(const CUtensorMap* tmapC, uint32_t taddr, int64_t m0, int64_t n0, int64_t n_limit, int q,
                                                 int lane, uint8_t* stage) {
  const int nch = (int)min((int64_t)(kTileN / 32), (n_limit - n0) >> 5);
  auto load = [&](int ch, uint32_t (&v)[32]) {
    tmem_ld_16x256b_x4(taddr + ch * 32, v);
    tmem_ld_16x256b_x4(taddr + ch * 32 + (16u << 16), v + 16);
  };
  // lane 8 k + j addresses eight features (16-byte unit k) of token j of eight: units swizzled as in store_chunk
  const uint32_t at = smem_u32(stage) + (lane & 7) * 64 + (((lane >> 3) ^ ((lane >> 1) & 3)) << 4);
  auto chunk = [&](int ch, uint32_t (&v)[32], uint32_t (&next)[32]) {
    tmem_ld_wait_on(v);
    if (ch + 1 < nch) load(ch + 1, next);
    uint32_t w[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t* x = v + 16 * (k >> 1) + 4 * i + 2 * (k & 1);
        w[i][k] = pack_bf16x2(__uint_as_float(x[0]), __uint_as_float(x[1]));
      }
    if (lane == 0) bulk_wait_read<0>();
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 4; ++i) stmatrix_x4_trans(at + i * 512, w[i][0], w[i][1], w[i][2], w[i][3]);
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) {
      tma_store_2d(tmapC, stage, (int)m0 + q * 32, (int)n0 + ch * 32);
      bulk_commit();
    }
  };
  uint32_t va[32], vb[32];
  load(0, va);
#pragma unroll 1
  for (int ch = 0; ch < nch; ch += 2) {
    chunk(ch, va, vb);
    if (ch + 1 < nch) chunk(ch + 1, vb, va);
  }
}

// ---- fused SquaredReLU + V:N:M selection (groups of eight) ---------------------------------------------
// Epilogue of the y1 product: the accumulator tile is y1^T (TMEM lane = feature, column = token), so a
// lane owns one feature column of every V x 8 block and eight neighbouring lanes own one block.
// A set of four warps works on a block of V tokens x the CTA's 128 features (16 groups):
//   pass 1  a warp reads its lanes' V accumulator columns into registers, rounded to bf16 (this is y1) as token pairs, and
//           sums the column score of Section 2.3 in float32, token by token in ascending order (the order is part of the
//           format);
//   rank    the eight lanes of a group exchange scores; the four best columns stay (ties to the lower column). Only they
//           go to shared memory, ReLU applied, four token pairs to a 16-byte store;
//   pass 2  one thread per (eight tokens, group): with the kept columns of two tokens in the halves of four words, one
//           selection serves both tokens; values, ReLU values, both metadata forms, the 2:4 view and the masked copy follow
//           by byte permutes. The masked copy's selectors belong to the group (a dropped column takes the sign byte of a
//           value that is not negative), the 2:4 view's come from a table over the pairs of columns.
// In pass 2 a warp serves all 16 groups of two tokens at a time: its stores are whole rows of the CTA's features (64 to
// 256 contiguous bytes a token).
// What bounds it: a set has two main loops' time for a tile, and what it moves through shared memory and the L1 is taken
// from theirs. With all columns parked in shared memory as [token][feature], selected token by token and the selectors
// worked out per block, a block took 7300 clocks of its set; this takes 4000. y1 at T 4096, D 2048, F 8192 102 -> 92 us,
// T 8192, D 4096, F 16384 608 -> 583 us, T 4096, D 512, F 8192 95 -> 78 us.
constexpr int kVnmStageBytes = 64 * 128;                                 // 64 tokens: [8][64 kept columns][4 token pairs]
constexpr int kVnmSetBytes = kVnmStageBytes + 16 * 4 + 16 * 8;
struct VnmTables {
  uint4 top2[16];            // of a keep mask: {Top2Entry::kept, selector of the two columns' numbers, half masks of the four}
  uint2 pair[64];            // of columns (a, b), at a + 8 b: {selectors of the 2:4 view's halves, its metadata byte}
};
__device__ __forceinline__ void vnm_tables_init(VnmTables* t, int tid) {               // 64 threads
  uint4 sel;
  uint32_t nib24;
  vnm8_pair_selectors((uint32_t)tid & 7u, (uint32_t)tid >> 3, sel, nib24);
  t->pair[tid] = make_uint2(sel.w, nib24);
  if (tid < 16) {
    const uint32_t m = (uint32_t)tid, p0 = __ffs(m) - 1u, p1 = 31u - __clz(m);
    t->top2[tid] = __popc(m) != 2 ? make_uint4(0u, 0u, 0u, 0u)
                                  : make_uint4(top2_lut_entry(m).kept, 0x4400u | p0 | (p1 << 4),
                                               (m & 1u) * 0xFFFFu | (m >> 1 & 1u) * 0xFFFF0000u,
                                               (m >> 2 & 1u) * 0xFFFFu | (m >> 3 & 1u) * 0xFFFF0000u);
  }
}
constexpr int kSetWarps = 8;                                     // two sets of four: one set per accumulator buffer
constexpr int kVnmEpiBytes = 2 * kVnmSetBytes + (int)sizeof(VnmTables);
// Byte permute with the sign mode: selector nibble 8 + i gives the sign of byte i in all eight bits.
__device__ __forceinline__ uint32_t prmt_signed(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
  return r;
}

// Barrier of one set of four epilogue warps.
__device__ __forceinline__ void set_sync(int set) { asm volatile("bar.sync %0, 128;" ::"r"(set + 1) : "memory"); }

// kCols: columns of the tile that this set takes at most; kStep: tokens in registers at a time (64: V = 64 only,
// with less code and fewer registers).
template <int kCols, int kStep>
__device__ __forceinline__ void epi_vnm8_tile(const GemmArgs& args, uint32_t taddr, int64_t m0, int64_t n0, int64_t n_limit, int q,
                                              int set, int lane, uint8_t* epi_stage, uint64_t* tmem_empty_bar) {
  const VnmTables* tables = reinterpret_cast<const VnmTables*>(epi_stage + 2 * kVnmSetBytes);
  const int64_t F = args.M;
  const int G = (int)(F >> 3);
  const int64_t g0 = m0 >> 3;                                             // the CTA's first group
  const int jm = lane & 7, gw = q * 4 + (lane >> 3);                      // pass 1: column of its group, group
  const int gl = lane & 15, psub = lane >> 4, odd = gl & 1;               // pass 2: group, which of two quads of token pairs
  const int cols = (int)min((int64_t)kCols, n_limit - n0);                // ragged last tile: whole blocks only
  if (cols <= 0) {
    release_accumulator(lane, tmem_empty_bar);
    return;
  }
  const bool tall = kStep == 128 && args.V == 128;                        // (64 otherwise)
  const uint32_t nib_mask = 0xF0000u << (4 * (gl & 3));                  // this group's nibble of its metadata word (high half)
  uint8_t* stage = epi_stage + set * kVnmSetBytes;
  uint8_t* cidx = stage + kVnmStageBytes;                                  // [16 groups][4] kept columns
  uint8_t* dsel = cidx + 16 * 4;                                           // [16 groups][8] selector byte of each column
#pragma unroll 1
  for (int c0 = 0; c0 < cols; c0 += kStep) {
    // ---- pass 1, kStep tokens (or the tile's last 64): the next 32 columns are on their way while these are worked on
    const bool both = kStep == 128 && cols - c0 > 64;
    uint32_t yp[kStep / 2], va[32], vb[32];
    auto take = [&](const uint32_t (&v)[32], int c) {
#pragma unroll
      for (int j = 0; j < 16; ++j) yp[c * 16 + j] = pack_bf16x2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
    };
    tmem_ld_32x32b_x32(taddr + (uint32_t)c0, va);
    tmem_ld_wait_on(va);
    tmem_ld_32x32b_x32(taddr + (uint32_t)(c0 + 32), vb);
    take(va, 0);
    tmem_ld_wait_on(vb);
    if (both) tmem_ld_32x32b_x32(taddr + (uint32_t)(c0 + 64), va);
    take(vb, 1);
    if constexpr (kStep == 128) {
      if (both) {
        tmem_ld_wait_on(va);
        tmem_ld_32x32b_x32(taddr + (uint32_t)(c0 + 96), vb);
        take(va, 2);
        tmem_ld_wait_on(vb);
        take(vb, 3);
      }
    }
    if (c0 + kStep >= cols) release_accumulator(lane, tmem_empty_bar);
    if (args.vn_y1) {
      if (c0 > 0) set_sync(set);
      // y1 itself, through this warp's quarter of the stage, 32 tokens at a time
      uint32_t* st = reinterpret_cast<uint32_t*>(stage + q * (kVnmStageBytes / 4));
#pragma unroll
      for (int c = 0; c < kStep / 32; ++c) {
        if (c >= 2 && !both) break;
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 16; ++j) st[j * 32 + lane] = yp[c * 16 + j];
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          uint32_t r0[4], r1[4];
          const int pr = i * 8 + (lane >> 2);
          pair_rows(st + pr * 32 + (lane & 3) * 8, lane, r0, r1);
          uint16_t* y = reinterpret_cast<uint16_t*>(args.vn_y1) + (n0 + c0 + c * 32 + 2 * pr) * F + m0 + q * 32 + (lane & 3) * 8;
          *reinterpret_cast<uint4*>(y) = make_uint4(r0[0], r0[1], r0[2], r0[3]);
          *reinterpret_cast<uint4*>(y + F) = make_uint4(r1[0], r1[1], r1[2], r1[3]);
        }
      }
      set_sync(set);                                                       // the quarters have been read
    }
    bool keep = false;
    int pos = 0;
#pragma unroll 1
    for (int h = 0; h < (both ? 2 : 1); ++h) {
      if (!tall || h == 0) {
        float score = 0.f;
        auto add = [&](int j0) {
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            yp[j0 + j] = bf2_relu(yp[j0 + j]);
            const uint32_t hp = bf2_sq(yp[j0 + j]);
            score = __fadd_rn(score, __uint_as_float(hp << 16));
            score = __fadd_rn(score, __uint_as_float(hp & 0xFFFF0000u));
          }
        };
        add(0);
        if constexpr (kStep == 128) {
          if (tall) add(32);
        }
        // ---- rank the eight columns of each group
        const uint32_t sb = __float_as_uint(score);                            // scores are >= 0: the pattern orders them
        int rank = 0;
#pragma unroll
        for (int i = 1; i < 8; ++i) {
          const uint32_t o = __shfl_xor_sync(0xFFFFFFFFu, sb, i);
          const int oj = jm ^ i;
          rank += (o > sb) || (o == sb && oj < jm);
        }
        keep = rank < 4;
        const uint32_t gbyte = (__ballot_sync(0xFFFFFFFFu, keep) >> (lane & 24)) & 0xFFu;
        pos = __popc(gbyte & ((1u << jm) - 1u));
      }
      if (c0 + h > 0) set_sync(set);                                       // the stage has been read
      if (!tall || h == 0) {
        // bytes 2 pos and 2 pos + 1 of the four kept values, or the sign (zero) of byte 1
        dsel[gw * 8 + jm] = keep ? (uint8_t)(0x10 + 0x22 * pos) : (uint8_t)0x99;
        if (keep) cidx[gw * 4 + pos] = (uint8_t)jm;
      }
      if (keep) {
        // unit of column pos: XOR-ed so that eight neighbouring groups' units of one column lie in different banks
        uint4* dst = reinterpret_cast<uint4*>(stage) + gw * 4 + (pos ^ ((gw >> 1) & 3));
#pragma unroll
        for (int u = 0; u < 8; ++u) dst[u * 64] = make_uint4(yp[4 * u], yp[4 * u + 1], yp[4 * u + 2], yp[4 * u + 3]);
      }
      if constexpr (kStep == 128) {
#pragma unroll
        for (int j = 0; j < 32; ++j) yp[j] = yp[32 + j];
      }
      set_sync(set);                                                       // the kept columns of all 128 features are in
      // ---- pass 2
      const uint32_t c4 = *reinterpret_cast<const uint32_t*>(cidx + gl * 4);
      const uint2 ds = *reinterpret_cast<const uint2*>(dsel + gl * 8);
      const int64_t t0 = n0 + c0 + 64 * h;
      if (q == 0 && psub == 0 && (!tall || h == 0))
        *reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(args.vn_colidx) + ((t0 >> (tall ? 7 : 6)) * G + g0 + gl) * 4) = c4;
      const int u = 2 * q + psub;                                            // eight tokens each
      const int64_t t = t0 + 8 * u;                                        // this thread's first token
      const int64_t at = t * G + g0 + gl;
      uint32_t* p_vals = reinterpret_cast<uint32_t*>(args.vn_vals) + at;
      uint32_t* p_relu = reinterpret_cast<uint32_t*>(args.vn_relu) + at;
      uint2* p_v24 = reinterpret_cast<uint2*>(args.vn_vals24) + at;
      uint2* p_r24 = reinterpret_cast<uint2*>(args.vn_relu24) + at;
      uint4* p_dense = args.vn_dense ? reinterpret_cast<uint4*>(args.vn_dense) + at : nullptr;
      // the metadata of four groups is one word: their first two lanes write a token each
      const int64_t atm = (t + odd) * (G >> 2) + ((g0 + gl) >> 2);
      uint16_t* p_meta = reinterpret_cast<uint16_t*>(args.vn_meta) + atm;
      uint32_t* p_m24 = reinterpret_cast<uint32_t*>(args.vn_meta24) + atm;
      // tensor-core-ordered copy: eight tokens are one column of 16-byte rows of an atom
      uint8_t* p_hw = reinterpret_cast<uint8_t*>(args.vn_meta24_hw) + meta_hw_offset(t, (m0 >> 4) + (gl >> 1), F) + odd * 16;
      const uint4* src = reinterpret_cast<const uint4*>(stage) + u * 64 + gl * 4;
      const int sw = (gl >> 1) & 3;
      uint4 x0 = src[sw], x1 = src[1 ^ sw], x2 = src[2 ^ sw], x3 = src[3 ^ sw];
      // two tokens: r_i holds kept column i of both
      auto emit = [&](uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3, int k) {
        const uint32_t e = 2u * top2_offsets_x2(bf2_sq(r0), bf2_sq(r1), bf2_sq(r2), bf2_sq(r3));
        const uint8_t* base = reinterpret_cast<const uint8_t*>(tables->top2);
        uint4 ent[2];
        ent[0] = *reinterpret_cast<const uint4*>(base + (e & 0xFFFFu));
        ent[1] = *reinterpret_cast<const uint4*>(base + (e >> 16));
        uint32_t mb[2];
#pragma unroll
        for (int d = 0; d < 2; ++d) {
          const uint32_t half = d ? 0x7632u : 0x5410u;
          const uint32_t ra = __byte_perm(r0, r1, half), rb = __byte_perm(r2, r3, half);
          const uint32_t ha = bf2_sq(ra), hb = bf2_sq(rb);
          const uint32_t packed = __byte_perm(ha, hb, ent[d].x), rpair = __byte_perm(ra, rb, ent[d].x);
          const int off = (2 * k + d) * G;
          p_vals[off] = packed;
          p_relu[off] = rpair;
          // {selectors, metadata byte} of the two columns: 8 a + 64 b
          const uint2 pe = *reinterpret_cast<const uint2*>(reinterpret_cast<const uint8_t*>(tables->pair) +
                                                           __dp4a(__byte_perm(c4, 0u, ent[d].y), 0x4008u, 0u));
          const uint32_t sel = pe.x;
          mb[d] = pe.y;
          p_v24[off] = make_uint2(__byte_perm(packed, 0u, sel), __byte_perm(packed, 0u, sel >> 16));
          p_r24[off] = make_uint2(__byte_perm(rpair, 0u, sel), __byte_perm(rpair, 0u, sel >> 16));
          if (p_dense) {
            const uint32_t za = ha & ent[d].z, zb = hb & ent[d].w;
            p_dense[off] = make_uint4(prmt_signed(za, zb, ds.x), prmt_signed(za, zb, ds.x >> 16), prmt_signed(za, zb, ds.y),
                                      prmt_signed(za, zb, ds.y >> 16));
          }
        }
        // even token in the low half, odd token in the high half
        uint32_t w = ((ent[0].x & nib_mask) >> 16) | (ent[1].x & nib_mask);
        w |= __shfl_xor_sync(0xFFFFFFFFu, w, 1);
        w |= __shfl_xor_sync(0xFFFFFFFFu, w, 2);
        uint32_t m = (mb[0] | (mb[1] << 16)) << (8 * odd);
        m |= __shfl_xor_sync(0xFFFFFFFFu, m, 1);
        const uint32_t m2 = __shfl_xor_sync(0xFFFFFFFFu, m, 2);
        *reinterpret_cast<uint16_t*>(p_hw + k * 32) = (uint16_t)(odd ? m >> 16 : m);
        if ((gl & 2) == 0) {
          const int off = 2 * k * (G >> 2);
          p_meta[off] = (uint16_t)(odd ? w >> 16 : w);
          p_m24[off] = __byte_perm(m, m2, odd ? 0x7632u : 0x5410u);
        }
      };
#pragma unroll(kStep == 128 ? 1 : 4)
      for (int k = 0; k < 4; ++k) {
        emit(x0.x, x1.x, x2.x, x3.x, k);
        x0.x = x0.y; x0.y = x0.z; x0.z = x0.w;
        x1.x = x1.y; x1.y = x1.z; x1.z = x1.w;
        x2.x = x2.y; x2.y = x2.z; x2.z = x2.w;
        x3.x = x3.y; x3.y = x3.z; x3.z = x3.w;
      }
    }
  }
}

// ---- dy1 = 2 dy2 ReLU(y1) on the activation's mask (Eq. 6) -----------------------------------------------
// Epilogue of the dy2 product: TMEM lane = feature, column = token. A chunk of 32 tokens x 32 features goes
// through shared memory as float32, [token][feature] with rows 33 words apart (conflict-free column stores);
// a lane then serves eight features of a token and fetches the accumulator values of the KEPT features only
// (EPI_DRELU24_T: two per four, positions from the metadata byte; EPI_DRELUV_T: the two of a wide V:N:M group,
// where they fall into its eight features). ReLU(y1) of the next chunk is requested while this one is worked on.
// The transposed-mask form that this replaces (every feature multiplied, 16-bit transposes both ways, one set
// of warps) issued twice the instructions and bound the product at small d_model: T 4096, D 2048, F 8192 (M = 8)
// 102 -> 82 us, T 8192, D 4096, F 16384 555 -> 523 us.
constexpr int kDreluRow = 33;
constexpr int kDreluWarpBytes = 32 * kDreluRow * 4;

// Byte-permute selectors of nibble n = p0 | p1 << 2: output byte pair of column c takes stored value 0 (bytes 1,0) if
// c == p0, value 1 (bytes 3,2) if c == p1, else the zero operand (byte 4).
__device__ __forceinline__ uint2 expand_lut_entry(uint32_t n) {
  const uint32_t sel = 0x44444444u ^ (0x54u << (8u * (n & 3u))) ^ (0x76u << (8u * (n >> 2)));
  return make_uint2(sel & 0xFFFFu, sel >> 16);
}
// One 2:4 group back to its four dense columns through the 16-entry selector table.
__device__ __forceinline__ void expand24_lut(const uint2* lut, uint32_t pair, uint32_t nib, uint32_t& w0, uint32_t& w1) {
  const uint2 s = lut[nib];
  w0 = __byte_perm(pair, 0u, s.x);
  w1 = __byte_perm(pair, 0u, s.y);
}

// kShare: the two sets work on one tile of 256 columns, four chunks each; the accumulator is handed back when the first chunk has
// been read, and the second set starts with its last one (see kOverlap in the kernel). The chunk is then staged in two halves.
template <int kEpi, int kTileN, bool kShare>
__device__ __forceinline__ bool epi_drelu_tile(const GemmArgs& args, uint32_t taddr, int64_t m0, int64_t n0, int64_t n_limit,
                                               bool live, int q, int set, int lane, float* stage, const uint2* lut,
                                               uint64_t* tmem_full_bar, uint32_t phase, volatile int* abort_flag,
                                               uint64_t* tmem_empty_bar) {
  constexpr bool kVenomMask = kEpi == EPI_DRELUV_T;
  const int t8 = lane >> 2, seg = lane & 3;
  const int64_t f = m0 + q * 32 + seg * 8;                                 // this lane's first feature
  const int nch = live ? (int)min((int64_t)(kShare ? 4 : kTileN / 32), (n_limit - n0) >> 5) : 0;
  auto at = [&](int i) { return kShare && set == 1 ? nch - 1 - i : i; };
  constexpr int kRows = kShare ? 16 : 32;                                  // tokens staged at a time
  const int64_t tok = n0 + t8;                                             // this lane's first token
  // per token: EPI_DRELU24_T four stored values + one metadata byte; EPI_DRELUV_T the group's pair + its nibble
  const int64_t g = kVenomMask ? f / args.Mv : 0;
  const int64_t s_relu = kVenomMask ? 2 * args.G : args.M >> 1, s_meta = kVenomMask ? args.G >> 1 : args.M >> 3;
  const uint8_t* p_relu = reinterpret_cast<const uint8_t*>(args.aux) + 2 * (tok * s_relu + (kVenomMask ? 2 * g : f >> 1));
  const uint8_t* p_meta = reinterpret_cast<const uint8_t*>(args.pack_meta) + tok * s_meta + (kVenomMask ? g >> 1 : f >> 3);
  uint2 r[4];
  uint32_t mb[4], c4 = 0, c4n = 0;
  auto fetch = [&](int ch) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t t = ch * 32 + i * 8;
      if (kVenomMask) r[i].x = __ldg(reinterpret_cast<const uint32_t*>(p_relu + 2 * t * s_relu));
      else            r[i] = __ldg(reinterpret_cast<const uint2*>(p_relu + 2 * t * s_relu));
      mb[i] = __ldg(p_meta + t * s_meta);
    }
    if (kVenomMask)      // a chunk lies inside one V-block (V is a multiple of 32)
      c4n = __ldg(reinterpret_cast<const uint32_t*>(args.colidx + ((n0 + ch * 32) / args.V * args.G + g) * 4));
  };
  if (nch > 0) fetch(at(0));
  if (!mbar_wait_warp(tmem_full_bar, phase, abort_flag)) return false;
  tc_fence_after();
  if (nch <= 0) {
    release_accumulator(lane, tmem_empty_bar);
    return true;
  }
  uint32_t v[32];
  tmem_ld_32x32b_x32(taddr + at(0) * 32, v);
  const float* row0 = stage + t8 * kDreluRow + seg * 8;
  uint16_t* p_dense = args.C ? reinterpret_cast<uint16_t*>(args.C) + tok * args.ldc + f : nullptr;
  const int off = kVenomMask ? (int)(f & (args.Mv - 1)) : 0;               // this lane's first column inside its group
#pragma unroll 1
  for (int ci = 0; ci < nch; ++ci) {
    const int ch = at(ci);
    tmem_ld_wait_on(v);
    if (kShare && ci == 0) release_accumulator(lane, tmem_empty_bar);
    uint2 rc[4];
    uint32_t mc[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) { rc[i] = r[i]; mc[i] = mb[i]; }
    c4 = c4n;
    if (ci + 1 < nch) fetch(at(ci + 1));
    // an off-mask entry is +0, also where the saved ReLU is zero
    auto prod = [](float x, uint32_t rb) {
      const float rv = bf16_bits_to_float(rb & 0xFFFFu);
      return rv == 0.f ? 0.f : __fmul_rn(__fmul_rn(2.f, x), rv);
    };
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (i % (kRows / 8) == 0) {                                          // the next kRows tokens
        __syncwarp();                                                      // the previous ones have been read
#pragma unroll
        for (int j = 0; j < kRows; ++j) stage[j * kDreluRow + lane] = __uint_as_float(v[i * 8 + j]);
        __syncwarp();
        if (i + kRows / 8 == 4) {
          if (ci + 1 < nch) tmem_ld_32x32b_x32(taddr + at(ci + 1) * 32, v);
          else if (!kShare) release_accumulator(lane, tmem_empty_bar);
        }
      }
      const float* row = row0 + (i % (kRows / 8)) * 8 * kDreluRow;
      const int64_t t = tok + ch * 32 + i * 8;
      uint4 o;
      if (!kVenomMask) {
        const uint32_t m = mc[i];
        const uint32_t pa = pack_bf16x2(prod(row[m & 3u], rc[i].x), prod(row[(m >> 2) & 3u], rc[i].x >> 16));
        const uint32_t pb = pack_bf16x2(prod(row[4u + ((m >> 4) & 3u)], rc[i].y), prod(row[4u + (m >> 6)], rc[i].y >> 16));
        *reinterpret_cast<uint2*>(reinterpret_cast<uint16_t*>(args.pack_vals) + t * (args.M >> 1) + (f >> 1)) = make_uint2(pa, pb);
        expand24_lut(lut, pa, m & 15u, o.x, o.y);
        expand24_lut(lut, pb, m >> 4, o.z, o.w);
      } else {
        const uint32_t nib = (mc[i] >> (4 * (g & 1))) & 15u;
        const uint32_t da = ((c4 >> (8 * (nib & 3u))) & 0xFFu) - (uint32_t)off, db = ((c4 >> (8 * (nib >> 2))) & 0xFFu) - (uint32_t)off;
        uint16_t* pv = reinterpret_cast<uint16_t*>(args.pack_vals) + t * (2 * args.G) + 2 * g;
        uint32_t va = 0, vb = 0;
        if (da < 8u) { va = float_to_bf16_bits(prod(row[da], rc[i].x)); pv[0] = (uint16_t)va; }
        if (db < 8u) { vb = float_to_bf16_bits(prod(row[db], rc[i].x >> 16)); pv[1] = (uint16_t)vb; }
        va <<= 16 * (da & 1u);
        vb <<= 16 * (db & 1u);
        const uint32_t wa = da >> 1, wb = db >> 1;                         // word of the kept column (beyond 3: not in this lane)
        o.x = (wa == 0u ? va : 0u) | (wb == 0u ? vb : 0u);
        o.y = (wa == 1u ? va : 0u) | (wb == 1u ? vb : 0u);
        o.z = (wa == 2u ? va : 0u) | (wb == 2u ? vb : 0u);
        o.w = (wa == 3u ? va : 0u) | (wb == 3u ? vb : 0u);
      }
      if (p_dense) *reinterpret_cast<uint4*>(p_dense + (int64_t)(ch * 32 + i * 8) * args.ldc) = o;
    }
  }
  return true;
}

// ---- fused SquaredReLU + 2:4 selection inside every four features of a token ------------------------------
// Epilogue of the routed y1 product and of the M = 4 step (a V x 4 block keeps all of its columns, so nothing
// but the row-wise choice is left): y1 goes through shared memory as token pairs; a lane serves eight features
// of two tokens and writes values, ReLU values, both metadata orders, the masked copy, and y1 if asked for.
// The M = 4 step ran this as a second kernel on a stored y1 before: T 1920, D 1408, F 5504, whole step 224 -> 194 us.
template <int kTileN>
__device__ __forceinline__ void epi_act24_tile(const GemmArgs& args, uint32_t taddr, int64_t m0, int64_t n0, int64_t n_limit,
                                               int q, int lane, uint32_t* stage, const uint2* lut, const Top2Entry* top2,
                                               uint64_t* tmem_empty_bar) {
  const int seg = lane & 3;
  const int64_t Fe = args.M, f = m0 + q * 32 + seg * 8;
  const int nch = (int)min((int64_t)(kTileN / 32), (n_limit - n0) >> 5);
  // Output addresses of this lane's first token; every store of the loop is a constant stride away from them. (Address
  // arithmetic written per store, with a division by V among it, was most of this epilogue's instructions.)
  const int64_t tok0 = n0 + (lane >> 2) * 2;
  uint2* p_vals = reinterpret_cast<uint2*>(args.vn_vals24) + ((tok0 * Fe + f) >> 3);           // 8-byte units: F / 8 per token
  uint2* p_relu = reinterpret_cast<uint2*>(args.vn_relu24) + ((tok0 * Fe + f) >> 3);
  uint4* p_dense = reinterpret_cast<uint4*>(args.vn_dense) + ((tok0 * Fe + f) >> 3);
  uint4* p_y1 = args.vn_y1 ? reinterpret_cast<uint4*>(args.vn_y1) + ((tok0 * Fe + f) >> 3) : nullptr;
  uint32_t* p_meta = reinterpret_cast<uint32_t*>(args.vn_meta24) + ((tok0 * Fe + f) >> 5);
  const int64_t s8 = Fe >> 3, s32 = Fe >> 5;
  // tensor-core order: a 16-token group is 256 bytes of an atom (tiles start at multiples of 32 tokens); see meta_hw_offset
  const int64_t kw = f >> 4;
  uint8_t* hw0 = reinterpret_cast<uint8_t*>(args.vn_meta24_hw) + (kw >> 3) * 2048 + (kw & 1) * 128 + ((kw >> 1) & 3) * 4 +
                 (((lane >> 2) * 2) & 7) * 16 + ((lane >> 2) >> 2) * 2;
  const uint32_t vmask = args.vn_colidx ? (uint32_t)args.V - 1u : 0u;      // V is 64 or 128
  uint32_t v[32];
  tmem_ld_32x32b_x32(taddr, v);
#pragma unroll 1
  for (int ch = 0; ch < nch; ++ch) {
    tmem_ld_wait_on(v);
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 16; ++j) stage[j * 32 + lane] = pack_bf16x2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
    __syncwarp();
    if (ch + 1 < nch) tmem_ld_32x32b_x32(taddr + (ch + 1) * 32, v);
    else              release_accumulator(lane, tmem_empty_bar);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      uint32_t y[2][4];
      pair_rows(stage + (i * 8 + (lane >> 2)) * 32 + seg * 8, lane, y[0], y[1]);
      const uint32_t t16 = (uint32_t)n0 + (uint32_t)(ch * 32 + i * 16);    // first token of this 16-token group
      uint8_t* hw = hw0 + (int64_t)(t16 >> 7) * (Fe >> 7) * 2048 + ((t16 >> 4) & 7u) * 256;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int64_t o8 = (i * 16 + k) * s8;
        uint32_t rw[4], hw4[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) { rw[j] = bf2_relu(y[k][j]); hw4[j] = bf2_sq(rw[j]); }
        Top2Entry ea, eb;
        top2of4_x2(__byte_perm(hw4[0], hw4[2], 0x5410u), __byte_perm(hw4[0], hw4[2], 0x7632u), __byte_perm(hw4[1], hw4[3], 0x5410u),
                   __byte_perm(hw4[1], hw4[3], 0x7632u), top2, ea, eb);
        const uint32_t pa = __byte_perm(hw4[0], hw4[1], ea.kept), pb = __byte_perm(hw4[2], hw4[3], eb.kept);
        const uint32_t na = (ea.kept >> 16) & 15u, nb = (eb.kept >> 16) & 15u;
        p_vals[o8] = make_uint2(pa, pb);
        p_relu[o8] = make_uint2(__byte_perm(rw[0], rw[1], ea.kept), __byte_perm(rw[2], rw[3], eb.kept));
        uint4 d;
        expand24_lut(lut, pa, na, d.x, d.y);
        expand24_lut(lut, pb, nb, d.z, d.w);
        p_dense[o8] = d;
        if (p_y1) p_y1[o8] = make_uint4(y[k][0], y[k][1], y[k][2], y[k][3]);
        // metadata: one byte per lane, four neighbouring lanes hold the warp's 32 features of this token
        uint32_t mb = na | (nb << 4);
        mb |= __shfl_down_sync(0xFFFFFFFFu, mb, 1) << 8;
        const uint32_t mb32 = (mb & 0xFFFFu) | (__shfl_down_sync(0xFFFFFFFFu, mb, 2) << 16);
        if (seg == 0) p_meta[(i * 16 + k) * s32] = mb32;
        if ((seg & 1) == 0) *reinterpret_cast<uint16_t*>(hw + k * 16) = (uint16_t)mb;
        // V:N:M with groups of four: every block keeps columns 0..3 of its two groups here
        const uint32_t token = t16 + (uint32_t)((lane >> 2) * 2 + k);
        if (vmask && (token & vmask) == 0)
          *reinterpret_cast<uint2*>(reinterpret_cast<uint8_t*>(args.vn_colidx) + (int64_t)(token >> (31 - __clz(vmask + 1u))) * Fe + f) =
              make_uint2(0x03020100u, 0x03020100u);
      }
    }
    p_vals += 32 * s8; p_relu += 32 * s8; p_dense += 32 * s8; p_meta += 32 * s32;
    if (p_y1) p_y1 += 32 * s8;
  }
}

template <int kMode, bool kAMN, bool kBMN, int kEpi>
__global__ void __launch_bounds__(kMode == MODE_VENOM ? kThreadsVenom : kThreads, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmapA, const __grid_constant__ CUtensorMap tmapB,
               const GemmArgs args) {
  extern __shared__ uint8_t smem_dyn[];
  uint8_t* smem = smem_dyn + align_pad(smem_dyn, 1024);
  constexpr bool kSparse = kMode != MODE_DENSE;
  constexpr int kStages = num_stages(kSparse);
  constexpr int kAStageBytes = a_stage_bytes(kSparse);
  constexpr int kStageBytes = stage_bytes(kSparse);
  uint8_t* epi_stage = smem + kStages * kStageBytes;
  SmemCtl* ctl = reinterpret_cast<SmemCtl*>(epi_stage + kEpiStageBytes);
  volatile int* abort_flag = &ctl->abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int kAccBufs = kSparse ? 1 : 2;
  constexpr int kMmaPerStage = kSparse ? 2 : 4;      // dense: K=16 x4 = 64; sparse: logical K=32 x2 = 64

  const int num_m_tiles = args.num_m_tiles, num_n_tiles_ = args.num_n_tiles;
  const int num_tiles = num_m_tiles * num_n_tiles_;
  const int nkb = args.num_k_blocks;                 // 64-wide (logical) k blocks per sweep
  const int sweeps = (kMode == MODE_VENOM && args.V == 64) ? 2 : 1;
  const int iters = nkb * sweeps;

  if (threadIdx.x == 0) {
    prefetch_tmap(&tmapA);
    prefetch_tmap(&tmapB);
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&ctl->full[s], kMode == MODE_VENOM ? 1 + 128 : 1);   // Venom: + one arrival per cp.async gather thread
      mbar_init(&ctl->empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&ctl->tmem_full[b], 1);
      mbar_init(&ctl->tmem_empty[b], 4);
    }
    ctl->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&ctl->tmem_base, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();
  pdl_trigger();
  const uint32_t tmem_base = ctl->tmem_base;

  if (warp == 0) {
    // =========================== TMA producer ===========================
    uint32_t stage = 0, phase = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
      int mt, nt;
      tile_coords(tile, num_m_tiles, num_n_tiles_, mt, nt);
      const int m0 = mt * BM, n0 = nt * BN;
      for (int it = 0; it < iters; ++it) {
        const int sweep = it / nkb, kb = it - sweep * nkb;
        if (!mbar_wait(&ctl->empty[stage], phase ^ 1, abort_flag)) { ok = false; break; }
        uint8_t* sA = smem + stage * kStageBytes;
        uint8_t* sB = sA + kAStageBytes;
        uint8_t* sM = sB + kBStageBytes;
        uint64_t* bar = &ctl->full[stage];
        const bool load_meta = kSparse && ((kb & 1) == 0);
        if (lane == 0) {
          const uint32_t b_tx = (kMode != MODE_VENOM) ? (uint32_t)kBStageBytes
                                                      : (uint32_t)args.gather_tma_groups * 2048u;  // TMA-gathered part
          uint32_t bytes = b_tx + (kSparse ? 8192u : 16384u) + (load_meta ? (uint32_t)kMetaStageBytes : 0u);
          mbar_arrive_expect_tx(bar, bytes);
          // ---- A
          if (kMode == MODE_DENSE) {
            if (!kAMN) {
              tma_load_2d(sA, &tmapA, bar, kb * 64, m0);                       // box {64 k, 128 m}
            } else {
              tma_load_2d(sA, &tmapA, bar, m0, kb * 64);                       // box {64 m, 64 k}
              tma_load_2d(sA + 8192, &tmapA, bar, m0 + 64, kb * 64);
            }
          } else if (kMode == MODE_SPARSE24 || sweeps == 1) {
            tma_load_2d(sA, &tmapA, bar, kb * 32, m0);                         // stored: box {32, 128}
          } else {
            // V = 64: this sweep owns one 64-row half of the tile; the other half reads the zero
            // fill of an out-of-range row coordinate. (box {32, 64})
            const int oob = (int)args.M + 64;
            tma_load_2d(sA, &tmapA, bar, kb * 32, sweep == 0 ? m0 : oob);
            tma_load_2d(sA + 4096, &tmapA, bar, kb * 32, sweep == 1 ? m0 + 64 : oob);
          }
          // ---- metadata atom (2 KB, contiguous in the hardware-ordered tensor)
          if (load_meta) {
            const uint8_t* src = args.meta_hw + ((size_t)mt * (size_t)(nkb >> 1) + (size_t)(kb >> 1)) * 2048;
            bulk_load(sM, src, kMetaStageBytes, bar);
          }
          // ---- B (non-gathered)
          if (kMode != MODE_VENOM) {
            if (!kBMN) {
              tma_load_2d(sB, &tmapB, bar, kb * 64, n0);                       // box {64 k, 256 n}
            } else {
#pragma unroll
              for (int c = 0; c < 4; ++c) tma_load_2d(sB + c * 8192, &tmapB, bar, n0 + c * 64, kb * 64);
            }
          }
        }
        if (++stage == kStages) { stage = 0; phase ^= 1; }
      }
    }
  } else if (warp == 1) {
    // =========================== MMA issuer ===========================
    if (lane == 0) {
      constexpr uint32_t idesc = idesc_bf16(BM, BN, kAMN, kBMN || kMode == MODE_VENOM, kSparse);
      uint32_t stage = 0, phase = 0;
      uint32_t acc = 0, acc_phase = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
        if (!mbar_wait(&ctl->tmem_empty[acc], acc_phase ^ 1, abort_flag)) { ok = false; break; }
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + acc * BN;
        for (int it = 0; it < iters; ++it) {
          const int kb = it % nkb;
          if (!mbar_wait(&ctl->full[stage], phase, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sA = smem_u32(smem + stage * kStageBytes);
          const uint32_t sB = sA + kAStageBytes;
          const uint32_t sM = sB + kBStageBytes;
          if (kSparse && (kb & 1) == 0) {
            // 128 rows x 16 B, no swizzle: 8-row core matrices 128 B apart
            tmem_cp_128x128b(tmem_base + kMetaTmemCol + 4u * ((uint32_t)(kb >> 1) & 1u),
                             smem_desc(sM, 128, 128, kSwizzleNone));
          }
#pragma unroll
          for (int k = 0; k < kMmaPerStage; ++k) {
            uint64_t adesc, bdesc;
            if (kMode == MODE_DENSE) {
              adesc = kAMN ? smem_desc(sA + k * 2048, 8192, 1024, kSwizzle128B)
                           : smem_desc(sA + k * 32, 16, 1024, kSwizzle128B);
            } else {
              adesc = smem_desc(sA + k * 32, 16, 512, 4 /* 64 B swizzle */);
            }
            if (kMode == MODE_VENOM || kBMN) {
              // MN-major: 16 (dense) or 32 (sparse) k rows of 128 B per instruction
              bdesc = smem_desc(sB + k * (kSparse ? 4096 : 2048), 8192, 1024, kSwizzle128B);
            } else {
              bdesc = smem_desc(sB + k * (kSparse ? 64 : 32), 16, 1024, kSwizzle128B);
            }
            const uint32_t accum = (it > 0 || k > 0) ? 1u : 0u;
            if (kSparse) {
              const uint32_t col = (uint32_t)((kb & 1) * 2 + k);              // metadata column of this k step
              const uint32_t mbuf = kMetaTmemCol + 4u * ((uint32_t)(kb >> 1) & 1u);   // metadata double buffer
              mma_sp_f16(tmem_d, adesc, bdesc, tmem_base + mbuf + (col & ~1u), idesc | (col & 1u), accum);
            } else {
              mma_f16(tmem_d, adesc, bdesc, idesc, accum);
            }
          }
          mma_commit(&ctl->empty[stage]);                                      // frees the smem stage
          if (++stage == kStages) { stage = 0; phase ^= 1; }
        }
        if (!ok) break;
        mma_commit(&ctl->tmem_full[acc]);                                      // accumulator ready
        if (++acc == (uint32_t)kAccBufs) { acc = 0; acc_phase ^= 1; }
      }
    }
  } else if (kMode == MODE_VENOM && warp >= 6) {
    // =========================== B gather (warps 6..17, Venom only) ===========================
    // Stage rows are the kept feature rows of Bt in condensed-k order: row r of the stage is
    // feature g*Mv + colidx[blk][g][r & 3] with g = kb*16 + r/4. Two engines work side by side:
    //   warps 6..13  TMA row gather (4 rows x 128 B per instruction) for the first `ntma` groups,
    //   warps 14..17 16-byte cp.async (one warp-wide copy = 512 B of one row) for the others.
    // Neither path alone keeps up with the tensor core; their in-flight limits are independent.
    const int gw = warp - 6;
    const int ntma = args.gather_tma_groups;
    const uint16_t* Bt = reinterpret_cast<const uint16_t*>(args.aux);
    uint32_t stage = 0, phase = 0;
    int pending = -1;                      // cp.async warps: stage whose copies are issued but not yet signalled
    bool ok = true;
    for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
      int mt, nt;
      tile_coords(tile, num_m_tiles, num_n_tiles_, mt, nt);
      const int64_t n0 = (int64_t)nt * BN;
      for (int it = 0; it < iters; ++it) {
        const int sweep = it / nkb, kb = it - sweep * nkb;
        if (!mbar_wait(&ctl->empty[stage], phase ^ 1, abort_flag)) { ok = false; break; }
        const uint32_t sB = smem_u32(smem + stage * kStageBytes + kAStageBytes);
        const int blk = (args.V == 64) ? (2 * mt + sweep) : mt;
        const uint8_t* cbase = args.colidx + ((int64_t)blk * args.G + (int64_t)kb * 16) * 4;
        if (gw < 8) {
          const int grp = gw + 8 * (lane >> 2), c = lane & 3;             // lanes 0..7: two groups x 4 chunks
          if (lane < 8 && grp < ntma) {
            const uint32_t cg = *reinterpret_cast<const uint32_t*>(cbase + grp * 4);
            const int base = (int)(((int64_t)kb * 16 + grp) * args.Mv);
            tma_gather4_2d(sB + c * 8192 + grp * 4 * 128, &tmapB, &ctl->full[stage], (int)n0 + c * 64,
                           base + (int)(cg & 0xFF), base + (int)((cg >> 8) & 0xFF), base + (int)((cg >> 16) & 0xFF),
                           base + (int)(cg >> 24));
          }
        } else {
          const int cw = gw - 8;                                          // 0..3
          for (int grp = ntma + cw; grp < 16; grp += 4) {
            const uint32_t cg = *reinterpret_cast<const uint32_t*>(cbase + grp * 4);
            const int64_t fbase = ((int64_t)kb * 16 + grp) * args.Mv;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int row = grp * 4 + i;
              const uint16_t* src = Bt + (fbase + ((cg >> (8 * i)) & 0xFFu)) * args.ldaux + n0 + lane * 8;
              const uint32_t dst = sB + (lane >> 3) * 8192 + row * 128 + (((lane & 7) ^ (row & 7)) << 4);
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
            }
          }
          asm volatile("cp.async.commit_group;" ::: "memory");
          // These copies are generic-proxy writes and the MMA reads the stage through the async proxy:
          // a stage is signalled only after its copies have landed and a proxy fence has ordered them.
          // The warps stay one stage ahead: signal the previous stage while this one is in flight.
          if (pending >= 0) {
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            fence_proxy_async_smem();
            mbar_arrive(&ctl->full[pending]);
          }
          pending = (int)stage;
        }
        if (++stage == kStages) { stage = 0; phase ^= 1; }
      }
    }
    if (gw >= 8) {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      if (pending >= 0) {
        fence_proxy_async_smem();
        mbar_arrive(&ctl->full[pending]);
      }
    }
  } else {
    // =========================== epilogue (warps 2..5) ===========================
    const int q = warp & 3;                                                    // TMEM lane quadrant
    uint8_t* my_stage = epi_stage + q * kEpiWarpBytes;
    uint32_t acc = 0, acc_phase = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < num_tiles && ok; tile += gridDim.x) {
      int mt, nt;
      tile_coords(tile, num_m_tiles, num_n_tiles_, mt, nt);
      const int64_t m0 = (int64_t)mt * BM, n0 = (int64_t)nt * BN;
      if (!mbar_wait_warp(&ctl->tmem_full[acc], acc_phase, abort_flag)) { ok = false; break; }
      tc_fence_after();
      const uint32_t taddr = tmem_base + acc * BN + ((uint32_t)(q * 32) << 16);
      epi_tile<kEpi>(args, taddr, m0, n0, args.N, q, lane, my_stage);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl->tmem_empty[acc]);
      if (++acc == (uint32_t)kAccBufs) { acc = 0; acc_phase ^= 1; }
    }
  }

  // =========================== teardown ===========================
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && ctl->abort_flag) atomicExch(args.status, 1);
  if (warp == 1) {
    if (ctl->abort_flag) drain_after_expiry();
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

// ---- two-CTA kernel (cta_group::2) -----------------------------------------------------------------
// A cluster of two CTAs computes one 256 x 256 tile: CTA r holds rows [128r, 128r+128) of A and of
// the accumulator, and columns [128r, 128r+128) of B; the leader (rank 0) issues MMAs that read both
// CTAs' shared memory. Each CTA therefore fetches half as much B per unit of tensor work as the
// one-CTA kernel. No TMA multicast is used: each CTA loads its own halves, with completion bytes
// routed to the leader's barrier.
// Stage = 64 K (dense, 4 MMAs of K=16) or 128 logical K (2:4, 4 MMAs of K=32 and one metadata atom):
// four MMAs per barrier round trip keep the single issuing thread ahead of the tensor pipe.
constexpr int kThreads2 = 192;
constexpr int kThreads2Expand = 448;                     // + eight warps that expand a packed operand into its stage
constexpr int kThreads2Sets = 320;                       // + a second set of four epilogue warps
__host__ __device__ constexpr int threads2(int mode, int epi, int expand, bool var) {
  return expand ? kThreads2Expand : (two_sets(epi) || split_sets(mode, epi, expand, var) ? kThreads2Sets : kThreads2);
}
constexpr int kPkStageBytes = 8192 + 1024;               // packed values [64 tokens][64] + metadata bytes [64][16]
// 8-bit operands (fp8 = true) keep the byte geometry of a stage (128-byte rows now hold 128 elements, so a
// 2:4 stage spans 256 logical K) and double its metadata: two 2 KB atoms.
__host__ __device__ constexpr int meta_stage_bytes2(bool fp8) { return fp8 ? 4096 : 2048; }
__host__ __device__ constexpr int stage_bytes2(bool sparse, int bn = BN, bool fp8 = false) {
  return sparse ? (16384 + 2 * (bn / 2) * 128 + meta_stage_bytes2(fp8)) : (16384 + 16384);
}
__host__ __device__ constexpr int num_stages2(bool sparse, int bn = BN, bool expand = false) {
  return sparse ? 4 : (expand ? 5 : 6);
}
// Plain stores of full-width tiles go through TMA, two chunk buffers to a warp (2:4 products, whose stages leave less room, one); narrow tiles (run-time width), where the latency
// of a chunk counts, and the kernels that expand an operand store from registers.
__host__ __device__ constexpr bool tma_store2(int epi, bool expand, bool var) {
  return (epi == EPI_STORE || epi == EPI_SQRELU || epi == EPI_DRELU) && !expand && !var;
}
// The store maps of a kernel: none, one, or two (two products, or two outputs). Only what it uses is a parameter, and only that is
// encoded: both cost the host's side of a launch, which is all of the smallest calls (dense 512 x 512 x 256 5.33 us with two maps
// that are not used and 5.21 without, 2:4 512 x 1280 x 512 7.44 and 7.21, E4M3 dense 512 x 1024 x 512 5.28 and 5.09). Without the
// alignment the arguments behind an empty one start inside a line of 64 bytes: T 1024, D 256, F 1024 38.66 us a step instead of 38.43.
template <int N> struct StoreMaps { CUtensorMap m[N]; };
template <> struct alignas(64) StoreMaps<0> {};
__host__ __device__ constexpr int store_maps2(int epi, bool expand, bool var, bool dual) {
  return !tma_store2(epi, expand, var) ? 0 : dual || epi == EPI_SQRELU ? 2 : 1;
}
template <int N>
__device__ __forceinline__ const CUtensorMap* store_map(const StoreMaps<N>& maps, int i) {
  if constexpr (N == 0) return nullptr;
  else return &maps.m[N > 1 ? i : 0];
}
__host__ __device__ constexpr int store_bufs2(bool sparse, int epi) { return sparse && epi == EPI_STORE ? 1 : 2; }
__host__ __device__ constexpr int epi_bytes2(int epi, int bn = BN, int store_bufs = 0) {
  return store_bufs > 0   ? store_bufs * kEpiWarpBytes
         : epi == EPI_VNM8 ? kVnmEpiBytes
         : is_drelu_t(epi) ? kSetWarps * kDreluWarpBytes / (bn == 256 ? 2 : 1)
         : epi == EPI_STORE || epi == EPI_ROUTE ? 0 : kSetWarps * kEpiWarpBytes;
}
__host__ __device__ constexpr int smem_bytes2(bool sparse, int bn = BN, int epi = EPI_STORE, bool expand = false,
                                              bool fp8 = false, int store_bufs = 0) {
  return 1024 + num_stages2(sparse, bn, expand) * (stage_bytes2(sparse, bn, fp8) + (expand ? kPkStageBytes : 0)) +
         epi_bytes2(epi, bn, store_bufs) + 1024;
}

struct SmemCtl2 {
  uint64_t full[8];
  uint64_t empty[8];
  uint64_t pk_full[8];
  uint64_t tmem_full[2];
  uint64_t tmem_empty[2];
  uint2 expand_lut[16];      // byte-permute selectors of a 2:4 nibble (see expand24_lut)
  Top2Entry top2_lut[16];    // EPI_ACT24_T
  uint32_t tmem_base;
  int abort_flag;
};

// Metadata of 128 rows and one stage (256 columns) of an 8-bit 2:4 operand, straight from the canonical [R, K/16] words: the
// instruction wants 16 bytes a row and 128 columns, rows in order. A box of 32 bytes a row brings both halves of the columns,
// 32-byte swizzled, and the copy to TMEM starts at either 16. A pass that wrote the words in this order first took 4 us at
// 4096 x 4096, and the product could not be set up beside it: E4M3 2:4 2048 x 2048 x 2048 11.6 -> 9.3 us, 8192 x 4096 x 16384 308 ->
// 288. Two boxes of 16 bytes a row are too many requests for 512-row tiles: 4096 x 16384 x 4096 154.1 us, 148.1 with one.
__device__ __forceinline__ void load_meta8(uint8_t* dst, const CUtensorMap* m, uint64_t* bar, int kb, int row) {
  tma_load_2d_2cta(dst, m, bar, kb * 16, row);             // box {16 words, 128 rows}
}

// The tile a CTA pair works on: from the regular raster, or from a device-built table (grouped products).
template <int kBN, bool kVar, bool kDual>
__device__ __forceinline__ GemmTile get_tile(const GemmArgs& args, int tile, int num_m, int num_n, int nkb_full) {
  if (args.tile_table) {
    const int4* p = reinterpret_cast<const int4*>(args.tile_table + tile);
    const int4 a = __ldg(p), b = __ldg(p + 1);
    return GemmTile{a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  }
  int mt, nt, N = (int)args.N;
  if (kDual && tile >= num_m * num_n) {                    // the second product's tiles follow the first one's
    tile -= num_m * num_n;
    num_m = args.num_m_tiles2; num_n = args.num_n_tiles2; N = (int)args.N2;
  }
  tile_coords(tile, num_m, num_n, mt, nt);
  const int n0 = nt * (kVar ? args.bn : kBN);
  return GemmTile{mt * 256, 0, n0, 0, nkb_full, mt * 256, n0, kVar ? min(N, n0 + args.bn) : N};
}

__device__ __forceinline__ uint64_t desc64(uint32_t lo, uint32_t hi) {
  return (static_cast<uint64_t>(hi) << 32) | lo;
}

// kExpand (dense mode with both operands MN-major only): 1 = operand A, 2 = operand B is not loaded as a
// dense tile; its 2:4-packed form (tmapPk: values, tmapMeta: metadata bytes) is staged by TMA and four
// extra warps expand it, zero-filled, into the swizzled layout the MMA reads.
// kFp8: E4M3 operands (both K-major). The kernel is unchanged in bytes: K, k-block counts and operand
// coordinates are given in 2-byte units (two codes each); only the instruction kind, the descriptor's formats
// and the amount of metadata per stage differ.
// kVar: the tile is args.bn (a multiple of 32, at most kBN) columns wide. Where there are few tiles, narrower ones put
// more SMs to work and shorten what one of them does: the eight kernels of a step at T 1024, D 256, F 1024 take 50 us
// instead of 61 (graph replay). A kernel of its own, because the run-time width costs the issuing threads instructions
// that the large products do not have (dense, 256 wide: 1.5 % and more).
// kDual: two independent products with the same reduction length in one launch (the weight gradients). The second one's
// operands are tmapMeta (A) and tmapPk (B), its output args.C2.
template <int kMode, bool kAMN, bool kBMN, int kEpi, int kBN = BN, int kExpand = 0, bool kFp8 = false, bool kVar = false, bool kDual = false>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(threads2(kMode, kEpi, kExpand, kVar), 1)
gemm_tc2_kernel(const __grid_constant__ CUtensorMap tmapA, const __grid_constant__ CUtensorMap tmapB,
                const __grid_constant__ CUtensorMap tmapMeta, const __grid_constant__ CUtensorMap tmapPk,
                const __grid_constant__ StoreMaps<store_maps2(kEpi, kExpand != 0, kVar, kDual)> tmapsC, const GemmArgs args) {
  extern __shared__ uint8_t smem_dyn[];
  uint8_t* smem = smem_dyn + align_pad(smem_dyn, 1024);
  constexpr bool kSparse = kMode == MODE_SPARSE24;
  constexpr int kStages = num_stages2(kSparse, kBN, kExpand != 0);
  constexpr int kBK = kSparse ? 128 : 64;                // logical K per stage
  static_assert(kExpand == 0 || (kMode == MODE_DENSE && kAMN && kBMN), "packed operands: weight-gradient products only");
  static_assert(!kDual || (kMode == MODE_DENSE && kExpand == 0 && kEpi == EPI_STORE), "pairs of plain dense products");
  static_assert(!kFp8 || (!kAMN && !kBMN && kExpand == 0 && kMode != MODE_VENOM), "8-bit operands are K-major");
  constexpr int kMetaBytes = meta_stage_bytes2(kFp8);
  constexpr uint32_t kMetaCols = kFp8 ? 8u : 4u;          // TMEM columns of one stage's metadata
  constexpr int kAStageBytes = 16384;
  constexpr int kBSlabBytes = (kBN / 2) * 128;            // this CTA's half of B for one 64-wide K slab
  constexpr int kBHalfBytes = kSparse ? 2 * kBSlabBytes : kBSlabBytes;
  constexpr int kStageBytes = stage_bytes2(kSparse, kBN, kFp8);
  // 2:4 mode: TMEM holds the metadata next to the accumulators. 224-column tiles fit two (448 columns + 8 of metadata), and
  // the epilogue of a tile overlaps the main loop of the next; 256-column tiles leave room for one. kOverlap: they alternate
  // between columns 0..255 and 224..479, and the next main loop starts when the 32 columns that both use have been read,
  // which the epilogue does first. One pair of barriers serves both positions: a warp hands tile n back when it has read
  // those columns, and by then it has read all of tile n - 1. It counts where k is short: the routed step at T 8192, D 4096,
  // F 16384 in four experts (32 k-stages a tile) 1309 -> 1293 us; with 64 stages and more, and in the fused activation
  // epilogue (more registers), nothing was gained: what the main loop loses by waiting it makes up from the full ring.
  // The dy1 epilogue holds on to its accumulator for long, so there it is what lets 256 columns be used.
  constexpr bool kOneAcc = kSparse && kBN > 248, kOverlap = kOneAcc && (kEpi == EPI_STORE || is_drelu_t(kEpi)) && !kVar;
  constexpr int kAccBufs = kOneAcc ? 1 : 2;
  constexpr uint32_t kMetaCol = kSparse ? (kOverlap ? 480u : (uint32_t)(kAccBufs * kBN)) : 0u;
  static_assert(kBN % 32 == 0 && kBN <= 256, "tile width");
  static_assert(!(kMode == MODE_DENSE) || kBN == BN, "dense mode uses 256-column tiles");
  static_assert(!kBMN || kBN == BN, "MN-major B is loaded in 64-column chunks");
  uint8_t* pk_stage = smem + kStages * kStageBytes;       // kExpand: ring of packed tiles, one per stage
  uint8_t* epi_stage = pk_stage + (kExpand ? kStages * kPkStageBytes : 0);
  constexpr bool kTmaStore = tma_store2(kEpi, kExpand != 0, kVar);
  constexpr bool kMapped = kTmaStore && kSparse && kEpi == EPI_STORE && !kFp8;   // may be given a row_map
  constexpr int kStoreBufs = kTmaStore ? (threads2(kMode, kEpi, kExpand, kVar) / 32 - 2) * store_bufs2(kSparse, kEpi) : 0;
  SmemCtl2* ctl = reinterpret_cast<SmemCtl2*>(epi_stage + epi_bytes2(kEpi, kBN, kStoreBufs));
  volatile int* abort_flag = &ctl->abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();               // 0 = leader
  const int pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;
  const int num_m_tiles = args.num_m_tiles, num_n_tiles_ = args.num_n_tiles;   // 256-row tiles
  const int half_n = kVar ? args.bn / 2 : kBN / 2;       // this CTA's columns of B
  const int b_chunks = (half_n + 63) >> 6;               // MN-major B: chunks of 64 columns
  const uint32_t b_bytes = kBMN ? (uint32_t)(b_chunks * (kSparse ? 16384 : 8192)) : (uint32_t)(half_n * (kSparse ? 256 : 128));
  const int nkb_full = (int)(args.K / kBK);

  if (threadIdx.x == 0) {
    prefetch_tmap(&tmapA);
    prefetch_tmap(&tmapB);
    if (kSparse || kExpand) prefetch_tmap(&tmapMeta);
    if (kExpand) prefetch_tmap(&tmapPk);
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&ctl->full[s], kExpand ? 1 + 16 : 1);    // + the eight expander warps of either CTA
      mbar_init(&ctl->empty[s], 1);
      mbar_init(&ctl->pk_full[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&ctl->tmem_full[b], 1);
      // the epilogue warps of both CTAs that read the accumulator
      mbar_init(&ctl->tmem_empty[b], split_sets(kMode, kEpi, kExpand, kVar) || (two_sets(kEpi) && kAccBufs == 1) ? 16 : 8);
    }
    ctl->abort_flag = 0;
    fence_mbar_init();
  }
  if ((kExpand || is_drelu_t(kEpi) || kEpi == EPI_ACT24_T) && threadIdx.x >= 64 && threadIdx.x < 80) {
    ctl->expand_lut[threadIdx.x - 64] = expand_lut_entry(threadIdx.x - 64);
  }
  if (kEpi == EPI_VNM8 && threadIdx.x >= 64 && threadIdx.x < 128)
    vnm_tables_init(reinterpret_cast<VnmTables*>(epi_stage + 2 * kVnmSetBytes), (int)threadIdx.x - 64);
  if (kEpi == EPI_ACT24_T && threadIdx.x >= 96) top2_lut_init(ctl->top2_lut, (int)threadIdx.x - 96);
  if (warp == 1) {
    tmem_alloc_2cta(&ctl->tmem_base, kTmemCols);
    tmem_relinquish_2cta();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                    // both CTAs' barriers and TMEM are ready
  tc_fence_after();
  pdl_wait();                                            // everything above overlaps the previous kernel's tail
  const int num_tiles = args.tile_table ? __ldg(args.num_tiles_dev)
                                        : num_m_tiles * num_n_tiles_ + (kDual ? args.num_m_tiles2 * args.num_n_tiles2 : 0);
  if (kMode == MODE_DENSE && !kVar && args.early_next) pdl_trigger();
  const uint32_t tmem_base = ctl->tmem_base;

  if (warp == 0) {
    // =========================== TMA producer (both CTAs) ===========================
    uint32_t stage = 0, phase = 0;
    bool ok = true;
    for (int tile = pair; tile < num_tiles && ok; tile += num_pairs) {
      const GemmTile tc = get_tile<kBN, kVar, kDual>(args, tile, num_m_tiles, num_n_tiles_, nkb_full);
      const int m0 = tc.a_row + (int)rank * 128;         // this CTA's rows of A / D
      const bool second = kDual && tile >= num_m_tiles * num_n_tiles_;
      const CUtensorMap *mapA = second ? &tmapMeta : &tmapA, *mapB = second ? &tmapPk : &tmapB;
      const int nb0 = tc.b_row + (int)rank * half_n;
      const int nkb = tc.nkb, ak0 = tc.a_k0, bk0 = tc.b_k0;
      for (int kb = 0; kb < nkb; ++kb) {
        if (!mbar_wait(&ctl->empty[stage], phase ^ 1, abort_flag)) { ok = false; break; }
        if (lane == 0) {
          uint8_t* sA = smem + stage * kStageBytes;
          uint8_t* sB = sA + kAStageBytes;
          uint8_t* sM = sB + kBHalfBytes;
          uint64_t* bar = &ctl->full[stage];
          if (rank == 0) {
            // the leader's barrier collects the bytes of both CTAs (an expanded operand arrives by
            // shared-memory stores, not by TMA)
            mbar_arrive_expect_tx(bar, 2u * ((kExpand == 1 ? 0u : (uint32_t)kAStageBytes) +
                                             (kExpand == 2 ? 0u : b_bytes) +
                                             (kSparse ? (uint32_t)kMetaBytes : 0u)));
          }
          if (kMode == MODE_DENSE) {
            if (kExpand == 1) {
              // packed A: this CTA's 128 features of 64 tokens, into the staging ring (own barrier)
            } else if (!kAMN) {
              tma_load_2d_2cta(sA, mapA, bar, ak0 + kb * 64, m0);
            } else {
              tma_load_2d_2cta(sA, mapA, bar, m0, ak0 + kb * 64);
              tma_load_2d_2cta(sA + 8192, mapA, bar, m0 + 64, ak0 + kb * 64);
            }
            if (kExpand == 2) {
            } else if (!kBMN) {
              tma_load_2d_2cta(sB, mapB, bar, bk0 + kb * 64, nb0);           // box {64 k, 128 n}
            } else {
              tma_load_2d_2cta(sB, mapB, bar, nb0, bk0 + kb * 64);           // box {64 n, 64 k}
              if (!kVar || b_chunks == 2) tma_load_2d_2cta(sB + 8192, mapB, bar, nb0 + 64, bk0 + kb * 64);
            }
            if (kExpand) {
              const int f0 = kExpand == 1 ? m0 : nb0;                          // first feature of this CTA's half
              uint8_t* sP = pk_stage + stage * kPkStageBytes;
              mbar_arrive_expect_tx(&ctl->pk_full[stage], (uint32_t)kPkStageBytes);
              tma_load_2d(sP, &tmapPk, &ctl->pk_full[stage], f0 >> 1, kb * 64);          // values: box {64, 64}
              tma_load_2d(sP + 8192, &tmapMeta, &ctl->pk_full[stage], f0 >> 4, kb * 64); // metadata: box {8, 64}
            }
          } else {
            tma_load_2d_2cta(sA, &tmapA, bar, (ak0 >> 1) + kb * 64, m0);       // stored values: box {64, 128}
            if (kFp8) {
              load_meta8(sM, &tmapMeta, bar, kb, m0);
            } else {
              // metadata atoms are rows of 2 x 1 KB in a [2 * atoms, 256] uint32 view
              const int atom = (m0 >> 7) * nkb_full + (ak0 >> 7) + kb;
              tma_load_2d_2cta(sM, &tmapMeta, bar, 0, 2 * atom);
            }
            if (!kBMN) {
              tma_load_2d_2cta(sB, &tmapB, bar, bk0 + kb * 128, nb0);          // two 64-wide K slabs
              tma_load_2d_2cta(sB + kBSlabBytes, &tmapB, bar, bk0 + kb * 128 + 64, nb0);
            } else {
              tma_load_2d_2cta(sB, &tmapB, bar, nb0, bk0 + kb * 128);          // two chunks {64 n, 128 k}
              if (!kVar || b_chunks == 2) tma_load_2d_2cta(sB + 16384, &tmapB, bar, nb0 + 64, bk0 + kb * 128);
            }
          }
        }
        if (++stage == kStages) { stage = 0; phase ^= 1; }
      }
    }
    // The next launch is let in when the last loads are on their way (long dense products: at the start, see long_dense). Let in at
    // the start, its CTAs sat in their wait on the SMs that were free (what that cost is measured, its cause is not). Whole steps:
    // T 1024, D 256, F 1024 39.85 -> 38.29 us, T 1920, D 1408, F 5504 180.2 -> 178.1, T 4096, D 2048, F 8192 554.6 -> 551.2. No early
    // start at all costs the first 3 us.
    pdl_trigger();
  } else if (warp == 1) {
    // =========================== MMA issuer (leader CTA only) ===========================
    if (rank == 0 && lane == 0) {
      constexpr uint32_t idesc_full = kFp8 ? idesc_e4m3(256, kBN, kSparse) : idesc_bf16(256, kBN, kAMN, kBMN, kSparse);
      const uint32_t idesc = kVar ? idesc_full - ((uint32_t)(kBN - args.bn) >> 3 << 17) : idesc_full;
      // Descriptor halves that never change: high word = stride offset, version, swizzle; the low
      // word is (address >> 4) | leading offset, advanced by plain 32-bit adds.
      const uint32_t smem0 = smem_u32(smem);
      const uint64_t a_proto = (kMode == MODE_DENSE && kAMN) ? smem_desc(0, 8192, 1024, kSwizzle128B)
                                                             : smem_desc(0, 16, 1024, kSwizzle128B);
      const uint64_t b_proto = kBMN ? smem_desc(0, kSparse ? 16384 : 8192, 1024, kSwizzle128B)
                                    : smem_desc(0, 16, 1024, kSwizzle128B);
      const uint64_t m_proto = kFp8 ? smem_desc(0, 16, 256, kSwizzle32B) : smem_desc(0, 128, 128, kSwizzleNone);
      const uint32_t a_hi = (uint32_t)(a_proto >> 32), b_hi = (uint32_t)(b_proto >> 32), m_hi = (uint32_t)(m_proto >> 32);
      const uint32_t a_lo0 = (uint32_t)a_proto + (smem0 >> 4);
      const uint32_t b_lo0 = (uint32_t)b_proto + ((smem0 + kAStageBytes) >> 4);
      const uint32_t m_lo0 = (uint32_t)m_proto + ((smem0 + kAStageBytes + kBHalfBytes) >> 4);
      // per-instruction advances of the low words (in 16-byte units)
      constexpr uint32_t a_step = (kMode == MODE_DENSE && kAMN) ? (2048 >> 4) : (32 >> 4);
      uint32_t stage = 0, phase = 0;
      uint32_t acc = 0, acc_phase = 0, shift = 0;
      bool ok = true;
      for (int tile = pair; tile < num_tiles && ok; tile += num_pairs, shift ^= kOverlap ? 224u : 0u) {
        const int nkb = args.tile_table ? __ldg(&args.tile_table[tile].nkb) : nkb_full;
        if (!mbar_wait(&ctl->tmem_empty[acc], acc_phase ^ 1, abort_flag)) { ok = false; break; }
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + acc * kBN + shift;
        for (int kb = 0; kb < nkb; ++kb) {
          if (!mbar_wait(&ctl->full[stage], phase, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t soff = stage * (uint32_t)(kStageBytes >> 4);
          const uint32_t a_lo = a_lo0 + soff, b_lo = b_lo0 + soff;
          const uint32_t mbuf = tmem_base + kMetaCol + kMetaCols * ((uint32_t)kb & 1u);   // metadata double buffer
          if (kSparse) tmem_cp_128x128b_2cta(mbuf, desc64(m_lo0 + soff, m_hi));
          if (kSparse && kFp8) tmem_cp_128x128b_2cta(mbuf + 4u, desc64(m_lo0 + soff + 1u, m_hi));
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint32_t accum = (kb > 0 || k > 0) ? 1u : 0u;
            if (kSparse) {
              // K = 32 per instruction: 32 B of stored A, 64 B of B inside a 64-wide K slab
              const uint32_t bk = kBMN ? (uint32_t)k * (4096 >> 4)      // 32 k rows of 128 B
                                       : (uint32_t)((k >> 1) * (kBSlabBytes >> 4) + (k & 1) * (64 >> 4));
              if (kFp8)      // 64 logical K per instruction: two metadata columns each
                mma_sp_f8_2cta(tmem_d, desc64(a_lo + k * a_step, a_hi), desc64(b_lo + bk, b_hi), mbuf + 2u * (uint32_t)k,
                               idesc, accum);
              else
                mma_sp_f16_2cta(tmem_d, desc64(a_lo + k * a_step, a_hi), desc64(b_lo + bk, b_hi),
                                mbuf + (uint32_t)(k & ~1), idesc | (uint32_t)(k & 1), accum);
            } else {
              const uint32_t bk = (uint32_t)k * (kBMN ? (2048 >> 4) : (32 >> 4));
              if (kFp8) mma_f8_2cta(tmem_d, desc64(a_lo + k * a_step, a_hi), desc64(b_lo + bk, b_hi), idesc, accum);
              else      mma_f16_2cta(tmem_d, desc64(a_lo + k * a_step, a_hi), desc64(b_lo + bk, b_hi), idesc, accum);
            }
          }
          mma_commit_2cta(&ctl->empty[stage]);             // frees the stage in both CTAs
          if (++stage == kStages) { stage = 0; phase ^= 1; }
        }
        if (!ok) break;
        mma_commit_2cta(&ctl->tmem_full[acc]);             // accumulator ready, both CTAs
        if (++acc == (uint32_t)kAccBufs) { acc = 0; acc_phase ^= 1; }
      }
    }
  } else if (kExpand != 0 && warp >= 6) {
    // =========================== operand expander (warps 6..13, both CTAs) ===========================
    // Stage tile = 64 tokens (K) x 128 features, MN-major, 128-byte swizzle: two chunks of 64 features,
    // a token row of a chunk is 128 bytes whose 16-byte units are XOR-ed with (token & 7). One unit is
    // eight features = two 2:4 groups = four stored values + one metadata byte in the packed tile.
    const int te = (int)threadIdx.x - 192;                 // 0..255
    const int seg = te & 15, tk0 = te >> 4;                // 16 units per token row; 16 tokens per pass
    const uint2* lut = ctl->expand_lut;
    uint32_t stage = 0, phase = 0;
    bool ok = true;
    for (int tile = pair; tile < num_tiles && ok; tile += num_pairs) {
      for (int kb = 0; kb < nkb_full; ++kb) {
        if (!mbar_wait_warp(&ctl->pk_full[stage], phase, abort_flag)) { ok = false; break; }
        const uint8_t* sP = pk_stage + stage * kPkStageBytes;
        uint8_t* dst = smem + stage * kStageBytes + (kExpand == 1 ? 0 : kAStageBytes) + (seg >> 3) * 8192;
        uint2 v[4];
        uint32_t mb[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int tk = tk0 + 16 * i;
          v[i] = *reinterpret_cast<const uint2*>(sP + tk * 128 + seg * 8);
          mb[i] = sP[8192 + tk * 16 + seg];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int tk = tk0 + 16 * i;
          const uint2 s0 = lut[mb[i] & 15u], s1 = lut[mb[i] >> 4];
          *reinterpret_cast<uint4*>(dst + tk * 128 + (((seg & 7) ^ (tk & 7)) << 4)) =
              make_uint4(__byte_perm(v[i].x, 0u, s0.x), __byte_perm(v[i].x, 0u, s0.y),
                         __byte_perm(v[i].y, 0u, s1.x), __byte_perm(v[i].y, 0u, s1.y));
        }
        // generic-proxy stores -> visible to the tensor core's async-proxy reads, then signal the stage
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive_leader(&ctl->full[stage]);
        if (++stage == kStages) { stage = 0; phase ^= 1; }
      }
    }
  } else if constexpr (two_sets(kEpi)) {
    // =========================== epilogue in two sets (warps 2..9, both CTAs) ===========================
    // Two sets of four warps, one per accumulator buffer: set 0 takes this pair's even tiles, set 1 the odd
    // ones, so each set has two main loops' time for one tile. With one accumulator they share every tile, 128 columns each.
    const int q = warp & 3, set = (warp - 2) >> 2;
    uint8_t* wsm = epi_stage + (set * 4 + q) * (epi_bytes2(kEpi, kBN) / kSetWarps);
    constexpr bool kShare = kAccBufs == 1;
    static_assert(!kShare || kEpi == EPI_VNM8 || is_drelu_t(kEpi), "the other epilogues walk whole tiles");
    const int acc = kShare ? 0 : set;
    const uint32_t taddr = tmem_base + set * (kShare ? 128 : kBN) + ((uint32_t)(q * 32) << 16);
    uint32_t acc_phase = 0;
    for (int tile = kShare ? pair : pair + set * num_pairs; tile < num_tiles; tile += kShare ? num_pairs : 2 * num_pairs) {
      const GemmTile tc = get_tile<kBN, kVar, kDual>(args, tile, num_m_tiles, num_n_tiles_, nkb_full);
      const int64_t m0 = (int64_t)tc.out_m + (int64_t)rank * 128, n0 = tc.out_n + (kShare ? set * 128 : 0), n_limit = tc.n_limit;
      // M % 256 == 128 (regular raster only): the second CTA of the last row of pairs holds no rows (its operand
      // loads were zero-filled); it only hands the accumulator back
      const bool live = args.tile_table != nullptr || m0 < args.M;
      if constexpr (is_drelu_t(kEpi)) {
        if (!epi_drelu_tile<kEpi, kBN, kShare>(args, taddr + (kOverlap ? acc_phase * 224u : 0u), m0, n0, n_limit, live, q, set, lane,
                                               reinterpret_cast<float*>(wsm), ctl->expand_lut, &ctl->tmem_full[acc], acc_phase,
                                               abort_flag, &ctl->tmem_empty[acc]))
          break;
      } else {
        bool ok = mbar_wait_warp(&ctl->tmem_full[acc], acc_phase, abort_flag);
        // the set's warps meet at barriers inside the tile: they go on, or leave, together
        if (kEpi == EPI_VNM8) ok = named_all(set + 1, 128, ok);
        if (!ok) break;
        tc_fence_after();
        if (!live) {
          release_accumulator(lane, &ctl->tmem_empty[acc]);
        } else if constexpr (kEpi == EPI_VNM8) {
          epi_vnm8_tile<kShare ? 128 : kBN, kBN == 192 ? 64 : 128>(args, taddr, m0, n0, n_limit, q, set, lane, epi_stage, &ctl->tmem_empty[acc]);
        } else {
          epi_act24_tile<kBN>(args, taddr, m0, n0, n_limit, q, lane, reinterpret_cast<uint32_t*>(wsm), ctl->expand_lut,
                              ctl->top2_lut, &ctl->tmem_empty[acc]);
        }
      }
      acc_phase ^= 1;
    }
  } else {
    // =========================== epilogue (warps 2..5 or 2..9, both CTAs) ===========================
    const int q = warp & 3, set = (warp - 2) >> 2;
    constexpr int kParts = split_sets(kMode, kEpi, kExpand, kVar) ? 2 : 1;
    uint8_t* my_stage = epi_stage + (set * 4 + q) * (kTmaStore ? store_bufs2(kSparse, kEpi) : 1) * kEpiWarpBytes;
    uint32_t acc = 0, acc_phase = 0, buf = 0;
    bool ok = true;
    for (int tile = pair; tile < num_tiles && ok; tile += num_pairs) {
      const GemmTile tc = get_tile<kBN, kVar, kDual>(args, tile, num_m_tiles, num_n_tiles_, nkb_full);
      const int64_t m0 = (int64_t)tc.out_m + (int64_t)rank * 128, n0 = tc.out_n, n_limit = tc.n_limit;
      const uint32_t taddr = tmem_base + acc * kBN + (kOverlap ? acc_phase * 224u : 0u) + ((uint32_t)(q * 32) << 16);
      // M % 256 == 128 (regular raster only): the second CTA of the last row of pairs holds no rows
      const bool second = kDual && tile >= num_m_tiles * num_n_tiles_;
      const bool live = args.tile_table != nullptr || m0 < (second ? args.M2 : args.M);
      if (!mbar_wait_warp(&ctl->tmem_full[acc], acc_phase, abort_flag)) { ok = false; break; }
      tc_fence_after();
      if (kEpi == EPI_STORE && kTmaStore && live && !(kMapped && args.row_map)) {
        epi_store_tile<kBN, store_bufs2(kSparse, kEpi), kOverlap>(args, store_map(tmapsC, second), taddr, m0, n0, n_limit, q, lane,
                                                                  my_stage, buf, set, kParts, &ctl->tmem_empty[0]);
      } else if (live) {
        epi_tile<kEpi, kBN, kOverlap, kMapped, kTmaStore>(
            args, taddr, m0, n0, n_limit, q, lane, my_stage, set, kParts, second, &ctl->tmem_empty[0], store_map(tmapsC, 0), store_map(tmapsC, 1), &buf);
      }
      if (!kOverlap || !live) release_accumulator(lane, &ctl->tmem_empty[acc]);
      if (++acc == (uint32_t)kAccBufs) { acc = 0; acc_phase ^= 1; }
    }
    if (kTmaStore && lane == 0) bulk_wait_all();
  }

  // =========================== teardown ===========================
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && ctl->abort_flag) {
    atomicExch(args.status, 1);
    drain_after_expiry();
  }
  cluster_sync_all();                                    // the peer is done with our shared memory and barriers
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_2cta(tmem_base, kTmemCols);
  }
}

// ---- 512-row tiles of the 2:4 products ---------------------------------------------------------------
// A CTA pair computes a 512 x 224 tile: two halves of 256 rows that share every stage's B columns, each with its own
// accumulator (448 TMEM columns + 16 of metadata) and its own set of four epilogue warps.
// Why: what bounds the 2:4 product is shared-memory bandwidth (128 B/clk). Per 128 logical K and SM a 256 x 256 tile
// writes 50 KB (TMA) and its MMAs read 48 KB: 768 clocks against 512 of the tensor pipe (735 measured, with the ring
// always full of data). Here B is written once for two halves: 64 KB written, 88 KB read, 1197 clocks against 896
// (1190 measured), 10 % less per column than 256 x 256 and 15 % less than 256 x 224. The price: one accumulator per
// half, so an epilogue overlaps the next main loop only as far as the halves are apart.
// Against 256-row tiles, same box: y3 at T 16384, D 8192, F 28672 3540 -> 3090 us, dX 3550 -> 3110, dy1 4030 -> 3680;
// 4096 x 16384 x 4096 296 -> 243 us, with E4M3 operands 196 -> 176.
constexpr int kTallBN = 224, kTallStages = 3;
constexpr int kTallThreads = 320;                         // producer, MMA issuer, two sets of four epilogue warps
__host__ __device__ constexpr int tall_b_bytes(bool bmn) { return bmn ? 32768 : 28672; }
__host__ __device__ constexpr int tall_stage_bytes(bool bmn, bool fp8) { return tall_b_bytes(bmn) + 2 * (16384 + meta_stage_bytes2(fp8)); }
__host__ __device__ constexpr int tall_epi_bytes(int epi) {
  return kSetWarps * (is_drelu_t(epi) ? kDreluWarpBytes : kEpiWarpBytes);
}
__host__ __device__ constexpr int tall_smem(int epi, bool bmn, bool fp8) {
  return 1024 + kTallStages * tall_stage_bytes(bmn, fp8) + tall_epi_bytes(epi) + 1024;
}

struct SmemCtlTall {
  uint64_t full[kTallStages], empty[kTallStages], tmem_full[2], tmem_empty[2];
  uint2 expand_lut[16];
  uint32_t tmem_base;
  int abort_flag;
};
static_assert(sizeof(SmemCtlTall) <= 1024, "control block");

// The l-th tile of CTA pair p (of P): -1 = no more. Full-width tiles are numbered first, the narrow ones of a ragged last
// column (one per tile row) after them. Full tiles go round robin; narrow ones fill up the pairs whose last round is
// empty, two each, where that takes all of them, else round robin too.
__device__ __forceinline__ int tall_nth(const GemmArgs& args, int l, int p, int P) {
  const int t = p + l * P, nfull = args.num_m_tiles * args.num_n_tiles;
  if (t < nfull) return t;
  const int nn = args.N % kTallBN ? args.num_m_tiles : 0;
  if (nn == 0) return -1;
  const int q = nfull / P, r = nfull - q * P, spare = P - r;
  const int k = l - (q + (p < r));
  int j;
  if (r != 0 && nn <= 2 * spare) j = p < r ? nn : (p - r) + k * spare;
  else                           j = (p < r ? p + spare : p - r) + k * P;
  return j < nn ? nfull + j : -1;
}

struct TallTile {
  int m0, n0, width, halves;   // first row and column, columns (a multiple of 32), 256-row halves that hold rows
};
__device__ __forceinline__ TallTile tall_tile(const GemmArgs& args, int tile) {
  const int nfull = args.num_m_tiles * args.num_n_tiles;
  int mt, nt;
  if (tile < nfull) {
    tile_coords(tile, args.num_m_tiles, args.num_n_tiles, mt, nt);
  } else {
    mt = tile - nfull;
    nt = args.num_n_tiles;
  }
  const int m0 = mt * 512, n0 = nt * kTallBN;
  return TallTile{m0, n0, min(kTallBN, (int)args.N - n0), m0 + 256 < (int)args.M ? 2 : 1};
}

// tmapB: B with boxes of 112 columns (K-major) or {64 n, 128 k} chunks (MN-major); tmapBn: K-major, boxes of half the
// narrow last column.
template <bool kBMN, int kEpi, bool kFp8>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kTallThreads, 1)
gemm_tall_kernel(const __grid_constant__ CUtensorMap tmapA, const __grid_constant__ CUtensorMap tmapB,
                 const __grid_constant__ CUtensorMap tmapBn, const __grid_constant__ CUtensorMap tmapMeta,
                 const __grid_constant__ CUtensorMap tmapC, const GemmArgs args) {
  extern __shared__ uint8_t smem_dyn[];
  uint8_t* smem = smem_dyn + align_pad(smem_dyn, 1024);
  constexpr int kBBytes = tall_b_bytes(kBMN), kMetaBytes = meta_stage_bytes2(kFp8), kStageBytes = tall_stage_bytes(kBMN, kFp8);
  constexpr int kMetaAt = kBBytes + 2 * 16384;            // stage: B columns, A of either half, metadata of either half
  constexpr int kSlab = (kTallBN / 2) * 128;              // K-major: this CTA's half of B for one 64-wide K slab
  constexpr uint32_t kMetaCol = 2 * kTallBN, kMetaCols = kFp8 ? 8u : 4u;
  static_assert(kMetaCol + 4 * kMetaCols <= kTmemCols, "TMEM columns");
  static_assert(!kFp8 || (!kBMN && kEpi == EPI_STORE), "8-bit operands are K-major");
  uint8_t* epi_stage = smem + kTallStages * kStageBytes;
  SmemCtlTall* ctl = reinterpret_cast<SmemCtlTall*>(epi_stage + tall_epi_bytes(kEpi));
  volatile int* abort_flag = &ctl->abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;
  const int nkb = (int)(args.K / 128);

  if (threadIdx.x == 0) {
    prefetch_tmap(&tmapA);
    prefetch_tmap(&tmapB);
    prefetch_tmap(&tmapMeta);
    for (int i = 0; i < kTallStages; ++i) { mbar_init(&ctl->full[i], 1); mbar_init(&ctl->empty[i], 1); }
    for (int h = 0; h < 2; ++h) { mbar_init(&ctl->tmem_full[h], 1); mbar_init(&ctl->tmem_empty[h], 8); }
    ctl->abort_flag = 0;
    fence_mbar_init();
  }
  if (is_drelu_t(kEpi) && threadIdx.x >= 64 && threadIdx.x < 80) ctl->expand_lut[threadIdx.x - 64] = expand_lut_entry(threadIdx.x - 64);
  if (warp == 1) {
    tmem_alloc_2cta(&ctl->tmem_base, kTmemCols);
    tmem_relinquish_2cta();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  tc_fence_after();
  pdl_wait();
  const uint32_t tmem_base = ctl->tmem_base;

  if (warp == 0) {
    // =========================== TMA producer (both CTAs) ===========================
    uint32_t stage = 0, phase = 0;
    bool ok = true;
    for (int l = 0, tile; ok && (tile = tall_nth(args, l, pair, num_pairs)) >= 0; ++l) {
      const TallTile t = tall_tile(args, tile);
      const int half_n = t.width / 2, m0 = t.m0 + (int)rank * 128, nb0 = t.n0 + (int)rank * half_n;
      const int chunks = (half_n + 63) >> 6, atom0 = (m0 >> 7) * nkb;
      const uint32_t tx = 2u * (t.halves * (16384u + (uint32_t)kMetaBytes) + (kBMN ? (uint32_t)chunks * 16384u : 256u * (uint32_t)half_n));
      auto load_a = [&](int kb, int h, uint8_t* st, uint64_t* bar) {
        tma_load_2d_2cta(st + kBBytes + h * 16384, &tmapA, bar, kb * 64, m0 + h * 256);           // stored values: box {64, 128}
        // metadata atoms are rows of 2 x 1 KB in a [2 * atoms, 256] uint32 view
        if (kFp8) load_meta8(st + kMetaAt + h * kMetaBytes, &tmapMeta, bar, kb, m0 + h * 256);
        else      tma_load_2d_2cta(st + kMetaAt + h * kMetaBytes, &tmapMeta, bar, 0, 2 * (atom0 + 2 * h * nkb + kb));
      };
      for (int kb = 0; kb < nkb; ++kb) {
        if (!mbar_wait(&ctl->empty[stage], phase ^ 1, abort_flag)) { ok = false; break; }
        if (lane == 0) {
          uint8_t* st = smem + stage * kStageBytes;
          uint64_t* bar = &ctl->full[stage];
          if (rank == 0) mbar_arrive_expect_tx(bar, tx);   // the leader's barrier collects the bytes of both CTAs
          load_a(kb, 0, st, bar);
          if (t.halves == 2) load_a(kb, 1, st, bar);
          if (kBMN) {
            tma_load_2d_2cta(st, &tmapB, bar, nb0, kb * 128);                                     // chunks {64 n, 128 k}
            if (chunks == 2) tma_load_2d_2cta(st + 16384, &tmapB, bar, nb0 + 64, kb * 128);
          } else if (t.width == kTallBN) {
            tma_load_2d_2cta(st, &tmapB, bar, kb * 128, nb0);                                     // two 64-wide K slabs
            tma_load_2d_2cta(st + kSlab, &tmapB, bar, kb * 128 + 64, nb0);
          } else {
            tma_load_2d_2cta(st, &tmapBn, bar, kb * 128, nb0);
            tma_load_2d_2cta(st + kSlab, &tmapBn, bar, kb * 128 + 64, nb0);
          }
        }
        if (++stage == kTallStages) { stage = 0; phase ^= 1; }
      }
    }
    pdl_trigger();
  } else if (warp == 1) {
    // =========================== MMA issuer (leader CTA only) ===========================
    if (rank == 0 && lane == 0) {
      constexpr uint32_t idesc0 = kFp8 ? idesc_e4m3(256, 0, true) : idesc_bf16(256, 0, false, kBMN, true);
      const uint32_t idesc_wide = idesc0 | ((uint32_t)(kTallBN >> 3) << 17);
      const uint32_t idesc_narrow = idesc0 | ((uint32_t)((int)args.N % kTallBN >> 3) << 17);
      const uint32_t s0 = smem_u32(smem) >> 4;
      const uint64_t a_proto = smem_desc(0, 16, 1024, kSwizzle128B), m_proto = kFp8 ? smem_desc(0, 16, 256, kSwizzle32B) : smem_desc(0, 128, 128, kSwizzleNone);
      const uint64_t b_proto = kBMN ? smem_desc(0, 16384, 1024, kSwizzle128B) : smem_desc(0, 16, 1024, kSwizzle128B);
      const uint32_t a_hi = (uint32_t)(a_proto >> 32), b_hi = (uint32_t)(b_proto >> 32), m_hi = (uint32_t)(m_proto >> 32);
      const int nfull = args.num_m_tiles * args.num_n_tiles;
      uint32_t stage = 0, phase = 0, acc_phase0 = 1, acc_phase1 = 1;
      bool ok = true;
      for (int l = 0, tile; ok && (tile = tall_nth(args, l, pair, num_pairs)) >= 0; ++l) {
        const int halves = tall_tile(args, tile).halves;
        const uint32_t idesc = tile < nfull ? idesc_wide : idesc_narrow;
        if (!mbar_wait(&ctl->tmem_empty[0], acc_phase0, abort_flag)) { ok = false; break; }
        for (int kb = 0; kb < nkb; ++kb) {
          if (!mbar_wait(&ctl->full[stage], phase, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t at = s0 + stage * (uint32_t)(kStageBytes >> 4), b_lo = (uint32_t)b_proto + at;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (h >= halves) break;
            if (h == 1 && kb == 0) {
              if (!mbar_wait(&ctl->tmem_empty[1], acc_phase1, abort_flag)) { ok = false; break; }
              tc_fence_after();
            }
            const uint32_t a_lo = (uint32_t)a_proto + at + (uint32_t)((kBBytes + h * 16384) >> 4);
            const uint32_t m_lo = (uint32_t)m_proto + at + (uint32_t)((kMetaAt + h * kMetaBytes) >> 4);
            const uint32_t mbuf = tmem_base + kMetaCol + kMetaCols * (uint32_t)(2 * (kb & 1) + h);   // metadata double buffer
            tmem_cp_128x128b_2cta(mbuf, desc64(m_lo, m_hi));
            if (kFp8) tmem_cp_128x128b_2cta(mbuf + 4u, desc64(m_lo + 1u, m_hi));
            const uint32_t tmem_d = tmem_base + (uint32_t)(h * kTallBN);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const uint32_t accum = (kb > 0 || k > 0) ? 1u : 0u;
              // K = 32 per instruction: 32 B of stored A, 64 B of B inside a 64-wide K slab, or 32 k rows of 128 B
              const uint32_t bk = kBMN ? (uint32_t)k * (4096 >> 4) : (uint32_t)((k >> 1) * (kSlab >> 4) + (k & 1) * (64 >> 4));
              if (kFp8)      // 64 logical K per instruction: two metadata columns each
                mma_sp_f8_2cta(tmem_d, desc64(a_lo + k * 2, a_hi), desc64(b_lo + bk, b_hi), mbuf + 2u * (uint32_t)k, idesc, accum);
              else
                mma_sp_f16_2cta(tmem_d, desc64(a_lo + k * 2, a_hi), desc64(b_lo + bk, b_hi), mbuf + (uint32_t)(k & ~1),
                                idesc | (uint32_t)(k & 1), accum);
            }
            if (h == 0 && kb == nkb - 1) mma_commit_2cta(&ctl->tmem_full[0]);
          }
          if (!ok) break;
          mma_commit_2cta(&ctl->empty[stage]);             // frees the stage in both CTAs
          if (++stage == kTallStages) { stage = 0; phase ^= 1; }
        }
        if (!ok) break;
        acc_phase0 ^= 1;
        if (halves == 2) {
          mma_commit_2cta(&ctl->tmem_full[1]);
          acc_phase1 ^= 1;
        }
      }
    }
  } else {
    // =========================== epilogue (warps 2..9, both CTAs): a set of four warps per half ===========================
    const int q = warp & 3, h = (warp - 2) >> 2;
    uint8_t* wsm = epi_stage + (h * 4 + q) * (tall_epi_bytes(kEpi) / kSetWarps);
    const uint32_t taddr = tmem_base + (uint32_t)(h * kTallBN) + ((uint32_t)(q * 32) << 16);
    uint32_t phase = 0, buf = 0;
    for (int l = 0, tile; (tile = tall_nth(args, l, pair, num_pairs)) >= 0; ++l) {
      const TallTile t = tall_tile(args, tile);
      if (h >= t.halves) continue;
      const int64_t m0 = (int64_t)t.m0 + h * 256 + (int64_t)rank * 128, n0 = t.n0, n_limit = t.n0 + t.width;
      // M % 256 == 128: the second CTA of the last half holds no rows; it only hands the accumulator back
      const bool live = m0 < args.M;
      if constexpr (is_drelu_t(kEpi)) {
        if (!epi_drelu_tile<kEpi, kTallBN, false>(args, taddr, m0, n0, n_limit, live, q, 0, lane, reinterpret_cast<float*>(wsm),
                                           ctl->expand_lut, &ctl->tmem_full[h], phase, abort_flag, &ctl->tmem_empty[h]))
          break;
      } else {
        if (!mbar_wait_warp(&ctl->tmem_full[h], phase, abort_flag)) break;
        tc_fence_after();
        if (kEpi == EPI_STORE_T && live) {
          epi_store_t_tile<kTallBN>(&tmapC, taddr, m0, n0, n_limit, q, lane, wsm);
        } else if (live) {
          epi_store_tile<kTallBN, 1, false>(args, &tmapC, taddr, m0, n0, n_limit, q, lane, wsm, buf, 0, 1, nullptr);
        }
        release_accumulator(lane, &ctl->tmem_empty[h]);
      }
      phase ^= 1;
    }
    if (!is_drelu_t(kEpi) && lane == 0) bulk_wait_all();
  }

  // =========================== teardown ===========================
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && ctl->abort_flag) {
    atomicExch(args.status, 1);
    drain_after_expiry();
  }
  cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_2cta(tmem_base, kTmemCols);
  }
}

// ---- host side -----------------------------------------------------------------------------------

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess)
      return nullptr;
    fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// 2D tensor map over a row-major [rows, cols] matrix of 2-byte (bf16, uint16) or 4-byte (uint32) elements;
// box = {box_cols, box_rows}.
int make_tmap(CUtensorMap* m, const void* base, int64_t rows, int64_t cols, int64_t ld, uint32_t box_cols,
              uint32_t box_rows, CUtensorMapSwizzle swz, int kind = 0 /* 0 bf16, 1 uint32, 2 uint16 */) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return cuda_fail(cudaErrorUnknown);
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const bool u32 = kind == 1;
  cuuint64_t strides[1] = {(cuuint64_t)ld * (u32 ? 4 : 2)};
  cuuint32_t box[2] = {box_cols, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(m, u32 ? CU_TENSOR_MAP_DATA_TYPE_UINT32 : (kind == 2 ? CU_TENSOR_MAP_DATA_TYPE_UINT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16), 2,
                  const_cast<void*>(base), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    g_last_cuda_error = (int)r;
    return SF_ERR_CUDA;
  }
  return SF_OK;
}

// Map of a plain store: C [rows, cols] bf16, chunks of 32 x 32 (see store_chunk).
int make_store_map(CUtensorMap* m, void* C, int64_t rows, int64_t cols, int64_t ld) {
  return make_tmap(m, C, rows, cols, ld, 32, 32, CU_TENSOR_MAP_SWIZZLE_64B);
}

int sm_count() {
  static int n[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
  if (n[dev] == 0) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 148;
    n[dev] = v;
  }
  return n[dev];
}

template <int kMode, bool kAMN, bool kBMN, int kEpi>
int launch_one(const CUtensorMap& ta, const CUtensorMap& tb, const GemmArgs& a, cudaStream_t s) {
  auto kern = gemm_tc_kernel<kMode, kAMN, kBMN, kEpi>;
  static bool attr_done[64] = {false};
  int dev = 0;
  SF_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64 || !attr_done[dev]) {
    SF_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(kMode != MODE_DENSE)));
    if (dev >= 0 && dev < 64) attr_done[dev] = true;
  }
  const int tiles = a.num_m_tiles * a.num_n_tiles;
  const int grid = tiles < sm_count() ? tiles : sm_count();
  return launch_pdl(kern, dim3(grid), kMode == MODE_VENOM ? kThreadsVenom : kThreads, smem_bytes(kMode != MODE_DENSE), s,
                    ta, tb, a);
}

// Dense products of several rounds of full-width tiles, 128 k-stages and more to a CTA pair (65 000 clocks): the next launch is let in
// at their start. Behind their last loads, call after call at the power cap, they took longer, at the same clocks and a lower rate: 8192
// x 8192 x 8192 874 us, at the start 846, 2048 x 12544 x 7360 309 and 296, 4096 x 16384 x 4096 424 and 421, E4M3 2048 x 12544 x 7424 165
// and 160; steps T 16384, D 8192, F 28672 26.73 ms and 26.05, the dense one at T 8192, D 4096, F 16384 5.16 and 5.08. 300 drawn sizes, at
// the start over behind the last loads: up to 64 stages 1.01, to 128 1.003, to 192 0.995, to 384 0.993, above 0.985 (4864 x 6144 x 448, 49
// stages, 28.9 us and 29.3; the step at T 1920, D 1408, F 5504, whose weight gradients have 120, 178.1 and 179.4). The 2:4 products gained
// nothing from it (0.996 to 1.005) and T 4096, D 2048, F 8192 lost 0.5 %; of its weight gradients (448 stages) it loses 0.2 %.
bool long_dense(int tiles, int pairs, int64_t stages) { return tiles > pairs && (int64_t)((tiles + pairs - 1) / pairs) * stages >= 128; }

template <int kMode, bool kAMN, bool kBMN, int kEpi, int kBN = BN, int kExpand = 0, bool kFp8 = false, bool kVar = false, bool kDual = false>
int launch_two(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& tm, GemmArgs a, cudaStream_t s,
               const CUtensorMap* tpk = nullptr, const CUtensorMap* tc = nullptr, const CUtensorMap* tc2 = nullptr) {
  auto kern = gemm_tc2_kernel<kMode, kAMN, kBMN, kEpi, kBN, kExpand, kFp8, kVar, kDual>;
  constexpr int threads = threads2(kMode, kEpi, kExpand, kVar);
  constexpr bool tma_store = tma_store2(kEpi, kExpand != 0, kVar);
  constexpr int smem = smem_bytes2(kMode != MODE_DENSE, kBN, kEpi, kExpand != 0, kFp8, tma_store ? (threads / 32 - 2) * store_bufs2(kMode != MODE_DENSE, kEpi) : 0);
  static_assert(smem <= 232448 && smem >= kExclusiveSmem, "shared memory per CTA: fits, and one CTA per SM");
  static bool attr_done[64] = {false};
  int dev = 0;
  SF_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64 || !attr_done[dev]) {
    SF_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    if (dev >= 0 && dev < 64) attr_done[dev] = true;
  }
  a.num_m_tiles = (int)((a.M + 255) / 256);
  const int bn = kVar ? a.bn : kBN;
  a.num_n_tiles = (int)((a.N + bn - 1) / bn);
  // table-driven products: the table's length is on the device; launch for its upper bound
  const int tiles = a.tile_table ? a.num_k_blocks /* upper bound, see the grouped launchers */
                                 : a.num_m_tiles * a.num_n_tiles + (kDual ? a.num_m_tiles2 * a.num_n_tiles2 : 0);
  const int max_pairs = sm_count() / 2;
  const int pairs = tiles < max_pairs ? tiles : max_pairs;
  a.early_next = kMode == MODE_DENSE && kEpi != EPI_ROUTE && kExpand == 0 && !kVar && !a.tile_table && long_dense(tiles, max_pairs, a.K / 64);
  constexpr int maps = store_maps2(kEpi, kExpand != 0, kVar, kDual);
  if (!a.row_map && ((maps > 0 && !tc) || (maps > 1 && !tc2))) return SF_ERR_UNSUPPORTED;
  StoreMaps<maps> cm;
  if constexpr (maps > 0) cm.m[0] = tc ? *tc : ta;
  if constexpr (maps > 1) cm.m[1] = *tc2;
  return launch_pdl(kern, dim3(2 * pairs), threads, smem, s, ta, tb, tm, tpk ? *tpk : ta, cm, a);
}

int64_t l2_bytes() {
  static int n[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 126 << 20;
  if (n[dev] == 0) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrL2CacheSize, dev) != cudaSuccess || v <= 0) v = 126 << 20;
    n[dev] = v;
  }
  return n[dev];
}

// Tile width of the two-accumulator 2:4 variant (transposed-output products): 2 x 224 accumulator
// columns + 8 metadata columns fit the 512 TMEM columns.
#ifndef SF_NARROW_BN
#define SF_NARROW_BN 224
#endif
constexpr int kNarrowBN = SF_NARROW_BN;

template <bool kBMN, int kEpi, bool kFp8 = false>
int launch_tall(const CUtensorMap& ta, const CUtensorMap& tb, const CUtensorMap& tbn, const CUtensorMap& tm, GemmArgs a,
                cudaStream_t s, const CUtensorMap* tc = nullptr) {
  if (!is_drelu_t(kEpi) && !tc) return SF_ERR_UNSUPPORTED;
  auto kern = gemm_tall_kernel<kBMN, kEpi, kFp8>;
  constexpr int smem = tall_smem(kEpi, kBMN, kFp8);
  static_assert(smem <= 232448 && smem >= kExclusiveSmem, "shared memory per CTA: fits, and one CTA per SM");
  static bool attr_done[64] = {false};
  int dev = 0;
  SF_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64 || !attr_done[dev]) {
    SF_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    if (dev >= 0 && dev < 64) attr_done[dev] = true;
  }
  a.num_m_tiles = (int)((a.M + 511) / 512);
  a.num_n_tiles = (int)(a.N / kTallBN);                                       // full-width columns
  const int tiles = a.num_m_tiles * (a.num_n_tiles + (a.N % kTallBN ? 1 : 0)), max_pairs = sm_count() / 2;
  return launch_pdl(kern, dim3(2 * (tiles < max_pairs ? tiles : max_pairs)), kTallThreads, smem, s, ta, tb, tbn, tm, tc ? *tc : ta, a);
}

// Map of the canonical metadata [R, K/16] of an 8-bit 2:4 operand; kw: K in 2-byte words.
int make_meta8_map(CUtensorMap* m, const void* meta, int64_t R, int64_t kw) {
  return make_tmap(m, meta, R, kw / 8, kw / 8, 16, 128, CU_TENSOR_MAP_SWIZZLE_32B, 2);
}

// Tensor maps of a tall product, lengths in 2-byte words (8-bit operands: two codes): vals [M, kw / 2] packed A, B [N, kw]
// K-major or [kw, N] MN-major. kind: 0 bf16 (metadata in tensor-core order), 2 words (canonical metadata).
int tall_maps(const void* vals, const void* meta, const void* B, bool b_kmajor, int64_t M, int64_t N, int64_t kw,
              int kind, CUtensorMap* ta, CUtensorMap* tb, CUtensorMap* tbn, CUtensorMap* tm) {
  int st = make_tmap(ta, vals, M, kw / 2, kw / 2, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B, kind);
  if (st == SF_OK)
    st = b_kmajor ? make_tmap(tb, B, N, kw, kw, 64, kTallBN / 2, CU_TENSOR_MAP_SWIZZLE_128B, kind)
                  : make_tmap(tb, B, kw, N, N, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B, kind);
  *tbn = *tb;
  if (st == SF_OK && b_kmajor && N % kTallBN)
    st = make_tmap(tbn, B, N, kw, kw, 64, (uint32_t)(N % kTallBN / 2), CU_TENSOR_MAP_SWIZZLE_128B, kind);
  if (st == SF_OK) st = kind == 2 ? make_meta8_map(tm, meta, M, kw) : make_tmap(tm, meta, 2 * (M / 128) * (kw / 128), 256, 256, 256, 2, CU_TENSOR_MAP_SWIZZLE_NONE, 1);
  return st;
}

// Tile width of a product on 256-row tiles: max_bn, or a narrower one where that ends sooner by the estimate: rounds of
// tiles over the CTA pairs x (k-stages x clocks per stage + epilogue). A stage's clocks are its shared-memory traffic
// (2:4: 0.93 x (272 + 2 w), measured 735 at w = 256 and 680 at 224; dense: 256 + w) or the tensor pipe's 2 w. chunk: epilogue
// clocks per 32 columns and `tile` per tile; exposed: nothing hides the epilogue of a tile (one accumulator), else only the
// last one counts. `tile`: hand-overs between the warps and the latency of the first TMEM load. It is what a short reduction
// is made of: transposed 2:4 product with K = 128, 28672 x 2048 37.6 us on 224 columns and 64.5 on the 32 that the estimate
// took without it, 4096 x 4096 14.7 and 22.1, K = 256 15.9 and 19.1 (64 columns); row-major 2048 x 5632, K = 512 19.9 and 21.1.
// A narrower width has to gain 10 %: its kernel takes the width at run time (at 6 % the weight gradients of D 2048 took 224
// columns, 0.94 by the estimate, and 1.02 of the time).
struct TileWidth { int cols; double clocks; };
TileWidth best_width(int64_t M, int64_t N, int64_t stages, bool sparse, int max_bn, int step, double chunk, bool exposed,
                     double tile = 0.0, int64_t M2 = 0, int64_t N2 = 0) {
  const int64_t P = sm_count() / 2, nm = (M + 255) / 256, nm2 = (M2 + 255) / 256;
  auto cost = [&](int w) {
    const int64_t tiles = nm * ((N + w - 1) / w) + nm2 * ((N2 + w - 1) / w);
    const double smem = sparse ? 0.93 * (272 + 2 * w) : 256.0 + w, main = stages * (smem > 2.0 * w ? smem : 2.0 * w);
    const double rounds = (double)((tiles + P - 1) / P), epi = chunk * (w / 32) + tile;
    return exposed ? rounds * (main + epi) : rounds * (main > epi ? main : epi) + epi;
  };
  int best = max_bn;
  double least = 0.90 * cost(max_bn);
  for (int w = max_bn - step; w >= step; w -= step)
    if (cost(w) < least) { least = cost(w); best = w; }
  return {best, cost(best)};
}

// 512 x 224 tiles, or 256-row tiles of `bn` columns (bn = 256: one accumulator, its epilogue exposed)? Estimated clocks
// of the busiest CTA pair: rounds of tiles x (k-stages x clocks per stage + the epilogue that nothing hides). A stage's
// clocks measured with clock stamps on all SMs: 735 (256 wide), 680 (224 wide), 1190 (512 x 224). A narrow tile of the
// last column takes nearly as long as a full one (three stages do not cover the load latency when there is so little
// to multiply: 64 columns 95 us against 97 at K = 16384), which is why 8192 x 4096 stays on 256-row tiles (434 us
// against 482 at K = 16384) while 16384 x 8192 does not.
// The comparison is with 256-row tiles of full width, not with the narrower ones that best_width would take: where those
// end sooner by the estimate (4 % of drawn sizes, few tokens or few rows of tiles), less is lost than it says: dy1 at T 256,
// D 3328, F 10752 takes 32.7 us on 512 x 224 tiles and 30.7 on 256 x 96, T 256, D 3456, F 12416 32.7 and 30.8. What the rule is
// for: y3 at T 1024, D 4096, F 16384 70.5 us on 512-row tiles and 78.2 without, dX 67.9 and 74.1.
bool use_tall(int64_t M, int64_t N, int64_t stages, int bn, double flat_epi, double tall_epi) {
  if (M < 512) return false;
  const int64_t P = sm_count() / 2;
  const int64_t flat_tiles = ((M + 255) / 256) * ((N + bn - 1) / bn);
  const double flat = (double)((flat_tiles + P - 1) / P) * (stages * (bn == 256 ? 735.0 : 680.0) + flat_epi);
  const int64_t nm = (M + 511) / 512, nfull = nm * (N / kTallBN), nn = N % kTallBN ? nm : 0, q = nfull / P, r = nfull % P, spare = P - r;
  const double full = stages * 1190.0 + tall_epi, narrow = 0.95 * full, last = r ? full : 0.0;
  double rest = last;
  if (nn) {
    if (r && nn <= 2 * spare) {
      const double on_spare = (double)((nn + spare - 1) / spare) * narrow;
      rest = on_spare > last ? on_spare : last;
    } else {
      const int64_t over = nn > spare ? (nn - spare + P - 1) / P : 0;
      const double a = last + over * narrow, b = (double)((nn + P - 1) / P) * narrow;
      rest = a > b ? a : b;
    }
  }
  return q * full + rest < 0.99 * flat;
}

// The same for the products that store row-major (y3, dX; E4M3). With an output beyond the L2 and a short reduction the kernel
// lasts as long as its writes, which the clocks above do not hold. With one stage 512-row tiles end first (8192 x 16384 67.5 us
// against 76.7), with two to six the two are equal in bf16 (K = 256 83.0 and 85.2, K = 512 109.5 and 109.1, K = 768 136.3
// and 136.1) and in E4M3 (K = 1024 113.7 and 113.9), and 256-row tiles are kept, which leave fewer idle at the end.
bool use_tall_plain(int64_t M, int64_t N, int64_t stages) {
  const bool write_bound = stages > 1 && stages < 7 && 2 * M * N > l2_bytes();
  return !write_bound && use_tall(M, N, stages, BN, 2500.0, 2500.0);
}

// CTA pairs work on 256-row tiles; with M % 256 == 128 the second CTA of the last row of pairs runs on
// zero-filled operand rows and stores nothing. A single 128-row block runs the one-CTA kernels.
bool use_two_cta(int64_t M) { return M >= 256; }

}  // namespace

int gemm_cta_pairs() { return sm_count() / 2; }

int make_tmap_2d(void* map, const void* base, int64_t rows, int64_t cols, int64_t ld, uint32_t box_cols,
                 uint32_t box_rows, bool swizzle128) {
  return make_tmap(reinterpret_cast<CUtensorMap*>(map), base, rows, cols, ld, box_cols, box_rows,
                   swizzle128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE);
}

int make_tmap_pairs(void* map, const void* base, int64_t rows, int64_t cols, uint32_t box_cols, uint32_t box_pairs) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return cuda_fail(cudaErrorUnknown);
  cuuint64_t dims[3] = {(cuuint64_t)cols, 2, (cuuint64_t)rows / 2};
  cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)cols * 4};
  cuuint32_t box[3] = {box_cols, 1, box_pairs}, estr[3] = {1, 1, 1};
  const CUresult r = fn(reinterpret_cast<CUtensorMap*>(map), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides,
                        box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r == CUDA_SUCCESS) return SF_OK;
  g_last_cuda_error = (int)r;
  return SF_ERR_CUDA;
}

int gemm_dense(const void* A, bool a_kmajor, const void* B, bool b_kmajor, int64_t M, int64_t N, int64_t K, int epi,
               void* C, int64_t ldc, void* C2, int64_t ldc2, const void* aux, int64_t ldaux, int* status,
               cudaStream_t s) {
  const bool two = use_two_cta(M);
  const int bn = two ? best_width(M, N, K / 64, false, BN, 32, epi == EPI_STORE ? 200.0 : 400.0, false).cols : BN;
  if (M % BM || N % (two ? 128 : BN) || K % 64) return SF_ERR_SHAPE;     // pairs: a ragged last tile of whole 32-column chunks
  if (M == 0 || N == 0) return SF_OK;
  CUtensorMap ta, tb;
  int st;
  if (a_kmajor) st = make_tmap(&ta, A, M, K, K, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B);
  else          st = make_tmap(&ta, A, K, M, M, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st != SF_OK) return st;
  if (b_kmajor) st = make_tmap(&tb, B, N, K, K, 64, two ? bn / 2 : 256, CU_TENSOR_MAP_SWIZZLE_128B);
  else          st = make_tmap(&tb, B, K, N, N, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st != SF_OK) return st;
  const bool tma = two && bn == BN;
  CUtensorMap tc, tc2;
  if (tma && (st = make_store_map(&tc, C, M, N, ldc)) != SF_OK) return st;
  if (tma && C2 && (st = make_store_map(&tc2, C2, M, N, ldc2)) != SF_OK) return st;
  GemmArgs a{};
  a.M = M; a.N = N; a.K = K;
  a.C = C; a.ldc = ldc; a.C2 = C2; a.ldc2 = ldc2; a.aux = aux; a.ldaux = ldaux;
  a.status = status;
  a.num_m_tiles = (int)(M / BM); a.num_n_tiles = (int)(N / BN); a.num_k_blocks = (int)(K / 64);
  a.bn = bn;
#define SF_DENSE_CASE(AMN, BMN, EPI)                                                                \
  return !two       ? launch_one<MODE_DENSE, AMN, BMN, EPI>(ta, tb, a, s)                             \
         : bn == BN ? launch_two<MODE_DENSE, AMN, BMN, EPI>(ta, tb, ta, a, s, nullptr, &tc, C2 ? &tc2 : nullptr) \
                    : launch_two<MODE_DENSE, AMN, BMN, EPI, BN, 0, false, true>(ta, tb, ta, a, s)
  const bool amn = !a_kmajor, bmn = !b_kmajor;
  if (epi == EPI_STORE) {
    if (!amn && !bmn) SF_DENSE_CASE(false, false, EPI_STORE);
    if (!amn && bmn) SF_DENSE_CASE(false, true, EPI_STORE);
    if (amn && !bmn) SF_DENSE_CASE(true, false, EPI_STORE);
    SF_DENSE_CASE(true, true, EPI_STORE);
  } else if (epi == EPI_SQRELU) {
    if (!amn && !bmn) SF_DENSE_CASE(false, false, EPI_SQRELU);
  } else if (epi == EPI_DRELU) {
    if (!amn && bmn) SF_DENSE_CASE(false, true, EPI_DRELU);
    if (!amn && !bmn) SF_DENSE_CASE(false, false, EPI_DRELU);
  }
#undef SF_DENSE_CASE
  return SF_ERR_UNSUPPORTED;
}

namespace {
// One or both weight gradients (M2 = N2 = 0: one), reduced over K.
TileWidth weight_grad_width(int64_t M1, int64_t N1, int64_t M2, int64_t N2, int64_t K) {
  return best_width(M1, N1, K / 64, false, BN, 32, 200.0, false, 0.0, M2, N2);
}
}  // namespace

// By the estimated clocks of the two launches, each on the width that suits it, and of the shared one, whose width is one for both.
// kLaunch is what the second launch costs next to its tiles. Whole steps, apart and together, with M = 8:
//   as many rounds: T 1920, D 1408, F 5504 174.7 us and 170.3;
//   together longer, by less than a launch: T 4096, D 1024, F 2816 (1000 clocks) 155.2 and 151.1, T 6272, D 512, F 7040 (5100)
//   296.2 and 292.0, T 10240, D 1920, F 1792 (9000) 326.4 and 324.7;
//   by more (one of the two fits fewer columns better): T 4096, D 384, F 28032 (11 100) 708 and 707, T 10112, D 384, F 18048 (19 000)
//   1031 and 1038, T 16256, D 384, F 28032 (47 600) 2390 and 2413.
// kShort: of two launches of that many clocks the one that is saved is half a percent; from there on nothing of it is left, and at the
// power cap the shared one takes fewer clocks at a lower rate. Together over apart, as many rounds: T 1536, D 2560, F 22272 (0.30
// million) 0.996, T 4096, D 3072, F 12288 (0.5) 1.000, T 8192, D 4096, F 16384 (1.8) 1.004, T 4096, D 8192, F 28672 (3.2) 1.005,
// T 16384, D 4096, F 16384 (3.7) 1.017, T 8192, D 8192, F 28672 (6.4) 1.033, T 16384, D 8192, F 28672 (12.8) 1.022. kLong: the same
// where rounds are saved: T 16384, D 1536, F 23040 (2.1; 15 instead of 16) 0.985 on one box and 1.004 on another, T 16384, D 2048,
// F 28672 (3.4; 25 instead of 26) 1.015.
bool gemm_dual_tn_pays(int64_t M1, int64_t N1, int64_t M2, int64_t N2, int64_t K) {
  constexpr double kLaunch = 10000.0, kShort = 1.6e6, kLong = 2.4e6;
  if (M1 < 256 || M2 < 256) return false;
  const double apart = weight_grad_width(M1, N1, 0, 0, K).clocks + weight_grad_width(M2, N2, 0, 0, K).clocks;
  const double together = weight_grad_width(M1, N1, M2, N2, K).clocks;
  return apart <= kShort ? together < apart + kLaunch : apart <= kLong && together <= 0.97 * apart;
}

TileShape gemm_dual_tn_tile(int64_t M1, int64_t N1, int64_t M2, int64_t N2, int64_t K) {
  return TileShape{256, weight_grad_width(M1, N1, M2, N2, K).cols};
}

int gemm_dual_tn(const void* A1, const void* B1, int64_t M1, int64_t N1, void* C1, const void* A2, const void* B2, int64_t M2,
                 int64_t N2, void* C2, int64_t K, int* status, cudaStream_t s) {
  if (M1 < 256 || M2 < 256 || M1 % 128 || N1 % 128 || M2 % 128 || N2 % 128 || K % 64) return SF_ERR_SHAPE;
  GemmArgs a{};
  a.bn = gemm_dual_tn_tile(M1, N1, M2, N2, K).cols;
  CUtensorMap ta, tb, ta2, tb2;
  int st = make_tmap(&ta, A1, K, M1, M1, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st == SF_OK) st = make_tmap(&tb, B1, K, N1, N1, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st == SF_OK) st = make_tmap(&ta2, A2, K, M2, M2, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st == SF_OK) st = make_tmap(&tb2, B2, K, N2, N2, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st != SF_OK) return st;
  a.M = M1; a.N = N1; a.K = K; a.C = C1; a.ldc = N1;
  a.M2 = M2; a.N2 = N2; a.C2 = C2; a.ldc2 = N2;
  a.num_m_tiles2 = (int)((M2 + 255) / 256);
  a.num_n_tiles2 = (int)((N2 + a.bn - 1) / a.bn);
  a.status = status;
  CUtensorMap tc, tc2;
  if (a.bn == BN) {
    st = make_store_map(&tc, C1, M1, N1, N1);
    if (st == SF_OK) st = make_store_map(&tc2, C2, M2, N2, N2);
    if (st != SF_OK) return st;
  }
  return a.bn == BN ? launch_two<MODE_DENSE, true, true, EPI_STORE, BN, 0, false, false, true>(ta, tb, ta2, a, s, &tb2, &tc, &tc2)
                    : launch_two<MODE_DENSE, true, true, EPI_STORE, BN, 0, false, true, true>(ta, tb, ta2, a, s, &tb2);
}

// Transposed-output products on CTA pairs run 224-column tiles with two accumulators.
TileShape gemm_sparse24_tile(int64_t M, int64_t N, int64_t K, int epi) {
  const bool plain = (epi == EPI_STORE);
  const int max_bn = plain ? BN : kNarrowBN;
  if (plain ? use_tall_plain(M, N, K / 128) : use_tall(M, N, K / 128, max_bn, 0.0, 2500.0)) return TileShape{512, kTallBN};
  return TileShape{256, best_width(M, N, K / 128, true, max_bn, 32, 400.0, plain, 700.0).cols};
}

int gemm_sparse24(const void* a_vals, const uint8_t* meta_hw, const void* B, bool b_kmajor, int64_t M, int64_t N,
                  int64_t K, int epi, void* C, int64_t ldc, int* status, cudaStream_t s) {
  const bool two = use_two_cta(M);
  if (M % BM || N % (two ? 128 : BN) || K % 128) return SF_ERR_SHAPE;
  if (M == 0 || N == 0) return SF_OK;
  const bool plain = (epi == EPI_STORE);                 // row-major output, either B layout: two-CTA kernel only
  if ((plain || !b_kmajor) && !two) return SF_ERR_UNSUPPORTED;
  CUtensorMap ta, tb, tm, tc;
  const TileShape tile = two ? gemm_sparse24_tile(M, N, K, epi) : TileShape{BM, BN};
  const int bn = tile.cols;
  const bool var = two && tile.rows != 512 && bn != (plain ? BN : kNarrowBN);
  if ((plain && !var) || tile.rows == 512) {
    const int st = plain ? make_store_map(&tc, C, M, N, ldc) : make_store_map(&tc, C, N, M, ldc);
    if (st != SF_OK) return st;
  }
  if (tile.rows == 512) {
    CUtensorMap tbn;
    const int st = tall_maps(a_vals, meta_hw, B, b_kmajor, M, N, K, 0, &ta, &tb, &tbn, &tm);
    if (st != SF_OK) return st;
    GemmArgs a{};
    a.M = M; a.N = N; a.K = K;
    a.C = C; a.ldc = ldc; a.status = status;
    if (!plain) return launch_tall<false, EPI_STORE_T>(ta, tb, tbn, tm, a, s, &tc);
    return b_kmajor ? launch_tall<false, EPI_STORE>(ta, tb, tbn, tm, a, s, &tc) : launch_tall<true, EPI_STORE>(ta, tb, tbn, tm, a, s, &tc);
  }
  int st = two ? make_tmap(&ta, a_vals, M, K / 2, K / 2, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B)
               : make_tmap(&ta, a_vals, M, K / 2, K / 2, 32, 128, CU_TENSOR_MAP_SWIZZLE_64B);
  if (st != SF_OK) return st;
  if (b_kmajor) st = make_tmap(&tb, B, N, K, K, 64, two ? bn / 2 : 256, CU_TENSOR_MAP_SWIZZLE_128B);
  else          st = make_tmap(&tb, B, K, N, N, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st != SF_OK) return st;
  tm = ta;
  if (two) {
    // hardware-ordered metadata: 2 KB atoms viewed as two rows of 256 uint32
    const int64_t atoms = (M / 128) * (K / 128);
    st = make_tmap(&tm, meta_hw, 2 * atoms, 256, 256, 256, 2, CU_TENSOR_MAP_SWIZZLE_NONE, 1);
    if (st != SF_OK) return st;
  }
  GemmArgs a{};
  a.M = M; a.N = N; a.K = K;
  a.C = C; a.ldc = ldc; a.meta_hw = meta_hw; a.status = status;
  a.num_m_tiles = (int)(M / BM); a.num_n_tiles = (int)(N / BN); a.num_k_blocks = (int)(K / 64);
  a.bn = bn;
  if (epi == EPI_STORE) {
    if (b_kmajor) return var ? launch_two<MODE_SPARSE24, false, false, EPI_STORE, BN, 0, false, true>(ta, tb, tm, a, s)
                             : launch_two<MODE_SPARSE24, false, false, EPI_STORE>(ta, tb, tm, a, s, nullptr, &tc);
    return var ? launch_two<MODE_SPARSE24, false, true, EPI_STORE, BN, 0, false, true>(ta, tb, tm, a, s)
               : launch_two<MODE_SPARSE24, false, true, EPI_STORE>(ta, tb, tm, a, s, nullptr, &tc);
  }
  if (epi == EPI_STORE_T)
    return !two ? launch_one<MODE_SPARSE24, false, false, EPI_STORE_T>(ta, tb, a, s)
           : var ? launch_two<MODE_SPARSE24, false, false, EPI_STORE_T, kNarrowBN, 0, false, true>(ta, tb, tm, a, s)
                 : launch_two<MODE_SPARSE24, false, false, EPI_STORE_T, kNarrowBN>(ta, tb, tm, a, s);
  return SF_ERR_UNSUPPORTED;
}

namespace {
// The 2:4 weight-times-token products whose epilogue works on the activation: W [F, D] packed, tokens [T, D],
// 224-column token tiles with two accumulators.
int weight_token_maps(const void* w_vals, const uint8_t* meta_hw, const void* tokens, int64_t F, int64_t T, int64_t D, int bn,
                      CUtensorMap* ta, CUtensorMap* tb, CUtensorMap* tm) {
  int st = make_tmap(ta, w_vals, F, D / 2, D / 2, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st == SF_OK) st = make_tmap(tb, tokens, T, D, D, 64, bn / 2, CU_TENSOR_MAP_SWIZZLE_128B);
  // hardware-ordered metadata: 2 KB atoms viewed as two rows of 256 uint32
  if (st == SF_OK) st = make_tmap(tm, meta_hw, 2 * (F / 128) * (D / 128), 256, 256, 256, 2, CU_TENSOR_MAP_SWIZZLE_NONE, 1);
  return st;
}
}  // namespace

TileShape gemm_sparse24_drelu_tile(int64_t F, int64_t T, int64_t D) {
  // 256-column tiles (one accumulator, 1000 clocks before the next main loop starts) or 224 and narrower (two), by estimated
  // clocks: T 4096, D 2048, F 8192 is 7 rounds of 256-column tiles or 9 of 224: 71.6 us against 79.3.
  // (At T 8192, D 4096, F 16384, 28 and 32 rounds, the two are equal: it has to gain 5 %.)
  // Fewer than eight k-stages (D < 1024) keep 224 columns. Sizes there for which the estimate prefers 256 are rare (11 of
  // 165 000 drawn); 256 columns take T 768, D 896, F 24832 from 43.0 to 38.9 us, T 1024, D 768, F 23296 from 49.1 to 45.1, T 2048,
  // D 896, F 11392 from 49.1 to 47.2 and T 768, D 768, F 23808 from 38.9 to 38.7, so the line could be lower.
  const int64_t stages = D / 128, P = sm_count() / 2, nm = (F + 255) / 256;
  auto rounds = [&](int64_t w) { return (double)((nm * ((T + w - 1) / w) + P - 1) / P); };
  const int bn = best_width(F, T, stages, true, kNarrowBN, 32, 500.0, false).cols;
  const bool wide = stages >= 8 && bn == kNarrowBN && rounds(256) * (stages * 735.0 + 1000.0) < 0.95 * rounds(kNarrowBN) * (stages * 680.0);
  if (use_tall(F, T, stages, wide ? 256 : kNarrowBN, wide ? 1000.0 : 0.0, 4000.0)) return TileShape{512, kTallBN};
  return TileShape{256, wide ? 256 : bn};
}

int gemm_sparse24_drelu(const void* w_vals, const uint8_t* meta_hw, const void* dY, int64_t F, int64_t T, int64_t D,
                        const ActMask& mask, void* dy1_vals, void* dy1_dense, int* status, cudaStream_t s) {
  if (F < 256 || F % 128 || T % 128 || D % 128) return SF_ERR_SHAPE;
  GemmArgs a{};
  a.M = F; a.N = T; a.K = D;
  a.C = dy1_dense; a.ldc = F; a.aux = mask.relu; a.pack_meta = mask.meta; a.pack_vals = dy1_vals; a.status = status;
  if (mask.colidx) {
    a.colidx = mask.colidx; a.V = mask.V; a.Mv = mask.Mv; a.G = F / mask.Mv;
  }
  CUtensorMap ta, tb, tbn, tm;
  const TileShape tile = gemm_sparse24_drelu_tile(F, T, D);
  if (tile.rows == 512) {
    const int st = tall_maps(w_vals, meta_hw, dY, true, F, T, D, 0, &ta, &tb, &tbn, &tm);
    if (st != SF_OK) return st;
    return mask.colidx ? launch_tall<false, EPI_DRELUV_T>(ta, tb, tbn, tm, a, s) : launch_tall<false, EPI_DRELU24_T>(ta, tb, tbn, tm, a, s);
  }
  a.bn = tile.cols;
  const int st = weight_token_maps(w_vals, meta_hw, dY, F, T, D, a.bn, &ta, &tb, &tm);
  if (st != SF_OK) return st;
  if (a.bn == 256)
    return mask.colidx ? launch_two<MODE_SPARSE24, false, false, EPI_DRELUV_T, 256>(ta, tb, tm, a, s)
                       : launch_two<MODE_SPARSE24, false, false, EPI_DRELU24_T, 256>(ta, tb, tm, a, s);
  if (a.bn != kNarrowBN)
    return mask.colidx ? launch_two<MODE_SPARSE24, false, false, EPI_DRELUV_T, kNarrowBN, 0, false, true>(ta, tb, tm, a, s)
                       : launch_two<MODE_SPARSE24, false, false, EPI_DRELU24_T, kNarrowBN, 0, false, true>(ta, tb, tm, a, s);
  return mask.colidx ? launch_two<MODE_SPARSE24, false, false, EPI_DRELUV_T, kNarrowBN>(ta, tb, tm, a, s)
                     : launch_two<MODE_SPARSE24, false, false, EPI_DRELU24_T, kNarrowBN>(ta, tb, tm, a, s);
}

TileShape gemm_sparse24_act4_tile(int64_t F, int64_t T, int64_t D) {
  return TileShape{256, best_width(F, T, D / 128, true, kNarrowBN, 32, 500.0, false).cols};
}

int gemm_sparse24_act4(const void* w_vals, const uint8_t* meta_hw, const void* X, int64_t F, int64_t T, int64_t D, int V,
                       const Act24Out& out, void* colidx, int* status, cudaStream_t s) {
  if (F < 256 || F % 128 || T % 128 || D % 128) return SF_ERR_SHAPE;
  GemmArgs a{};
  a.bn = gemm_sparse24_act4_tile(F, T, D).cols;
  CUtensorMap ta, tb, tm;
  const int st = weight_token_maps(w_vals, meta_hw, X, F, T, D, a.bn, &ta, &tb, &tm);
  if (st != SF_OK) return st;
  a.M = F; a.N = T; a.K = D; a.V = V;
  a.status = status;
  a.vn_vals24 = out.vals; a.vn_relu24 = out.relu; a.vn_meta24 = out.meta; a.vn_meta24_hw = out.meta_hw;
  a.vn_dense = out.dense; a.vn_y1 = out.y1; a.vn_colidx = colidx;
  return a.bn == kNarrowBN ? launch_two<MODE_SPARSE24, false, false, EPI_ACT24_T, kNarrowBN>(ta, tb, tm, a, s)
                           : launch_two<MODE_SPARSE24, false, false, EPI_ACT24_T, kNarrowBN, 0, false, true>(ta, tb, tm, a, s);
}

int gemm_route(const void* X, const void* means, int64_t T, int64_t D, int E, int* expert, float* logits, int* status,
               cudaStream_t s) {
  if (T % 256 || D % 64 || E < 1 || E > 16) return SF_ERR_SHAPE;
  if (T == 0) return SF_OK;
  CUtensorMap ta, tb;
  int st = make_tmap(&ta, X, T, D, D, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st != SF_OK) return st;
  st = make_tmap(&tb, means, E, D, D, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B);     // rows beyond E arrive as zeros
  if (st != SF_OK) return st;
  GemmArgs a{};
  a.M = T; a.N = 256; a.K = D;
  a.status = status;
  a.route_expert = expert; a.route_logits = logits; a.route_E = E;
  a.num_k_blocks = (int)(D / 64);
  return launch_two<MODE_DENSE, false, false, EPI_ROUTE>(ta, tb, ta, a, s);
}

int gemm_fp8(bool sparse, const void* A, const void* meta, const void* B, int64_t M, int64_t N, int64_t K,
             float alpha, void* C, int64_t ldc, int* status, cudaStream_t s) {
  if (M % 256 || N % 32 || K % (sparse ? 256 : 128) || (sparse && !meta)) return SF_ERR_SHAPE;
  if (M == 0 || N == 0) return SF_OK;
  // the operands in 2-byte units: [M, K/2] (dense) or [M, K/4] (2:4 values), [N, K/2]
  const int64_t K2 = K / 2;
  CUtensorMap ta, tb, tm, tc;
  const bool tall = sparse && use_tall_plain(M, N, K / 256);
  const int bn = tall ? kTallBN : best_width(M, N, K2 / (sparse ? 128 : 64), sparse, BN, 32, sparse ? 400.0 : 200.0, sparse, sparse ? 700.0 : 0.0).cols;
  int st = SF_OK;
  if ((tall || bn == BN) && (st = make_store_map(&tc, C, M, N, ldc)) != SF_OK) return st;
  if (tall) {
    CUtensorMap tbn;
    st = tall_maps(A, meta, B, true, M, N, K2, 2, &ta, &tb, &tbn, &tm);
    if (st != SF_OK) return st;
    GemmArgs a{};
    a.M = M; a.N = N; a.K = K2;
    a.C = C; a.ldc = ldc; a.status = status; a.out_scale = alpha;
    return launch_tall<false, EPI_STORE, true>(ta, tb, tbn, tm, a, s, &tc);
  }
  st = sparse ? make_tmap(&ta, A, M, K2 / 2, K2 / 2, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B, 2)
              : make_tmap(&ta, A, M, K2, K2, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B, 2);
  if (st != SF_OK) return st;
  st = make_tmap(&tb, B, N, K2, K2, 64, bn / 2, CU_TENSOR_MAP_SWIZZLE_128B, 2);
  if (st != SF_OK) return st;
  tm = ta;
  if (sparse) {
    st = make_meta8_map(&tm, meta, M, K2);
    if (st != SF_OK) return st;
  }
  GemmArgs a{};
  a.M = M; a.N = N; a.K = K2;
  a.C = C; a.ldc = ldc; a.status = status; a.out_scale = alpha;
  a.num_k_blocks = (int)(K2 / 64);
  a.bn = bn;
  if (bn != BN)
    return sparse ? launch_two<MODE_SPARSE24, false, false, EPI_STORE, BN, 0, true, true>(ta, tb, tm, a, s)
                  : launch_two<MODE_DENSE, false, false, EPI_STORE, BN, 0, true, true>(ta, tb, tm, a, s);
  return sparse ? launch_two<MODE_SPARSE24, false, false, EPI_STORE, BN, 0, true>(ta, tb, tm, a, s, nullptr, &tc)
                : launch_two<MODE_DENSE, false, false, EPI_STORE, BN, 0, true>(ta, tb, tm, a, s, nullptr, &tc);
}

bool gemm_sparse24_vnm8_supported(int64_t F, int64_t T, int64_t D, int V) {
  return F >= 256 && T > 0 && F % 128 == 0 && D % 128 == 0 && (V == 64 || V == 128) && T % V == 0;
}

// Token columns of a tile. 256 (one accumulator, shared by both sets of epilogue warps) costs 16 % less shared-memory traffic a
// column than 192 (two accumulators): y1 at T 8192, D 4096, F 16384 578 -> 558 us, T 16384, D 8192, F 28672 4.41 -> 3.95 ms.
// With few k-stages or few tiles the narrower ones end sooner: T 4096, D 2048, F 8192 90 us at 192 columns and 92 at 256,
// D 512 79 and 89. Estimated clocks: rounds of tiles x the longer of main loop and epilogue, plus the last epilogue; per 64
// tokens the epilogue takes 3000 where two tiles' overlap and 6500 where both sets work on one tile; reading a shared
// accumulator, 2500, is exposed. Tiles hold whole V-blocks: the narrow width for V = 128 is 128.
TileShape gemm_sparse24_vnm8_tile(int64_t F, int64_t T, int64_t D, int V) {
  const int64_t stages = D / 128, P = sm_count() / 2, nm = (F + 255) / 256;
  auto rounds = [&](int w) { return (double)((nm * ((T + w - 1) / w) + P - 1) / P); };
  const int narrow = V == 128 ? 128 : best_width(F, T, stages, true, 192, 64, 1500.0, false).cols;
  const double epi = 1500.0 * (narrow / 32), main = stages * 0.93 * (272 + 2 * narrow), wide = stages * 735.0 + 2500.0;
  const double cost_narrow = rounds(narrow) * (main > epi ? main : epi) + epi;
  const double cost_wide = rounds(256) * (wide > 13000.0 ? wide : 13000.0) + 9000.0;
  return TileShape{256, cost_wide < cost_narrow ? 256 : narrow};
}

int gemm_sparse24_vnm8(const void* a_vals, const uint8_t* meta_hw, const void* X, int64_t F, int64_t T, int64_t D,
                       int V, const Vnm8Out& out, int* status, cudaStream_t s) {
  if (!gemm_sparse24_vnm8_supported(F, T, D, V)) return SF_ERR_SHAPE;
  GemmArgs a{};
  a.bn = gemm_sparse24_vnm8_tile(F, T, D, V).cols;
  CUtensorMap ta, tb, tm;
  const int st = weight_token_maps(a_vals, meta_hw, X, F, T, D, a.bn, &ta, &tb, &tm);
  if (st != SF_OK) return st;
  a.M = F; a.N = T; a.K = D; a.V = V;
  a.meta_hw = meta_hw; a.status = status;
  a.vn_vals = out.vals; a.vn_relu = out.relu; a.vn_meta = out.meta; a.vn_colidx = out.colidx;
  a.vn_vals24 = out.vals24; a.vn_relu24 = out.relu24; a.vn_meta24 = out.meta24; a.vn_meta24_hw = out.meta24_hw;
  a.vn_y1 = out.y1; a.vn_dense = out.dense;
  return a.bn == 256 ? launch_two<MODE_SPARSE24, false, false, EPI_VNM8, 256>(ta, tb, tm, a, s)
         : V == 128  ? launch_two<MODE_SPARSE24, false, false, EPI_VNM8, 128>(ta, tb, tm, a, s)
                     : launch_two<MODE_SPARSE24, false, false, EPI_VNM8, 192, 0, false, true>(ta, tb, tm, a, s);
}

// ---- grouped (table-driven) products of the routed step --------------------------------------------------
// All of them run on CTA pairs; the caller's tables hold one entry per output tile and `max_tiles` bounds
// their length (it sizes the grid; GemmArgs::num_k_blocks carries it to the launcher).

int gemm_grouped_act24(const void* a_vals, const uint8_t* meta_hw, const void* Xp, int64_t rows, int64_t F, int64_t Fe,
                       int64_t D, const Act24Out& out, const GemmTile* tiles, const int* num_tiles, int max_tiles,
                       int* status, cudaStream_t s) {
  if (F % 256 || Fe % 256 || D % 128 || rows % 32 || max_tiles <= 0) return SF_ERR_SHAPE;
  CUtensorMap ta, tb, tm;
  const int st = weight_token_maps(a_vals, meta_hw, Xp, F, rows, D, kNarrowBN, &ta, &tb, &tm);
  if (st != SF_OK) return st;
  GemmArgs a{};
  a.M = Fe; a.N = rows; a.K = D;                           // M: width of the outputs (features per expert)
  a.status = status;
  a.vn_vals24 = out.vals; a.vn_relu24 = out.relu; a.vn_meta24 = out.meta; a.vn_meta24_hw = out.meta_hw;
  a.vn_dense = out.dense; a.vn_y1 = out.y1;
  a.tile_table = tiles; a.num_tiles_dev = num_tiles; a.num_k_blocks = max_tiles;
  return launch_two<MODE_SPARSE24, false, false, EPI_ACT24_T, kNarrowBN>(ta, tb, tm, a, s);
}

int gemm_grouped_drelu24(const void* a_vals, const uint8_t* meta_hw, const void* dYp, int64_t rows, int64_t F,
                         int64_t Fe, int64_t D, const void* relu_vals, const void* meta, void* pack_vals, void* dense,
                         const GemmTile* tiles, const int* num_tiles, int max_tiles, int* status, cudaStream_t s) {
  if (F % 256 || Fe % 256 || D % 128 || rows % 32 || max_tiles <= 0) return SF_ERR_SHAPE;
  CUtensorMap ta, tb, tm;
  const int st = weight_token_maps(a_vals, meta_hw, dYp, F, rows, D, kNarrowBN, &ta, &tb, &tm);
  if (st != SF_OK) return st;
  GemmArgs a{};
  a.M = Fe; a.N = rows; a.K = D;
  a.C = dense; a.ldc = Fe; a.aux = relu_vals; a.pack_meta = meta; a.pack_vals = pack_vals;
  a.status = status;
  a.tile_table = tiles; a.num_tiles_dev = num_tiles; a.num_k_blocks = max_tiles;
  return launch_two<MODE_SPARSE24, false, false, EPI_DRELU24_T, kNarrowBN>(ta, tb, tm, a, s);
}

int gemm_grouped_sparse24_rm(const void* a_vals, const uint8_t* meta_hw, const void* B, bool b_kmajor, int64_t rows,
                             int64_t N, int64_t Fe, int64_t Ktot, void* C, const int* row_map, const GemmTile* tiles,
                             const int* num_tiles, int max_tiles, int* status, cudaStream_t s) {
  if (rows % 256 || N % 256 || Fe % 128 || Ktot % Fe || max_tiles <= 0) return SF_ERR_SHAPE;
  CUtensorMap ta, tb, tm;
  int st = make_tmap(&ta, a_vals, rows, Fe / 2, Fe / 2, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st != SF_OK) return st;
  if (b_kmajor) st = make_tmap(&tb, B, N, Ktot, Ktot, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B);
  else          st = make_tmap(&tb, B, Ktot, N, N, 64, 128, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st != SF_OK) return st;
  st = make_tmap(&tm, meta_hw, 2 * (rows / 128) * (Fe / 128), 256, 256, 256, 2, CU_TENSOR_MAP_SWIZZLE_NONE, 1);
  if (st != SF_OK) return st;
  GemmArgs a{};
  a.M = rows; a.N = N; a.K = Fe;                           // K of the packed operand: its metadata atoms follow it
  a.C = C; a.ldc = N; a.status = status; a.row_map = row_map;
  a.tile_table = tiles; a.num_tiles_dev = num_tiles; a.num_k_blocks = max_tiles;
  if (b_kmajor) return launch_two<MODE_SPARSE24, false, false, EPI_STORE>(ta, tb, tm, a, s);
  return launch_two<MODE_SPARSE24, false, true, EPI_STORE>(ta, tb, tm, a, s);
}

int gemm_grouped_dense_tn(const void* A, int64_t Ma, const void* B, int64_t Nb, int64_t rows, void* C, int64_t c_rows, int64_t ldc,
                          const GemmTile* tiles, const int* num_tiles, int max_tiles, int* status, cudaStream_t s) {
  if (Ma % 256 || Nb % 256 || rows % 64 || max_tiles <= 0) return SF_ERR_SHAPE;
  CUtensorMap ta, tb;
  int st = make_tmap(&ta, A, rows, Ma, Ma, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st != SF_OK) return st;
  st = make_tmap(&tb, B, rows, Nb, Nb, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B);
  CUtensorMap tc;
  if (st == SF_OK) st = make_store_map(&tc, C, c_rows, ldc, ldc);
  if (st != SF_OK) return st;
  GemmArgs a{};
  a.M = Ma; a.N = ldc; a.K = rows;                         // N bounds the stored columns: the whole output row
  a.C = C; a.ldc = ldc; a.status = status;
  a.tile_table = tiles; a.num_tiles_dev = num_tiles; a.num_k_blocks = max_tiles;
  return launch_two<MODE_DENSE, true, true, EPI_STORE>(ta, tb, ta, a, s, nullptr, &tc);
}

int gemm_dense_expand(const void* dense_op, int packed_operand, const void* pk_vals, const void* pk_meta, int64_t M,
                      int64_t N, int64_t K, void* C, int64_t ldc, int* status, cudaStream_t s) {
  if (M % 256 || N % 256 || K % 64 || (packed_operand != 1 && packed_operand != 2)) return SF_ERR_SHAPE;
  if (M == 0 || N == 0) return SF_OK;
  const int64_t X = packed_operand == 1 ? M : N;                              // width of the packed operand
  CUtensorMap ta, tb, tm, tp;
  // the dense operand: [K, M] or [K, N] row-major, 64 x 64 boxes
  int st = make_tmap(packed_operand == 1 ? &tb : &ta, dense_op, K, packed_operand == 1 ? N : M,
                     packed_operand == 1 ? N : M, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st != SF_OK) return st;
  if (packed_operand == 1) ta = tb; else tb = ta;                             // the unused map only has to be valid
  st = make_tmap(&tp, pk_vals, K, X / 2, X / 2, 64, 64, CU_TENSOR_MAP_SWIZZLE_NONE);
  if (st != SF_OK) return st;
  st = make_tmap(&tm, pk_meta, K, X / 16, X / 16, 8, 64, CU_TENSOR_MAP_SWIZZLE_NONE, 2);
  if (st != SF_OK) return st;
  GemmArgs a{};
  a.M = M; a.N = N; a.K = K;
  a.C = C; a.ldc = ldc; a.status = status;
  a.num_m_tiles = (int)(M / BM); a.num_n_tiles = (int)(N / BN); a.num_k_blocks = (int)(K / 64);
  if (packed_operand == 1) return launch_two<MODE_DENSE, true, true, EPI_STORE, BN, 1>(ta, tb, tm, a, s, &tp);
  return launch_two<MODE_DENSE, true, true, EPI_STORE, BN, 2>(ta, tb, tm, a, s, &tp);
}

int gemm_venom(const void* a_vals, const uint8_t* meta_hw, const uint8_t* colidx, const void* Bt, int64_t T,
               int64_t F, int64_t N, int V, int Mv, void* C, int64_t ldc, int* status, cudaStream_t s) {
  const int64_t Kc = 4 * F / Mv;                                               // condensed reduction length
  if (T % BM || N % BN || Kc % 128 || (V != 64 && V != 128)) return SF_ERR_SHAPE;
  if (T == 0 || N == 0) return SF_OK;
  CUtensorMap ta, tb;
  int st = make_tmap(&ta, a_vals, T, Kc / 2, Kc / 2, 32, V == 64 ? 64 : 128, CU_TENSOR_MAP_SWIZZLE_64B);
  if (st != SF_OK) return st;
  st = make_tmap(&tb, Bt, F, N, N, 64, 1, CU_TENSOR_MAP_SWIZZLE_128B);        // row gather: one row per box
  if (st != SF_OK) return st;
  GemmArgs a{};
  a.gather_tma_groups = 12;      // measured optimum of the TMA : cp.async split (of 16 groups per stage)
  a.M = T; a.N = N; a.K = Kc;
  a.aux = Bt; a.ldaux = N;
  a.C = C; a.ldc = ldc; a.meta_hw = meta_hw; a.colidx = colidx; a.V = V; a.Mv = Mv; a.G = F / Mv;
  a.status = status;
  a.num_m_tiles = (int)(T / BM); a.num_n_tiles = (int)(N / BN); a.num_k_blocks = (int)(Kc / 64);
  return launch_one<MODE_VENOM, false, true, EPI_STORE>(ta, tb, a, s);
}

}  // namespace sf
