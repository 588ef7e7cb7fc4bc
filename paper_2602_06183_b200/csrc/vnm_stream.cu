// SquaredReLU + V:N:M sparsification, streaming form (Eq. 2, Section 2.3), for M in {8, 16, 32, 64}.
// (Groups of eight have a kernel of their own further down, built the same way.)
//
// Same selection rule and outputs as the kernels of vnm.cu (values, ReLU values, canonical metadata, colidx), organised
// as a pipeline so that loading, scoring and emitting overlap inside one CTA instead of alternating:
//   warp 0        TMA producer: one bulk tensor load per V x 256 strip into a three-slot ring
//   warps 1..4    column scores (sequential float32 sums, two columns per thread), ranking of the eight columns
//                 of every group, colidx
//   warps 5..12   emit: one thread per (row, group): 2:4 among the kept columns, packed stores
// Persistent CTAs walk the strips; every mbarrier wait is bounded (a role that gives up makes the others leave too).
#include "sf_common.cuh"
#include "sparse_fmt.cuh"
#include "tc_ptx.cuh"
#include "gemm_tc.cuh"

namespace sf {
namespace {

using namespace ptx;

constexpr int kSlots = 3;
constexpr int kThreadsS = 32 + 128 + 256;

// kSW = columns per strip: 256 for V <= 64, 128 for taller blocks (three slots then still leave room for two
// CTAs per SM).
template <int kSW>
struct StripAux {
  uint32_t score[kSW];
  uint8_t keep[kSW];
  uint8_t cidx[kSW / 8 * 4];             // [groups of the strip][4]; sized for the narrowest group
};

struct StreamCtl {
  uint64_t full[kSlots], scored[kSlots], empty[kSlots];
  int abort_flag;
};

__device__ __forceinline__ void named_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

template <int kSW, int kM>
__global__ void __launch_bounds__(kThreadsS)
vnm_stream_kernel(const __grid_constant__ CUtensorMap tmapP, int64_t T, int64_t F, int V, int apply,
                   uint16_t* __restrict__ vals, uint16_t* __restrict__ meta, uint8_t* __restrict__ colidx,
                   uint16_t* __restrict__ relu_vals) {
  extern __shared__ uint8_t smem_dyn[];
  uint8_t* smem = smem_dyn + align_pad(smem_dyn, 128);
  const int strip_bytes = V * kSW * 2;
  using Aux = StripAux<kSW>;
  Aux* aux = reinterpret_cast<Aux*>(smem + kSlots * strip_bytes);
  StreamCtl* ctl = reinterpret_cast<StreamCtl*>(aux + kSlots);
  volatile int* abort_flag = &ctl->abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nsx = (int)((F + kSW - 1) / kSW);
  const int64_t nstrips = (T / V) * nsx;
  const int64_t G = F / kM;

  if (tid == 0) {
    prefetch_tmap(&tmapP);
    for (int s = 0; s < kSlots; ++s) {
      mbar_init(&ctl->full[s], 1);
      mbar_init(&ctl->scored[s], 4);
      mbar_init(&ctl->empty[s], 8);
    }
    ctl->abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  pdl_wait();
  pdl_trigger();

  if (warp == 0) {
    // =========================== producer ===========================
    uint32_t slot = 0, phase = 0;
    for (int64_t i = blockIdx.x; i < nstrips; i += gridDim.x) {
      if (!mbar_wait(&ctl->empty[slot], phase ^ 1, abort_flag)) break;
      if (lane == 0) {
        const int64_t blk = i / nsx, cx = i - blk * nsx;
        mbar_arrive_expect_tx(&ctl->full[slot], (uint32_t)strip_bytes);
        tma_load_2d(smem + slot * strip_bytes, &tmapP, &ctl->full[slot], (int)(cx * kSW), (int)(blk * V));
      }
      if (++slot == kSlots) { slot = 0; phase ^= 1; }
    }
  } else if (warp <= 4) {
    // =========================== score + rank (128 threads) ===========================
    const int ts = tid - 32;
    uint32_t slot = 0, phase = 0;
    for (int64_t i = blockIdx.x; i < nstrips; i += gridDim.x) {
      const int64_t blk = i / nsx, cx = i - blk * nsx;
      const int cvalid = (int)min((int64_t)kSW, F - cx * kSW);
      Aux& a = aux[slot];
      const bool ok = mbar_wait_warp(&ctl->full[slot], phase, abort_flag);
      // rows first to last, one float32 add per element: two columns per thread (256-column strips) or one
      if (ok && kSW == 256) {
        const uint32_t* col = reinterpret_cast<const uint32_t*>(smem + slot * strip_bytes) + ts;
        float s0 = 0.f, s1 = 0.f;
        for (int r = 0; r < V; r += 8) {
          uint32_t h[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const uint32_t w = col[(r + u) * (kSW / 2)];
            h[u] = apply ? bf2_sq(bf2_relu(w)) : (w & 0x7FFF7FFFu);
          }
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            s0 = __fadd_rn(s0, __uint_as_float(h[u] << 16));
            s1 = __fadd_rn(s1, __uint_as_float(h[u] & 0xFFFF0000u));
          }
        }
        a.score[2 * ts] = __float_as_uint(s0);
        a.score[2 * ts + 1] = __float_as_uint(s1);
      } else if (ok) {
        const uint16_t* col = reinterpret_cast<const uint16_t*>(smem + slot * strip_bytes) + ts;
        float s0 = 0.f;
        for (int r = 0; r < V; r += 16) {
          uint32_t h[16];
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            const uint32_t w = col[(r + u) * kSW];
            h[u] = apply ? bf2_sq(bf2_relu(w)) : (w & 0x7FFFu);
          }
#pragma unroll
          for (int u = 0; u < 16; ++u) s0 = __fadd_rn(s0, __uint_as_float(h[u] << 16));
        }
        a.score[ts] = __float_as_uint(s0);
      }
      if (!named_all(1, 128, ok)) break;                       // the four warps go on, or leave, together
      constexpr int kCPT = kSW / 128;                          // columns per scoring thread
#pragma unroll
      for (int c = 0; c < kCPT; ++c) {
        const int j = kCPT * ts + c, jm = j & (kM - 1), base = j - jm;
        const uint32_t s = a.score[j];
        int rank = 0;
#pragma unroll 8
        for (int k = 0; k < kM; ++k) {
          const uint32_t sk = a.score[base + k];
          rank += (sk > s) || (sk == s && k < jm);
        }
        a.keep[j] = rank < 4;
      }
      named_sync(1, 128);
#pragma unroll
      for (int c = 0; c < kCPT; ++c) {
        const int j = kCPT * ts + c, jm = j & (kM - 1), base = j - jm;
        if (a.keep[j]) {
          int pos = 0;
          for (int k = 0; k < jm; ++k) pos += a.keep[base + k];
          a.cidx[(j / kM) * 4 + pos] = (uint8_t)jm;
        }
      }
      named_sync(1, 128);
      const int ng = cvalid / kM;
      if (ts < ng)
        *reinterpret_cast<uint32_t*>(colidx + (blk * G + cx * (kSW / kM) + ts) * 4) =
            *reinterpret_cast<const uint32_t*>(a.cidx + ts * 4);
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl->scored[slot]);
      if (++slot == kSlots) { slot = 0; phase ^= 1; }
    }
  } else {
    // =========================== emit (256 threads) ===========================
    constexpr int kGS = kSW / kM, kRows = 256 / kGS;         // groups per strip row, rows in flight
    const int te = tid - 160, g = te & (kGS - 1), r0 = te / kGS;
    const bool want_relu = relu_vals != nullptr && apply;
    uint32_t slot = 0, phase = 0;
    for (int64_t i = blockIdx.x; i < nstrips; i += gridDim.x) {
      const int64_t blk = i / nsx, cx = i - blk * nsx;
      const int cvalid = (int)min((int64_t)kSW, F - cx * kSW);
      const bool live = g < cvalid / kM;
      const Aux& a = aux[slot];
      if (!mbar_wait_warp(&ctl->scored[slot], phase, abort_flag)) break;
      const uint32_t c4 = *reinterpret_cast<const uint32_t*>(a.cidx + g * 4);
      const int64_t gg = cx * (kSW / kM) + g, trow = blk * V + r0;
      const uint8_t* tp = smem + slot * strip_bytes + r0 * (kSW * 2) + g * (kM * 2);
      const int o0 = 2 * (int)(c4 & 0xFFu), o1 = 2 * (int)((c4 >> 8) & 0xFFu), o2 = 2 * (int)((c4 >> 16) & 0xFFu),
                o3 = 2 * (int)(c4 >> 24);                      // byte offsets of the kept columns inside the group
      uint32_t* p_vals = reinterpret_cast<uint32_t*>(vals) + trow * G + gg;
      uint32_t* p_relu = want_relu ? reinterpret_cast<uint32_t*>(relu_vals) + trow * G + gg : nullptr;
      uint16_t* p_meta = meta + trow * (G >> 2) + (gg >> 2);
      const int64_t s_vals = kRows * G, s_meta = kRows * (G >> 2);
      const bool lead4 = (g & 3) == 0;
      // the four kept columns of a row as two packed pairs, then the activation on those only
      auto kept = [&](const uint8_t* rowp, uint32_t& rk0, uint32_t& rk1, uint32_t& hk0, uint32_t& hk1) {
        rk0 = (uint32_t)*reinterpret_cast<const uint16_t*>(rowp + o0) |
              ((uint32_t)*reinterpret_cast<const uint16_t*>(rowp + o1) << 16);
        rk1 = (uint32_t)*reinterpret_cast<const uint16_t*>(rowp + o2) |
              ((uint32_t)*reinterpret_cast<const uint16_t*>(rowp + o3) << 16);
        hk0 = rk0; hk1 = rk1;
        if (apply) {
          rk0 = bf2_relu(rk0); rk1 = bf2_relu(rk1);
          hk0 = bf2_sq(rk0); hk1 = bf2_sq(rk1);
        }
      };
      auto put = [&](uint32_t packed, uint32_t rpair, uint32_t nib) {
        if (live) *p_vals = packed;
        if (want_relu) {
          if (live) *p_relu = rpair;
          p_relu += s_vals;
        }
        uint32_t word = nib;
        word |= __shfl_down_sync(0xFFFFFFFFu, word, 1) << 4;
        word |= __shfl_down_sync(0xFFFFFFFFu, word, 2) << 8;
        if (lead4 && live) *p_meta = (uint16_t)word;
        p_vals += s_vals;
        p_meta += s_meta;
      };
      for (int r = r0; r < V; r += kRows) {
        uint32_t rk0, rk1, hk0, hk1, packed, psel;
        kept(tp, rk0, rk1, hk0, hk1);
        const uint32_t nib = top2of4_packed(hk0, hk1, &packed, nullptr, &psel);
        put(packed, __byte_perm(rk0, rk1, psel), nib);
        tp += kRows * kSW * 2;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl->empty[slot]);
      if (++slot == kSlots) { slot = 0; phase ^= 1; }
    }
  }
  if (*abort_flag) drain_after_expiry();
}

// ---- groups of eight ----------------------------------------------------------------------------------------------
// The same pipeline with another split of the work. What bounds it is instruction issue, not memory, so an emitting
// thread takes four neighbouring groups of a row: one 16-byte store of values instead of four of four bytes, one of ReLU
// values, the metadata word put together in registers, and the byte-permute selectors of a group read from shared
// memory, where the ranking warp left them, instead of derived by every thread. Strips are loaded as 128-byte-swizzled
// boxes of 64 columns, so that eight rows at the same columns (a quarter-warp) sit in different banks. Ranking runs on
// shuffles; the float32 sums of a column pair are one packed addition.
// 16384 x 16384: V = 64 174 -> 154 us (5.3 TB/s of the bytes it cannot do without), V = 128 180 -> 153, V = 32 241 -> 191 (the
// ring holds as many strips as fit: a short one with three slots had too few bytes in flight).
constexpr int kMaxSlots8 = 8;                               // strips in the ring: as many as half of an SM's memory holds, 3 to 8
struct Stream8Ctl {
  uint64_t full[kMaxSlots8], scored[kMaxSlots8], empty[kMaxSlots8];
  int abort_flag;
};
struct Stream8Sel { uint32_t selp0, selp1, mhi0, mhi1; };   // of a group: permute selectors and half masks of its kept pairs

// Kept columns (four set bits of `mask`) of a group, ascending, one byte each.
__device__ __forceinline__ uint32_t kept_bytes(uint32_t mask) {
  uint32_t c = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    c |= (uint32_t)(__ffs(mask) - 1) << (8 * i);
    mask &= mask - 1;
  }
  return c;
}
__device__ __forceinline__ Stream8Sel kept_selectors(uint32_t c4) {
  uint32_t selp[2], mhi[2];
#pragma unroll
  for (int pr = 0; pr < 2; ++pr) {
    const uint32_t ca = (c4 >> (16 * pr)) & 0xFFu, cb = (c4 >> (16 * pr + 8)) & 0xFFu;
    const uint32_t sa = 2u * (ca & 3u), sb = 2u * (cb & 3u);
    selp[pr] = sa | ((sa + 1u) << 4) | (sb << 8) | ((sb + 1u) << 12);
    mhi[pr] = ((ca & 4u) ? 0x0000FFFFu : 0u) | ((cb & 4u) ? 0xFFFF0000u : 0u);
  }
  return Stream8Sel{selp[0], selp[1], mhi[0], mhi[1]};
}
// (a, b) += (x, y), two rounded float32 additions in one instruction
__device__ __forceinline__ void add2(float& a, float& b, float x, float y) {
  uint64_t s, t;
  asm("mov.b64 %0, {%1, %2};" : "=l"(s) : "f"(a), "f"(b));
  asm("mov.b64 %0, {%1, %2};" : "=l"(t) : "f"(x), "f"(y));
  asm("add.rn.f32x2 %0, %0, %1;" : "+l"(s) : "l"(t));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(s));
}

// kSW = columns per strip: 256 for V <= 64, 128 for taller blocks.
template <int kSW>
__global__ void __launch_bounds__(kThreadsS)
vnm8_stream_kernel(const __grid_constant__ CUtensorMap tmapP, int64_t T, int64_t F, int V, int nslots, int apply,
                   uint4* __restrict__ vals, uint16_t* __restrict__ meta, uint32_t* __restrict__ colidx,
                   uint4* __restrict__ relu_vals) {
  extern __shared__ uint8_t smem_dyn[];
  uint8_t* smem = smem_dyn + align_pad(smem_dyn, 1024);
  const int strip_bytes = V * kSW * 2, seg_bytes = V * 128;
  constexpr int kGS = kSW / 8;                              // groups per strip
  Stream8Sel* sel = reinterpret_cast<Stream8Sel*>(smem + nslots * strip_bytes);     // [nslots][kGS]
  Stream8Ctl* ctl = reinterpret_cast<Stream8Ctl*>(sel + nslots * kGS);
  volatile int* abort_flag = &ctl->abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nsx = (int)((F + kSW - 1) / kSW);
  const int nstrips = (int)(T / V) * nsx;
  const int G = (int)(F >> 3);

  __shared__ Top2Entry lut[16];
  top2_lut_init(lut, tid);
  if (tid == 0) {
    prefetch_tmap(&tmapP);
    for (int s = 0; s < nslots; ++s) {
      mbar_init(&ctl->full[s], 1);
      mbar_init(&ctl->scored[s], kSW == 256 ? 4 : 2);
      mbar_init(&ctl->empty[s], 8);
    }
    ctl->abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  pdl_wait();
  pdl_trigger();

  uint32_t slot = 0, phase = 0;
  if (warp == 0) {
    // =========================== producer ===========================
    for (int i = blockIdx.x; i < nstrips; i += gridDim.x) {
      if (!mbar_wait(&ctl->empty[slot], phase ^ 1, abort_flag)) break;
      if (lane == 0) {
        const int blk = i / nsx, cx = i - blk * nsx;
        mbar_arrive_expect_tx(&ctl->full[slot], (uint32_t)strip_bytes);
#pragma unroll
        for (int g = 0; g < kSW / 64; ++g)                  // columns beyond F arrive as zeros
          tma_load_2d(smem + slot * strip_bytes + g * seg_bytes, &tmapP, &ctl->full[slot], cx * kSW + g * 64, blk * V);
      }
      if (++slot == (uint32_t)nslots) { slot = 0; phase ^= 1; }
    }
  } else if (warp <= 4) {
    // =========================== score + rank (128 threads) ===========================
    // A thread scores a pair of columns. 256-column strips take all 128 threads; of 128-column ones two are in work at
    // a time, 64 threads each.
    const int ts = kSW == 256 ? tid - 32 : (tid - 32) & 63, turn = kSW == 256 ? 0 : (tid - 32) >> 6;
    // word of row r: the 16-byte unit inside the 128-byte row is XOR-ed with r & 7
    const int unit = (ts & 31) >> 2, seg = ts >> 5;
    int off[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) off[u] = seg * seg_bytes + u * 128 + ((unit ^ u) << 4) + (ts & 3) * 4;
    int n = 0;
    for (int i = blockIdx.x; i < nstrips; i += gridDim.x, ++n) {
      if (kSW == 128 && (n & 1) != turn) {
        if (++slot == (uint32_t)nslots) { slot = 0; phase ^= 1; }
        continue;
      }
      const int blk = i / nsx, cx = i - blk * nsx;
      if (!mbar_wait_warp(&ctl->full[slot], phase, abort_flag)) break;
      const uint8_t* base = smem + slot * strip_bytes;
      // rows first to last, one float32 addition per element
      float s0 = 0.f, s1 = 0.f;
      for (int r = 0; r < V; r += 8, base += 1024) {
        uint32_t h[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const uint32_t w = *reinterpret_cast<const uint32_t*>(base + off[u]);
          h[u] = apply ? bf2_sq(bf2_relu(w)) : (w & 0x7FFF7FFFu);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) add2(s0, s1, __uint_as_float(h[u] << 16), __uint_as_float(h[u] & 0xFFFF0000u));
      }
      // the four best columns of each group (ties to the lower column); scores are >= 0: their patterns order them
      const uint32_t a = __float_as_uint(s0), b = __float_as_uint(s1);
      int ra = b > a, rb = a >= b;
#pragma unroll
      for (int x = 1; x < 4; ++x) {
        const uint32_t oa = __shfl_xor_sync(0xFFFFFFFFu, a, x), ob = __shfl_xor_sync(0xFFFFFFFFu, b, x);
        const bool lower = ((lane ^ x) & 3) < (lane & 3);    // the other pair's columns come first
        ra += (oa > a || (lower && oa == a)) + (ob > a || (lower && ob == a));
        rb += (oa > b || (lower && oa == b)) + (ob > b || (lower && ob == b));
      }
      const uint32_t ea = __ballot_sync(0xFFFFFFFFu, ra < 4) >> (lane & 28), eb = __ballot_sync(0xFFFFFFFFu, rb < 4) >> (lane & 28);
      if ((lane & 3) == 0) {
        const uint32_t mask = (ea & 1u) | ((eb & 1u) << 1) | ((ea & 2u) << 1) | ((eb & 2u) << 2) | ((ea & 4u) << 2) |
                              ((eb & 4u) << 3) | ((ea & 8u) << 3) | ((eb & 8u) << 4);
        const int g = ts >> 2, gg = cx * kGS + g;
        const uint32_t c4 = kept_bytes(mask);
        sel[slot * kGS + g] = kept_selectors(c4);
        if (gg < G) colidx[(int64_t)blk * G + gg] = c4;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl->scored[slot]);
      if (++slot == (uint32_t)nslots) { slot = 0; phase ^= 1; }
    }
  } else {
    // =========================== emit (256 threads) ===========================
    // a lane serves the four groups of one 32-column quad in row (row block) + (lane & 7)
    const int ew = warp - 5, r8 = lane & 7;
    const int quad = kSW == 256 ? (ew & 1) * 4 + (lane >> 3) : lane >> 3;
    const int r0 = (kSW == 256 ? ew >> 1 : ew) * 8 + r8;
    constexpr int kStep = kSW == 256 ? 32 : 64;
    int off[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) off[j] = (quad >> 1) * seg_bytes + ((((quad & 1) * 4 + j) ^ r8) << 4);
    const int64_t step = (int64_t)kStep * (G >> 2);
    for (int i = blockIdx.x; i < nstrips; i += gridDim.x) {
      const int blk = i / nsx, cx = i - blk * nsx;
      const bool live = cx * kSW + quad * 32 < F;
      if (!mbar_wait_warp(&ctl->scored[slot], phase, abort_flag)) break;
      Stream8Sel sl[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) sl[j] = sel[slot * kGS + quad * 4 + j];
      const uint8_t* tp = smem + slot * strip_bytes + r0 * 128;
      int64_t at = ((int64_t)blk * V + r0) * (G >> 2) + cx * (kSW / 32) + quad;     // in quads
      for (int r = r0; r < V; r += kStep, tp += kStep * 128, at += step) {
        uint32_t rk[4][2], hk[4][2];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint4 q = *reinterpret_cast<const uint4*>(tp + off[j]);
          const uint32_t a0 = __byte_perm(q.x, q.y, sl[j].selp0), b0 = __byte_perm(q.z, q.w, sl[j].selp0);
          const uint32_t a1 = __byte_perm(q.x, q.y, sl[j].selp1), b1 = __byte_perm(q.z, q.w, sl[j].selp1);
          rk[j][0] = (a0 & ~sl[j].mhi0) | (b0 & sl[j].mhi0);
          rk[j][1] = (a1 & ~sl[j].mhi1) | (b1 & sl[j].mhi1);
          hk[j][0] = rk[j][0]; hk[j][1] = rk[j][1];
          if (apply) {
#pragma unroll
            for (int k = 0; k < 2; ++k) { rk[j][k] = bf2_relu(rk[j][k]); hk[j][k] = bf2_sq(rk[j][k]); }
          }
        }
        Top2Entry e[4];
#pragma unroll
        for (int j = 0; j < 4; j += 2)
          top2of4_x2(__byte_perm(hk[j][0], hk[j + 1][0], 0x5410u), __byte_perm(hk[j][0], hk[j + 1][0], 0x7632u),
                     __byte_perm(hk[j][1], hk[j + 1][1], 0x5410u), __byte_perm(hk[j][1], hk[j + 1][1], 0x7632u), lut, e[j], e[j + 1]);
        if (live) {
          vals[at] = make_uint4(__byte_perm(hk[0][0], hk[0][1], e[0].kept), __byte_perm(hk[1][0], hk[1][1], e[1].kept),
                                __byte_perm(hk[2][0], hk[2][1], e[2].kept), __byte_perm(hk[3][0], hk[3][1], e[3].kept));
          if (relu_vals)
            relu_vals[at] = make_uint4(__byte_perm(rk[0][0], rk[0][1], e[0].kept), __byte_perm(rk[1][0], rk[1][1], e[1].kept),
                                       __byte_perm(rk[2][0], rk[2][1], e[2].kept), __byte_perm(rk[3][0], rk[3][1], e[3].kept));
          // the entry's high half holds the nibble four times over
          meta[at] = (uint16_t)(((e[0].kept & 0x000F0000u) | (e[1].kept & 0x00F00000u) | (e[2].kept & 0x0F000000u) |
                                 (e[3].kept & 0xF0000000u)) >> 16);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&ctl->empty[slot]);
      if (++slot == (uint32_t)nslots) { slot = 0; phase ^= 1; }
    }
  }
  if (*abort_flag) drain_after_expiry();
}

}  // namespace

bool vnm_stream_supported(int64_t F, int64_t ld, int V, int M, const void* P) {
  // TMA: 16-byte aligned base and row pitch; box rows = V; emit threads take rows in steps of 256 * M / strip width
  if (!(M == 8 || M == 16 || M == 32 || M == 64)) return false;
  // 256 emit threads over (strip width / M) groups; M = 64 always takes 256-column strips (a metadata word
  // spans four groups)
  const int rows_in_flight = (V <= 64 || M == 64) ? M : 2 * M;
  return V >= 16 && V <= 128 && V % 16 == 0 && V % rows_in_flight == 0 && F % (4 * M) == 0 && ld % 8 == 0 && aligned16(P);
}

template <int kSW, int kM>
static int launch_stream_t(const void* P, int64_t T, int64_t F, int64_t ld, int V, int apply_sqrelu, void* vals, void* meta,
                           void* colidx, void* relu_vals, cudaStream_t s) {
  alignas(64) CUtensorMap tm;
  int st = make_tmap_2d(&tm, P, T, F, ld, kSW, (uint32_t)V, false);
  if (st != SF_OK) return st;
  const size_t smem = 128 + (size_t)kSlots * V * kSW * 2 + kSlots * sizeof(StripAux<kSW>) + sizeof(StreamCtl);
  static bool attr_done[64] = {false};
  static int sms[64] = {0};
  int dev = 0;
  SF_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return SF_ERR_UNSUPPORTED;
  if (!attr_done[dev]) {
    SF_CUDA_TRY(cudaFuncSetAttribute(vnm_stream_kernel<kSW, kM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     128 + kSlots * 128 * kSW * 2 + kSlots * (int)sizeof(StripAux<kSW>) +
                                         (int)sizeof(StreamCtl)));
    SF_CUDA_TRY(cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev));
    attr_done[dev] = true;
  }
  const int64_t nstrips = (T / V) * ((F + kSW - 1) / kSW);
  const int per_sm = smem <= 110 * 1024 ? 2 : 1;
  const int64_t resident = (int64_t)sms[dev] * per_sm;
  const unsigned grid = (unsigned)(nstrips < resident ? nstrips : resident);
  return launch_pdl(vnm_stream_kernel<kSW, kM>, dim3(grid), kThreadsS, smem, s, tm, T, F, V, apply_sqrelu,
                    (uint16_t*)vals, (uint16_t*)meta, (uint8_t*)colidx, (uint16_t*)relu_vals);
}

template <int kSW>
static int launch_stream8(const void* P, int64_t T, int64_t F, int64_t ld, int V, int apply_sqrelu, void* vals, void* meta,
                          void* colidx, void* relu_vals, cudaStream_t s) {
  alignas(64) CUtensorMap tm;
  int st = make_tmap_2d(&tm, P, T, F, ld, 64, (uint32_t)V, true);
  if (st != SF_OK) return st;
  constexpr int kSlotAux = (kSW / 8) * (int)sizeof(Stream8Sel), kMost = 96 * 1024 + 8 * 1024;
  const int strip = V * kSW * 2, fit = 96 * 1024 / strip, nslots = fit < 3 ? 3 : fit > kMaxSlots8 ? kMaxSlots8 : fit;
  const size_t smem = 1024 + (size_t)nslots * (strip + kSlotAux) + sizeof(Stream8Ctl);
  static bool attr_done[64] = {false};
  static int sms[64] = {0};
  int dev = 0;
  SF_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return SF_ERR_UNSUPPORTED;
  if (!attr_done[dev]) {
    SF_CUDA_TRY(cudaFuncSetAttribute(vnm8_stream_kernel<kSW>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost));
    SF_CUDA_TRY(cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev));
    attr_done[dev] = true;
  }
  const int64_t nstrips = (T / V) * ((F + kSW - 1) / kSW), resident = (int64_t)sms[dev] * 2;     // two CTAs of 101 KB at most
  const unsigned grid = (unsigned)(nstrips < resident ? nstrips : resident);
  return launch_pdl(vnm8_stream_kernel<kSW>, dim3(grid), kThreadsS, smem, s, tm, T, F, V, nslots, apply_sqrelu, (uint4*)vals,
                    (uint16_t*)meta, (uint32_t*)colidx, (uint4*)(apply_sqrelu ? relu_vals : nullptr));
}

int launch_vnm_stream(const void* P, int64_t T, int64_t F, int64_t ld, int V, int M, int apply_sqrelu, void* vals,
                      void* meta, void* colidx, void* relu_vals, cudaStream_t s) {
  if (T == 0 || F == 0) return SF_OK;
  if (M == 8)
    return V <= 64 ? launch_stream8<256>(P, T, F, ld, V, apply_sqrelu, vals, meta, colidx, relu_vals, s)
                   : launch_stream8<128>(P, T, F, ld, V, apply_sqrelu, vals, meta, colidx, relu_vals, s);
#define SF_STREAM_CASE(MM)                                                                                      \
  if (M == MM)                                                                                                  \
    return V <= 64 ? launch_stream_t<256, MM>(P, T, F, ld, V, apply_sqrelu, vals, meta, colidx, relu_vals, s)   \
                   : launch_stream_t<128, MM>(P, T, F, ld, V, apply_sqrelu, vals, meta, colidx, relu_vals, s);
  SF_STREAM_CASE(16)
  SF_STREAM_CASE(32)
#undef SF_STREAM_CASE
  if (M == 64) return launch_stream_t<256, 64>(P, T, F, ld, V, apply_sqrelu, vals, meta, colidx, relu_vals, s);
  return SF_ERR_UNSUPPORTED;
}

}  // namespace sf
