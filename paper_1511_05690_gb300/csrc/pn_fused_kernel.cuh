// A whole small product in one launch (template; instantiated per operand
// format in pn_fused_*.cu).
//
// One CTA per 128 x BN output tile keeps its tile through every level of P:
//   1. the maxima of the tile's 128 rows of A and BN columns of B (domain
//      test, power-of-two scales), unless the caller knows them to be 1;
//   2. per level, largest p first: the FP32 operands (from L2 after the first
//      pass) go through a ring of raw 32-column blocks in shared memory, are
//      scaled, powered and cast straight into the operand ring -- no images in
//      global memory -- and one thread issues the MMAs of the blocks that are
//      complete;
//   3. the level kernel's epilogue on the tile; entries left take the CTA to
//      the next level.  Tiles never wait on one another.
// The level launches (maxima, and an image kernel and a GEMM per level) cost
// about 1.3 us on the GPU and 3.5 us on the host each, 78 us for a 256^3
// product whose work takes a few; their images are built once per operand
// block, here once per tile.  What bounds this kernel is that building: about
// 270 instructions per warp and block of 32 columns in 3xTF32 and a barrier
// per block, 40 % of the issue slots used (0.8 us per block and level in
// BF16, 1.2 us in 3xTF32 at 64 columns), so it serves outputs of at most one
// tile per SM and moderate contractions (the rule is in pn_api.cu).
#pragma once
#include "pn_gemm_kernel.cuh"
#include "pn_image.cuh"

namespace pn {
namespace gemm {

// Every warp builds operands; warp 0 also issues the MMAs and warps 2-9 finish
// the tile.
constexpr int FUSED_WORKERS = 16;
constexpr int FUSED_BUILD = 32 * FUSED_WORKERS;

// Raw operand blocks: 32 columns of A's 128 rows (128-byte rows, 16-byte
// groups XORed with the row modulo 8) and 32 rows of B's BN columns, zeros past
// M, N and K.  Held in shared memory rather than loaded ahead into registers,
// several blocks stay in flight (a block is 24 or 32 KB; one SM needs about
// 50 KB to cover L2's latency), and the build loop has no bounds to check.
// Operands with 16-byte aligned rows arrive by two tensor copies per block; the
// others by per-thread asynchronous copies of 4 bytes, which fill the load
// pipe (1.5 to 2 times slower per block).
constexpr int RAW_K = 32;
__host__ __device__ constexpr int raw_bytes(int BN) { return (TILE_M + BN) * RAW_K * 4; }
__host__ __device__ constexpr int raw_stages(int mode, int BN) {
  return num_stages(mode, BN, 1, 2, true) * stage_bytes(mode, BN) > 100000 ? 3 : 4;
}
__host__ __device__ constexpr int fused_smem(int mode, int BN) {
  return num_stages(mode, BN, 1, 2, true) * stage_bytes(mode, BN) + 1024 /*align*/ +
         LOCAL_CTRL_BYTES + raw_stages(mode, BN) * raw_bytes(BN);
}

// The copies of raw block i (columns 32 i .. of A, rows 32 i .. of B) by the
// workers; one group per thread.
struct RawSrc {
  const float* a;   // the tile's first row of A, first column of B
  const float* b;
  int64_t lda, ldb;
  int32_t rows, cols, K;   // rows of A and columns of B that exist (> 0)
  bool vec_a, vec_b;       // rows are 16-byte aligned
};

template <int BN>
__device__ __noinline__ void raw_issue(const RawSrc& rs, uint32_t dst, int i, int t) {
  const int k0 = i * RAW_K;
  if (rs.vec_a) {
#pragma unroll
    for (int u = 0; u < TILE_M * 8 / FUSED_BUILD; ++u) {
      const int r = (t >> 3) + (FUSED_BUILD / 8) * u, c = t & 7;
      const int room = r < rs.rows ? 4 * max(0, min(4, rs.K - k0 - 4 * c)) : 0;
      cp_async16(dst + r * 128 + ((c ^ (r & 7)) << 4),
                 rs.a + (room ? r * rs.lda + k0 + 4 * c : 0), room);
    }
  } else {
#pragma unroll 4
    for (int u = 0; u < TILE_M * 32 / FUSED_BUILD; ++u) {
      const int r = (t >> 5) + FUSED_WORKERS * u, k = t & 31;
      const int room = r < rs.rows && k0 + k < rs.K ? 4 : 0;
      cp_async4(dst + r * 128 + (((k >> 2) ^ (r & 7)) << 4) + (k & 3) * 4,
                rs.a + (room ? r * rs.lda + k0 + k : 0), room);
    }
  }
  const uint32_t db = dst + TILE_M * 128;
  if (rs.vec_b) {
    constexpr int CH = BN / 4;  // 16-byte groups per row
#pragma unroll
    for (int u = 0; u < RAW_K * CH / FUSED_BUILD; ++u) {
      const int k = t / CH + (FUSED_BUILD / CH) * u, c = t & (CH - 1);
      const int room = k0 + k < rs.K ? 4 * max(0, min(4, rs.cols - 4 * c)) : 0;
      cp_async16(db + k * BN * 4 + c * 16, rs.b + (room ? (k0 + k) * rs.ldb + 4 * c : 0), room);
    }
  } else {
#pragma unroll 4
    for (int u = 0; u < RAW_K * BN / FUSED_BUILD; ++u) {
      const int k = t / BN + (FUSED_BUILD / BN) * u, n = t & (BN - 1);
      const int room = k0 + k < rs.K && n < rs.cols ? 4 : 0;
      cp_async4(db + (k * BN + n) * 4, rs.b + (room ? (k0 + k) * rs.ldb + n : 0), room);
    }
  }
}

// The same copies for whole blocks (32 (i + 1) <= K), with everything that
// does not depend on the block worked out once: about five instructions per
// copy instead of 25, which otherwise took half of the kernel's issue slots.
template <int BN>
struct RawWalk {
  static constexpr int CH = BN / 4;
  static constexpr int UA4 = TILE_M * 8 / FUSED_BUILD, UB4 = RAW_K * CH / FUSED_BUILD;
  static constexpr int UA1 = TILE_M * 32 / FUSED_BUILD, UB1 = RAW_K * BN / FUSED_BUILD;
  const float* pa[UA4];   // 16-byte copies: the rows' next group; else pa[0]: column
  const float* pb;        // the thread's first row and column of the next block
  int64_t sb;             // rows of B between the thread's copies
  uint32_t da, db;        // offsets of the thread's first copies in a block
  uint32_t na[UA4], nb;   // bytes per copy (0: past the operand)

  __device__ __forceinline__ void init(const RawSrc& rs, int t) {
    if (rs.vec_a) {
      const int r0 = t >> 3, c = t & 7;
      da = r0 * 128 + ((c ^ (r0 & 7)) << 4);
#pragma unroll
      for (int u = 0; u < UA4; ++u) {
        const int r = r0 + (FUSED_BUILD / 8) * u;
        pa[u] = rs.a + (int64_t)min(r, rs.rows - 1) * rs.lda + 4 * c;
        na[u] = r < rs.rows ? 16u : 0u;
      }
    } else {
      const int r0 = t >> 5, k = t & 31;
      da = r0 * 128 + (((k >> 2) ^ (r0 & 7)) << 4) + (k & 3) * 4;
      pa[0] = rs.a + k;
    }
    if (rs.vec_b) {
      const int c = t & (CH - 1);
      nb = 4 * max(0, min(4, rs.cols - 4 * c));
      pb = rs.b + (int64_t)(t / CH) * rs.ldb + (nb ? 4 * c : 0);
      sb = (int64_t)(FUSED_BUILD / CH) * rs.ldb;
      db = TILE_M * 128 + (t / CH) * BN * 4 + c * 16;
    } else {
      const int n = t & (BN - 1);
      nb = n < rs.cols ? 4u : 0u;
      pb = rs.b + (int64_t)(t / BN) * rs.ldb + (nb ? n : 0);
      sb = (int64_t)(FUSED_BUILD / BN) * rs.ldb;
      db = TILE_M * 128 + (t / BN) * BN * 4 + n * 4;
    }
  }

  // Block i (the blocks in order) into the ring slot dst.
  __device__ __forceinline__ void issue(const RawSrc& rs, uint32_t dst, int i, int t) {
    if ((i + 1) * RAW_K > rs.K) {  // the last block, or past it
      raw_issue<BN>(rs, dst, i, t);
      return;
    }
    if (rs.vec_a) {
#pragma unroll
      for (int u = 0; u < UA4; ++u) {
        cp_async16(dst + da + u * (FUSED_BUILD / 8) * 128, pa[u], na[u]);
        pa[u] += RAW_K;
      }
    } else {
      const int r0 = t >> 5;
#pragma unroll
      for (int u = 0; u < UA1; ++u) {
        const int r = r0 + FUSED_WORKERS * u;
        cp_async4(dst + da + u * FUSED_WORKERS * 128,
                  pa[0] + (int64_t)min(r, rs.rows - 1) * rs.lda, r < rs.rows ? 4u : 0u);
      }
      pa[0] += RAW_K;
    }
    if (rs.vec_b) {
#pragma unroll
      for (int u = 0; u < UB4; ++u) {
        cp_async16(dst + db + u * (FUSED_BUILD / CH) * BN * 4, pb, nb);
        pb += sb;
      }
    } else {
#pragma unroll
      for (int u = 0; u < UB1; ++u) {
        cp_async4(dst + db + u * (FUSED_BUILD / BN) * BN * 4, pb, nb);
        pb += sb;
      }
    }
  }
};

// Ring position of the raw blocks (carried over from walk to walk) and the
// tensor copies' barriers.
struct RawRing {
  uint32_t base;
  uint64_t* full;   // [RAW], tensor copies only
  int slot;         // the slot of the next block to read
  uint32_t phase;   // its barrier's parity
  bool tma;
};

// Walks the raw blocks 0 .. count - 1 of tile (tm, tn): body(i, addr) with all
// of block i in shared memory at addr, RAW - 1 blocks ahead in flight; done(i)
// once every thread has finished the body of block i (and fenced its
// shared-memory writes for the async proxy).  Called by every thread.  drop_first
// (test hook): block 0 is never copied.
template <int BN, int RAW, typename Body, typename Done>
__device__ __forceinline__ void raw_walk(const RawSrc& rs, RawRing& rr, const OperandMaps& maps,
                                         const Ctx& cx, int32_t* status, bool drop_first, int tm,
                                         int tn, int count, int t, const Body& body,
                                         const Done& done) {
  RawWalk<BN> w;
  if (!rr.tma) w.init(rs, t);
  int put = rr.slot;
#pragma unroll 1
  for (int i = 1 - RAW; i < count; ++i) {
    if (i >= 0) {
      if (!rr.tma) {
        cp_async_wait<RAW - 2>();
      } else if (!mbar_wait(&rr.full[rr.slot], rr.phase, cx.tmo, cx.abort_flag)) {
        *cx.abort_flag = 1;
        set_status(status, PN_ETIMEOUT);
        // the walk goes on to its end: thread 0 still waits for every block, so
        // that no copy outlives the CTA's memory
        if (t == 0 && !mbar_wait_drain(&rr.full[rr.slot], rr.phase, cx.tmo) && drop_first)
          mbar_arrive(&rr.full[rr.slot]);  // in place of the block that was left out
      }
      __syncthreads();  // block i has landed, block i - 1 is finished, for every thread
      if (i > 0) done(i - 1);
    }
    const int n = i + RAW - 1;
    const uint32_t dst = rr.base + put * raw_bytes(BN);
    if (n < count) {
      if (!rr.tma) {
        w.issue(rs, dst, n, t);
      } else if (t == 0 && !(drop_first && n == 0)) {
        mbar_arrive_expect_tx(&rr.full[put], raw_bytes(BN));
        tma_load_2d(dst, &maps.a, n * RAW_K, tm * TILE_M, &rr.full[put]);
        tma_load_2d(dst + TILE_M * 128, &maps.b, tn * BN, n * RAW_K, &rr.full[put]);
      }
      put = put + 1 == RAW ? 0 : put + 1;
    }
    if (!rr.tma) cp_async_commit();
    if (i >= 0) {
      body(i, rr.base + rr.slot * raw_bytes(BN));
      if (++rr.slot == RAW) {
        rr.slot = 0;
        rr.phase ^= 1u;
      }
    }
  }
  if (!rr.tma) cp_async_wait<0>();
  __syncthreads();
  done(count - 1);
}

__device__ __forceinline__ void lds_pairs(uint32_t addr, uint64_t& a, uint64_t& b) {
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(addr) : "memory");
}
__device__ __forceinline__ uint4 lds_u4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
__device__ __forceinline__ float lds_f32(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void sts_u4(uint32_t addr, uint4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y),
               "r"(v.z), "r"(v.w)
               : "memory");
}

// The MMAs of one image block (128 bytes of K): K steps of 32 bytes, 3xTF32 as
// lo hi + hi lo + hi hi (small terms first), the order of run_mma.
template <int MODE, int BN>
__device__ __forceinline__ void fused_mma(uint32_t acc, uint32_t sa, uint32_t sb, int lo_off,
                                          bool accumulate) {
  constexpr int KIND = mma_kind(MODE);
  constexpr uint32_t IDESC = idesc_make(ab_format(MODE), TILE_M, BN);
  // the address field counts 16-byte units, so offsets add to the descriptor
  const uint64_t da = sdesc_sw128(sa), db = sdesc_sw128(sb);
  const uint32_t lo = lo_off >> 4;
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) {
    const uint64_t ad = da + 2 * kk, bd = db + 2 * kk;
    const uint32_t on = accumulate || kk != 0;
    if constexpr (mode_planes(MODE) == 1) {
      mma_ss<KIND>(acc, ad, bd, IDESC, on);
    } else {
      mma_ss<KIND>(acc, ad + lo, bd, IDESC, on);
      mma_ss<KIND>(acc, ad, bd + lo, IDESC, 1u);
      mma_ss<KIND>(acc, ad, bd, IDESC, 1u);
    }
  }
}

// x / s for scales whose reciprocal is no normal float.
static __device__ __noinline__ uint64_t div2(uint64_t v, float s) {
  float a, b;
  f32x2_unpack(v, a, b);
  return f32x2_pack(a / s, b / s);
}

// Scales and powers U chunks of EPC values.  inv: the scales' reciprocals, or
// (!exact) the scales, which then divide.
template <int U, int E2>
__device__ __forceinline__ void fused_scale(uint64_t (&v)[U][E2], const float (&inv)[U],
                                            bool exact) {
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int e = 0; e < E2; ++e)
      v[u][e] = exact ? f32x2_mul(v[u][e], f32x2_pack(inv[u], inv[u])) : div2(v[u][e], inv[u]);
}
template <int U, int E2>
__device__ __forceinline__ void fused_times(uint64_t (&v)[U][E2], bool square, float f) {
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int e = 0; e < E2; ++e) v[u][e] = f32x2_mul(v[u][e], square ? v[u][e] : f32x2_pack(f, f));
}

// Casts and stores U chunks at the image addresses dst[u] + at (3xTF32: the lo
// plane lo_off further).
template <int MODE, int U>
__device__ __forceinline__ void fused_store(const uint32_t (&dst)[U], uint32_t sx, uint32_t at,
                                            int lo_off,
                                            const uint64_t (&v)[U][Packer<MODE>::EPC / 2]) {
  using PK = Packer<MODE>;
  constexpr int EPC = PK::EPC;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    float f[EPC];
#pragma unroll
    for (int e = 0; e < EPC / 2; ++e) f32x2_unpack(v[u][e], f[2 * e], f[2 * e + 1]);
    uint4 hi, lo;
    PK::pack(f, hi, lo);
    const uint32_t d = (dst[u] ^ sx) + at;
    sts_u4(d, hi);
    if constexpr (mode_planes(MODE) == 2) sts_u4(d + lo_off, lo);
  }
}

template <int MODE, int BN>
__global__ void __launch_bounds__(FUSED_BUILD, 1)
    k_fused_product(const __grid_constant__ Common cm, const __grid_constant__ FusedArgs fa,
                    const __grid_constant__ OperandMaps maps) {
  constexpr int NG = 2;
  constexpr int STAGES = num_stages(MODE, BN, 1, NG, true);
  constexpr int STAGE_BYTES = stage_bytes(MODE, BN);
  constexpr int A_BYTES = IMG_BYTES, LO_OFF = IMG_BYTES + IMG_BYTES * BN / TILE_M;
  constexpr int RAW = raw_stages(MODE, BN);
  constexpr int EPC = Packer<MODE>::EPC;
  constexpr int SLOTS = RAW_K / EPC;           // image slots per raw block
  constexpr int SUBS = mode_bk(MODE) / RAW_K;  // raw blocks per image block
  constexpr int NA = TILE_M * SLOTS, NB = BN * SLOTS;  // chunks of A and B per raw block
  constexpr int UA = NA > FUSED_BUILD ? NA / FUSED_BUILD : 1;
  constexpr int UB = NB > FUSED_BUILD ? NB / FUSED_BUILD : 1;
  constexpr int ACC_BUFS = acc_bufs(BN);
  static_assert(raw_stages(MODE, BN) * raw_bytes(BN) >= EPI_WARPS * STG_BYTES,
                "the epilogue's staging lies in the raw ring");
  pdl_wait();
  pdl_trigger();
  Ctx cx = ctx_setup<MODE, BN, 1, NG, true>(false, cm.timeout_ns);
  cx.wid = 0;
  cx.wstride = 1;
  cx.tile = blockIdx.x;
  const uint32_t img = smem_u32(cx.smem);
  // control block: ctx_setup's barriers (256 bytes), the raw ring's, the scales
  uint8_t* const ctrl = cx.smem + STAGES * STAGE_BYTES;
  RawRing rr;
  rr.base = img + STAGES * STAGE_BYTES + LOCAL_CTRL_BYTES;
  rr.full = reinterpret_cast<uint64_t*>(ctrl + 256);
  rr.slot = 0;
  rr.phase = 0;
  rr.tma = maps.has_a && maps.has_b;
  const bool drop_first = (cm.debug_flags & 16) != 0;
  int32_t* const s_left = reinterpret_cast<int32_t*>(ctrl + 320);
  float* const s_scale = reinterpret_cast<float*>(ctrl + 512);  // maxima as bits first
  cx.rs = s_scale;
  cx.cs = s_scale + TILE_M;
  cx.left = s_left;
  const Prob& P = cm.single;
  const int t = threadIdx.x, warp = t >> 5;
  int tm, tn;
  tile_coords<1>(P, cx.tile, 0, tm, tn);
  RawSrc rs;
  rs.a = P.A + (int64_t)tm * TILE_M * P.lda;
  rs.b = P.B + tn * BN;
  rs.lda = P.lda;
  rs.ldb = P.ldb;
  rs.rows = min(TILE_M, P.M - tm * TILE_M);
  rs.cols = min(BN, P.N - tn * BN);
  rs.K = P.K;
  rs.vec_a = (P.lda & 3) == 0 && (reinterpret_cast<uintptr_t>(P.A) & 15) == 0;
  rs.vec_b = (P.ldb & 3) == 0 && (reinterpret_cast<uintptr_t>(P.B) & 15) == 0;

  uint32_t* const smax = reinterpret_cast<uint32_t*>(s_scale);
  for (int i = t; i < TILE_M + BN; i += FUSED_BUILD) smax[i] = fa.unit_scales ? 0x3f800000u : 0u;
  if (t == 0) {
    *s_left = 0;
    for (int i = 0; i < RAW; ++i) mbar_init(&rr.full[i], 1);
    fence_barrier_init();
  }
  __syncthreads();
  if (!fa.unit_scales) {
    // maxima on raw bits (the domain test as in k_maxes): a thread's quarter
    // of a row of A and its part of a column of B
    constexpr int KB_T = RAW_K * BN / FUSED_BUILD;  // values of B per thread and block
    const int ra = t >> 2, n = t & (BN - 1);
    uint32_t ua = 0u, ub = 0u, oa[2];
    bool bad = false;
#pragma unroll
    for (int j = 0; j < 2; ++j) oa[j] = ra * 128 + ((((t & 3) * 2 + j) ^ (ra & 7)) << 4);
    const uint32_t ob = TILE_M * 128 + ((t / BN) * KB_T * BN + n) * 4;
    raw_walk<BN, RAW>(
        rs, rr, maps, cx, cm.status, drop_first, tm, tn, (P.K + RAW_K - 1) / RAW_K, t,
        [&](int, uint32_t blk) {
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const uint4 v = lds_u4(blk + oa[j]);
            ua = umax3(ua, max(v.x, v.y), max(v.z, v.w));
          }
#pragma unroll
          for (int e = 0; e < KB_T; ++e)
            ub = max(ub, __float_as_uint(lds_f32(blk + ob + e * BN * 4)));
        },
        [](int) {});
    // over the whole row or column (others are zeros, but after a copy that never landed)
    if (ua > DOMAIN_MAX_BITS && ra < rs.rows)
      ua = take_exact(exact_max_bits(rs.a + ra * rs.lda, 1, P.K), bad);
    if (ub > DOMAIN_MAX_BITS && n < rs.cols) ub = take_exact(exact_max_bits(rs.b + n, rs.ldb, P.K), bad);
    ua = max(ua, __shfl_xor_sync(0xffffffffu, ua, 1));
    ua = max(ua, __shfl_xor_sync(0xffffffffu, ua, 2));
    if ((t & 3) == 0) smax[ra] = ua;
    atomicMax(smax + TILE_M + n, ub);
    if (__syncthreads_or(bad) && t == 0) set_status(cm.status, PN_EDOMAIN);
    for (int i = t; i < TILE_M + BN; i += FUSED_BUILD) s_scale[i] = scale_from_bits(cm, smax[i]);
    __syncthreads();
  }

  // the thread's chunks of a raw block: where they lie in it and in an image
  // stage (raw block sub of an image block: the slot's upper bits, see below),
  // and their scales.  Where A has fewer chunks than there are threads, B's go
  // to the others first.
  const int tb = NA < FUSED_BUILD ? (t - NA) & (FUSED_BUILD - 1) : t;
  const bool live_a = t < NA, live_b = tb < NB;
  uint32_t src_a[UA], src_b[UB], dst_a[UA], dst_b[UB];
  float inv_a[UA], inv_b[UB];
  bool exact = true;
#pragma unroll
  for (int u = 0; u < UA; ++u) {
    const int row = (t / SLOTS + (FUSED_BUILD / SLOTS) * u) & (TILE_M - 1), slot = t & (SLOTS - 1);
    src_a[u] = row * 128 + (((slot * (EPC / 4)) ^ (row & 7)) << 4);
    dst_a[u] = img + sw128_offset(row, slot * 16);
    inv_a[u] = cx.rs[row];
    exact = exact && recip_exact(inv_a[u]);
  }
#pragma unroll
  for (int u = 0; u < UB; ++u) {
    const int row = tb & (BN - 1), slot = (tb / BN + (FUSED_BUILD / BN) * u) & (SLOTS - 1);
    src_b[u] = TILE_M * 128 + (slot * EPC * BN + row) * 4;
    dst_b[u] = img + A_BYTES + sw128_offset(row, slot * 16);
    inv_b[u] = cx.cs[row];
    exact = exact && recip_exact(inv_b[u]);
  }
  exact = __all_sync(0xffffffffu, exact);
  if (exact) {
#pragma unroll
    for (int u = 0; u < UA; ++u) inv_a[u] = 1.0f / inv_a[u];
#pragma unroll
    for (int u = 0; u < UB; ++u) inv_b[u] = 1.0f / inv_b[u];
  }

  const float opscale = ldexpf(1.0f, cm.s_op);
  int stage = 0;
  uint32_t phase = 0;
  bool aborted = false;
  for (int s = 0; s < fa.n_p; ++s) {
    Level lv{};
    lv.q = fa.n_p - 1 - s;
    lv.plog = fa.p_log2[lv.q];
    lv.is_top = s == 0;
    lv.is_bottom = lv.q == 0;
    // r = 1 projection: as set_projection
    lv.proj_next = fa.estimator == 1 && lv.q > 0 && fa.p_log2[lv.q - 1] == lv.plog - 1;
    lv.proj_here =
        fa.estimator == 1 && lv.q + 1 < fa.n_p && fa.p_log2[lv.q + 1] == lv.plog + 1;
    const uint32_t acc = cx.tmem_base + (s & (ACC_BUFS - 1)) * BN;
    int mma_stage = stage;  // the stage of the next block to multiply
    raw_walk<BN, RAW>(
        rs, rr, maps, cx, cm.status, drop_first, tm, tn, P.KB * SUBS, t,
        [&](int i, uint32_t blk) {
          const int sub = SUBS == 1 ? 0 : i % SUBS;
          if (sub == 0 && !aborted &&
              !mbar_wait(&cx.empty[stage], phase ^ 1u, cx.tmo, cx.abort_flag)) {
            *cx.abort_flag = 1;
            set_status(cm.status, PN_ETIMEOUT);
            aborted = true;
          }
          if (aborted) return;
          // slots SLOTS sub ..: these bits of the slot pass through the
          // swizzle's XOR unchanged
          const uint32_t at = stage * STAGE_BYTES, sx = (SLOTS * sub) << 4;
          const bool do_a = NA >= FUSED_BUILD || live_a, do_b = NB >= FUSED_BUILD || live_b;
          uint64_t va[UA][EPC / 2], vb[UB][EPC / 2];
          if (do_a) {
#pragma unroll
            for (int u = 0; u < UA; ++u)
#pragma unroll
              for (int e = 0; e < EPC / 4; ++e)
                lds_pairs(blk + (src_a[u] ^ (e << 4)), va[u][2 * e], va[u][2 * e + 1]);
          }
          if (do_b) {
#pragma unroll
            for (int u = 0; u < UB; ++u) {
              const uint32_t b0 = blk + src_b[u];
#pragma unroll
              for (int e = 0; e < EPC; e += 2)
                vb[u][e / 2] = f32x2_pack(lds_f32(b0 + e * BN * 4), lds_f32(b0 + (e + 1) * BN * 4));
            }
          }
          if (do_a && do_b) {  // their chains of squarings interleaved
            fused_scale(va, inv_a, exact);
            fused_scale(vb, inv_b, exact);
#pragma unroll 1
            for (int p = 0; p < lv.plog; ++p) {
              fused_times(va, true, 0.0f);
              fused_times(vb, true, 0.0f);
            }
          } else if (do_a) {
            fused_scale(va, inv_a, exact);
#pragma unroll 1
            for (int p = 0; p < lv.plog; ++p) fused_times(va, true, 0.0f);
          } else if (do_b) {
            fused_scale(vb, inv_b, exact);
#pragma unroll 1
            for (int p = 0; p < lv.plog; ++p) fused_times(vb, true, 0.0f);
          }
          if (mode_op_shift(MODE) != 0) {
            if (do_a) fused_times(va, false, opscale);
            if (do_b) fused_times(vb, false, opscale);
          }
          if (do_a) fused_store<MODE>(dst_a, sx, at, LO_OFF, va);
          if (do_b) fused_store<MODE>(dst_b, sx, at, LO_OFF, vb);
          fence_proxy_async_smem();  // before the MMAs (async proxy) read the stage
          if (sub == SUBS - 1 && ++stage == STAGES) {
            stage = 0;
            phase ^= 1u;
          }
        },
        [&](int i) {
          // an image block is complete: its MMAs, and the stage's release
          if (t != 0 || (SUBS > 1 && i % SUBS != SUBS - 1) || *cx.abort_flag) return;
          tc_fence_after();
          const uint32_t sa = img + mma_stage * STAGE_BYTES;
          fused_mma<MODE, BN>(acc, sa, sa + A_BYTES, LO_OFF, i >= SUBS);
          mma_commit(&cx.empty[mma_stage]);
          if (++mma_stage == STAGES) mma_stage = 0;
        });
    const int buf = s & (ACC_BUFS - 1);
    if (t == 0) mma_commit(&cx.acc_full[buf]);
    if (warp >= 2 && warp < 2 + 4 * NG) {
      run_epilogue<MODE, BN, 0, 1, NG, false, true>(cm, lv, cx, 1, false, s, Ready{nullptr, 0, 0});
      // the staging buffers were written by ordinary stores, and the next
      // level's tensor copies (async proxy) write the same bytes of the raw ring
      fence_proxy_async_smem();
    }
    __syncthreads();
    if (*cx.abort_flag || !*s_left) break;  // uniform: nothing writes either before the next barrier
    __syncthreads();
  }
  if (*cx.abort_flag && t == 0) {
    // no MMA may outlive the CTA's memory (raw_walk has waited for the copies)
    mma_commit(cx.drain);
    mbar_wait_drain(cx.drain, 0, cx.tmo);
  }
  ctx_teardown<BN>(cx);
}

template <int MODE, int BN>
inline int launch_fused_t(const Common& cm, const FusedArgs& fa, void* stream) {
  constexpr int smem = fused_smem(MODE, BN);
  static_assert(smem <= 232448, "shared memory of one CTA");
  if (const cudaError_t e = allow_smem<k_fused_product<MODE, BN>>(smem)) return e;
  OperandMaps maps;
  make_raw_maps(cm, RAW_K, maps);
  const cudaError_t e = launch_pdl(k_fused_product<MODE, BN>, dim3(cm.total_tiles),
                                   dim3(FUSED_BUILD), smem, stream, cm, fa, maps);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace gemm
}  // namespace pn
