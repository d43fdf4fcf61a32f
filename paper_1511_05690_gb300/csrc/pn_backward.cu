// Device side of the adjoint of the p-norm product (maxprod_pnorm_backward).
//
// With p = p*_ij held fixed per entry, C_ij = (sum_k (a_ik b_kj)^p)^(1/p) is
// differentiable (the p-norm rings are, Sec. 4), and in the forward's scaled
// variables a' = a / r_i, b' = b / c_j, S = sum_k (a'_ik b'_kj)^p:
//   dC_ij / da_ik = (C_ij / S_ij) (a'_ik^(p-1) / r_i) b'_kj^p.
// Hence, with W_ij = dC_ij C_ij / S_ij and W^(p) = W masked to p*_ij = p,
//   dA = sum_p (a'^(p-1) / r) (.) (W^(p) B'^p^T),
//   dB = sum_p (b'^(p-1) / c) (.) (A'^p^T W^(p)),
// two ring GEMMs per p that occurs in p_sel.  This file builds their operand
// images (recomputed from A, B, C, S_sel, p_sel rather than stored) and the
// mask of the p values that occur; the GEMMs are the tensor-core level kernel
// with its gradient epilogue.
#include "pn_launch.h"
#include "pn_pack.cuh"

namespace pn {

namespace {

constexpr int BW_THREADS = 256;

// Bit q of *mask is set when some entry of p_sel selected p = 2^plog_list[q].
struct PList {
  int32_t n_p;
  int32_t plog[PN_MAX_P];
};

// Row and column scales from the maxima (same rule as the forward), and the
// mask of the p that occur in p_sel.
__global__ void __launch_bounds__(BW_THREADS)
    k_bw_prep(const __grid_constant__ Common cm, const uint8_t* __restrict__ psel, int64_t count,
              PList pl, uint32_t* mask) {
  pdl_wait();
  pdl_trigger();
  const Prob& P = cm.single;
  const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = first; e < (int64_t)P.M + P.N; e += stride) {
    const bool col = e >= P.M;
    const int64_t idx = col ? e - P.M : e;
    float s = 1.0f;
    if (cm.scaling != 0) {
      const uint32_t bits = cm.scaling == 1 ? cm.gmax[col ? 1 : 0] : (col ? cm.cmax : cm.rmax)[idx];
      s = pow2_ceil_f(__uint_as_float(bits));
    }
    (col ? cm.c : cm.r)[idx] = s;
  }
  // bit log2 p of every entry, 16 entries per load where p_sel is aligned
  uint32_t seen = 0;
  auto take = [&](uint32_t byte) { seen |= 1u << min(byte & 0x7Fu, 31u); };
  const int64_t vecs = (reinterpret_cast<uintptr_t>(psel) & 15) == 0 ? count >> 4 : 0;
  for (int64_t e = first; e < vecs; e += stride) {
    const uint4 v = __ldg(reinterpret_cast<const uint4*>(psel) + e);
#pragma unroll
    for (int b = 0; b < 32; b += 8) {
      take(v.x >> b); take(v.y >> b); take(v.z >> b); take(v.w >> b);
    }
  }
  for (int64_t e = (vecs << 4) + first; e < count; e += stride) take(psel[e]);
  seen = __reduce_or_sync(0xffffffffu, seen);
  if ((threadIdx.x & 31) == 0) {
    uint32_t bits = 0;
    for (int q = 0; q < pl.n_p; ++q) bits |= ((seen >> pl.plog[q]) & 1u) << q;
    if (bits) atomicOr(mask, bits);
  }
}

// The operand images of one p, all four in one launch.  A block takes 128 x 128
// values of W^(p) (job 0), of the powered B (job 1) or of the powered A (job 2)
// through shared memory and writes them as image tiles: W in both
// orientations (rows i, contraction j, and the reverse), so that its four
// sources (13 bytes per entry) are read and divided once, B' as rows k and
// A' as its transpose.  What bounds it is HBM: at 2048^2 in 3xTF32 the four
// images are 134 MB of writes and 88 MB of reads; 44 us, 98 us as four launches of
// one block per 16 KB tile (W formed twice, a division per value in each).
template <int MODE>
__global__ void __launch_bounds__(BW_THREADS) k_bw_images(const __grid_constant__ BwImages im) {
  pdl_wait();
  pdl_trigger();
  if (!((*im.pmask >> im.q) & 1u)) return;  // no entry selected this p
  using PK = Packer<MODE>;
  constexpr int EPC = PK::EPC, BK = mode_bk(MODE), KBS = 128 / BK, LD = 129;
  extern __shared__ float tile[];  // [128][LD]
  int id = blockIdx.x, job = 0;
  while (job < 2 && id >= im.blocks[job]) id -= im.blocks[job++];
  const int rb = id / im.cols[job], cb = id - rb * im.cols[job];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rows = job == 0 ? im.M : job == 1 ? im.K : im.M;  // source rows, columns
  const int cols = job == 0 ? im.N : job == 1 ? im.N : im.K;
  // columns cb 128 + lane + 32 c; all loads are issued, unconditionally, before
  // any is used: past the source they read its last row or column and are zeroed
  int col[4];
  bool cin[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    cin[c] = cb * 128 + lane + 32 * c < cols;
    col[c] = min(cb * 128 + lane + 32 * c, cols - 1);
  }
  constexpr int U = 2;  // rows per step
  if (job == 0) {
#pragma unroll 1
    for (int i = 0; i < 16; i += U) {
      float S[U][4], d[U][4], C[U][4];
      int p[U][4];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int64_t e = (int64_t)min(rb * 128 + warp + 8 * (i + u), rows - 1) * im.N;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          S[u][c] = __ldg(im.S + e + col[c]);
          d[u][c] = __ldg(im.dC + e + col[c]);
          C[u][c] = __ldg(im.Cv + e + col[c]);
          p[u][c] = __ldg(im.psel + e + col[c]) & 0x7F;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int rr = warp + 8 * (i + u);
        const bool rin = rb * 128 + rr < rows;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const bool take = rin && cin[c] && p[u][c] == im.plog && S[u][c] > 0.0f;
          tile[rr * LD + lane + 32 * c] = take ? d[u][c] * C[u][c] / S[u][c] : 0.0f;
        }
      }
    }
  } else {
    const float* src = job == 1 ? im.B : im.A;
    float cs[4], ci[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      cs[c] = job == 1 ? __ldg(im.c + col[c]) : 1.0f;
      ci[c] = 1.0f / cs[c];
    }
#pragma unroll 1
    for (int i = 0; i < 16; i += 2 * U) {
      float v[2 * U][4], rs[2 * U];
#pragma unroll
      for (int u = 0; u < 2 * U; ++u) {
        const int r = min(rb * 128 + warp + 8 * (i + u), rows - 1);
        rs[u] = job == 2 ? __ldg(im.r + r) : 1.0f;
#pragma unroll
        for (int c = 0; c < 4; ++c) v[u][c] = __ldg(src + (int64_t)r * cols + col[c]);
      }
#pragma unroll
      for (int u = 0; u < 2 * U; ++u) {
        const bool rin = rb * 128 + warp + 8 * (i + u) < rows;
        const float ri = 1.0f / rs[u];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float s = job == 2 ? rs[u] : cs[c], inv = job == 2 ? ri : ci[c];
          v[u][c] = rin && cin[c] ? div_pow2(v[u][c], s, inv, recip_exact(s)) : 0.0f;
        }
      }
#pragma unroll 1
      for (int t = 0; t < im.plog; ++t) {
#pragma unroll
        for (int u = 0; u < 2 * U; ++u)
#pragma unroll
          for (int c = 0; c < 4; ++c) v[u][c] *= v[u][c];
      }
#pragma unroll
      for (int u = 0; u < 2 * U; ++u)
#pragma unroll
        for (int c = 0; c < 4; ++c) tile[(warp + 8 * (i + u)) * LD + lane + 32 * c] = v[u][c];
    }
  }
  __syncthreads();
  // rows as image rows (jobs 0, 1), columns as image rows (jobs 0, 2)
#pragma unroll 1
  for (int o = 0; o < 2; ++o) {
    const BwDst& d = im.dst[job][o];
    const int row_blk = o == 0 ? rb : cb, k_blk = (o == 0 ? cb : rb) * KBS;
    if (d.img == nullptr || row_blk >= d.RB) continue;
#pragma unroll 1
    for (int k = 0; k < KBS; ++k) {
      if (k_blk + k >= d.KB) break;
      uint8_t* dst = d.img + ((int64_t)(row_blk * d.KB + k_blk + k) << 14);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int ch = threadIdx.x + BW_THREADS * u, rr = ch >> 3, cc = ch & 7;
        float v[EPC];
#pragma unroll
        for (int e = 0; e < EPC; ++e) {
          const int kk = k * BK + cc * EPC + e;
          v[e] = o == 0 ? tile[rr * LD + kk] : tile[kk * LD + rr];
        }
        uint4 hi, lo;
        PK::pack(v, hi, lo);
        const uint32_t off = sw128_offset(rr, cc * 16);
        *reinterpret_cast<uint4*>(dst + off) = hi;
        if constexpr (MODE == MODE_3XTF32) *reinterpret_cast<uint4*>(dst + d.plane + off) = lo;
      }
    }
  }
}

template <int MODE>
int launch_images_t(const BwImages& im, void* stream) {
  constexpr int smem = 128 * 129 * 4;
  if (const cudaError_t e = allow_smem<k_bw_images<MODE>>(smem)) return e;
  const int blocks = im.blocks[0] + im.blocks[1] + im.blocks[2];
  if (blocks <= 0) return 0;
  const cudaError_t e = launch_pdl(k_bw_images<MODE>, dim3(blocks), dim3(BW_THREADS), smem, stream,
                                   im);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

int launch_bw_prep(const Common& cm, const uint8_t* psel, int64_t count, const int32_t* plog_list,
                   int n_p, uint32_t* mask, void* stream) {
  PList pl{};
  pl.n_p = n_p;
  for (int q = 0; q < n_p; ++q) pl.plog[q] = plog_list[q];
  const int64_t work = count / 16 > (int64_t)cm.single.M + cm.single.N
                           ? count / 16 : (int64_t)cm.single.M + cm.single.N;
  int64_t blocks = (work + BW_THREADS - 1) / BW_THREADS;
  if (blocks > 152 * 8) blocks = 152 * 8;
  if (blocks < 1) blocks = 1;
  const cudaError_t e = launch_pdl(k_bw_prep, dim3(static_cast<unsigned>(blocks)),
                                   dim3(BW_THREADS), 0, stream, cm, psel, count, pl, mask);
  return e != cudaSuccess ? e : cudaGetLastError();
}

int launch_bw_images(int mode, const BwImages& im, void* stream) {
  switch (mode) {
    case MODE_3XTF32: return launch_images_t<MODE_3XTF32>(im, stream);
    case MODE_TF32: return launch_images_t<MODE_TF32>(im, stream);
    case MODE_BF16: return launch_images_t<MODE_BF16>(im, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pn
