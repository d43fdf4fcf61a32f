// Bias corrections of the p-norm estimate.
//
// correction 1 (Sec. 2.1, the envelope ||u||_inf <= ||u||_p <= K^(1/p) ||u||_inf):
//   the estimate divided by K^(1/p*), applied in the GEMM epilogue.
// correction 2 (Discussion: an affine model fitted to a few exact
//   sub-solutions): at caller-chosen sample entries the exact max and the
//   estimate are computed directly here; a least-squares line
//   exact = a_q * est + b_q per p* class q, in the scaled space
//   (value / (r_i c_j)), is applied to every entry by the GEMM epilogue.
#include <cstdint>

#include "pn_device.cuh"
#include "pn_launch.h"

namespace pn {

namespace {

constexpr int FIT_THREADS = 256;  // one block per sample

// S[q] += u^p for every p of P.
__device__ __forceinline__ void fit_add(const FitArgs& fa, float u, float (&S)[PN_MAX_P]) {
  float t = u;
  int lg = 0;
#pragma unroll
  for (int q = 0; q < PN_MAX_P; ++q) {
    if (q < fa.n_p) {
      while (lg < fa.p_log2[q]) {
        t = t * t;
        ++lg;
      }
      S[q] += t;
    }
  }
}

// The same where P = {1, 2, 4, ...}: one product and one sum per p.
__device__ __forceinline__ void fit_add_dense(int n_p, float u, float (&S)[PN_MAX_P]) {
#pragma unroll
  for (int q = 0; q < PN_MAX_P; ++q) {
    if (q >= n_p) break;
    S[q] += u;
    u = u * u;
  }
}

// A sample's record from its sums: its p* and estimate (the epilogue's rule) and
// the exact value.
__device__ __forceinline__ void fit_record(float tau, const FitArgs& fa, int s,
                                           const float (&S)[PN_MAX_P], float mx) {
  int qs = -1;
  for (int q = fa.n_p - 1; q >= 0; --q) {
    float sq = 0.0f;
#pragma unroll
    for (int t = 0; t < PN_MAX_P; ++t)
      if (t == q) sq = S[t];
    if (sq >= tau) {
      qs = q;
      break;
    }
  }
  const bool unstable = qs < 0;
  if (unstable) qs = 0;
  float s_sel = 0.0f, s_half = 0.0f;
#pragma unroll
  for (int t = 0; t < PN_MAX_P; ++t) {
    if (t == qs) s_sel = S[t];
    if (t == qs - 1) s_half = S[t];
  }
  const double p = ldexp(1.0, fa.p_log2[qs]);
  double est = s_sel > 0.0f ? pow(static_cast<double>(s_sel), 1.0 / p) : 0.0;
  if (fa.estimator == 1 && !unstable && qs > 0 && fa.p_log2[qs - 1] == fa.p_log2[qs] - 1) {
    // r = 1 projection, with the epilogue's clamp of the ratio to <= 1
    const double ratio = static_cast<double>(s_sel) / fmax(static_cast<double>(s_half),
                                                           static_cast<double>(s_sel));
    est = pow(ratio, 2.0 / p);
  }
  fa.samp[2 * s] = est;
  fa.samp[2 * s + 1] = static_cast<double>(mx);
  fa.scls[s] = qs;
}

// One block per sample entry (i, j): u_k = (a_ik / r_i)(b_kj / c_j) in FP32,
// the exact max over k and the p-sums S^(p) for every p of P (each thread a
// strided part of k, then warp and block reductions), the sample's own p* and
// estimate (the same rule as the epilogue); the sample's record (estimate,
// exact value, class) goes to its own slot, so that the class sums can be
// formed in a fixed order (deterministic results).
__global__ void __launch_bounds__(FIT_THREADS)
    k_fit_samples(const __grid_constant__ Common cm, const __grid_constant__ FitArgs fa) {
  __shared__ float red[FIT_THREADS / 32][PN_MAX_P + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int s = blockIdx.x;
  const Prob& P = cm.single;
  const int i = fa.fi[s], j = fa.fj[s];
  if (i < 0 || i >= P.M || j < 0 || j >= P.N) {
    if (threadIdx.x == 0) {
      set_status(cm.status, PN_EINVAL);
      fa.scls[s] = -1;
    }
    return;
  }
  const float ri = cm.r[P.rc_r + i], cj = cm.c[P.rc_c + j];
  float mx = 0.0f;
  float S[PN_MAX_P];
#pragma unroll
  for (int q = 0; q < PN_MAX_P; ++q) S[q] = 0.0f;
  const float* arow = P.A + (int64_t)i * P.lda;
  for (int k = threadIdx.x; k < P.K; k += FIT_THREADS) {
    const float u = (__ldg(arow + k) / ri) * (__ldg(P.B + (int64_t)k * P.ldb + j) / cj);
    mx = fmaxf(mx, u);
    fit_add(fa, u, S);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
#pragma unroll
    for (int q = 0; q < PN_MAX_P; ++q) S[q] += __shfl_xor_sync(0xffffffffu, S[q], off);
  }
  if (lane == 0) {
#pragma unroll
    for (int q = 0; q < PN_MAX_P; ++q) red[warp][q] = S[q];
    red[warp][PN_MAX_P] = mx;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
#pragma unroll
  for (int q = 0; q < PN_MAX_P; ++q) {
    S[q] = 0.0f;
    for (int w = 0; w < FIT_THREADS / 32; ++w) S[q] += red[w][q];
  }
  mx = 0.0f;
  for (int w = 0; w < FIT_THREADS / 32; ++w) mx = fmaxf(mx, red[w][PN_MAX_P]);
  fit_record(P.tau, fa, s, S, mx);
}

// The same sums for many samples, as a stream over B: CTA x takes the
// contraction indices [per x, per (x + 1)), copies these rows of B whole through
// a ring in shared memory, and thread s takes its sample's value from each; the
// samples' values of A come 16 indices at a time, transposed through shared
// memory.  k_fit_samples' reads of B are scattered, a 32-byte sector each, and
// bound per SM (about 4.7 clocks each: 136 us for 1024 samples at n = 8192); here
// B is read once: 67 us, and 24 for the merge.  The partial sums go to
// part[x][value][sample].
// (STREAM_K indices of A per load, STREAM_LD floats between them.)
__global__ void __launch_bounds__(STREAM_THREADS, 1)
    k_fit_stream(const __grid_constant__ Common cm, const __grid_constant__ FitArgs fa, int per,
                 int stages) {
  extern __shared__ __align__(128) uint8_t sm_fit[];
  __shared__ uint64_t full[STREAM_MAX_STAGES], empty[STREAM_MAX_STAGES];
  __shared__ int32_t abort_flag, arow[STREAM_THREADS];
  const Prob& P = cm.single;
  const int s = threadIdx.x, lane = s & 31, warp = s >> 5;
  const int row_floats = P.N;
  float* const as = reinterpret_cast<float*>(sm_fit);  // [STREAM_K][STREAM_LD]
  float* const ring = as + STREAM_A_FLOATS;
  const int k0 = blockIdx.x * per, k1 = min(P.K, k0 + per);
  const int i = s < fa.n_fit ? fa.fi[s] : 0, j = s < fa.n_fit ? fa.fj[s] : 0;
  const bool valid = s < fa.n_fit && i >= 0 && i < P.M && j >= 0 && j < P.N;
  const int ic = valid ? i : 0, jc = valid ? j : 0;  // k_fit_merge reports the others
  arow[s] = ic;
  if (s == 0) {
    abort_flag = 0;
    for (int t = 0; t < stages; ++t) {
      mbar_init(&full[t], 1);
      mbar_init(&empty[t], STREAM_THREADS / 32);
    }
    fence_barrier_init();
  }
  __syncthreads();
  auto copy = [&](int k, int st) {
    mbar_arrive_expect_tx(&full[st], row_floats * 4);
    bulk_g2s(smem_u32(ring + st * row_floats), P.B + (int64_t)k * P.ldb, row_floats * 4, &full[st]);
  };
  int issued = k0;  // thread 0: rows copied so far
  if (s == 0)
    for (; issued < k1 && issued < k0 + stages; ++issued) copy(issued, issued - k0);
  const float ri = cm.r[P.rc_r + ic], cj = cm.c[P.rc_c + jc];
  const float rinv = 1.0f / ri, cinv = 1.0f / cj;
  const bool exact = __all_sync(0xffffffffu, recip_exact(ri) && recip_exact(cj));
  bool dense = true;
  for (int q = 0; q < fa.n_p; ++q) dense = dense && fa.p_log2[q] == q;
  float mx = 0.0f, S[PN_MAX_P];
#pragma unroll
  for (int q = 0; q < PN_MAX_P; ++q) S[q] = 0.0f;
  int st = 0, prev = 0;       // the row's stage, the stage of the row before
  uint32_t phase = 0, prev_phase = 0;
  bool ok = true;
  for (int c0 = k0; c0 < k1 && ok; c0 += STREAM_K) {
    __syncthreads();  // the last indices' values are read
    float v[STREAM_K];
#pragma unroll
    for (int u = 0; u < STREAM_K; ++u) {  // two samples per instruction, 16 indices each
      const int t = warp * 32 + 2 * u + (lane >> 4), k = min(c0 + (lane & 15), P.K - 1);
      v[u] = __ldg(P.A + (int64_t)arow[t] * P.lda + k);
    }
#pragma unroll
    for (int u = 0; u < STREAM_K; ++u)
      as[(lane & 15) * STREAM_LD + warp * 32 + 2 * u + (lane >> 4)] = v[u];
    __syncthreads();
    const int ce = min(c0 + STREAM_K, k1);
    // (a wait that gave up leaves no thread behind: every thread goes on through
    // the same barriers to the end of the block, the other waits giving up at once)
    for (int k = c0; k < ce; ++k) {
      if (!mbar_wait(&full[st], phase, cm.timeout_ns, &abort_flag)) ok = false;
      const float b = ok ? ring[st * row_floats + jc] : 0.0f;
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[st]);
      const float a = as[(k - c0) * STREAM_LD + s];
      const float u = exact ? (a * rinv) * (b * cinv) : (a / ri) * (b / cj);
      mx = fmaxf(mx, u);
      if (dense) fit_add_dense(fa.n_p, u, S);
      else fit_add(fa, u, S);
      // the row before is read by most warps by now: its stage's next copy
      if (s == 0 && k > k0 && issued < k1) {
        if (ok && mbar_wait(&empty[prev], prev_phase, cm.timeout_ns, &abort_flag)) {
          copy(issued++, prev);
        } else {
          ok = false;
          *const_cast<volatile int32_t*>(&abort_flag) = 1;
        }
      }
      prev = st;
      prev_phase = phase;
      if (++st == stages) {
        st = 0;
        phase ^= 1u;
      }
    }
    ok = __syncthreads_and(ok);
  }
  if (!ok) {  // let the copies in flight land before the memory goes
    if (s == 0) {
      set_status(cm.status, PN_ETIMEOUT);
      abort_flag = 1;
      int32_t never = 0;
      for (int k = issued - stages < k0 ? k0 : issued - stages; k < issued; ++k)
        mbar_wait(&full[(k - k0) % stages], ((k - k0) / stages) & 1, cm.timeout_ns, &never);
    }
    return;
  }
  if (s >= fa.n_fit) return;
  float* out = fa.part + (int64_t)blockIdx.x * (fa.n_p + 1) * fa.n_fit + s;
#pragma unroll
  for (int q = 0; q < PN_MAX_P; ++q)
    if (q < fa.n_p) out[(int64_t)q * fa.n_fit] = S[q];
  out[(int64_t)fa.n_p * fa.n_fit] = mx;
}

// The partial sums of eight samples per block in a fixed order (warp w: ranges w,
// w + 8, ..., then the warps in FP64), and the samples' records.
constexpr int MERGE_WARPS = 8, MERGE_SAMPLES = 8;
__global__ void __launch_bounds__(32 * MERGE_WARPS)
    k_fit_merge(const __grid_constant__ Common cm, const __grid_constant__ FitArgs fa, int ranges) {
  constexpr int VALUES = PN_MAX_P + 1, PER_LANE = (VALUES + 3) / 4;
  __shared__ double red[MERGE_WARPS][VALUES][MERGE_SAMPLES];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int e = lane & 7, v0 = lane >> 3, s = blockIdx.x * MERGE_SAMPLES + e;
  float acc[PER_LANE];
#pragma unroll
  for (int u = 0; u < PER_LANE; ++u) acc[u] = 0.0f;
  if (s < fa.n_fit) {
#pragma unroll 4
    for (int x = warp; x < ranges; x += MERGE_WARPS) {
#pragma unroll
      for (int u = 0; u < PER_LANE; ++u) {
        const int v = v0 + 4 * u;
        if (v > fa.n_p) break;
        const float t = __ldg(fa.part + ((int64_t)x * (fa.n_p + 1) + v) * fa.n_fit + s);
        acc[u] = v == fa.n_p ? fmaxf(acc[u], t) : acc[u] + t;
      }
    }
  }
#pragma unroll
  for (int u = 0; u < PER_LANE; ++u)
    if (v0 + 4 * u < VALUES) red[warp][v0 + 4 * u][e] = acc[u];
  __syncthreads();
  if (threadIdx.x >= MERGE_SAMPLES || s >= fa.n_fit) return;
  const Prob& P = cm.single;
  if (fa.fi[s] < 0 || fa.fi[s] >= P.M || fa.fj[s] < 0 || fa.fj[s] >= P.N) {
    set_status(cm.status, PN_EINVAL);
    fa.scls[s] = -1;
    return;
  }
  float S[PN_MAX_P];
  double mx = 0.0;
#pragma unroll
  for (int q = 0; q < PN_MAX_P; ++q) {
    double t = 0.0;
    for (int w = 0; w < MERGE_WARPS; ++w) t += red[w][q][e];
    S[q] = q < fa.n_p ? static_cast<float>(t) : 0.0f;
  }
  for (int w = 0; w < MERGE_WARPS; ++w) mx = fmax(mx, red[w][fa.n_p][e]);
  fit_record(P.tau, fa, s, S, static_cast<float>(mx));
}

// One warp per class q: the FP64 sums n, x, y, x^2, x y over the samples of
// the class (x = estimate, y = exact value), lane l taking samples l, l + 32,
// ... in order and a fixed butterfly combining the lanes, so the sums and the
// line are the same on every run; then the least-squares line (the oracle's
// rule, including the degenerate cases).
__global__ void k_fit_solve(const __grid_constant__ FitArgs fa) {
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (q >= fa.n_p) return;
  double c5[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int s = lane; s < fa.n_fit; s += 32) {
    if (fa.scls[s] != q) continue;
    const double x = fa.samp[2 * s], y = fa.samp[2 * s + 1];
    c5[0] += 1.0;
    c5[1] += x;
    c5[2] += y;
    c5[3] += x * x;
    c5[4] += x * y;
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
#pragma unroll
    for (int t = 0; t < 5; ++t) c5[t] += __shfl_xor_sync(0xffffffffu, c5[t], off);
  if (lane != 0) return;
  const double n = c5[0], sx = c5[1], sy = c5[2], sxx = c5[3], sxy = c5[4];
  double a = 1.0, b = 0.0;
  if (n >= 2.0 && sxx - sx * sx / n > 1e-12 * sxx) {
    a = (sxy - sx * sy / n) / (sxx - sx * sx / n);
    b = (sy - a * sx) / n;
  } else if (n >= 1.0 && sx > 0.0) {
    a = sy / sx;
  }
  fa.coef[2 * q] = static_cast<float>(a);
  fa.coef[2 * q + 1] = static_cast<float>(b);
  if (fa.user_coef) {
    fa.user_coef[2 * q] = static_cast<float>(a);
    fa.user_coef[2 * q + 1] = static_cast<float>(b);
  }
}

}  // namespace

int launch_fit(const Common& cm, const FitArgs& fa, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const Prob& P = cm.single;
  const bool whole_rows = (P.N & 3) == 0 && (P.ldb & 3) == 0 &&
                          (reinterpret_cast<uintptr_t>(P.B) & 15) == 0;
  int stages = 0;
  const int ranges = whole_rows ? fit_stream_ranges(P.N, P.K, fa.n_fit, fa.n_p, fa.part_floats,
                                                    host_device_sms(), &stages)
                                : 0;
  if (ranges > 0) {
    const int smem = 4 * (STREAM_A_FLOATS + stages * P.N);
    cudaError_t e = allow_smem<k_fit_stream>(STREAM_SMEM);
    if (e != cudaSuccess) return e;
    const int per = (P.K + ranges - 1) / ranges, n = (P.K + per - 1) / per;
    k_fit_stream<<<n, STREAM_THREADS, smem, s>>>(cm, fa, per, stages);
    k_fit_merge<<<(fa.n_fit + MERGE_SAMPLES - 1) / MERGE_SAMPLES, 32 * MERGE_WARPS, 0, s>>>(cm, fa, n);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  } else if (fa.n_fit > 0) {
    // (plain launches: placed early on the SMs that drain first, the blocks of a
    // kernel that is bound per SM pile up there: 190 us instead of 136)
    k_fit_samples<<<fa.n_fit, FIT_THREADS, 0, s>>>(cm, fa);
    const int e = cudaGetLastError();
    if (e) return e;
  }
  k_fit_solve<<<1, 32 * PN_MAX_P, 0, s>>>(fa);
  return cudaGetLastError();
}

}  // namespace pn
