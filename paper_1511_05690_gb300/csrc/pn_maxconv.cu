// Max-convolution z_m = max_i x_i y_(m-i) (Sec. 1) and its p-norm estimate
// with H = FFT convolution (Sec. 1; the scaled H' and the threshold tau of
// Sec. 2.1).
//
// k_maxconv_fft: one CTA per problem, everything in shared memory.  Per p
// (largest first): x' = x / max x and y' = y / max y raised to p in FP32
// (relative error (p - 1) 2^-24), packed as one complex sequence
// a = x'^p + i y'^p and transformed by one radix-2 FFT (decimation in time);
// the spectra X, Y are separated from A by Hermitian symmetry, Z = X Y, and the
// inverse FFT gives the ring convolution S^(p) = x'^p * y'^p.  Each index m takes
// the first p with S^(p)_m >= tau; z_m = max x max y (S^(p*)_m)^(1/p*).  The CTA
// stops as soon as every index is resolved.  An FFT's absolute error goes with
// the norms of the powered vectors (about log2(N) 2^-53 of them in FP64), which
// is what the paper's tau = 1e-12 guards.  GB300 issues FP64 at 1/64 of the
// FP32 rate, so the transforms run in two floats per value, and the indices
// whose sums are so small that their error would show get FP64 sums (below);
// the roots of S >= 1e-30 are FP32 square roots.  When the indices still open after
// a level hold few terms in total (typically the edges of the convolution),
// their p-sums for every remaining p are summed directly in FP64 (the naive
// ring convolution, which the FFT only reproduces) instead of running more
// FFT levels.
//
// k_maxconv_exact: the exact comparison on the CUDA cores, one CTA per 1792
// outputs and 8192 terms of one problem, 7 consecutive outputs per thread;
// each FP32 product is correctly rounded and the max is exact, so the result
// is bit-identical to any sequential evaluation.
#include <cstdint>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "pn_device.cuh"
#include "pn_launch.h"

namespace pn {

namespace {

constexpr int FFT_THREADS = 512;
constexpr int FFT_LOG_NMAX = MAXCONV_LOG_NMAX;
constexpr int FFT_NMAX = 1 << FFT_LOG_NMAX;

// exp(-2 pi i k / NMAX), k < NMAX / 2; a transform of length N uses every
// (NMAX / N)-th entry.
__device__ double2 g_twiddle[FFT_NMAX / 2];
__device__ float4 g_twiddle_ff[FFT_NMAX / 2];  // the same in two floats per part (cff)

__global__ void k_twiddle_init() {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= FFT_NMAX / 2) return;
  double s, c;
  sincospi(-2.0 * static_cast<double>(k) / FFT_NMAX, &s, &c);
  g_twiddle[k] = make_double2(c, s);
  const float ch = static_cast<float>(c), sh = static_cast<float>(s);
  g_twiddle_ff[k] = make_float4(ch, sh, static_cast<float>(c - ch), static_cast<float>(s - sh));
}

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -__dmul_rn(a.y, b.y)), fma(a.x, b.y, __dmul_rn(a.y, b.x)));
}

// conj(a) * b
__device__ __forceinline__ double2 cmulc(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, __dmul_rn(a.y, b.y)), fma(a.x, b.y, -__dmul_rn(a.y, b.x)));
}

// (S)^(1/2^plog): plog correctly rounded FP32 square roots of float(S) for
// S >= 1e-30 (the output is FP32; relative error about (plog + 1) 2^-24),
// FP64 square roots below that (only unstable indices at the smallest p).
// (Compared as integers: positive values order alike, and no FP64 slot is taken.)
__device__ __forceinline__ bool ge_pos(double v, double bound) {  // bound > 0, v no NaN
  return __double_as_longlong(v) >= __double_as_longlong(bound);
}
__device__ __forceinline__ double root_pow2(double S, int plog) {
  if (ge_pos(S, 1e-30)) {
    float r = static_cast<float>(S);
    for (int s = 0; s < plog; ++s) r = sqrtf(r);
    return r;
  }
  double r = S > 0.0 ? S : 0.0;
  for (int s = 0; s < plog; ++s) r = sqrt(r);
  return r;
}

// Number of terms x_i y_(m-i) of output m.
__device__ __forceinline__ int terms_of(int m, int nx, int ny) {
  const int lo = m - ny + 1 > 0 ? m - ny + 1 : 0;
  const int hi = m < nx - 1 ? m : nx - 1;
  return hi - lo + 1;
}

// v >= 0 in FP64; a normal value without the conversion, which takes an FP64 slot.
__device__ __forceinline__ double widen(float v) {
  const unsigned b = __float_as_uint(v);
  if (b != 0u && b < 0x00800000u) return static_cast<double>(v);
  return b == 0u ? 0.0 : __hiloint2double((b >> 3) + 0x38000000u, b << 29);
}

// Index m still open after level q <= Q: its p-sums for levels q-1 .. 0 summed
// directly, sum_i (x'_i y'_(m-i))^p in FP64, then the selection rule, by G = 1 lane or
// the G = 32 of a warp (the terms in turn).  iss = the scales' reciprocals multiplied
// (exactly), so that a term takes two FP64 products and no conversion, of about 16
// FP64 instructions, which bound it.  The Q sums are held in registers: 16 of them
// spill in a kernel of 64 registers.
template <int G, int Q>
__device__ __forceinline__ void direct_levels_q(const MaxconvArgs& ma, const float* x,
                                                const float* y, double iss, double sxy,
                                                int m, int q, float* z, uint8_t* res) {
  double S[Q];
#pragma unroll
  for (int t = 0; t < Q; ++t) S[t] = 0.0;
  const int lane = threadIdx.x & (G - 1);
  const int lo = m - ma.ny + 1 > 0 ? m - ma.ny + 1 : 0;
  const int hi = m < ma.nx - 1 ? m : ma.nx - 1;
  for (int i = lo + lane; i <= hi; i += G) {
    double t = (widen(x[i]) * widen(y[m - i])) * iss;  // = x'_i y'_(m-i): both products are exact
    int lg = 0;
#pragma unroll
    for (int u = 0; u < Q; ++u) {
      if (u < q) {
        while (lg < ma.p_log2[u]) {
          t *= t;
          ++lg;
        }
        S[u] += t;
      }
    }
  }
  int qs = -1;
  double s_sel = 0.0;
#pragma unroll
  for (int u = Q - 1; u >= 0; --u) {
    if (u < q && qs < 0) {
      if constexpr (G == 32) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) S[u] += __shfl_xor_sync(0xffffffffu, S[u], off);
      }
      if (u == 0 || S[u] >= ma.tau) {
        qs = u;
        s_sel = S[u];
      }
    }
  }
  if (lane == 0) {
    z[m] = static_cast<float>(sxy * root_pow2(s_sel, ma.p_log2[qs]));
    res[m] = static_cast<uint8_t>(ma.p_log2[qs] | (s_sel >= ma.tau ? 0 : 0x80));
  }
}
template <int G = 1>
__device__ __forceinline__ void direct_levels(const MaxconvArgs& ma, const float* x,
                                              const float* y, double iss, double sxy,
                                              int m, int q, float* z, uint8_t* res) {
  if (q <= 6) direct_levels_q<G, 6>(ma, x, y, iss, sxy, m, q, z, res);
  else direct_levels_q<G, PN_MAX_P>(ma, x, y, iss, sxy, m, q, z, res);
}

// 4 Z_k = 4 X_k Y_k from a = A_k and b = A_(N-k), the spectra of the packed real
// pair: X = (a + conj b) / 2, Y = (a - conj b) / (2i); the halves are left out
// (powers of two, exact).
__device__ __forceinline__ double2 spec_z4(double2 a, double2 b) {
  const double2 s = make_double2(a.x + b.x, a.y - b.y);
  const double dy = a.y + b.y, ndx = b.x - a.x;  // -i (a - conj b) = (dy, ndx)
  return make_double2(fma(s.x, dy, -__dmul_rn(s.y, ndx)), fma(s.x, ndx, __dmul_rn(s.y, dy)));
}

__device__ __forceinline__ float pow_f32(float v, int plog) {
  for (int s = 0; s < plog; ++s) v *= v;
  return v;
}

// One level of the FFT convolution in shared memory: a = x'^p + i y'^p (zero
// padded; powers in FP32), forward FFT of length N, the spectrum of the ring
// convolution, inverse at half length.
//
// The spectrum: X_k = (A_k + conj A_(N-k)) / 2, Y_k = (A_k - conj A_(N-k)) /
// (2i), Z = X Y (Hermitian: the convolution is real).  Its inverse runs at
// half length M = N / 2: with E, O the length-M DFTs of the even and odd
// samples of S, Z_k = E_k + W^k O_k and Z_(k+M) = conj Z_(M-k) = E_k - W^k O_k
// (W = exp(-2 pi i / N)), so
// V_k = E_k + i O_k = (Z_k + conj Z_(M-k)) / 2 + i W^-k (Z_k - conj Z_(M-k)) / 2
// is the DFT of v_j = S_2j + i S_(2j+1).  Thread work: k and M - k together
// (reads A at k, N - k, M - k, M + k).
//
// Radix-2 butterflies, decimation in time, eight values per thread in registers
// for three stages, so that a level of N = 2^13 makes 9 passes over shared memory
// with a barrier each instead of 28 (one per stage), and nothing is permuted: the
// forward transform reads natural
// order and leaves frequency k at address bitrev(k); the last forward stage
// pairs the addresses of k and k + N/2, which the spectrum needs together
// with those of N - k and N/2 - k, so it is fused into the spectrum; the
// spectrum's half-length sequence, left in the even addresses in
// bit-reversed order, is what the decimation in time starts from.
//
// Values are double2, or cff, each part the unevaluated sum of two floats: an
// addition (8 FP32 operations) and a product (4) keep about 2^-46 of their
// operands' magnitude, and GB300 issues 64 FP32 operations per FP64 one, so a
// butterfly takes 64 lane slots instead of 8 x 64.
// What bounds the double2 form is the FP64 issue rate (two lanes per clock and
// SM): about 6.8e5 FP64 instructions per level at N = 2^13.

// Shared-memory slot of element i: bits 1-2 are XORed with bits 4-5, so that
// the passes with a stride of two or eight elements spread over the banks.
__device__ __forceinline__ int slot(int i) { return i ^ (((i >> 4) & 3) << 1); }

// A complex value in two floats per part: h = (x.h, y.h), l = (x.l, y.l), each
// pair one operand of the packed FP32 instructions (two operations, rounded
// as by themselves, in one issue slot; the kernel runs out of slots and of
// instruction cache, not of FP32 lanes).
struct alignas(16) cff {
  uint64_t h, l;
};
__device__ __forceinline__ float2 f2_unpack(uint64_t v) {
  float2 r;
  f32x2_unpack(v, r.x, r.y);
  return r;
}
constexpr uint64_t F2_NEG = 0xbf800000bf800000ull;  // (-1, -1)
__device__ __forceinline__ uint64_t f2_sub(uint64_t a, uint64_t b) { return f32x2_fma(b, F2_NEG, a); }
__device__ __forceinline__ uint64_t f2_neg(uint64_t a) { return a ^ 0x8000000080000000ull; }

// a + b: the rounding error of the high parts by Knuth's two-sum, the low parts
// added to it (not renormalised).
__device__ __forceinline__ cff ff_add(uint64_t ah, uint64_t al, uint64_t bh, uint64_t bl) {
  const uint64_t s = f32x2_add(ah, bh), t = f2_sub(s, ah);
  const uint64_t e = f32x2_add(f2_sub(ah, f2_sub(s, t)), f2_sub(bh, t));
  return cff{s, f32x2_add(e, f32x2_add(al, bl))};
}
// a - b
__device__ __forceinline__ cff ff_sub(uint64_t ah, uint64_t al, uint64_t bh, uint64_t bl) {
  const uint64_t s = f2_sub(ah, bh), t = f2_sub(s, ah);
  const uint64_t e = f2_sub(f2_sub(ah, f2_sub(s, t)), f32x2_add(bh, t));
  return cff{s, f32x2_add(e, f2_sub(al, bl))};
}

__device__ __forceinline__ double2 c_add(double2 a, double2 b) {
  return make_double2(a.x + b.x, a.y + b.y);
}
__device__ __forceinline__ double2 c_sub(double2 a, double2 b) {
  return make_double2(a.x - b.x, a.y - b.y);
}
// a + conj b, a - conj b, a + i b, -i a
__device__ __forceinline__ double2 c_add_conj(double2 a, double2 b) {
  return make_double2(a.x + b.x, a.y - b.y);
}
__device__ __forceinline__ double2 c_sub_conj(double2 a, double2 b) {
  return make_double2(a.x - b.x, a.y + b.y);
}
__device__ __forceinline__ double2 c_add_i(double2 a, double2 b) {
  return make_double2(a.x - b.y, a.y + b.x);
}
__device__ __forceinline__ cff c_add(cff a, cff b) { return ff_add(a.h, a.l, b.h, b.l); }
__device__ __forceinline__ cff c_sub(cff a, cff b) { return ff_sub(a.h, a.l, b.h, b.l); }
__device__ __forceinline__ cff c_conj(cff a) {
  return cff{a.h ^ 0x8000000000000000ull, a.l ^ 0x8000000000000000ull};
}
// i a = (-y, x)
__device__ __forceinline__ cff c_muli(cff a) {
  const float2 h = f2_unpack(a.h), l = f2_unpack(a.l);
  return cff{f32x2_pack(-h.y, h.x), f32x2_pack(-l.y, l.x)};
}
__device__ __forceinline__ cff c_add_conj(cff a, cff b) { return c_add(a, c_conj(b)); }
__device__ __forceinline__ cff c_sub_conj(cff a, cff b) { return c_sub(a, c_conj(b)); }
__device__ __forceinline__ cff c_add_i(cff a, cff b) { return c_add(a, c_muli(b)); }
__device__ __forceinline__ cff c_mul_mi(cff a) {
  const cff b = c_muli(a);
  return cff{f2_neg(b.h), f2_neg(b.l)};
}
// w v = v.x (w.x, w.y) + v.y (-w.y, w.x)
__device__ __forceinline__ cff cmul(cff w, cff v) {
  const cff iw = c_muli(w);
  const float2 vh = f2_unpack(v.h), vl = f2_unpack(v.l);
  const uint64_t xh = f32x2_pack(vh.x, vh.x), xl = f32x2_pack(vl.x, vl.x);
  const uint64_t yh = f32x2_pack(vh.y, vh.y), yl = f32x2_pack(vl.y, vl.y);
  const uint64_t p = f32x2_mul(xh, w.h), q = f32x2_mul(yh, iw.h);
  uint64_t e = f32x2_fma(xh, w.h, f2_neg(p)), f = f32x2_fma(yh, iw.h, f2_neg(q));
  e = f32x2_fma(xh, w.l, f32x2_fma(xl, w.h, e));
  f = f32x2_fma(yh, iw.l, f32x2_fma(yl, iw.h, f));
  return ff_add(p, e, q, f);
}
__device__ __forceinline__ cff cmulc(cff w, cff v) { return cmul(c_conj(w), v); }

// Twiddle k of the table.  The two-float table is stored with the low three
// index bits XORed with the higher ones, three at a time: the passes read it
// with strides of powers of two, which would meet in a few banks (the FP64
// form has time for that: its arithmetic takes eight times as long).
__device__ __forceinline__ int tw_slot(int k) {
  return k ^ (((k >> 3) ^ (k >> 6) ^ (k >> 9)) & 7);
}
__device__ __forceinline__ double2 tw_at(const double2* tw, int k) { return tw[k]; }
__device__ __forceinline__ cff tw_at(const cff* tw, int k) { return tw[tw_slot(k)]; }

template <typename C>
__device__ __forceinline__ void bfly(C& u, C& v, C t) {
  const C a = u;
  u = c_add(a, t);
  v = c_sub(a, t);
}

// The butterfly with the twiddle -i (INV: +i).  (A negated FP64 value costs an
// FP64 instruction unless it is the subtrahend of the operation that uses it.)
template <bool INV = false>
__device__ __forceinline__ void bfly_mi(double2& u, double2& v) {
  const double2 a = u, b = v;
  const double2 p = make_double2(a.x + b.y, a.y - b.x), m = make_double2(a.x - b.y, a.y + b.x);
  u = INV ? m : p;
  v = INV ? p : m;
}

// Stages 0 to 2 of a transform on the 8 values of positions 0..7 of a block,
// w1 and w3 = exp(-2 pi i / 8), exp(-6 pi i / 8) as tabled: the twiddles 1 and
// -+i take no product (their products are exact).  HALF: the values of odd
// positions, the upper half of the input, are zero and not read.
template <bool INV, bool HALF>
__device__ __forceinline__ void first_stages8(double2 (&v)[8], double2 w1, double2 w3) {
#pragma unroll
  for (int r = 0; r < 8; r += 2) {
    if constexpr (HALF) v[r + 1] = v[r];
    else bfly(v[r], v[r + 1], v[r + 1]);
  }
#pragma unroll
  for (int r = 0; r < 8; r += 4) {
    bfly(v[r], v[r + 2], v[r + 2]);
    bfly_mi<INV>(v[r + 1], v[r + 3]);
  }
  bfly(v[0], v[4], v[4]);
  bfly(v[1], v[5], INV ? cmulc(w1, v[5]) : cmul(w1, v[5]));
  bfly_mi<INV>(v[2], v[6]);
  bfly(v[3], v[7], INV ? cmulc(w3, v[7]) : cmul(w3, v[7]));
}

// R stages s .. s + R - 1 of a transform of 2^lg values on the 2^R values
// v[r] of one group; v[r] sits at position j + (r << s) within its block of
// 2^(s + R) (position: the bit-reversed sample index).  tw[k << tsh] = exp(-2 pi i k / 2^lg).
template <int R, bool INV, typename C>
__device__ __forceinline__ void group_stages(C (&v)[1 << R], const C* tw, int lg, int tsh, int s,
                                             int j) {
#pragma unroll
  for (int t = 0; t < R; ++t) {
    const int sh = lg - 1 - s - t + tsh;
#pragma unroll
    for (int o = 0; o < (1 << t); ++o) {
      const C w = tw_at(tw, (j + (o << s)) << sh);
#pragma unroll
      for (int r = 0; r < (1 << R); r += 2 << t) {
        const C b = v[r + o + (1 << t)];
        bfly(v[r + o], v[r + o + (1 << t)], INV ? cmulc(w, b) : cmul(w, b));
      }
    }
  }
}

__device__ __forceinline__ int rev_bits(int k, int n) {
  return n == 0 ? 0 : static_cast<int>(__brev(static_cast<unsigned>(k)) >> (32 - n));
}

// Stages s .. s + R - 1 in place, by threads t of nt: the address of a position
// is its bit reversal, so stage t pairs addresses that differ in bit lg - 1 - t.
template <int R, bool INV = false, typename C>
__device__ __forceinline__ void fwd_pass(C* a, const C* tw, int lg, int s, int t = threadIdx.x,
                                         int nt = blockDim.x) {
  const int low = lg - s - R;  // address bits below the group's
  for (int g = t; g < (1 << (lg - R)); g += nt) {
    const int hi = g >> low, base = (hi << (low + R)) | (g & ((1 << low) - 1));
    C v[1 << R];
#pragma unroll
    for (int r = 0; r < (1 << R); ++r) v[r] = a[slot(base + (rev_bits(r, R) << low))];
    group_stages<R, INV>(v, tw, lg, 0, s, rev_bits(hi, s));
#pragma unroll
    for (int r = 0; r < (1 << R); ++r) a[slot(base + (rev_bits(r, R) << low))] = v[r];
  }
  __syncthreads();
}

// Inverse stages s .. s + R - 1 of the 2^lg values in the even addresses.
template <int R, typename C>
__device__ __forceinline__ void inv_pass(C* a, const C* tw, int lg, int s) {
  for (int g = threadIdx.x; g < (1 << (lg - R)); g += blockDim.x) {
    const int j = g & ((1 << s) - 1), base = ((g >> s) << (s + R)) | j;
    C v[1 << R];
#pragma unroll
    for (int r = 0; r < (1 << R); ++r) v[r] = a[slot(2 * (base + (r << s)))];
    group_stages<R, true>(v, tw, lg, 1, s, j);
#pragma unroll
    for (int r = 0; r < (1 << R); ++r) a[slot(2 * (base + (r << s)))] = v[r];
  }
  __syncthreads();
}

// Stages 0 to 2 (first_stages8), FP64: forward; inverse on the even addresses.
__device__ __forceinline__ void fwd_first_pass(double2* a, const double2* tw, int lg) {
  const int ng = 1 << (lg - 3);
  for (int g = threadIdx.x; g < ng; g += blockDim.x) {
    double2 v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = a[slot(g + rev_bits(r, 3) * ng)];
    first_stages8<false, false>(v, tw[ng], tw[3 * ng]);
#pragma unroll
    for (int r = 0; r < 8; ++r) a[slot(g + rev_bits(r, 3) * ng)] = v[r];
  }
  __syncthreads();
}
__device__ __forceinline__ void inv_first_pass(double2* a, const double2* tw, int lg) {
  const double2 w1 = tw[2 << (lg - 3)], w3 = tw[6 << (lg - 3)];
  for (int g = threadIdx.x; g < (1 << (lg - 3)); g += blockDim.x) {
    double2 v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = a[slot(2 * (8 * g + r))];
    first_stages8<true, false>(v, w1, w3);
#pragma unroll
    for (int r = 0; r < 8; ++r) a[slot(2 * (8 * g + r))] = v[r];
  }
  __syncthreads();
}

// The spectrum from the packed pair's transform (all but its last stage done)
// to the half-length sequence 8 V_k in the even addresses (formulas above).
// Their halves are left out: a power of two, exact.
template <typename C>
__device__ __forceinline__ void spectrum_pass(C* a, const C* tw, int lg) {
  const int lm = lg - 1, M = 1 << lm;
  for (int e = threadIdx.x; e <= (M >> 1); e += blockDim.x) {
    // p = bitrev(k): 0, then the lower half of every [2^h, 2^(h + 1)); the
    // address of M - k mirrors p within that range
    int p = e, pm = e;
    if (e > 1) {
      const int f = e - 1, hb = 1 << (31 - __clz(f));
      p = f + hb;
      pm = p ^ (2 * hb - 1);
    }
    const int k = rev_bits(p, lm);
    C ak = a[slot(2 * p)], amk = a[slot(2 * p + 1)];  // frequencies k, k + M
    const C wk = tw_at(tw, k);
    bfly(ak, amk, cmul(wk, amk));
    C am = ak, an = amk;                              // M - k, N - k
    if (k == 0) {
      an = ak;  // N - 0 = 0 and M - 0 = M
      am = amk;
    } else if (pm != p) {
      am = a[slot(2 * pm)];
      an = a[slot(2 * pm + 1)];
      bfly(am, an, cmul(tw_at(tw, M - k), an));
    }
    auto z4 = [](C u, C v) {  // 4 spec_z: (u + conj v) (-i (u - conj v))
      if constexpr (std::is_same_v<C, double2>) return spec_z4(u, v);
      else return cmul(c_add_conj(u, v), c_mul_mi(c_sub_conj(u, v)));
    };
    auto v8 = [](C zk, C zm, C w) {  // 8 spec_v
      return c_add_i(c_add_conj(zk, zm), cmulc(w, c_sub_conj(zk, zm)));
    };
    const C zk = z4(ak, an), zm = z4(am, amk);
    a[slot(2 * p)] = v8(zk, zm, wk);
    if (k != 0 && pm != p) a[slot(2 * pm)] = v8(zm, zk, tw_at(tw, M - k));
  }
  __syncthreads();
}

// The passes after the first forward stages (s of them done): the rest of the
// forward transform, the spectrum, the inverse.  On return S_m = 8 N / 2 times
// part m & 1 of a[slot(m & ~1)].  Three stages per pass in FP64; two in two
// floats, whose butterflies are five times as many instructions: with three, a
// pass's loop outgrows the instruction cache (a third of the fetches missed)
// and its registers allow half the warps.
__device__ __forceinline__ void conv_passes(double2* a, const double2* tw, int lg, int s) {
  if (s == 0 && lg >= 4) {
    fwd_first_pass(a, tw, lg);
    s = 3;
  }
  for (; s + 3 <= lg - 1; s += 3) fwd_pass<3>(a, tw, lg, s);
  if (s + 2 == lg - 1) fwd_pass<2>(a, tw, lg, s);
  else if (s + 1 == lg - 1) fwd_pass<1>(a, tw, lg, s);
  spectrum_pass(a, tw, lg);
  const int lm = lg - 1;
  s = 0;
  if (lm >= 3) {
    inv_first_pass(a, tw, lm);
    s = 3;
  }
  for (; s + 3 <= lm; s += 3) inv_pass<3>(a, tw, lm, s);
  if (s + 2 == lm) inv_pass<2>(a, tw, lm, s);
  else if (s + 1 == lm) inv_pass<1>(a, tw, lm, s);
}
__device__ __forceinline__ void conv_passes(cff* a, const cff* tw, int lg) {
  int s = (lg - 1) & 1;
  if (s) fwd_pass<1>(a, tw, lg, 0);
  for (; s < lg - 1; s += 2) fwd_pass<2>(a, tw, lg, s);
  spectrum_pass(a, tw, lg);
  const int lm = lg - 1;
  s = lm & 1;
  if (s) inv_pass<1>(a, tw, lm, 0);
  for (; s < lm; s += 2) inv_pass<2>(a, tw, lm, s);
}

// Whether the remaining p-sums of open indices with W terms in all are cheaper
// summed directly (about W (8 + 2 q) FP64 operations) than by one more FFT
// level (about 10 N log2 N).
__device__ __forceinline__ bool few_terms(unsigned long long W, int q, int logN) {
  return W * static_cast<unsigned long long>(8 + 2 * q) <=
         10ull * (1ull << logN) * static_cast<unsigned long long>(logN);
}

// Sum over a warp, the same on every lane.
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// The `count` open indices of list after level q, block-wide: those of 64 terms or
// more by a warp each, the others by a thread each (an FP64 instruction of a warp
// takes the same time however many lanes have work, and a warp's sums meet at the
// end).  1024 problems of 4096 values in [1/16, 1]: 2.8 ms, 6.6 with a thread for
// every index, 5.0 when 512 threads of twice the registers ran them.
__device__ void direct_open(const MaxconvArgs& ma, const float* x, const float* y, double iss,
                            double sxy, const int* list, int count, int q, float* z,
                            uint8_t* res) {
  const int tid = threadIdx.x, nt = static_cast<int>(blockDim.x);
  for (int e = tid >> 5; e < count; e += nt >> 5)
    if (terms_of(list[e], ma.nx, ma.ny) >= 64)
      direct_levels<32>(ma, x, y, iss, sxy, list[e], q, z, res);
  for (int e = tid; e < count; e += nt)
    if (terms_of(list[e], ma.nx, ma.ny) < 64)
      direct_levels<1>(ma, x, y, iss, sxy, list[e], q, z, res);
}

// The levels q .. 0 of one problem by FP64 transforms, for the indices still
// open in res (0xFF); block-wide.
__device__ void maxconv_levels64(const MaxconvArgs& ma, double2* a, double2* tw, uint8_t* res,
                                 const float* x, const float* y, float isx, float isy, double sxy,
                                 float* z, int q) {
  __shared__ unsigned long long open_terms;
  __shared__ int n_open;
  const int N = 1 << ma.logN, tid = threadIdx.x, nt = static_cast<int>(blockDim.x);
  const double scale = 0.25 / N;  // 2 / N, and the spectrum's 8
  __syncthreads();
  for (int k = tid; k < (N >> 1); k += nt) tw[k] = g_twiddle[k << (FFT_LOG_NMAX - ma.logN)];
  for (; q >= 0; --q) {
    const int plog = ma.p_log2[q];
    for (int k = tid; k < N; k += nt)
      a[slot(k)] = make_double2(k < ma.nx ? pow_f32(x[k] * isx, plog) : 0.0f,
                                k < ma.ny ? pow_f32(y[k] * isy, plog) : 0.0f);
    __syncthreads();
    conv_passes(a, tw, ma.logN, 0);
    // selection: first (largest) p with S >= tau; the smallest p takes the rest
    if (tid == 0) {
      open_terms = 0ull;
      n_open = 0;
    }
    __syncthreads();
    unsigned long long my_terms = 0ull;
    for (int m = tid; m < ma.nz; m += nt) {
      if (res[m] != 0xFF) continue;
      const double2 v = a[slot(m & ~1)];
      const double S = ((m & 1) ? v.y : v.x) * scale;
      const bool stable = S >= ma.tau;
      if (stable || q == 0) {
        z[m] = static_cast<float>(sxy * root_pow2(S, plog));
        res[m] = static_cast<uint8_t>(plog | (stable ? 0 : 0x80));
      } else {
        my_terms += static_cast<unsigned long long>(terms_of(m, ma.nx, ma.ny));
      }
    }
    if (my_terms) atomicAdd(&open_terms, my_terms);
    __syncthreads();
    const unsigned long long W = open_terms;
    if (W == 0ull) break;
    if (few_terms(W, q, ma.logN)) {
      // compact list of the open indices (the FFT buffer is free now)
      int* list = reinterpret_cast<int*>(a);
      for (int m = tid; m < ma.nz; m += nt)
        if (res[m] == 0xFF) list[atomicAdd(&n_open, 1)] = m;
      __syncthreads();
      const int cnt = n_open;
      direct_open(ma, x, y, static_cast<double>(isx) * isy, sxy, list, cnt, q, z, res);
      break;
    }
  }
}

// One CTA per problem.  Per level the transforms run in two floats per value
// (see above).  Their rounding adds noise to every S_m, independent of S_m's
// own size.  Its scale R: the products' and the inverse transform's rounding goes
// with the root mean square of the S_m; x'^p and y'^p are transformed together, so
// each spectrum has an error that goes with both their norms, which multiplied by
// the spectra and transformed back comes to (|x'^p|^2 + |y'^p|^2) / sqrt(N) (more
// than the first only where one vector outweighs the other); R^2 is the sum of
// the squares.  The noise's standard deviation is at most sigma = 2^-45
// sqrt(log2 N) R (measured 0.12 to 0.28 sigma, largest value 1.2 sigma, N = 2^13),
// that of FP64 transforms sigma64 = 2^-53 sqrt(log2 N) R (measured 0.6).  An index
// with S_m >= theta = 2^28 sigma (16 sigma below 2^-24 of S_m) is rooted from it.
// The others -- the outermost few, which sum few terms -- get S_m by a direct
// FP64 sum, which has no such noise.  Where that sum lies within 4 sigma64 of tau,
// more than six of the noise's standard deviations (about one problem in 300), or
// where too many indices lie below theta (wide ranges of values), the problem's
// level and the rest run in FP64 transforms, so that p_sel is what FP64
// transforms give.
// Per problem of n = 4096 (one CTA, P = {1..64}): 62 us, of which the transforms
// take 37 (issue slots: about 50 instructions per butterfly), against 240 by
// FP64 transforms at 78 % of the FP64 pipe; 1024 problems 0.55 to 0.62 ms (0.43
// where no problem falls back to FP64), all by FP64 transforms 1.49.
constexpr int MC_THREADS = 1024;
constexpr int FF_SMALL_MAX = 512;  // indices summed directly, at most
__global__ void __launch_bounds__(MC_THREADS, 1)
    k_maxconv_fft(const __grid_constant__ MaxconvArgs ma) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lg = ma.logN, N = 1 << lg;
  cff* a = reinterpret_cast<cff*>(smem);
  cff* tw = a + N;
  uint8_t* res = reinterpret_cast<uint8_t*>(tw + (N >> 1));  // p_sel, 0xFF = open
  __shared__ float red[2][MC_THREADS / 32];
  __shared__ unsigned long long s_terms;
  __shared__ int n_small, n_open, redo;
  __shared__ int small[FF_SMALL_MAX];
  __shared__ double small_S[FF_SMALL_MAX];
  __shared__ unsigned s_large[2];
  const int b = blockIdx.x;
  const float* x = ma.x + (int64_t)b * ma.ldx;
  const float* y = ma.y + (int64_t)b * ma.ldy;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nt = static_cast<int>(blockDim.x), nw = nt >> 5;

  for (int k = tid; k < (N >> 1); k += nt) 
    *reinterpret_cast<float4*>(tw + tw_slot(k)) = g_twiddle_ff[k << (FFT_LOG_NMAX - lg)];
  // maxima and domain (R+, finite)
  float mx = 0.0f, my = 0.0f;
  bool bad = false;
  for (int k = tid; k < ma.nx; k += nt) {
    const float v = x[k];
    bad |= !(v >= 0.0f && v <= 3.4028235e38f);
    mx = fmaxf(mx, v);
  }
  for (int k = tid; k < ma.ny; k += nt) {
    const float v = y[k];
    bad |= !(v >= 0.0f && v <= 3.4028235e38f);
    my = fmaxf(my, v);
  }
  if (__syncthreads_or(bad)) {
    if (tid == 0) set_status(ma.status, PN_EDOMAIN);
    return;
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    my = fmaxf(my, __shfl_xor_sync(0xffffffffu, my, off));
  }
  if (lane == 0) {
    red[0][warp] = mx;
    red[1][warp] = my;
  }
  for (int m = tid; m < ma.nz; m += nt) res[m] = 0xFF;
  if (tid < 2) s_large[tid] = 0u;
  __syncthreads();
  mx = my = 0.0f;
  for (int w = 0; w < nw; ++w) {
    mx = fmaxf(mx, red[0][w]);
    my = fmaxf(my, red[1][w]);
  }
  // the FP64 scalars by one warp (one FP64 instruction takes a warp 64 cycles)
  __shared__ double s_sxy;
  __shared__ float s_f[4];
  if (warp == 0) {
    // a zero vector keeps scale 1
    const double sx = mx == 0.0f ? 1.0 : static_cast<double>(mx);
    const double sy = my == 0.0f ? 1.0 : static_cast<double>(my);
    const double p = sx * sy;
    const float ph = static_cast<float>(p);
    if (lane == 0) {
      s_sxy = p;
      s_f[0] = static_cast<float>(1.0 / sx);
      s_f[1] = static_cast<float>(1.0 / sy);
      s_f[2] = ph;
      s_f[3] = static_cast<float>(p - ph);
    }
  }
  __syncthreads();
  const double sxy = s_sxy;
  const float isx = s_f[0], isy = s_f[1], sxy_h = s_f[2], sxy_l = s_f[3];
  float* z = ma.z + (int64_t)b * ma.ldz;
  const float scale = 0.25f / N;  // 2 / N, and the spectrum's 8
  const float tau = static_cast<float>(ma.tau);
  // products of the scales outside FP32's comfortable range, tiny transforms and
  // thresholds beyond FP32: FP64 from the start
  bool ff = lg >= 5 && sxy_h >= 1e-30f && sxy_h <= 1e30f && tau >= 1e-30f && tau <= 1e6f;
  int q = ma.n_p - 1;
  // A term of a sum that reaches theta (below, at least 2^-17 sqrt(log2 N / N), as the
  // largest x'^p and y'^p are 1) has both its factors at or above least, so at
  // most as many sums reach it as there are pairs of such factors.  Where the
  // largest p leaves too few pairs, its transforms in two floats are not begun:
  // they took 37 of the 232 us of a problem that falls back (1024 problems with
  // one value in 100 not zero: 11.6 ms, 11.1 so).
  const float least = 7.0e-6f * sqrtf(static_cast<float>(lg) / N) / min(ma.nx, ma.ny);
  for (; ff && q >= 0; --q) {
    const int plog = ma.p_log2[q];
    unsigned large_x = 0, large_y = 0;
    float sq = 0.0f;  // |x'^p|^2 + |y'^p|^2
    for (int k = tid; k < N; k += nt) {
      const float xr = k < ma.nx ? pow_f32(x[k] * isx, plog) : 0.0f;
      const float yr = k < ma.ny ? pow_f32(y[k] * isy, plog) : 0.0f;
      a[slot(k)] = cff{f32x2_pack(xr, yr), 0ull};
      sq = fmaf(xr, xr, fmaf(yr, yr, sq));
      large_x += xr >= least;
      large_y += yr >= least;
    }
    if (q == ma.n_p - 1) {
      large_x = __reduce_add_sync(0xffffffffu, large_x);
      large_y = __reduce_add_sync(0xffffffffu, large_y);
      if (lane == 0) {
        atomicAdd(&s_large[0], large_x);
        atomicAdd(&s_large[1], large_y);
      }
    }
    __syncthreads();
    if (q == ma.n_p - 1 && s_large[0] * s_large[1] + FF_SMALL_MAX < static_cast<unsigned>(ma.nz)) {
      ff = false;
      break;
    }
    conv_passes(a, tw, lg);
    // the sums' root mean square
    constexpr int PER = FFT_NMAX / MC_THREADS;
    float S[PER], ss = 0.0f;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int m = tid + u * nt;
      S[u] = 0.0f;
      if (m < ma.nz) {
        const cff v = a[slot(m & ~1)];
        const float2 h = f2_unpack(v.h), l = f2_unpack(v.l);
        S[u] = ((m & 1) ? __fadd_rn(h.y, l.y) : __fadd_rn(h.x, l.x)) * scale;
        ss = fmaf(S[u], S[u], ss);
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      ss += __shfl_xor_sync(0xffffffffu, ss, off);
      sq += __shfl_xor_sync(0xffffffffu, sq, off);
    }
    if (lane == 0) {
      red[0][warp] = ss;
      red[1][warp] = sq;
    }
    if (tid == 0) {
      s_terms = 0ull;
      n_small = n_open = redo = 0;
    }
    __syncthreads();
    ss = sq = 0.0f;
    for (int w = 0; w < nw; ++w) {
      ss += red[0][w];
      sq += red[1][w];
    }
    const float noise = sqrtf(static_cast<float>(lg) * fmaf(sq, sq, ss) / N);  // sqrt(log2 N) R
    const float theta = fmaxf(noise * 7.62939453e-6f, 4.0f * tau);           // 2^28 2^-45
    const float near = noise * 4.44089210e-16f;  // 4 2^-53
    unsigned long long terms = 0ull;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int m = tid + u * nt;
      if (m >= ma.nz || res[m] != 0xFF) continue;
      if (S[u] >= theta) {
        float r = S[u];
        for (int s = 0; s < plog; ++s) r = sqrtf(r);
        z[m] = fmaf(sxy_h, r, sxy_l * r);
        res[m] = static_cast<uint8_t>(plog);
      } else {
        const int at = atomicAdd(&n_small, 1);
        if (at < FF_SMALL_MAX) small[at] = m;
        terms += static_cast<unsigned long long>(terms_of(m, ma.nx, ma.ny));
      }
    }
    if (terms) atomicAdd(&s_terms, terms);
    __syncthreads();
    const int cnt = n_small;
    // too many terms to sum directly (against an FP64 level)
    if (cnt > FF_SMALL_MAX || s_terms > 2ull * N) {
      ff = false;
      break;
    }
    __syncthreads();
    if (tid == 0) s_terms = 0ull;
    __syncthreads();
    for (int e = warp; e < cnt; e += nw) {  // a warp per index
      const int m = small[e];
      const int lo = m - ma.ny + 1 > 0 ? m - ma.ny + 1 : 0, hi = m < ma.nx - 1 ? m : ma.nx - 1;
      double t = 0.0;
      for (int i = lo + lane; i <= hi; i += 32)
        t = fma(static_cast<double>(pow_f32(x[i] * isx, plog)),
                static_cast<double>(pow_f32(y[m - i] * isy, plog)), t);
      t = warp_sum(t);
      if (lane == 0) {
        small_S[e] = t;
        if (fabsf(static_cast<float>(t - ma.tau)) <= near) redo = 1;
      }
    }
    __syncthreads();
    if (redo) {
      ff = false;
      break;
    }
    terms = 0ull;
    for (int e = tid; e < cnt; e += nt) {
      const int m = small[e];
      const double t = small_S[e];
      const bool stable = t >= ma.tau;
      if (stable || q == 0) {
        z[m] = static_cast<float>(sxy * root_pow2(t, plog));
        res[m] = static_cast<uint8_t>(plog | (stable ? 0 : 0x80));
      } else {
        terms += static_cast<unsigned long long>(terms_of(m, ma.nx, ma.ny));
      }
    }
    if (terms) atomicAdd(&s_terms, terms);
    __syncthreads();
    const unsigned long long W = s_terms;
    if (W == 0ull) break;
    if (few_terms(W, q, lg)) {
      int* list = reinterpret_cast<int*>(a);  // the FFT buffer is free now
      for (int m = tid; m < ma.nz; m += nt)
        if (res[m] == 0xFF) list[atomicAdd(&n_open, 1)] = m;
      __syncthreads();
      const int open = n_open;
      direct_open(ma, x, y, static_cast<double>(isx) * isy, sxy, list, open, q, z, res);
      break;
    }
    __syncthreads();
  }
  if (!ff && q >= 0)
    maxconv_levels64(ma, reinterpret_cast<double2*>(a), reinterpret_cast<double2*>(tw), res, x, y,
                     isx, isy, sxy, z, q);
  __syncthreads();
  if (ma.psel) {
    uint8_t* ps = ma.psel + (int64_t)b * ma.ldp;
    for (int m = tid; m < ma.nz; m += nt) ps[m] = res[m];
  }
}

// ---------------------------------------------------------------- exact ---
constexpr int MCX_THREADS = 256;
constexpr int MCX_OUT = 7;                              // outputs per thread
constexpr int MCX_SPAN = MCX_THREADS * MCX_OUT;         // outputs per CTA
constexpr int MCX_IB = 8192;                            // terms i per CTA

// z_m for m in [m0, m0 + MCX_SPAN), terms i in [i0, i0 + MCX_IB), problems
// blockIdx.z, + gridDim.z, ...  Shared memory holds x[i0 .. i0 + IB + 8) and
// the y values those terms reach, zero outside [0, ny), so invalid terms
// contribute 0 (every product is >= 0, and the max over the nonempty set of
// valid terms is unchanged; terms counted by two CTAs are harmless for a max).
// Thread t owns outputs m0 + 7t .. m0 + 7t + 6: 7 is coprime with the 32
// banks, so the threads of a warp read their y windows without conflicts,
// and the warp walks one common range of i, so x is read by broadcast.
// Several i-blocks combine by atomicMax on the float bits (non-negative
// floats order like their bit patterns; z is zeroed first).
__global__ void __launch_bounds__(MCX_THREADS)
    k_maxconv_exact(const __grid_constant__ MaxconvArgs ma) {
  extern __shared__ __align__(16) float sm[];
  const int m0 = blockIdx.x * MCX_SPAN;
  const int i0 = blockIdx.y * MCX_IB;
  const int warp = threadIdx.x >> 5;
  float* xs = sm;                        // MCX_IB + 8 values: x[i0 + k]
  float* ys = sm + MCX_IB + 8;           // MCX_SPAN + MCX_IB + 16 values: y[tb + u]
  const int tb = m0 - i0 - MCX_IB - 8;   // y index of ys[0]
  const bool atomic = gridDim.y > 1;
  // terms of this CTA: i in [max(i0, m0 - ny + 1), min(i0 + IB, m0 + SPAN, nx))
  const int c_lo = max(i0, m0 - ma.ny + 1);
  const int c_hi = min(min(i0 + MCX_IB, m0 + MCX_SPAN), ma.nx);
  if (c_lo >= c_hi || m0 >= ma.nz) return;
  // the warp's outputs and terms
  const int mw = m0 + warp * 32 * MCX_OUT;
  const int w_lo = max(c_lo, mw - ma.ny + 1);
  const int w_hi = min(c_hi, mw + 32 * MCX_OUT);
  const int mt = m0 + threadIdx.x * MCX_OUT;
  for (int64_t b = blockIdx.z; b < ma.batch; b += gridDim.z) {
    __syncthreads();  // the previous problem's reads are done
    const float* x = ma.x + b * ma.ldx;
    const float* y = ma.y + b * ma.ldy;
    for (int k = threadIdx.x; k < MCX_IB + 8; k += MCX_THREADS)
      xs[k] = (i0 + k < ma.nx) ? x[i0 + k] : 0.0f;
    for (int u = threadIdx.x; u < MCX_SPAN + MCX_IB + 16; u += MCX_THREADS) {
      const int t = tb + u;
      ys[u] = (t >= 0 && t < ma.ny) ? y[t] : 0.0f;
    }
    __syncthreads();
    float acc[MCX_OUT];
#pragma unroll
    for (int r = 0; r < MCX_OUT; ++r) acc[r] = 0.0f;
#pragma unroll 1
    for (int i = w_lo; i < w_hi; i += 8) {
      const int k = i - i0;
      float xv[8], yv[MCX_OUT + 7];
#pragma unroll
      for (int e = 0; e < 8; ++e) xv[e] = xs[k + e];
      // yv[u] = y_(mt - i - 7 + u), i.e. ys[(mt - i - 7 + u) - tb]
      const float* yp = ys + (mt - i - 7 - tb);
#pragma unroll
      for (int u = 0; u < MCX_OUT + 7; ++u) yv[u] = yp[u];
#pragma unroll
      for (int r = 0; r < MCX_OUT; ++r) {
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
          // terms i+e and i+e+1 of output mt + r
          const float p0 = xv[e] * yv[r - e + 7];
          const float p1 = xv[e + 1] * yv[r - e + 6];
          float t;
          asm("max.f32 %0, %1, %2, %3;" : "=f"(t) : "f"(acc[r]), "f"(p0), "f"(p1));
          acc[r] = t;
        }
      }
    }
    float* z = ma.z + b * ma.ldz;
#pragma unroll
    for (int r = 0; r < MCX_OUT; ++r) {
      const int m = mt + r;
      if (m >= ma.nz) continue;
      if (atomic) {
        if (acc[r] > 0.0f) atomicMax(reinterpret_cast<unsigned int*>(z + m), __float_as_uint(acc[r]));
      } else {
        z[m] = acc[r];
      }
    }
  }
}

// ------------------------------------------------------- long problems ---
// One max-convolution of any length up to N = 2^22 (nz = nx + ny - 1 <= N),
// four-step FFT over the N1 x N2 view of the length-N buffer (index
// n = N2 n1 + n2, N1 = 2^min(10, floor(log2 N / 2))):
//   forward  A[k1 + N1 k2] = sum_n2 W_N2^(n2 k2) [W_N^(n2 k1) sum_n1 a[n] W_N1^(n1 k1)]
//   inverse  s[n] = sum_k1 W_N1^-(n1 k1) [W_N^-(n2 k1) sum_k2 Z[k1 + N1 k2] W_N2^-(n2 k2)]
// Three kernels per level: columns forward (the powered inputs are formed on
// the fly), rows (forward row, spectrum, inverse row; row k1 holds the
// partners N - k of row N1 - k1, so two CTAs of a cluster take these two rows
// and read each other's spectrum), columns inverse with the selection.  A
// fourth kernel ends the level loop (nothing open) or sums the remaining
// levels directly for few open terms.  All kernels of a finished call return
// at once (device flag), so every launch is issued unconditionally.
//
// The transforms are radix-2 butterflies in FP64 throughout (the values near
// tau at the edges carry their rounding, and p_sel depends on it), eight values
// per thread in registers for three stages; the first and last three stages
// read from and write to global memory.  What bounds them is the FP64 rate,
// two lanes per clock and SM: 7.5e8 instructions at N = 2^22, 1.3 ms.  Hence
// no products with 1 and -+i, no first stage where the upper half of the input
// is zero, two CTAs per SM to fill each other's barriers, and pieces small
// enough for a full last wave (1024 of each kind on 152 SMs, 6.7 per SM, against 512
// in 3.4 waves).  n = 2^21 per vector: 1538 us per call (column kernels about 315 each, rows 815), 2160 with a barrier
// per stage, 8 columns or a pair of rows per CTA.
constexpr int LONG_CC = 4;   // columns per CTA of the column kernels
constexpr int LONG_THREADS = 512;

struct LongArgs {
  const float* x;
  const float* y;
  float* z;
  uint8_t* res;            // p_sel, 0xFF while open
  int32_t nx, ny, nz;
  int32_t logN, l1, l2;    // N = 2^logN = N1 N2
  int32_t n_p;
  int32_t p_log2[PN_MAX_P];
  double tau;
  int32_t* status;
  double2* buf;            // N complex
  const double2* tlo;      // W_N^m, m < 2048
  const double2* thi;      // W_N^(2048 m), m < N / 2048
  unsigned long long* open_terms;  // per level
  int32_t* done;                   // 0; 1 + the level that was the last; -1 on bad input
  uint32_t* mxy;           // max x, max y (float bits)
};

__device__ __forceinline__ double2 w_n(const LongArgs& la, int m) {
  return cmul(la.thi[m >> 11], la.tlo[m & 2047]);
}

constexpr int LONG_TAB_BLOCKS = 8, LONG_MAX_BLOCKS = 152 * 4;  // of 256 threads

// The tables of W_N^m (the first blocks), the maxima and the domain test (the rest).
__global__ void k_long_init(const __grid_constant__ LongArgs la, double2* tlo, double2* thi) {
  if (blockIdx.x < LONG_TAB_BLOCKS) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const double N = static_cast<double>(1 << la.logN);
    double s, c;
    if (k < 2048) {
      sincospi(-2.0 * k / N, &s, &c);
      tlo[k] = make_double2(c, s);
    }
    if (k < ((1 << la.logN) >> 11)) {
      sincospi(-2.0 * (2048.0 * k) / N, &s, &c);
      thi[k] = make_double2(c, s);
    }
    return;
  }
  const int first = (blockIdx.x - LONG_TAB_BLOCKS) * blockDim.x + threadIdx.x;
  float mx = 0.0f, my = 0.0f;
  bool bad = false;
  const int stride = LONG_MAX_BLOCKS * blockDim.x;
  for (int k = first; k < la.nx; k += stride) {
    const float v = la.x[k];
    bad |= !(v >= 0.0f && v <= 3.4028235e38f);
    mx = fmaxf(mx, v);
  }
  for (int k = first; k < la.ny; k += stride) {
    const float v = la.y[k];
    bad |= !(v >= 0.0f && v <= 3.4028235e38f);
    my = fmaxf(my, v);
  }
  if (bad) {
    set_status(la.status, PN_EDOMAIN);
    *la.done = -1;  // nothing more runs
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    my = fmaxf(my, __shfl_xor_sync(0xffffffffu, my, off));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(la.mxy, __float_as_uint(mx));
    atomicMax(la.mxy + 1, __float_as_uint(my));
  }
}

__device__ __forceinline__ void long_scales(const LongArgs& la, double& sx, double& sy) {
  sx = __uint_as_float(la.mxy[0]);
  sy = __uint_as_float(la.mxy[1]);
  if (sx == 0.0) sx = 1.0;
  if (sy == 0.0) sy = 1.0;
}

// Elements between the columns in shared memory: columns of the same address
// two slots apart.
__device__ __forceinline__ int long_col_stride(int l1) { return (1 << l1) + 2; }

__device__ __forceinline__ void long_twiddles(double2* tw, int lg) {
  for (int k = threadIdx.x; k < (1 << (lg - 1)); k += blockDim.x)
    tw[k] = g_twiddle[k << (FFT_LOG_NMAX - lg)];
}

// Stages 3 .. lg - 4 of a transform whose first three stages are done.
template <bool INV>
__device__ __forceinline__ void long_middle(double2* a, const double2* tw, int lg, int t, int nt) {
  int s = 3;
  const int end = lg - 3;
  while (s < end) {
    if (end - s == 3 || end - s >= 5) {
      fwd_pass<3, INV>(a, tw, lg, s, t, nt);
      s += 3;
    } else if (end - s >= 2) {
      fwd_pass<2, INV>(a, tw, lg, s, t, nt);
      s += 2;
    } else {
      fwd_pass<1, INV>(a, tw, lg, s, t, nt);
      s += 1;
    }
  }
}

// columns [c0, c0 + CC): a[N2 n1 + n2] = x'^p + i y'^p, DFT over n1 (length
// N1), times W_N^(n2 k1), stored row-major as buf[k1 N2 + n2].  CC N1 / 8 threads.
__global__ void __launch_bounds__(LONG_THREADS, 2)
    k_long_col_fwd(const __grid_constant__ LongArgs la, int q) {
  pdl_wait();
  pdl_trigger();
  if (*la.done) return;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ float inv[2];
  const int l1 = la.l1, N1 = 1 << l1, N2 = 1 << la.l2;
  const int tid = threadIdx.x, c = tid & (LONG_CC - 1), g = tid / LONG_CC, ng = N1 >> 3;
  double2* col = reinterpret_cast<double2*>(smem);   // [CC][stride]
  double2* tw = col + LONG_CC * long_col_stride(l1);  // N1 / 2
  col += c * long_col_stride(l1);
  long_twiddles(tw, l1);
  if (tid == 0) {
    double sx, sy;
    long_scales(la, sx, sy);
    inv[0] = static_cast<float>(1.0 / sx);
    inv[1] = static_cast<float>(1.0 / sy);
  }
  const int n2 = blockIdx.x * LONG_CC + c;
  // v[r]: position r of the first three stages, n1 = g + rev3(r) N1 / 8
  float xr[8], yr[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int n = (g + rev_bits(r, 3) * ng) * N2 + n2;
    xr[r] = n < la.nx ? __ldg(la.x + n) : 0.0f;
    yr[r] = n < la.ny ? __ldg(la.y + n) : 0.0f;
  }
  __syncthreads();
  const float isx = inv[0], isy = inv[1];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    xr[r] *= isx;
    yr[r] *= isy;
  }
  const int plog = la.p_log2[q];
#pragma unroll 1
  for (int s = 0; s < plog; ++s) {
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      xr[r] *= xr[r];
      yr[r] *= yr[r];
    }
  }
  double2 v[8];
  if (max(la.nx, la.ny) <= (1 << (la.logN - 1))) {
#pragma unroll
    for (int r = 0; r < 8; r += 2) v[r] = make_double2(xr[r], yr[r]);
    first_stages8<false, true>(v, tw[ng], tw[3 * ng]);
  } else {
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = make_double2(xr[r], yr[r]);
    first_stages8<false, false>(v, tw[ng], tw[3 * ng]);
  }
#pragma unroll
  for (int r = 0; r < 8; ++r) col[slot(g + rev_bits(r, 3) * ng)] = v[r];
  __syncthreads();
  long_middle<false>(col, tw, l1, g, ng);
#pragma unroll
  for (int r = 0; r < 8; ++r) v[r] = col[slot(8 * g + rev_bits(r, 3))];
  const int rg = rev_bits(g, l1 - 3);
  group_stages<3, false>(v, tw, l1, 0, l1 - 3, rg);
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int k1 = r * ng + rg;
    la.buf[(int64_t)k1 * N2 + n2] = cmul(w_n(la, n2 * k1), v[r]);
  }
}

// R decimation-in-frequency stages of the inverse transform, in the natural
// order of the addresses: position k sits at address bitrev(k), stage s = lg - 1
// - b pairs addresses that differ in bit b; the result of address n is sample
// n.  v[r] is at address (hi << (b0 + R)) + (r << b0) + any lower bits.
template <int R>
__device__ __forceinline__ void dif_stages(double2 (&v)[1 << R], const double2* tw, int lg, int b0,
                                           int hi) {
  const int nh = lg - b0 - R, rh = rev_bits(hi, nh);
#pragma unroll
  for (int t = 0; t < R; ++t) {
#pragma unroll
    for (int o = 0; o < (1 << (R - 1 - t)); ++o) {
      const double2 w = tw[(rh + (rev_bits(o, R - 1 - t) << nh)) << (b0 + t)];
#pragma unroll
      for (int l = 0; l < (1 << t); ++l) {
        const int r = (o << (t + 1)) + l, u = r + (1 << t);
        const double2 d = c_sub(v[r], v[u]);
        v[r] = c_add(v[r], v[u]);
        v[u] = cmulc(w, d);
      }
    }
  }
}

template <int R>
__device__ __forceinline__ void dif_pass(double2* a, const double2* tw, int lg, int b0) {
  for (int g = threadIdx.x; g < (1 << (lg - R)); g += blockDim.x) {
    const int hi = g >> b0, base = (hi << (b0 + R)) | (g & ((1 << b0) - 1));
    double2 v[1 << R];
#pragma unroll
    for (int r = 0; r < (1 << R); ++r) v[r] = a[slot(base + (r << b0))];
    dif_stages<R>(v, tw, lg, b0, hi);
#pragma unroll
    for (int r = 0; r < (1 << R); ++r) a[slot(base + (r << b0))] = v[r];
  }
  __syncthreads();
}

// The last three of them (twiddles as in first_stages8): v[u] becomes i (v[r] -
// v[u]) or the plain difference where the twiddle is conj(-i) or 1.
__device__ __forceinline__ void dif_last8(double2 (&v)[8], double2 w1, double2 w3) {
  auto one = [&](int r, int u) {
    const double2 d = c_sub(v[r], v[u]);
    v[r] = c_add(v[r], v[u]);
    v[u] = d;
  };
  auto by_i = [&](int r, int u) {
    const double2 d = make_double2(v[u].y - v[r].y, v[r].x - v[u].x);
    v[r] = c_add(v[r], v[u]);
    v[u] = d;
  };
  one(0, 1);
  by_i(2, 3);
  one(4, 5);
  v[5] = cmulc(w1, v[5]);
  one(6, 7);
  v[7] = cmulc(w3, v[7]);
  one(0, 2);
  one(1, 3);
  by_i(4, 6);
  by_i(5, 7);
#pragma unroll
  for (int r = 0; r < 4; ++r) one(r, r + 4);
}

__device__ __forceinline__ double2 ld_cluster(uint32_t addr) {
  double2 v;
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(addr));
  return v;
}

// Rows k1 and N1 - k1 by the two CTAs of cluster k1 (cluster 0: the rows 0 and
// N1 / 2, each its own partner), N2 / 8 threads (a warp at least).
__global__ void __launch_bounds__(LONG_THREADS, 2)
    k_long_rows(const __grid_constant__ LongArgs la) {
  pdl_wait();
  pdl_trigger();
  if (*la.done) return;
  extern __shared__ __align__(16) unsigned char smem[];
  const int l2 = la.l2, N1 = 1 << la.l1, N2 = 1 << l2;
  double2* a = reinterpret_cast<double2*>(smem);  // the row
  double2* tw = a + N2;                            // N2 / 2
  const int g = threadIdx.x, ng = N2 >> 3;
  const uint32_t rank = cluster_ctarank();
  const int id = static_cast<int>(cluster_id_x());
  const int k1 = rank == 0 ? id : id == 0 ? N1 >> 1 : N1 - id;
  double2* row = la.buf + (int64_t)k1 * N2;
  long_twiddles(tw, l2);
  double2 v[8];
  if (g < ng) {
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = row[g + rev_bits(r, 3) * ng];
  }
  __syncthreads();
  if (g < ng) {
    first_stages8<false, false>(v, tw[ng], tw[3 * ng]);
#pragma unroll
    for (int r = 0; r < 8; ++r) a[slot(g + rev_bits(r, 3) * ng)] = v[r];
  }
  __syncthreads();
  long_middle<false>(a, tw, l2, threadIdx.x, blockDim.x);
  if (g < ng) {  // the last three stages; the values stay in registers too
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = a[slot(8 * g + rev_bits(r, 3))];
    group_stages<3, false>(v, tw, l2, 0, l2 - 3, rev_bits(g, l2 - 3));
#pragma unroll
    for (int r = 0; r < 8; ++r) a[slot(8 * g + rev_bits(r, 3))] = v[r];
  }
  __syncwarp();
  cluster_sync_all();
  // the spectrum: frequency k2 is at address bitrev(k2); the partner of
  // (k1, k2) is (N1 - k1, N2 - 1 - k2), the complement of the address, of (0, k2)
  // it is (0, (N2 - k2) mod N2)
  double2 z[8];  // by address 8 g + r
  if (g < ng) {
    const uint32_t peer = mapa_shared(smem_u32(a), id == 0 ? rank : rank ^ 1u);
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int at = 8 * g + r;
      const int pa = k1 == 0 ? rev_bits((N2 - rev_bits(at, l2)) & (N2 - 1), l2) : N2 - 1 - at;
      z[r] = spec_z4(v[rev_bits(r, 3)], ld_cluster(peer + 16u * static_cast<uint32_t>(slot(pa))));
    }
  }
  __syncwarp();
  cluster_sync_all();  // both rows are read
  if (g < ng) {
    dif_stages<3>(z, tw, l2, 0, g);
#pragma unroll
    for (int r = 0; r < 8; ++r) a[slot(8 * g + r)] = z[r];
  }
  __syncthreads();
  int b0 = 3;
  const int end = l2 - 3;
  while (b0 < end) {
    if (end - b0 == 3 || end - b0 >= 5) {
      dif_pass<3>(a, tw, l2, b0);
      b0 += 3;
    } else if (end - b0 >= 2) {
      dif_pass<2>(a, tw, l2, b0);
      b0 += 2;
    } else {
      dif_pass<1>(a, tw, l2, b0);
      b0 += 1;
    }
  }
  if (g < ng) {
#pragma unroll
    for (int r = 0; r < 8; ++r) z[r] = a[slot(g + r * ng)];
    dif_last8(z, tw[ng], tw[3 * ng]);
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const int n2 = g + r * ng;
      row[n2] = cmulc(w_n(la, n2 * k1), z[r]);
    }
  }
}

// columns [c0, c0 + CC): inverse DFT over k1 gives 4 s[N2 n1 + n2]; the
// selection of level q for every open index; open terms counted for the
// direct-sum decision.
__global__ void __launch_bounds__(LONG_THREADS, 2)
    k_long_col_inv(const __grid_constant__ LongArgs la, int q) {
  pdl_wait();
  pdl_trigger();
  if (*la.done) return;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double scale;
  const int l1 = la.l1, N1 = 1 << l1, N2 = 1 << la.l2;
  const int tid = threadIdx.x, c = tid & (LONG_CC - 1), g = tid / LONG_CC, ng = N1 >> 3;
  double2* col = reinterpret_cast<double2*>(smem);
  double2* tw = col + LONG_CC * long_col_stride(l1);
  col += c * long_col_stride(l1);
  long_twiddles(tw, l1);
  if (tid == 0) {
    double sx, sy;
    long_scales(la, sx, sy);
    scale = sx * sy;
  }
  const int n2 = blockIdx.x * LONG_CC + c;
  double2 v[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) v[r] = la.buf[(int64_t)(g + rev_bits(r, 3) * ng) * N2 + n2];
  __syncthreads();
  first_stages8<true, false>(v, tw[ng], tw[3 * ng]);
#pragma unroll
  for (int r = 0; r < 8; ++r) col[slot(g + rev_bits(r, 3) * ng)] = v[r];
  __syncthreads();
  long_middle<true>(col, tw, l1, g, ng);
#pragma unroll
  for (int r = 0; r < 8; ++r) v[r] = col[slot(8 * g + rev_bits(r, 3))];
  const int rg = rev_bits(g, l1 - 3);
  group_stages<3, true>(v, tw, l1, 0, l1 - 3, rg);
  const double sxy = scale;
  const double inv4n = __hiloint2double((1023 - 2 - la.logN) << 20, 0);  // 1 / (4 N)
  const int plog = la.p_log2[q];
  unsigned terms = 0u;  // at most 8 x 2^21, 2^29 in a warp
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int m = (r * ng + rg) * N2 + n2;
    if (m >= la.nz || la.res[m] != 0xFF) continue;
    const double S = v[r].x * inv4n;
    const bool stable = ge_pos(S, la.tau);
    if (stable || q == 0) {
      la.z[m] = static_cast<float>(sxy * root_pow2(S, plog));
      la.res[m] = static_cast<uint8_t>(plog | (stable ? 0 : 0x80));
    } else {
      terms += static_cast<unsigned>(terms_of(m, la.nx, la.ny));
    }
  }
  // one atomic per warp (one per thread, all on one address: 5 us more for a level
  // of 2^19 with every index open)
  terms = __reduce_add_sync(0xffffffffu, terms);
  if ((tid & 31) == 0 && terms) atomicAdd(la.open_terms + q, static_cast<unsigned long long>(terms));
}

// After level q: nothing open ends the call; few open terms are summed
// directly for every remaining level (then the call ends); otherwise the
// next level runs.
__global__ void k_long_direct(const __grid_constant__ LongArgs la, int q) {
  pdl_wait();
  pdl_trigger();
  const int done = *la.done;  // may already be this level's, by block 0
  if (done != 0 && done != q + 1) return;
  const unsigned long long W = la.open_terms[q];
  const int N = 1 << la.logN;
  if (W == 0ull || q == 0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *la.done = q + 1;
    return;
  }
  if (W * static_cast<unsigned long long>(8 + 2 * q) >
      10ull * static_cast<unsigned long long>(N) * static_cast<unsigned long long>(la.logN))
    return;
  double sx, sy;
  long_scales(la, sx, sy);
  MaxconvArgs ma;
  ma.nx = la.nx;
  ma.ny = la.ny;
  ma.tau = la.tau;
  for (int t = 0; t < PN_MAX_P; ++t) ma.p_log2[t] = la.p_log2[t];
  const double isx = static_cast<double>(static_cast<float>(1.0 / sx));
  const double isy = static_cast<double>(static_cast<float>(1.0 / sy));
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < la.nz; m += gridDim.x * blockDim.x)
    if (la.res[m] == 0xFF) direct_levels(ma, la.x, la.y, isx * isy, sx * sy, m, q, la.z, la.res);
  if (blockIdx.x == 0 && threadIdx.x == 0) *la.done = q + 1;
}

// ------------------------------------------------------------ top-k x y ---
// Approximate top-k of the products x_i y_j (Alg. 9 with the NormQueue), for
// `batch` independent pairs of length n (2n - 1 <= 8192), each run twice (y,
// and y reversed for the index recovery):
//   k_topk_sums  the p-sums of every p of P for every diagonal m = i + j (one
//                FFT convolution per problem, direction and p);
//   k_topk_merge k <= TOPK_KMAX NormQueue pops, every diagonal's at once: a pop
//                takes the diagonal with the largest estimate psi, subtracts
//                psi^p from every p-sum of that diagonal and re-estimates,
//                clamped to the value just popped; a diagonal is exhausted
//                after as many pops as it has terms;
//   k_topk_first, k_topk_pop  the same pops for larger k, one after another
//                (one warp per problem and direction, a two-level argmax over
//                blocks of 32 diagonals);
//   k_topk_index i = (m1 + m2 - n + 1) / 2, j = m1 - i from the diagonals of
//                the two calls' pops of equal rank, kept when x_i y_j agrees
//                with the popped value within TOPK_VERIFY.
constexpr double TOPK_VERIFY = 1e-2;

struct TopkArgs {
  const float* x;
  const float* y;
  int64_t ldx, ldy;
  int32_t batch, n, nz, logN, n_p, k;
  int32_t p_log2[PN_MAX_P];
  double tau;
  double* sig;     // [batch][2][n_p][nz]
  double* psi0;    // [batch][2][nz] estimates (the first, then kept by the pops)
  double* bmax0;   // [batch][2][nb] the largest estimate of each block of 32 diagonals
  uint16_t* left;  // [batch][2][nz] terms of each diagonal not yet popped
  double* scale;   // [batch] max x * max y, -1 where the input is out of the domain
  int32_t* diag;   // [batch][2][k]
  float* vals;     // [batch][ldk]
  int32_t* out_i;
  int32_t* out_j;
  int64_t ldk;
  int32_t* status;
};

// sigma^(1/2^plog) in FP64: FP32 square roots, then two Newton steps on
// r^p = sigma (sigma >= tau > 0 is in the FP32 range for the default tau).
__device__ double root_fp64(double sig, int plog) {
  if (!(sig > 0.0)) return 0.0;
  float rf = static_cast<float>(sig);
  for (int s = 0; s < plog; ++s) rf = sqrtf(rf);
  double r = rf;
  if (!(r > 0.0)) {  // below the FP32 range: FP64 square roots
    r = sig;
    for (int s = 0; s < plog; ++s) r = sqrt(r);
    return r;
  }
  const double p = ldexp(1.0, plog);
  for (int it = 0; it < 2; ++it) {
    double rp = r;
    for (int s = 0; s < plog; ++s) rp *= rp;
    r = r * (1.0 + (sig / rp - 1.0) / p);
  }
  return r;
}

__device__ __forceinline__ double pow_pow2(double a, int plog) {
  for (int s = 0; s < plog; ++s) a *= a;
  return a;
}

// First forward pass of R = 3 stages straight from the powered values: group j
// holds the addresses j + t N / 8, of which t >= 4 are zero (n <= N / 2), so
// stage 0 copies, stage 1 multiplies by 1 and -i, and half of stage 2 does.
__device__ __forceinline__ void first_pass8(double2* a, const double2* tw, int lg, int j,
                                            const double (&x)[4], const double (&y)[4]) {
  double2 v[8];
#pragma unroll
  for (int r = 0; r < 8; r += 2) {
    const int t = ((r >> 1) & 1) * 2 + (r >> 2);  // rev3(r), r even
    v[r] = make_double2(x[t], y[t]);
  }
  first_stages8<false, true>(v, tw[1 << (lg - 3)], tw[3 << (lg - 3)]);
#pragma unroll
  for (int r = 0; r < 8; ++r) a[slot(j + (rev_bits(r, 3) << (lg - 3)))] = v[r];
}

// The p-sums.  Work items (problem, direction, level) in this order, each CTA
// a contiguous run of them: the items spread over all SMs (one CTA per
// problem and direction ran 512 pairs of the 256-problem batch as 3.37 waves
// of 152, the last one mostly empty), and the values x'^p, y'^p of a pair stay
// in registers and are squared from level to level.
// 256 problems of n = 4096, 13 levels: 7.99 ms (12.29 ms with one CTA per
// problem and direction and two stages per pass).
__global__ void __launch_bounds__(FFT_THREADS, 1)
    k_topk_sums(const __grid_constant__ TopkArgs ta) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lg = ta.logN, N = 1 << lg;
  double2* a = reinterpret_cast<double2*>(smem);
  double2* tw = a + N;
  __shared__ float red[2][FFT_THREADS / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nt = static_cast<int>(blockDim.x), nw = nt >> 5;
  for (int k = tid; k < (N >> 1); k += nt) tw[k] = g_twiddle[k << (FFT_LOG_NMAX - lg)];
  const int64_t items = (int64_t)2 * ta.batch * ta.n_p;
  const int64_t first = items * blockIdx.x / gridDim.x, last = items * (blockIdx.x + 1) / gridDim.x;
  const int groups = N >> 3;  // of the first pass (N >= 8)
  double xv[2][4], yv[2][4];  // the thread's values of the current pair (N >= 8)
  double sx = 1.0, sy = 1.0;
  int plog = 0;
  bool skip = false;          // the pair's input is out of the domain
  for (int64_t it = first; it < last; ++it) {
    const int pd = static_cast<int>(it / ta.n_p), q = static_cast<int>(it - (int64_t)pd * ta.n_p);
    const int b = pd >> 1, dir = pd & 1;
    const float* x = ta.x + (int64_t)b * ta.ldx;
    const float* y = ta.y + (int64_t)b * ta.ldy;
    if (it == first || q == 0) {
      float mx = 0.0f, my = 0.0f;
      bool bad = false;
      for (int k = tid; k < ta.n; k += nt) {
        const float u = x[k], v = y[k];
        bad |= !(u >= 0.0f && u <= 3.4028235e38f) || !(v >= 0.0f && v <= 3.4028235e38f);
        mx = fmaxf(mx, u);
        my = fmaxf(my, v);
      }
      skip = __syncthreads_or(bad);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
        my = fmaxf(my, __shfl_xor_sync(0xffffffffu, my, off));
      }
      if (lane == 0) {
        red[0][warp] = mx;
        red[1][warp] = my;
      }
      __syncthreads();
      sx = sy = 0.0;
      for (int w = 0; w < nw; ++w) {
        sx = fmax(sx, static_cast<double>(red[0][w]));
        sy = fmax(sy, static_cast<double>(red[1][w]));
      }
      if (sx == 0.0) sx = 1.0;
      if (sy == 0.0) sy = 1.0;
      if (tid == 0 && q == 0) {
        if (skip) set_status(ta.status, PN_EDOMAIN);
        if (dir == 0) ta.scale[b] = skip ? -1.0 : sx * sy;
      }
      plog = 0;
      if (lg >= 3) {
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            const int j = tid + u * nt, k = j + t * groups;
            const bool in = j < groups && k < ta.n && !skip;
            xv[u][t] = in ? static_cast<double>(x[k]) * (1.0 / sx) : 0.0;
            yv[u][t] = in ? static_cast<double>(y[dir ? ta.n - 1 - k : k]) * (1.0 / sy) : 0.0;
          }
      }
    }
    if (skip) continue;
    if (lg >= 3) {
      for (; plog < ta.p_log2[q]; ++plog) {
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            xv[u][t] = __dmul_rn(xv[u][t], xv[u][t]);
            yv[u][t] = __dmul_rn(yv[u][t], yv[u][t]);
          }
      }
    }
    int s = 0;
    if (lg >= 4) {
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (tid + u * nt < groups) first_pass8(a, tw, lg, tid + u * nt, xv[u], yv[u]);
      s = 3;
    } else {  // N <= 8: every stage below
      for (int k = tid; k < N; k += nt) {
        double u = 0.0, v = 0.0;
        if (k < ta.n) {
          u = static_cast<double>(x[k]) * (1.0 / sx);
          v = static_cast<double>(y[dir ? ta.n - 1 - k : k]) * (1.0 / sy);
          for (int t = 0; t < ta.p_log2[q]; ++t) {
            u = __dmul_rn(u, u);
            v = __dmul_rn(v, v);
          }
        }
        a[slot(k)] = make_double2(u, v);
      }
    }
    __syncthreads();
    conv_passes(a, tw, lg, s);
    const double scale = 0.25 / N;  // 2 / N, and the spectrum's 8
    double* sig = ta.sig + ((int64_t)pd * ta.n_p + q) * ta.nz;
    for (int m = tid; m < ta.nz; m += nt) {
      const double2 v = a[slot(m & ~1)];
      sig[m] = ((m & 1) ? v.y : v.x) * scale;
    }
    __syncthreads();
  }
}

// First estimate psi_m: the largest p with sigma >= tau (none: 0).
__device__ __forceinline__ int first_level(const TopkArgs& ta, const double* sig, int m, double& v) {
  for (int q = ta.n_p - 1; q >= 0; --q) {
    v = sig[(int64_t)q * ta.nz + m];
    if (v >= ta.tau) return q;
  }
  return -1;
}

// First estimates, term counts and block maxima for k_topk_pop (large k).
__global__ void __launch_bounds__(FFT_THREADS, 1)
    k_topk_first(const __grid_constant__ TopkArgs ta) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double* sig = ta.sig + (int64_t)blockIdx.x * ta.n_p * ta.nz;
  double* psi = ta.psi0 + (int64_t)blockIdx.x * ta.nz;
  uint16_t* left = ta.left + (int64_t)blockIdx.x * ta.nz;
  const bool ok = ta.scale[blockIdx.x >> 1] >= 0.0;  // else no p-sums were written: no pops
  for (int m = tid; m < ta.nz; m += FFT_THREADS) {
    double v = 0.0;
    const int q = ok ? first_level(ta, sig, m, v) : -1;
    psi[m] = q >= 0 ? root_fp64(v, ta.p_log2[q]) : 0.0;
    left[m] = static_cast<uint16_t>(terms_of(m, ta.n, ta.n));
  }
  __syncthreads();
  // the largest estimate of each block of 32 diagonals (-1 past the last)
  const int nb = (ta.nz + 31) >> 5;
  double* bmax = ta.bmax0 + (int64_t)blockIdx.x * nb;
  for (int blk = warp; blk < nb; blk += FFT_THREADS / 32) {
    const int m = blk * 32 + lane;
    double v = m < ta.nz ? psi[m] : -1.0;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, off));
    if (lane == 0) bmax[blk] = v;
  }
}

// k NormQueue pops of one (problem, direction), k <= TOPK_KMAX, for all
// diagonals at once.  A diagonal's pops depend on that diagonal alone: its
// values alpha_1 = psi_m >= alpha_2 >= ... (each re-estimate is clamped to the
// value popped before it), each from the diagonal's p-sums after the pops
// before.  The queue always takes the largest value at hand, the smallest
// diagonal among equals, so its k pops are the k first of all diagonals'
// values in the order (value descending, diagonal ascending), and equal
// pairs are interchangeable.  Hence: keep the k first values known so far;
// a diagonal whose last known value is among them makes its next value (one
// thread per diagonal); repeat until no last value is left among the k.  The
// values are the sequential loop's bit for bit.
// What bounds the sequential loop (k_topk_pop) is latency: 1024 dependent pops
// of about 90 FP64 instructions of one warp, 64 cycles each at two FP64 lanes
// per clock and SM.  Here a warp instruction serves 32 diagonals, and about
// three rounds replace the 1024 steps.  256 problems of n = 4096, k = 1024:
// 0.90 ms (6.34 ms with k_topk_pop).
constexpr int TOPK_KMAX = 2048;
constexpr int TOPK_THREADS = 256;

// Values held at most: every diagonal at first, later k kept and as many new.
__host__ __device__ inline int topk_cap(int nz, int k) {
  int cap = 2;
  while (cap < nz || cap < 2 * k) cap <<= 1;
  return cap;
}
__host__ __device__ inline int topk_merge_smem(int nz, int k) {
  return topk_cap(nz, k) * (8 + 2) + 2 * k;
}

// Sorts (val, dm) [0, count) by value descending, then diagonal ascending;
// the arrays hold a power of two >= count entries.  Values are positive
// doubles as their bits, which order alike, so that no compare takes the FP64
// pipe.
__device__ void topk_sort(uint64_t* val, uint16_t* dm, int count) {
  int n2 = 2;
  while (n2 < count) n2 <<= 1;
  for (int i = count + threadIdx.x; i < n2; i += TOPK_THREADS) {
    val[i] = 0u;
    dm[i] = 0;
  }
  __syncthreads();
  for (int size = 2; size <= n2; size <<= 1) {
    for (int d = size >> 1; d > 0; d >>= 1) {
      for (int e = threadIdx.x; e < (n2 >> 1); e += TOPK_THREADS) {
        const int i = ((e & ~(d - 1)) << 1) | (e & (d - 1)), j = i + d;
        const uint64_t vi = val[i], vj = val[j];
        const uint16_t mi = dm[i], mj = dm[j];
        const bool same = vi == vj;
        const int di = mi & 0x1fff, dj = mj & 0x1fff;
        if ((i & size) == 0 ? (vj > vi || (same && dj < di)) : (vi > vj || (same && di < dj))) {
          val[i] = vj;
          val[j] = vi;
          dm[i] = mj;
          dm[j] = mi;
        }
      }
      __syncthreads();
    }
  }
}

__global__ void __launch_bounds__(TOPK_THREADS)
    k_topk_merge(const __grid_constant__ TopkArgs ta) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr uint16_t TAIL = 0x2000;  // the last value made of its diagonal
  const int cap = topk_cap(ta.nz, ta.k);
  uint64_t* val = reinterpret_cast<uint64_t*>(smem);        // [cap] values, as bits
  float* f = reinterpret_cast<float*>(smem);                // [nz], before val is used
  uint16_t* dm = reinterpret_cast<uint16_t*>(val + cap);    // [cap] diagonal | TAIL
  uint16_t* act = dm + cap;                                 // [k] entries to go on from
  __shared__ int cnt, n_act;
  const int tid = threadIdx.x, lane = tid & 31;
  const int b = blockIdx.x >> 1, dir = blockIdx.x & 1;
  double* sig = ta.sig + (int64_t)blockIdx.x * ta.n_p * ta.nz;
  uint16_t* left = ta.left + (int64_t)blockIdx.x * ta.nz;
  int32_t* diag = ta.diag + (int64_t)blockIdx.x * ta.k;
  const double scale = ta.scale[b];
  int kept = 0;
  if (scale >= 0.0) {  // else: the input is out of the domain, no pops
    // candidates: the first estimates to FP32 accuracy, and the diagonals at
    // or above the k-th largest of them (less a margin far above FP32's error)
    for (int m = tid; m < ta.nz; m += TOPK_THREADS) {
      double v;
      const int q = first_level(ta, sig, m, v);
      float r = 0.0f;
      if (q >= 0) {
        r = static_cast<float>(v);
        for (int s = 0; s < ta.p_log2[q]; ++s) r = sqrtf(r);
        if (!(r > 0.0f)) r = static_cast<float>(root_fp64(v, ta.p_log2[q]));
      }
      f[m] = r;
    }
    if (tid == 0) cnt = 0;
    __syncthreads();
    // largest bit pattern T >= 1 that k values reach (1: fewer than k are positive)
    uint32_t T = 1u;
    if (ta.nz > ta.k) {
      uint32_t lo = 1u, hi = 0x7f800001u;  // reached by >= k (or lo = 1), by < k
      while (hi - lo > 1u) {
        const uint32_t mid = lo + (hi - lo) / 2u;
        int c = 0;
        for (int m = tid; m < ta.nz; m += TOPK_THREADS) c += __float_as_uint(f[m]) >= mid;
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0 && c) atomicAdd(&cnt, c);
        __syncthreads();
        const int total = cnt;
        __syncthreads();
        if (tid == 0) cnt = 0;
        if (total >= ta.k) lo = mid;
        else hi = mid;
        __syncthreads();
      }
      T = lo;
    }
    const float thr = __uint_as_float(T) * (1.0f - 1e-5f);
    for (int m0 = 0; m0 < ta.nz; m0 += TOPK_THREADS) {
      const int m = m0 + tid;
      const bool take = m < ta.nz && f[m] > 0.0f && f[m] >= thr;
      const unsigned bal = __ballot_sync(0xffffffffu, take);
      int at = 0;
      if (lane == 0 && bal) at = atomicAdd(&cnt, __popc(bal));
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(bal & ((1u << lane) - 1u));
      if (take) dm[at] = static_cast<uint16_t>(m);
    }
    __syncthreads();
    int total = cnt;
    for (int c = tid; c < total; c += TOPK_THREADS) {
      const int m = dm[c];
      double v;
      const int q = first_level(ta, sig, m, v);
      val[c] = __double_as_longlong(q >= 0 ? root_fp64(v, ta.p_log2[q]) : 0.0);
      left[m] = static_cast<uint16_t>(terms_of(m, ta.n, ta.n));
      dm[c] = static_cast<uint16_t>(m | TAIL);
    }
    __syncthreads();
    while (true) {
      topk_sort(val, dm, total);
      kept = min(total, ta.k);
      const double theta = kept == ta.k ? __longlong_as_double(val[kept - 1]) : 0.0;
      if (tid == 0) {
        n_act = 0;
        cnt = kept;
      }
      __syncthreads();
      for (int e = tid; e < kept; e += TOPK_THREADS)
        if (dm[e] & TAIL) act[atomicAdd(&n_act, 1)] = static_cast<uint16_t>(e);
      __syncthreads();
      const int A = n_act;
      if (A == 0) break;
      const int pops = (cap - kept) / A;  // per diagonal, at most: their values fit
      for (int c = tid; c < A; c += TOPK_THREADS) {
        const int e0 = act[c], m = dm[e0] & 0x1fff;
        dm[e0] = static_cast<uint16_t>(m);
        double alpha = __longlong_as_double(val[e0]), sg[PN_MAX_P];
#pragma unroll
        for (int q = 0; q < PN_MAX_P; ++q)
          sg[q] = q < ta.n_p ? sig[(int64_t)q * ta.nz + m] : 0.0;
        int rem = left[m];
        int at = -1;
        for (int t = 0; t < pops; ++t) {
          // sigma^(p)_m -= alpha^p for every p, and the largest stable p
          --rem;
          double pw = alpha, sv = 0.0;
          int lg = 0, pl = -1;
#pragma unroll
          for (int q = 0; q < PN_MAX_P; ++q) {
            if (q < ta.n_p) {
              for (; lg < ta.p_log2[q]; ++lg) pw = __dmul_rn(pw, pw);
              sg[q] = __dsub_rn(sg[q], pw);
              if (sg[q] >= ta.tau) {
                sv = sg[q];
                pl = lg;
              }
            }
          }
          const double e = rem > 0 && pl >= 0 ? fmin(root_fp64(sv, pl), alpha) : 0.0;
          if (!(e > 0.0) || e < theta) {  // the diagonal makes no more of the k values
            at = -1;
            break;
          }
          at = atomicAdd(&cnt, 1);
          val[at] = __double_as_longlong(e);
          dm[at] = static_cast<uint16_t>(m);
          alpha = e;
        }
        if (at >= 0) {
          dm[at] = static_cast<uint16_t>(m | TAIL);
          left[m] = static_cast<uint16_t>(rem);
#pragma unroll
          for (int q = 0; q < PN_MAX_P; ++q)
            if (q < ta.n_p) sig[(int64_t)q * ta.nz + m] = sg[q];
        }
      }
      __syncthreads();
      total = cnt;
      __syncthreads();
    }
  }
  for (int t = tid; t < ta.k; t += TOPK_THREADS) {
    diag[t] = t < kept ? (dm[t] & 0x1fff) : -1;
    if (dir == 0)
      ta.vals[(int64_t)b * ta.ldk + t] =
          t < kept ? static_cast<float>(__longlong_as_double(val[t]) * scale) : 0.0f;
  }
}

// (value, index) argmax across a warp: larger value, then smaller index.
__device__ __forceinline__ void warp_argmax(double& v, int& i) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const double ov = __shfl_xor_sync(0xffffffffu, v, off);
    const int oi = __shfl_xor_sync(0xffffffffu, i, off);
    if (ov > v || (ov == v && oi < i)) {
      v = ov;
      i = oi;
    }
  }
}

// One warp per (problem, direction).  The estimates psi and the counts of
// terms left live in the workspace; shared memory holds only the largest
// estimate of each block of 32 diagonals, so every warp of the launch is
// resident at once.  A pop reads the chosen block's 32 estimates with one
// coalesced load.
__global__ void __launch_bounds__(32) k_topk_pop(const __grid_constant__ TopkArgs ta) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int nb = (ta.nz + 31) >> 5;
  double* bmax = reinterpret_cast<double*>(smem);  // nb
  const int lane = threadIdx.x;
  const int b = blockIdx.x >> 1, dir = blockIdx.x & 1;
  double* sig = ta.sig + (int64_t)blockIdx.x * ta.n_p * ta.nz;
  double* psi = ta.psi0 + (int64_t)blockIdx.x * ta.nz;
  uint16_t* left = ta.left + (int64_t)blockIdx.x * ta.nz;
  int32_t* diag = ta.diag + (int64_t)blockIdx.x * ta.k;
  const double* bmax0 = ta.bmax0 + (int64_t)blockIdx.x * nb;
  for (int blk = lane; blk < nb; blk += 32) bmax[blk] = bmax0[blk];
  __syncwarp();
  const double scale = dir == 0 ? ta.scale[b] : 0.0;
  for (int t = 0; t < ta.k; ++t) {
    // the block, then the diagonal, with the largest psi
    double v = -2.0;
    int bi = 0x7fffffff;
    for (int blk = lane; blk < nb; blk += 32) {
      const double w = bmax[blk];
      if (w > v) {
        v = w;
        bi = blk;
      }
    }
    warp_argmax(v, bi);
    const int mcand = bi * 32 + lane;
    double pv = mcand < ta.nz ? psi[mcand] : -1.0;
    const int lf = mcand < ta.nz ? left[mcand] : 0;
    double pm = pv;
    int m = mcand;
    warp_argmax(pm, m);
    if (!(pm > 0.0)) {  // every diagonal exhausted or without a stable p
      for (int r = t + lane; r < ta.k; r += 32) {
        diag[r] = -1;
        if (dir == 0) ta.vals[(int64_t)b * ta.ldk + r] = 0.0f;
      }
      break;
    }
    const double alpha = pm;
    if (lane == 0) {
      diag[t] = m;
      if (dir == 0) ta.vals[(int64_t)b * ta.ldk + t] = static_cast<float>(alpha * scale);
    }
    const int mi = m - bi * 32;  // the popped diagonal's lane
    const int rem = __shfl_sync(0xffffffffu, lf, mi) - 1;
    // NormQueue pop: sigma^(p)_m -= alpha^p for every p (one lane per p)
    double sq = 0.0;
    if (lane < ta.n_p) {
      const int64_t at = (int64_t)lane * ta.nz + m;
      sq = sig[at] - pow_pow2(alpha, ta.p_log2[lane]);
      sig[at] = sq;
    }
    // re-estimate: the largest p whose sigma is >= tau, clamped to alpha
    const unsigned stable = __ballot_sync(0xffffffffu, lane < ta.n_p && sq >= ta.tau);
    double e = 0.0;
    if (rem > 0 && stable) {
      const int qs = 31 - __clz(stable);
      const double sv = __shfl_sync(0xffffffffu, sq, qs);
      e = fmin(root_fp64(sv, ta.p_log2[qs]), alpha);
    }
    if (lane == mi) {
      pv = e;
      psi[m] = e;
      left[m] = static_cast<uint16_t>(rem);
    }
    double w = pv;
    int wi = lane;
    warp_argmax(w, wi);
    if (lane == 0) bmax[bi] = w;
    __syncwarp();
  }
}

__global__ void k_topk_index(const __grid_constant__ TopkArgs ta) {
  const int b = blockIdx.x;
  const int32_t* d1 = ta.diag + (int64_t)(2 * b) * ta.k;
  const int32_t* d2 = ta.diag + (int64_t)(2 * b + 1) * ta.k;
  const float* x = ta.x + (int64_t)b * ta.ldx;
  const float* y = ta.y + (int64_t)b * ta.ldy;
  for (int t = threadIdx.x; t < ta.k; t += blockDim.x) {
    int i = -1, j = -1;
    const int m1 = d1[t], m2 = d2[t];
    const int s = m1 + m2 - ta.n + 1;
    if (m1 >= 0 && m2 >= 0 && (s & 1) == 0) {
      const int ii = s >> 1, jj = m1 - ii;
      if (ii >= 0 && ii < ta.n && jj >= 0 && jj < ta.n) {
        const double v = ta.vals[(int64_t)b * ta.ldk + t];
        const double prod = static_cast<double>(x[ii]) * static_cast<double>(y[jj]);
        if (fabs(prod - v) <= TOPK_VERIFY * v) {
          i = ii;
          j = jj;
        }
      }
    }
    if (ta.out_i) ta.out_i[(int64_t)b * ta.ldk + t] = i;
    if (ta.out_j) ta.out_j[(int64_t)b * ta.ldk + t] = j;
  }
}

std::mutex g_tw_mu;
bool g_tw_ready[64];

}  // namespace

int maxconv_fft_smem_bytes(int logN) {
  const int N = 1 << logN;
  return N * 16 + (N / 2) * 16 + N;  // data, twiddles, p_sel of up to N indices
}

// The device's tables of FFT twiddle factors, filled on the first use: on a stream of
// their own that is waited for, so that the tables are there for every stream and
// thread once they are marked ready, and so that a first call under stream
// capture fills them at once instead of recording the fill into its graph.
int ensure_twiddles() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_tw_mu);
  if (g_tw_ready[dev]) return 0;
  // (a capture elsewhere in the process does not forbid what follows: none of it
  // touches a capturing stream)
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  cudaError_t e = cudaThreadExchangeStreamCaptureMode(&mode);
  if (e != cudaSuccess) return e;
  cudaStream_t s = nullptr;
  e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
  if (e == cudaSuccess) {
    k_twiddle_init<<<(FFT_NMAX / 2 + 255) / 256, 256, 0, s>>>();
    e = cudaGetLastError();
    const cudaError_t done = cudaStreamSynchronize(s);
    if (e == cudaSuccess) e = done;
    cudaStreamDestroy(s);
  }
  const cudaError_t back = cudaThreadExchangeStreamCaptureMode(&mode);
  if (e == cudaSuccess) e = back;
  if (e == cudaSuccess) g_tw_ready[dev] = true;
  return e;
}

int launch_maxconv_fft(const MaxconvArgs& ma, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int te = ensure_twiddles();
  if (te) return te;
  const int smem = maxconv_fft_smem_bytes(ma.logN);
  if (const cudaError_t e = allow_smem<k_maxconv_fft>(maxconv_fft_smem_bytes(FFT_LOG_NMAX))) return e;
  // eight values per thread: several CTAs per SM on short problems
  const int N = 1 << ma.logN;
  const int threads = N / 8 < 64 ? 64 : N / 8;
  k_maxconv_fft<<<static_cast<unsigned>(ma.batch), threads, smem, s>>>(ma);
  return cudaGetLastError();
}

int maxconv_exact_smem_bytes() {
  return static_cast<int>(sizeof(float)) * (MCX_IB + 8 + MCX_SPAN + MCX_IB + 16);
}

int launch_maxconv_exact(const MaxconvArgs& ma, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int smem = maxconv_exact_smem_bytes();
  if (const cudaError_t e = allow_smem<k_maxconv_exact>(smem)) return e;
  const int iblocks = (ma.nx + MCX_IB - 1) / MCX_IB;
  if (iblocks > 1) {  // partial maxima meet in z by atomicMax: start from 0
    const cudaError_t me = cudaMemset2DAsync(ma.z, sizeof(float) * ma.ldz, 0,
                                             sizeof(float) * ma.nz, ma.batch, s);
    if (me != cudaSuccess) return me;
  }
  const dim3 grid(static_cast<unsigned>((ma.nz + MCX_SPAN - 1) / MCX_SPAN),
                  static_cast<unsigned>(iblocks),
                  static_cast<unsigned>(ma.batch < 65535 ? ma.batch : 65535));
  k_maxconv_exact<<<grid, MCX_THREADS, smem, s>>>(ma);
  return cudaGetLastError();
}

// Workspace of a long problem: control words, the W_N^m tables, the
// complex buffer of N, and p_sel when the caller passes none.
struct LongLayout {
  size_t off_ctrl = 0, off_tlo = 0, off_thi = 0, off_buf = 0, off_res = 0, total = 0;
};

LongLayout long_layout(int64_t nz, int logN, bool own_res) {
  LongLayout L;
  size_t off = 0;
  L.off_ctrl = off; off += 256;  // open_terms[16] (128 B), done, max x, max y
  L.off_tlo = off; off += 2048 * sizeof(double2);
  L.off_thi = off; off += 2048 * sizeof(double2);
  L.off_buf = off; off += (size_t(1) << logN) * sizeof(double2);
  if (own_res) { L.off_res = off; off += (static_cast<size_t>(nz) + 255) & ~size_t(255); }
  L.total = off;
  return L;
}

int long_logN(int64_t nz) {
  int logN = 1;
  while ((int64_t(1) << logN) < nz) ++logN;
  return logN < 14 ? 14 : logN;
}

int launch_maxconv_long(const pn_opts* o, int64_t nx, const float* x, int64_t ny, const float* y,
                        float* z, uint8_t* p_sel, uint8_t* ws, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int e = ensure_twiddles();
  if (e) return e;
  const int64_t nz = nx + ny - 1;
  LongArgs la;
  std::memset(&la, 0, sizeof(la));
  la.logN = long_logN(nz);
  la.l1 = la.logN / 2 < 10 ? la.logN / 2 : 10;
  la.l2 = la.logN - la.l1;
  const LongLayout L = long_layout(nz, la.logN, p_sel == nullptr);
  la.x = x; la.y = y; la.z = z;
  la.res = p_sel ? p_sel : ws + L.off_res;
  la.nx = static_cast<int32_t>(nx);
  la.ny = static_cast<int32_t>(ny);
  la.nz = static_cast<int32_t>(nz);
  la.n_p = o->n_p;
  for (int q = 0; q < o->n_p; ++q) la.p_log2[q] = o->p_log2[q];
  la.tau = o->tau > 0.0 ? o->tau : 1e-12;
  la.status = o->dev_status;
  la.buf = reinterpret_cast<double2*>(ws + L.off_buf);
  la.tlo = reinterpret_cast<const double2*>(ws + L.off_tlo);
  la.thi = reinterpret_cast<const double2*>(ws + L.off_thi);
  la.open_terms = reinterpret_cast<unsigned long long*>(ws + L.off_ctrl);
  la.done = reinterpret_cast<int32_t*>(ws + L.off_ctrl + 128);
  la.mxy = reinterpret_cast<uint32_t*>(ws + L.off_ctrl + 136);
  if ((e = cudaMemsetAsync(ws + L.off_ctrl, 0, 256, s))) return e;
  if ((e = cudaMemsetAsync(la.res, 0xFF, static_cast<size_t>(nz), s))) return e;
  k_long_init<<<LONG_TAB_BLOCKS + LONG_MAX_BLOCKS, 256, 0, s>>>(
      la, reinterpret_cast<double2*>(ws + L.off_tlo), reinterpret_cast<double2*>(ws + L.off_thi));
  if ((e = cudaGetLastError())) return e;
  const int N1 = 1 << la.l1, N2 = 1 << la.l2;
  const auto col_bytes = [](int n) { return (LONG_CC * (n + 2) + n / 2) * static_cast<int>(sizeof(double2)); };
  const auto row_bytes = [](int n) { return (n + n / 2) * static_cast<int>(sizeof(double2)); };
  const int col_threads = LONG_CC * N1 / 8, row_threads = N2 / 8 < 32 ? 32 : N2 / 8;
  const dim3 cols(N2 / LONG_CC);
  const int sms = host_device_sms();
  const int smem_col = even_share_smem(col_bytes(N1), N2 / LONG_CC, col_threads, sms);
  const int smem_row = even_share_smem(row_bytes(N2), N1, row_threads, sms);
  constexpr int DIRECT_CTAS = 152 * 4, DIRECT_THREADS = 256;
  const int smem_direct = even_share_smem(0, DIRECT_CTAS, DIRECT_THREADS, sms);
  if ((e = allow_smem<k_long_col_fwd>(CTA_SMEM_MAX))) return e;
  if ((e = allow_smem<k_long_col_inv>(CTA_SMEM_MAX))) return e;
  if ((e = allow_smem<k_long_rows>(CTA_SMEM_MAX))) return e;
  if ((e = allow_smem<k_long_direct>(CTA_SMEM_MAX))) return e;
  cudaLaunchConfig_t rows = {};
  rows.gridDim = dim3(N1);
  rows.blockDim = dim3(row_threads);
  rows.dynamicSmemBytes = smem_row;
  rows.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see launch_pdl
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  rows.attrs = attr;
  rows.numAttrs = 2;
  for (int q = o->n_p - 1; q >= 0; --q) {
    if ((e = launch_pdl(k_long_col_fwd, cols, dim3(col_threads), smem_col, s, la, q))) return e;
    if ((e = cudaLaunchKernelEx(&rows, k_long_rows, la))) return e;
    if ((e = launch_pdl(k_long_col_inv, cols, dim3(col_threads), smem_col, s, la, q))) return e;
    if ((e = launch_pdl(k_long_direct, dim3(DIRECT_CTAS), dim3(DIRECT_THREADS), smem_direct, s, la, q)))
      return e;
  }
  return cudaGetLastError();
}

struct TopkLayout {
  size_t off_sig = 0, off_psi = 0, off_bmax = 0, off_left = 0, off_scale = 0, off_diag = 0,
         total = 0;
};

TopkLayout topk_layout(int64_t batch, int64_t n, int64_t k, int n_p) {
  TopkLayout L;
  const int64_t nz = 2 * n - 1;
  size_t off = 0;
  L.off_sig = off; off += static_cast<size_t>(batch) * 2 * n_p * nz * sizeof(double);
  off = (off + 255) & ~size_t(255);
  L.off_psi = off; off += static_cast<size_t>(batch) * 2 * nz * sizeof(double);
  off = (off + 255) & ~size_t(255);
  L.off_bmax = off; off += static_cast<size_t>(batch) * 2 * ((nz + 31) / 32) * sizeof(double);
  off = (off + 255) & ~size_t(255);
  L.off_left = off; off += static_cast<size_t>(batch) * 2 * nz * sizeof(uint16_t);
  off = (off + 255) & ~size_t(255);
  L.off_scale = off; off += static_cast<size_t>(batch) * sizeof(double);
  off = (off + 255) & ~size_t(255);
  L.off_diag = off; off += static_cast<size_t>(batch) * 2 * k * sizeof(int32_t);
  L.total = (off + 255) & ~size_t(255);
  return L;
}

int launch_topk(const TopkArgs& ta0, uint8_t* ws, void* stream) {
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int e = ensure_twiddles();
  if (e) return e;
  TopkArgs ta = ta0;
  const TopkLayout L = topk_layout(ta.batch, ta.n, ta.k, ta.n_p);
  ta.sig = reinterpret_cast<double*>(ws + L.off_sig);
  ta.psi0 = reinterpret_cast<double*>(ws + L.off_psi);
  ta.bmax0 = reinterpret_cast<double*>(ws + L.off_bmax);
  ta.left = reinterpret_cast<uint16_t*>(ws + L.off_left);
  ta.scale = reinterpret_cast<double*>(ws + L.off_scale);
  ta.diag = reinterpret_cast<int32_t*>(ws + L.off_diag);
  const int N = 1 << ta.logN;
  const int smem_sums = (N + N / 2) * static_cast<int>(sizeof(double2));
  if ((e = allow_smem<k_topk_sums>((FFT_NMAX + FFT_NMAX / 2) * static_cast<int>(sizeof(double2)))))
    return e;
  const int nb = (ta.nz + 31) / 32;
  const int smem_pop = nb * 8;  // at most 2 KB
  // threads: two groups of eight values each in the first pass; as many CTAs
  // as fit on the SMs, each with a run of the work items
  const int threads = N / 16 < 64 ? 64 : N / 16 > FFT_THREADS ? FFT_THREADS : N / 16;
  int per_sm = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_topk_sums, threads, smem_sums)))
    return e;
  const int64_t items = (int64_t)2 * ta.batch * ta.n_p;
  const int64_t room = static_cast<int64_t>(host_device_sms()) * (per_sm > 0 ? per_sm : 1);
  k_topk_sums<<<static_cast<unsigned>(items < room ? items : room), threads, smem_sums, s>>>(ta);
  if (ta.k <= TOPK_KMAX) {
    const int smem = topk_merge_smem(ta.nz, ta.k);
    if ((e = allow_smem<k_topk_merge>(topk_merge_smem(FFT_NMAX - 1, TOPK_KMAX)))) return e;
    k_topk_merge<<<2 * ta.batch, TOPK_THREADS, smem, s>>>(ta);
  } else {
    k_topk_first<<<2 * ta.batch, FFT_THREADS, 0, s>>>(ta);
    k_topk_pop<<<2 * ta.batch, 32, smem_pop, s>>>(ta);
  }
  k_topk_index<<<ta.batch, 256, 0, s>>>(ta);
  return cudaGetLastError();
}

}  // namespace pn

using namespace pn;

extern "C" {

size_t pn_topk_xy_workspace_size(int64_t batch, int64_t n, int64_t k, const pn_opts* opts) {
  if (!host_opts_valid(opts) || batch < 1 || n < 1 || 2 * n - 1 > (int64_t(1) << MAXCONV_LOG_NMAX) ||
      k < 1 || batch > (1 << 20) || k > (int64_t(1) << 30))
    return 0;
  return topk_layout(batch, n, k, opts->n_p).total;
}

pn_status topk_xy(int64_t batch, int64_t n, const float* x, int64_t ldx, const float* y,
                  int64_t ldy, int64_t k, float* vals, int32_t* idx_i, int32_t* idx_j,
                  int64_t ldk, const pn_opts* opts, void* ws, size_t ws_bytes, void* stream) {
  if (!host_opts_valid(opts)) return PN_EINVAL;
  if (opts->estimator != 0 || opts->correction != 0) return PN_EUNSUPPORTED;
  if (batch < 0 || n < 1 || k < 1) return PN_EINVAL;
  if (batch == 0) return PN_OK;
  if (2 * n - 1 > (int64_t(1) << MAXCONV_LOG_NMAX) || batch > (1 << 20) || k > (int64_t(1) << 30))
    return PN_EUNSUPPORTED;
  if (!x || !y || !vals || ldx < n || ldy < n || ldk < k) return PN_EINVAL;
  const size_t need = pn_topk_xy_workspace_size(batch, n, k, opts);
  if (!ws || ws_bytes < need) return PN_EWORKSPACE;
  if (reinterpret_cast<uintptr_t>(ws) % 256) return PN_EALIGN;
  if (host_device_sms() <= 0) return PN_EUNSUPPORTED;
  TopkArgs ta;
  std::memset(&ta, 0, sizeof(ta));
  ta.x = x; ta.y = y; ta.ldx = ldx; ta.ldy = ldy;
  ta.batch = static_cast<int32_t>(batch);
  ta.n = static_cast<int32_t>(n);
  ta.nz = static_cast<int32_t>(2 * n - 1);
  int logN = 1;
  while ((int64_t(1) << logN) < 2 * n - 1) ++logN;
  ta.logN = logN;
  ta.n_p = opts->n_p;
  for (int q = 0; q < opts->n_p; ++q) ta.p_log2[q] = opts->p_log2[q];
  ta.tau = opts->tau > 0.0 ? opts->tau : pn_maxconv_default_tau();
  ta.k = static_cast<int32_t>(k);
  ta.vals = vals; ta.out_i = idx_i; ta.out_j = idx_j; ta.ldk = ldk;
  ta.status = opts->dev_status;
  return launch_topk(ta, static_cast<uint8_t*>(ws), stream) == 0 ? PN_OK : PN_ECUDA;
}


size_t pn_maxconv_long_workspace_size(int64_t nx, int64_t ny, int32_t with_p_sel) {
  if (nx < 1 || ny < 1 || nx + ny - 1 > (int64_t(1) << 22)) return 0;
  const int64_t nz = nx + ny - 1;
  return long_layout(nz, long_logN(nz), with_p_sel == 0).total;
}

pn_status maxconv_pnorm_long(int64_t nx, const float* x, int64_t ny, const float* y, float* z,
                             uint8_t* p_sel, const pn_opts* opts, void* ws, size_t ws_bytes,
                             void* stream) {
  if (!host_opts_valid(opts)) return PN_EINVAL;
  if (opts->estimator != 0 || opts->correction != 0) return PN_EUNSUPPORTED;
  if (nx < 1 || ny < 1) return PN_EINVAL;
  if (nx + ny - 1 > (int64_t(1) << 22)) return PN_EUNSUPPORTED;
  if (!x || !y || !z) return PN_EINVAL;
  const size_t need = pn_maxconv_long_workspace_size(nx, ny, p_sel != nullptr);
  if (!ws || ws_bytes < need) return PN_EWORKSPACE;
  if (reinterpret_cast<uintptr_t>(ws) % 256) return PN_EALIGN;
  if (host_device_sms() <= 0) return PN_EUNSUPPORTED;
  return launch_maxconv_long(opts, nx, x, ny, y, z, p_sel, static_cast<uint8_t*>(ws), stream) == 0
             ? PN_OK
             : PN_ECUDA;
}


double pn_maxconv_default_tau(void) { return 1e-12; }

pn_status maxconv_pnorm(int64_t batch, int64_t nx, const float* x, int64_t ldx, int64_t ny,
                        const float* y, int64_t ldy, float* z, int64_t ldz, uint8_t* p_sel,
                        int64_t ldp, const pn_opts* opts, void* stream) {
  if (!host_opts_valid(opts)) return PN_EINVAL;
  if (opts->estimator != 0 || opts->correction != 0) return PN_EUNSUPPORTED;
  if (batch < 0 || batch > 0x7fffffff || nx < 1 || ny < 1) return PN_EINVAL;
  if (batch == 0) return PN_OK;
  const int64_t nz = nx + ny - 1;
  if (nz > (int64_t(1) << MAXCONV_LOG_NMAX)) return PN_EUNSUPPORTED;
  if (!x || !y || !z || ldx < nx || ldy < ny || ldz < nz || (p_sel && ldp < nz)) return PN_EINVAL;
  if (host_device_sms() <= 0) return PN_EUNSUPPORTED;
  MaxconvArgs ma;
  std::memset(&ma, 0, sizeof(ma));
  ma.x = x; ma.y = y; ma.z = z; ma.psel = p_sel;
  ma.ldx = ldx; ma.ldy = ldy; ma.ldz = ldz; ma.ldp = ldp;
  ma.batch = batch;
  ma.nx = static_cast<int32_t>(nx);
  ma.ny = static_cast<int32_t>(ny);
  ma.nz = static_cast<int32_t>(nz);
  int logN = 1;
  while ((int64_t(1) << logN) < nz) ++logN;
  ma.logN = logN;
  ma.n_p = opts->n_p;
  for (int q = 0; q < opts->n_p; ++q) ma.p_log2[q] = opts->p_log2[q];
  ma.tau = opts->tau > 0.0 ? opts->tau : pn_maxconv_default_tau();
  ma.status = opts->dev_status;
  return launch_maxconv_fft(ma, stream) == 0 ? PN_OK : PN_ECUDA;
}

pn_status maxconv_exact(int64_t batch, int64_t nx, const float* x, int64_t ldx, int64_t ny,
                        const float* y, int64_t ldy, float* z, int64_t ldz, void* stream) {
  if (batch < 0 || nx < 1 || ny < 1) return PN_EINVAL;
  if (batch == 0) return PN_OK;
  if (nx + ny > (int64_t(1) << 30)) return PN_EUNSUPPORTED;
  const int64_t nz = nx + ny - 1;
  if (!x || !y || !z || ldx < nx || ldy < ny || ldz < nz) return PN_EINVAL;
  if (host_device_sms() <= 0) return PN_EUNSUPPORTED;
  MaxconvArgs ma;
  std::memset(&ma, 0, sizeof(ma));
  ma.x = x; ma.y = y; ma.z = z;
  ma.ldx = ldx; ma.ldy = ldy; ma.ldz = ldz;
  ma.batch = batch;
  ma.nx = static_cast<int32_t>(nx);
  ma.ny = static_cast<int32_t>(ny);
  ma.nz = static_cast<int32_t>(nz);
  return launch_maxconv_exact(ma, stream) == 0 ? PN_OK : PN_ECUDA;
}

}  // extern "C"
