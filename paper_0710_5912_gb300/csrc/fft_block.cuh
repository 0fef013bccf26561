// Block-level complex FFTs for the row and column passes.
//
// The paper's transforms (Appendix B: real <-> reciprocal space "x -> q_x and
// y -> q_y", done with a CPU library) are done here by a hand-written
// Stockham auto-sort FFT: every stage reads R values at stride N/R, applies the
// stage twiddles, performs a radix-R DFT in registers and writes the results to
// their auto-sorted positions, so the output comes out in natural order with no
// bit reversal.
//
// - fft_reg (the step kernels): each thread holds P = 8 (FP64) or 16 (FP32)
//   complex values in registers; a stage is radix P (one butterfly per
//   thread), or radix 8 / 4 / 2 for the last stage; stages exchange through a
//   padded shared buffer.  Twiddles come from per-stage tables (below), copied
//   once per CTA into shared memory in a compact per-length form.
// - fft_smem (the structure-factor diagnostics): in-place in shared memory,
//   8 values per thread per stage, twiddles from one table
//   W[k] = exp(+2 pi i k / NMAX) read with stride NMAX / N.
//
// Conventions (shared with the host code): forward uses exp(-2 pi i jk / N),
// inverse uses exp(+2 pi i jk / N) without scaling.  All tables are computed on
// the host in double precision and rounded once to the working precision.
#pragma once
#include <cuda_runtime.h>

namespace shf {

constexpr int LOG2_NMAX = 12;          // largest supported transform: 4096 points
constexpr int NMAX = 1 << LOG2_NMAX;

template <class T> struct cplx_of;
template <> struct cplx_of<float> { using type = float2; };
template <> struct cplx_of<double> { using type = double2; };
template <class T> using cplx = typename cplx_of<T>::type;

template <class C> __device__ __forceinline__ C cadd(C a, C b) { return C{a.x + b.x, a.y + b.y}; }
template <class C> __device__ __forceinline__ C csub(C a, C b) { return C{a.x - b.x, a.y - b.y}; }
template <class C> __device__ __forceinline__ C cmul(C a, C b) {
  return C{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <class C> __device__ __forceinline__ C cconj(C a) { return C{a.x, -a.y}; }
template <class C, class T> __device__ __forceinline__ C cscale(C a, T s) { return C{a.x * s, a.y * s}; }

// multiply by sigma*i, sigma = +1 (inverse) or -1 (forward)
template <bool INV, class C> __device__ __forceinline__ C mul_si(C a) {
  return INV ? C{-a.y, a.x} : C{a.y, -a.x};
}

template <bool INV, class C>
__device__ __forceinline__ void dft2(C& a, C& b) {
  C t = a;
  a = cadd(t, b);
  b = csub(t, b);
}

// X_k = sum_r v_r w^{rk}, w = sigma*i
template <bool INV, class C>
__device__ __forceinline__ void dft4(C& v0, C& v1, C& v2, C& v3) {
  C s02 = cadd(v0, v2), d02 = csub(v0, v2);
  C s13 = cadd(v1, v3), d13 = csub(v1, v3);
  C wd = mul_si<INV>(d13);
  v0 = cadd(s02, s13);
  v2 = csub(s02, s13);
  v1 = cadd(d02, wd);
  v3 = csub(d02, wd);
}

// radix 8 as two radix-4 DFTs (even / odd inputs) joined by powers of
// w8 = exp(sigma 2 pi i / 8) = (1 + sigma i) / sqrt(2)
template <bool INV, class C>
__device__ __forceinline__ void dft8(C* v) {
  using T = decltype(v[0].x);
  const T c = T(0.70710678118654752440084436210484904);  // 1/sqrt(2)
  C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
  C o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4<INV>(e0, e1, e2, e3);
  dft4<INV>(o0, o1, o2, o3);
  const T sg = INV ? T(1) : T(-1);
  // w8^1 * o1 = c (1 + sigma i) o1
  C t1 = C{c * (o1.x - sg * o1.y), c * (o1.y + sg * o1.x)};
  // w8^2 * o2 = sigma i o2
  C t2 = mul_si<INV>(o2);
  // w8^3 * o3 = c (-1 + sigma i) o3
  C t3 = C{c * (-o3.x - sg * o3.y), c * (-o3.y + sg * o3.x)};
  v[0] = cadd(e0, o0);
  v[4] = csub(e0, o0);
  v[1] = cadd(e1, t1);
  v[5] = csub(e1, t1);
  v[2] = cadd(e2, t2);
  v[6] = csub(e2, t2);
  v[3] = cadd(e3, t3);
  v[7] = csub(e3, t3);
}

template <bool INV, class C>
__device__ __forceinline__ C twiddle(const C* __restrict__ tw, int idx) {
  C w = __ldg(tw + idx);
  return INV ? w : cconj(w);
}

// One Stockham stage of radix R = 2^LR on NB buffers: each thread does 8/R
// butterflies j = tid + b*T (T = N/8 threads per instance), reading inputs at
// j + r*N/R and writing the radix-R outputs to ((j - k) R + k) + r Ns with
// k = j mod Ns, Ns being the length of the sub-transforms already done.
template <bool INV, int NB, int LR, class C>
__device__ __forceinline__ void fft_stage(C* const (&buf)[NB], int log2N, int log2Ns, int tid,
                                          const C* __restrict__ tw) {
  constexpr int R = 1 << LR;
  constexpr int B = 8 >> LR;
  const int N = 1 << log2N;
  const int T = N >> 3;
  const int stride = N >> LR;
  C v[NB][8];
#pragma unroll
  for (int q = 0; q < NB; ++q)
#pragma unroll
    for (int b = 0; b < B; ++b)
#pragma unroll
      for (int r = 0; r < R; ++r) v[q][b * R + r] = buf[q][tid + b * T + r * stride];
  __syncthreads();
  const int Ns = 1 << log2Ns;
  const int twShift = LOG2_NMAX - log2Ns - LR;
#pragma unroll
  for (int b = 0; b < B; ++b) {
    const int j = tid + b * T;
    const int k = j & (Ns - 1);
    const int base = ((j - k) << LR) + k;
    if (log2Ns > 0) {
#pragma unroll
      for (int r = 1; r < R; ++r) {
        const C w = twiddle<INV>(tw, (k * r) << twShift);
#pragma unroll
        for (int q = 0; q < NB; ++q) v[q][b * R + r] = cmul(v[q][b * R + r], w);
      }
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      if (LR == 3) {
        dft8<INV>(&v[q][b * R]);
      } else if (LR == 2) {
        dft4<INV>(v[q][b * R], v[q][b * R + 1], v[q][b * R + 2], v[q][b * R + 3]);
      } else {
        dft2<INV>(v[q][b * R], v[q][b * R + 1]);
      }
#pragma unroll
      for (int r = 0; r < R; ++r) buf[q][base + r * Ns] = v[q][b * R + r];
    }
  }
  __syncthreads();
}

// In-place FFT of NB buffers of length N = 2^log2N (N >= 8) held in shared
// memory.  tid in [0, N/8) is this thread's index within its FFT instance;
// every thread of the CTA must call this (it contains __syncthreads), and all
// instances in the CTA must share N.  The routine starts with a barrier, so
// the caller's writes to the buffers need no barrier of their own, and it
// ends with one, so the results may be read right away.
template <bool INV, int NB, class C>
__device__ void fft_smem(C* const (&buf)[NB], int log2N, int tid, const C* __restrict__ tw) {
  __syncthreads();
  int log2Ns = 0;
  while (log2N - log2Ns >= 3) {
    fft_stage<INV, NB, 3>(buf, log2N, log2Ns, tid, tw);
    log2Ns += 3;
  }
  if (log2N - log2Ns == 2) fft_stage<INV, NB, 2>(buf, log2N, log2Ns, tid, tw);
  else if (log2N - log2Ns == 1) fft_stage<INV, NB, 1>(buf, log2N, log2Ns, tid, tw);
}

// ---------------------------------------------------------------------------
// Register-resident FFT (P = 8 or 16 points per thread).
//
// Thread t of an instance (0 <= t < T = N/P) holds v[q] = x[t + T q],
// q = 0..P-1.  Each Stockham stage is radix P except possibly the last (radix
// 4 or 2 when log2 N is not a multiple of log2 P).  A stage's butterflies
// j = t + b T (b < P/R) read x[j + r N/R] = v[b + r P/R] -- exactly the
// register layout -- so the first stage needs no exchange, and the last
// stage's outputs (positions j + r N/R) land in that same layout, so the
// transform ends in registers with v[q] = X[t + T q].  Only the stages in
// between exchange through shared memory.  Exchange buffers are padded by one
// element per 16 (index i -> i + i/16), which keeps the scatter of the early
// stages free of bank conflicts.  FP32 uses sixteen points per thread, one
// exchange fewer, which measured faster; FP64, with twice the registers per
// point, eight.
constexpr int kP = 8;
constexpr int kLogP = 3;

__device__ __forceinline__ int pad16(int i) { return i + (i >> 4); }
// elements of a padded exchange buffer for an N-point transform
__host__ __device__ constexpr int padded_len(int N) { return N + N / 16; }

// Per-stage twiddle tables.  A stage of radix R = 2^LR after sub-transforms of
// length Ns = 2^a multiplies input r of butterfly k = j mod Ns by W_L^{k r},
// L = Ns R.  For each (a, LR) with a + LR <= 12 the table holds 2 Ns entries
// from [2 stage_table_offset(a, LR)] on.
// FP32: the pairs (exp(+2 pi i k / L), exp(+2 pi i 2k / L)), k = 0..Ns-1: one
// 16-byte load per butterfly, and the warp's loads are one contiguous run; the
// other factors are products of these two (stage_factors).
// FP64: exp(+2 pi i j / L), j = 0..2Ns-1, in which dit_twiddled finds all four
// of its factors, each rounded once.
__host__ __device__ constexpr int stage_table_offset(int a, int LR) {
  return 4 * ((1 << a) - 1) + (LR - 1) * (1 << a);
}
// complex entries of the whole table (pairs for a = 0..11, LR = 1..4)
__host__ __device__ constexpr int stage_table_len() { return 2 * 4 * ((1 << 12) - 1); }

// Compact per-length tables in shared memory.  A register transform with
// 2^LP points per thread multiplies by twiddles only in its stages a = LP,
// 2 LP, ... (a = log2 Ns < log2 N; the last one of radix 2^(log2 N - a) <=
// 2^LP).  The compact table holds the 2 Ns entries of exactly these stages, in
// stage order: stage a starts at pair (2^a - 2^LP) / (2^LP - 1), the sum of
// the earlier stages' 2^b.  Each transform kernel copies it from the global
// table once per CTA, so the butterflies read their pair from shared memory.
__host__ __device__ constexpr int compact_stage_offset(int a, int LP) {
  return a < LP ? 0 : ((1 << a) - (1 << LP)) / ((1 << LP) - 1);
}
// pairs of the compact table of an N = 2^log2N transform
__host__ __device__ constexpr int compact_stage_pairs(int log2N, int LP) {
  return compact_stage_offset(((log2N - 1) / LP) * LP + LP, LP);
}
template <class C>
__device__ __forceinline__ void stage_tables_to_smem(C* dst, const C* __restrict__ tw, int log2N, int LP, int tid,
                                                     int nthr) {
  for (int a = LP; a < log2N; a += LP) {
    const int LR = log2N - a < LP ? log2N - a : LP;
    const C* src = tw + 2 * stage_table_offset(a, LR);
    C* d = dst + 2 * compact_stage_offset(a, LP);
    for (int i = tid; i < (2 << a); i += nthr) d[i] = __ldg(src + i);
  }
}

__device__ __forceinline__ void load_pair(const float2* p, float2& w1, float2& w2) {
  const float4 x = *reinterpret_cast<const float4*>(p);
  w1 = float2{x.x, x.y};
  w2 = float2{x.z, x.w};
}

// ---- the arithmetic of the register FFT.  Products whose contraction would
// depend on their surroundings are spelled out, so that kernels that share a
// formula give the same bits.
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// -- FP32: radix-R DFTs of additions, the inputs multiplied by W^r first.
// radix 16 as 4 x 4: radix-4 DFTs over n1 (n = 4 n1 + n2), the factors
// w16^{n2 k1}, w16 = exp(sigma 2 pi i / 16), then radix-4 DFTs over n2;
// X[k1 + 4 k2] lands in v[k1 + 4 k2]
template <bool INV>
__device__ __forceinline__ float2 w16_times(float2 x, int e) {
  const float c1 = 0.92387953251128675612818318939678828682f, s1 = 0.38268343236508977172845998403039886676f;
  const float r2 = 0.70710678118654752440084436210484903928f;
  const float sg = INV ? 1.f : -1.f;                   // sign of the imaginary part of w16
  float cr, ci;                                        // w16^e = cr + i sg ci
  switch (e) {
    case 1: cr = c1; ci = s1; break;
    case 2: cr = r2; ci = r2; break;
    case 3: cr = s1; ci = c1; break;
    case 4: return mul_si<INV>(x);
    case 6: cr = -r2; ci = r2; break;
    case 9: cr = -c1; ci = -s1; break;
    default: return x;
  }
  const float wi = sg * ci;
  return float2{x.x * cr - x.y * wi, x.x * wi + x.y * cr};
}
template <bool INV>
__device__ __forceinline__ void dft16(float2* v) {
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) dft4<INV>(v[n2], v[4 + n2], v[8 + n2], v[12 + n2]);   // -> v[4 k1 + n2]
#pragma unroll
  for (int n2 = 1; n2 < 4; ++n2)
#pragma unroll
    for (int k1 = 1; k1 < 4; ++k1) v[4 * k1 + n2] = w16_times<INV>(v[4 * k1 + n2], n2 * k1);
  float2 o[16];
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    float2 a = v[4 * k1], b = v[4 * k1 + 1], c = v[4 * k1 + 2], d = v[4 * k1 + 3];
    dft4<INV>(a, b, c, d);
    o[k1] = a;
    o[k1 + 4] = b;
    o[k1 + 8] = c;
    o[k1 + 12] = d;
  }
#pragma unroll
  for (int q = 0; q < 16; ++q) v[q] = o[q];
}
// the R factors W^r, r = 1..R-1, from W and W^2 (at most three roundings deep)
template <int R>
__device__ __forceinline__ void stage_factors(float2 w1, float2 w2, float2 (&f)[R]) {
  f[1] = w1;
  if (R > 2) {
    f[2] = w2;
    f[3] = cmul(w1, w2);
  }
  if (R > 4) {
    f[4] = cmul(w2, w2);
    f[5] = cmul(f[4], w1);
    f[6] = cmul(f[4], w2);
    f[7] = cmul(f[4], f[3]);
  }
  if (R > 8) {                                          // w8 = w4 w4, w(8+r) = w8 wr
    f[8] = cmul(f[4], f[4]);
#pragma unroll
    for (int r = 1; r < 8; ++r) f[8 + r] = cmul(f[8], f[r]);
  }
}
template <bool INV, int LR>
__device__ __forceinline__ void dft_radix(float2* v) {
  if (LR == 4) dft16<INV>(v);
  else if (LR == 3) dft8<INV>(v);
  else if (LR == 2) dft4<INV>(v[0], v[1], v[2], v[3]);
  else dft2<INV>(v[0], v[1]);
}

// -- FP64: X[k] = sum_r x_r W^r w_R^{r k} by decimation in time: with E, O the
// transforms of the even and odd inputs (factor W^2),
//   X[k] = E[k] + (W w_R^k) O[k],  X[k + R/2] = E[k] - (W w_R^k) O[k],
// so a level of length len has the factors W^{R/len} w_len^k, and each
// two-point butterfly takes its factor in six fused multiply-adds: four for
// a + w b and one per component for a - w b = 2a - (a + w b).  9 FP64
// instructions per point of a radix-8 stage, where separate factors (R - 1
// products and their powers) and additions took 13; these passes are bound by
// the FP64 pipe (about 16 cycles of an SM per warp instruction).  a - w b carries
// its partner's rounding as well; the factors come rounded once from the table
// instead of as products, which more than makes up for it: rms error against
// 128 bits 1.53e-16 of the result at 64 points and 2.14e-16 at 1024, with
// separate factors 1.74 and 2.34 (with fused ones from products 1.80 and 2.42).
// An inertial step of 1024^2: 941 us with separate factors and one stencil per
// item of stage 2, 745 with factors from products, 732 now.  In FP32 the same butterflies gained 3% at
// 4096^2 and nothing below, and re-drew the rounding noise of phi; it keeps the
// form above.
// (a, b) <- (a + w b, a - w b)
template <class C> __device__ __forceinline__ void bfly(C& a, C& b, C w) {
  using T = decltype(a.x);
  const C p = C{fma_rn(w.x, b.x, fma_rn(-w.y, b.y, a.x)), fma_rn(w.x, b.y, fma_rn(w.y, b.x, a.y))};
  b = C{fma_rn(T(2), a.x, -p.x), fma_rn(T(2), a.y, -p.y)};
  a = p;
}
// the same with a - w b formed by itself: for the short last stages of radix 2
// and 4, whose few factors leave the table nothing to make up for
template <class C> __device__ __forceinline__ void bfly_apart(C& a, C& b, C w) {
  const C p = C{fma_rn(w.x, b.x, fma_rn(-w.y, b.y, a.x)), fma_rn(w.x, b.y, fma_rn(w.y, b.x, a.y))};
  b = C{fma_rn(-w.x, b.x, fma_rn(w.y, b.y, a.x)), fma_rn(-w.x, b.y, fma_rn(-w.y, b.x, a.y))};
  a = p;
}
// w = 1, w = sigma i, and w = (1 + sigma i) / sqrt(2) turned by Q quarters
template <class C> __device__ __forceinline__ void bfly_one(C& a, C& b) { dft2<false>(a, b); }
template <bool INV, int Q, class C> __device__ __forceinline__ void bfly_eighth(C& a, C& b) {
  using T = decltype(a.x);
  const T c = T(0.70710678118654752440084436210484904);
  const T sg = INV ? T(1) : T(-1);
  // (1 + sg i) b, for Q = 1 sg i (1 + sg i) b = (-1 + sg i) b
  const C d = Q == 0 ? C{b.x - sg * b.y, b.y + sg * b.x} : C{-b.x - sg * b.y, sg * b.x - b.y};
  b = C{fma_rn(-c, d.x, a.x), fma_rn(-c, d.y, a.y)};
  a = C{fma_rn(c, d.x, a.x), fma_rn(c, d.y, a.y)};
}
template <int LR> __host__ __device__ constexpr int bit_reversed(int r) {
  int v = 0;
  for (int i = 0; i < LR; ++i) v |= ((r >> i) & 1) << (LR - 1 - i);
  return v;
}
// y holds the R inputs in bit-reversed places, factors all one; X in natural order
template <bool INV, int LR, class C>
__device__ __forceinline__ void dit_plain(C* y) {
  constexpr int R = 1 << LR;
#pragma unroll
  for (int i = 0; i < R; i += 2) bfly_one(y[i], y[i + 1]);
  if (LR >= 2)
#pragma unroll
    for (int i = 0; i < R; i += 4) {
      bfly_one(y[i], y[i + 2]);
      y[i + 3] = mul_si<INV>(y[i + 3]);
      bfly_one(y[i + 1], y[i + 3]);
    }
  if (LR >= 3)
#pragma unroll
    for (int i = 0; i < R; i += 8) {
      bfly_one(y[i], y[i + 4]);
      bfly_eighth<INV, 0>(y[i + 1], y[i + 5]);
      y[i + 6] = mul_si<INV>(y[i + 6]);
      bfly_one(y[i + 2], y[i + 6]);
      bfly_eighth<INV, 1>(y[i + 3], y[i + 7]);
    }
}
// the same with the factors W^r, W = W_L^k: w1 = W, w2 = W^2, w4 = W^4 and w1
// turned by an eighth are entries k, 2k, 4k (a quarter turn on from 2 Ns) and
// k + Ns of the stage's table
template <bool INV, int LR, class C>
__device__ __forceinline__ void dit_twiddled(C* y, const C* tab, int Ns, int k) {
  constexpr int R = 1 << LR;
  auto factor = [&](int j) { return INV ? tab[j] : cconj(tab[j]); };
  if constexpr (LR == 3) {
    C w4 = factor((4 * k) & (2 * Ns - 1));
    if (4 * k >= 2 * Ns) w4 = mul_si<INV>(w4);
#pragma unroll
    for (int i = 0; i < R; i += 2) bfly(y[i], y[i + 1], w4);
    const C w2 = factor(2 * k);
#pragma unroll
    for (int i = 0; i < R; i += 4) {
      bfly(y[i], y[i + 2], w2);
      bfly(y[i + 1], y[i + 3], mul_si<INV>(w2));
    }
    const C w1 = factor(k);
    bfly(y[0], y[4], w1);
    bfly(y[2], y[6], mul_si<INV>(w1));
    const C we = factor(k + Ns);
    bfly(y[1], y[5], we);
    bfly(y[3], y[7], mul_si<INV>(we));
  } else {
    if constexpr (LR == 2) {
      const C w2 = factor(2 * k);
      bfly_apart(y[0], y[1], w2);
      bfly_apart(y[2], y[3], w2);
    }
    const C w1 = factor(k);
    bfly_apart(y[0], y[R / 2], w1);
    if constexpr (LR == 2) bfly_apart(y[1], y[3], mul_si<INV>(w1));
  }
}

// One stage on the register layout.  LAST: keep the outputs in registers;
// otherwise scatter them to buf (padded), barrier, gather the next stage's
// inputs, barrier (so the buffer can be written again).  The barrier is the
// CTA's (CtaSync) or, for a transform owned by a whole-warp subset of the CTA,
// a named barrier of that subset (NamedSync), so that several transforms in
// one CTA need not wait for each other.
template <int P> constexpr int log2_points() { return P == 16 ? 4 : 3; }

struct CtaSync {
  __device__ __forceinline__ void operator()() const { __syncthreads(); }
};
struct NamedSync {
  int id, nthreads;                                    // barrier 1..15, a multiple of 32 threads
  __device__ __forceinline__ void operator()() const {
    asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(nthreads) : "memory");
  }
};
// a group's barrier where a kernel runs as thread groups, else the CTA's
template <bool GROUPED> struct GroupSync : NamedSync {};
template <> struct GroupSync<false> : CtaSync {
  __device__ __forceinline__ GroupSync(NamedSync) {}
};

template <bool INV, int LR, bool LAST, int P, class C, class Sync = CtaSync>
__device__ __forceinline__ void fft_reg_stage(C (&v)[P], int log2N, int log2Ns, int t, C* buf, const C* twt,
                                              const Sync& sync = Sync{}) {
  constexpr int R = 1 << LR;
  constexpr int B = P >> LR;
  const int T = 1 << (log2N - log2_points<P>());
  const int Ns = 1 << log2Ns;
  C w[R];
#pragma unroll
  for (int b = 0; b < B; ++b) {
    const int j = t + b * T;
    const int k = j & (Ns - 1);
#pragma unroll
    for (int r = 0; r < R; ++r) w[sizeof(w[0].x) == 4 ? r : bit_reversed<LR>(r)] = v[b + r * B];
    const C* tab = twt + 2 * compact_stage_offset(log2Ns, log2_points<P>());
    if constexpr (sizeof(w[0].x) == 4) {
      if (log2Ns > 0) {
        C w1, w2, f[R];
        load_pair(tab + 2 * k, w1, w2);
        stage_factors<R>(w1, w2, f);
#pragma unroll
        for (int r = 1; r < R; ++r) w[r] = cmul(w[r], INV ? f[r] : cconj(f[r]));
      }
      dft_radix<INV, LR>(w);
    } else {
      if (log2Ns > 0) dit_twiddled<INV, LR>(w, tab, Ns, k);
      else dit_plain<INV, LR>(w);
    }
    if (LAST) {
#pragma unroll
      for (int r = 0; r < R; ++r) v[b + r * B] = w[r];
    } else {
      const int base = ((j - k) << LR) + k;
#pragma unroll
      for (int r = 0; r < R; ++r) buf[pad16(base + r * Ns)] = w[r];
    }
  }
  if (!LAST) {
    sync();
#pragma unroll
    for (int q = 0; q < P; ++q) v[q] = buf[pad16(t + q * T)];
    sync();
  }
}

// Transform of N = 2^log2N points (16 <= N <= NMAX) held as v[q] = x[t + T q].
// buf: this instance's padded exchange buffer (padded_len(N) elements); tw:
// the compact stage table of this length and P (compact_stage_offset) in
// shared memory.  All threads of the CTA must call it (barriers) with the same
// log2N.
template <bool INV, int P, class C, class Sync = CtaSync>
__device__ __forceinline__ void fft_reg(C (&v)[P], int log2N, int t, C* buf, const C* tw, const Sync& sync = Sync{}) {
  constexpr int LP = log2_points<P>();
  int log2Ns = 0;
  while (log2N - log2Ns > LP) {
    fft_reg_stage<INV, LP, false>(v, log2N, log2Ns, t, buf, tw, sync);
    log2Ns += LP;
  }
  switch (log2N - log2Ns) {
    case 4: if constexpr (P == 16) fft_reg_stage<INV, 4, true>(v, log2N, log2Ns, t, buf, tw, sync); break;
    case 3: fft_reg_stage<INV, 3, true>(v, log2N, log2Ns, t, buf, tw, sync); break;
    case 2: fft_reg_stage<INV, 2, true>(v, log2N, log2Ns, t, buf, tw, sync); break;
    default: fft_reg_stage<INV, 1, true>(v, log2N, log2Ns, t, buf, tw, sync); break;
  }
}

// v[q] = X[t + T q] -> buf (padded, natural order), followed by a barrier.
template <int P, class C, class Sync = CtaSync>
__device__ __forceinline__ void reg_to_smem(const C (&v)[P], int log2N, int t, C* buf, const Sync& sync = Sync{}) {
  const int T = 1 << (log2N - log2_points<P>());
#pragma unroll
  for (int q = 0; q < P; ++q) buf[pad16(t + q * T)] = v[q];
  sync();
}

}  // namespace shf
