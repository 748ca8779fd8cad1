// FFT plans of the multislice passes: two super-stages and one shared-memory exchange for
// every grid side.
//
// A super-stage is one radix (8, 16, 24, 32) or two consecutive small radices A, B run on
// A B values of a thread, with the twiddle factors between them read from a table: the
// arithmetic of a three- or four-stage plan with the data movement of a two-stage one.
//
//   N      forward        reverse (inverse transforms)    sequences per warp (row pass)
//   64     8 | 8          8 | 8                           4
//   128    8 | 4.4        4.4 | 8                         4
//   256    16 | 16        16 | 16                         2
//   384    3.8 | 4.4      4.4 | 8.3                       2
//   512    16 | 32        32 | 16                         2
//   768    24 | 32        32 | 24                         1
//   1024   32 | 32        32 | 32                         1
//
// The last super-stage of a transform leaves x[b + q N/R], the layout the first
// super-stage of the reversed plan reads, so inverse and forward transforms chain
// without a second exchange.  Every sum and product is written with its rounding
// (__fadd_rn, __fmaf_rn): results do not depend on which products the compiler fuses.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace eels {
namespace pf {

// ---------------------------------------------------------------------------
// complex arithmetic with fixed rounding

__device__ __forceinline__ float2 add(float2 a, float2 b) {
  return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
}
__device__ __forceinline__ float2 sub(float2 a, float2 b) {
  return make_float2(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y));
}
// a w, with the products of a.y rounded first
__device__ __forceinline__ float2 mul(float2 a, float2 w) {
  return make_float2(__fmaf_rn(a.x, w.x, -__fmul_rn(a.y, w.y)),
                     __fmaf_rn(a.x, w.y, __fmul_rn(a.y, w.x)));
}
// a conj(w), with the products a.y w.y and a.x w.y rounded first
__device__ __forceinline__ float2 mulc(float2 a, float2 w) {
  return make_float2(__fmaf_rn(a.x, w.x, __fmul_rn(a.y, w.y)),
                     __fmaf_rn(a.y, w.x, -__fmul_rn(a.x, w.y)));
}
template <bool CONJ>
__device__ __forceinline__ float2 mul_c(float2 a, float2 w) {
  return CONJ ? mulc(a, w) : mul(a, w);
}
// e + h d
__device__ __forceinline__ float2 axpy(float h, float2 d, float2 e) {
  return make_float2(__fmaf_rn(h, d.x, e.x), __fmaf_rn(h, d.y, e.y));
}
// a + i b (S = +1) or a - i b (S = -1)
template <int S>
__device__ __forceinline__ float2 add_i(float2 a, float2 b) {
  return S > 0 ? make_float2(__fsub_rn(a.x, b.y), __fadd_rn(a.y, b.x))
               : make_float2(__fadd_rn(a.x, b.y), __fsub_rn(a.y, b.x));
}

// ---------------------------------------------------------------------------
// In-register DFTs.  INV: the + sign in the exponent.  EDGE: the input is band-limited
// (the first stage of an inverse transform), only its first and last quarter are nonzero.

template <bool INV, bool EDGE>
__device__ __forceinline__ void dft4(float2& u0, float2& u1, float2& u2, float2& u3) {
  constexpr int S = INV ? 1 : -1;
  if constexpr (EDGE) {   // u1 = u2 = 0
    const float2 a = u0, d = u3;
    u0 = add(a, d);
    u2 = sub(a, d);
    u1 = add_i<-S>(a, d);   // the odd difference is -u3
    u3 = add_i<S>(a, d);
  } else {
    const float2 t0 = add(u0, u2), t1 = sub(u0, u2);
    const float2 t2 = add(u1, u3), t3 = sub(u1, u3);
    u0 = add(t0, t2);
    u2 = sub(t0, t2);
    u1 = add_i<S>(t1, t3);
    u3 = add_i<-S>(t1, t3);
  }
}

template <bool INV, bool EDGE>
__device__ __forceinline__ void dft8(float2* u) {
  constexpr int S = INV ? 1 : -1;
  constexpr float H = 0.70710678118654752440f;   // 1/sqrt(2)
  float2 e0 = u[0], e1 = u[2], e2 = u[4], e3 = u[6];
  float2 o0 = u[1], o1 = u[3], o2 = u[5], o3 = u[7];
  dft4<INV, EDGE>(e0, e1, e2, e3);
  dft4<INV, EDGE>(o0, o1, o2, o3);
  u[0] = add(e0, o0);
  u[4] = sub(e0, o0);
  // o1 exp(S i pi / 4) = H (x - S y, y + S x), added with one fused rounding
  const float2 d1 = add_i<S>(o1, o1);
  u[1] = axpy(H, d1, e1);
  u[5] = axpy(-H, d1, e1);
  u[2] = add_i<S>(e2, o2);
  u[6] = add_i<-S>(e2, o2);
  // o3 exp(3 S i pi / 4) = -H (x + S y, y - S x)
  const float2 d3 = add_i<-S>(o3, o3);
  u[3] = axpy(-H, d3, e3);
  u[7] = axpy(H, d3, e3);
}

template <bool INV>
__device__ __forceinline__ void dft3(float2* u) {
  constexpr float S3 = (INV ? 1.0f : -1.0f) * 0.86602540378443864676f;   // sign * sqrt(3)/2
  const float2 t1 = add(u[1], u[2]), t2 = sub(u[1], u[2]);
  const float2 m = axpy(-0.5f, t1, u[0]);
  u[0] = add(u[0], t1);
  u[1] = make_float2(__fmaf_rn(-S3, t2.y, m.x), __fmaf_rn(S3, t2.x, m.y));
  u[2] = make_float2(__fmaf_rn(S3, t2.y, m.x), __fmaf_rn(-S3, t2.x, m.y));
}

// a exp(+-2 pi i m / R) (+ for INV); quarter turns are exact
template <int R, bool INV>
__device__ __forceinline__ float2 rotate(float2 a, int m) {
  if ((4 * m) % R == 0) {
    const int quarter = ((INV ? 4 * m : -4 * m) / R) & 3;
    return quarter == 0 ? a
         : quarter == 2 ? make_float2(-a.x, -a.y)
         : quarter == 1 ? make_float2(-a.y, a.x)
                        : make_float2(a.y, -a.x);
  }
  return mul(a, croot<R>(m, INV ? 1.f : -1.f));
}

template <int R, bool INV, bool EDGE>
__device__ __forceinline__ void dft(float2* x);

// R = R1 R2: n = R2 n1 + n2, k = k1 + R1 k2
template <int R1, int R2, bool INV, bool EDGE>
__device__ __forceinline__ void dft_composite(float2* x) {
  constexpr int R = R1 * R2;
  float2 y[R];
#pragma unroll
  for (int n2 = 0; n2 < R2; ++n2) {
    float2 t[R1];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) t[n1] = x[R2 * n1 + n2];
    dft<R1, INV, EDGE>(t);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) y[n2 * R1 + k1] = rotate<R, INV>(t[k1], (n2 * k1) % R);
  }
#pragma unroll
  for (int k1 = 0; k1 < R1; ++k1) {
    float2 t[R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) t[n2] = y[n2 * R1 + k1];
    dft<R2, INV, false>(t);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) x[k1 + R1 * k2] = t[k2];
  }
}

template <int R, bool INV, bool EDGE>
__device__ __forceinline__ void dft(float2* x) {
  if constexpr (R == 3) dft3<INV>(x);
  else if constexpr (R == 4) dft4<INV, EDGE>(x[0], x[1], x[2], x[3]);
  else if constexpr (R == 8) dft8<INV, EDGE>(x);
  else if constexpr (R == 16) dft_composite<4, 4, INV, EDGE>(x);
  else if constexpr (R == 24) dft_composite<8, 3, INV, EDGE>(x);
  else dft_composite<8, 4, INV, EDGE>(x);
}

// ---------------------------------------------------------------------------
// plans

// radices of the forward plan: super-stage s is a(s) b(s), b = 1 for a single radix
__host__ __device__ constexpr int fwd_a(int n, int s) {
  return n == 64 ? 8 : n == 128 ? (s == 0 ? 8 : 4) : n == 256 ? 16 : n == 384 ? (s == 0 ? 3 : 4)
       : n == 512 ? (s == 0 ? 16 : 32) : n == 768 ? (s == 0 ? 24 : 32) : 32;
}
__host__ __device__ constexpr int fwd_b(int n, int s) {
  return n == 128 ? (s == 0 ? 1 : 4) : n == 384 ? (s == 0 ? 8 : 4) : 1;
}
__host__ __device__ constexpr int seqs_per_warp(int n) {
  return n <= 128 ? 4 : n <= 512 ? 2 : 1;
}
__host__ __device__ constexpr int plan_a(int n, bool rev, int s) {
  return !rev ? fwd_a(n, s) : fwd_b(n, 1 - s) > 1 ? fwd_b(n, 1 - s) : fwd_a(n, 1 - s);
}
__host__ __device__ constexpr int plan_b(int n, bool rev, int s) {
  return !rev ? fwd_b(n, s) : fwd_b(n, 1 - s) > 1 ? fwd_a(n, 1 - s) : 1;
}

template <int N, bool REV>
struct Plan2 {
  static constexpr int A0 = plan_a(N, REV, 0), B0 = plan_b(N, REV, 0), R0 = A0 * B0;
  static constexpr int A1 = plan_a(N, REV, 1), B1 = plan_b(N, REV, 1), R1 = A1 * B1;
  static constexpr int SEQ = seqs_per_warp(N);
  static constexpr int NB0 = N / R0, NB1 = N / R1;   // butterflies per sequence; NB1 = R0
  static constexpr int PER0 = (SEQ * NB0 + 31) / 32, PER1 = (SEQ * NB1 + 31) / 32;
  static constexpr int E = PER0 * R0 > PER1 * R1 ? PER0 * R0 : PER1 * R1;
  static constexpr int PADDED = N + N / R0;          // exchange buffer, one spare per R0 values
  static_assert(R0 * R1 == N, "plan");
};
// Column pass: threads per column, each holding E values of it.
__host__ __device__ constexpr int col_threads(int n) {
  return n == 64 ? 8 : n <= 256 ? 16 : n == 384 ? 24 : n == 512 ? 16 : 32;
}
template <int N>
struct Seqs {
  static constexpr int SEQ = seqs_per_warp(N);
  static constexpr int E = Plan2<N, false>::E > Plan2<N, true>::E ? Plan2<N, false>::E
                                                                  : Plan2<N, true>::E;
  static constexpr int PADDED = Plan2<N, false>::PADDED > Plan2<N, true>::PADDED
                                    ? Plan2<N, false>::PADDED
                                    : Plan2<N, true>::PADDED;
};

// Twiddle tables, appended to the table of N roots: per pass (row, column) and direction
// (forward plan, reversed plan) one set of
//   [0, 32)         factors between the two radices of the first super-stage, [m][q1]
//   [32, 32 + N)    factors before radix A1 of the second super-stage, [q][k], k < R0
//   [32 + N, ...)   factors between A1 and B1 of the second super-stage, [m][k2], k2 < R0 A1
// so that a warp's read of one factor index is a contiguous run.
__host__ __device__ constexpr int set_len(int n) { return 32 + 2 * n; }
__host__ __device__ constexpr int set_offset(int n, bool col, bool rev) {
  return twiddle_table_len(n) + ((col ? 2 : 0) + (rev ? 1 : 0)) * set_len(n);
}
__host__ __device__ constexpr int table_len(int n) { return twiddle_table_len(n) + 4 * set_len(n); }

// The part of a set that a plan reads, as it lies in shared memory: all of it where a
// super-stage has two radices, otherwise only the factors before A1.
template <int N>
struct SetPart {
  static constexpr bool ALL = fwd_b(N, 0) > 1 || fwd_b(N, 1) > 1;
  static constexpr int FROM = ALL ? 0 : 32, LEN = ALL ? set_len(N) : N;
  static constexpr int AT0 = 0, AT1 = ALL ? 32 : 0, AT2 = ALL ? 32 + N : 0;
  static constexpr bool SAME = fwd_a(N, 0) == fwd_a(N, 1) && !ALL;   // one set for both plans
  static constexpr int BOTH = SAME ? LEN : 2 * LEN;
};
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(smem)),
               "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// count values (a multiple of 2) from global to shared memory, both 16-byte aligned; the
// caller waits (cp_async_wait) and synchronises
__device__ __forceinline__ void copy_async(float2* dst, const float2* src, int count) {
  for (int i = 2 * threadIdx.x; i < count; i += 2 * blockDim.x) cp_async16(dst + i, src + i);
}
// Both plans' sets of a pass into shared memory (BOTH values), asynchronously.
template <int N>
__device__ __forceinline__ void load_sets(float2* dst, const float2* tw, bool col) {
  copy_async(dst, tw + set_offset(N, col, false) + SetPart<N>::FROM, SetPart<N>::LEN);
  if constexpr (!SetPart<N>::SAME)
    copy_async(dst + SetPart<N>::LEN, tw + set_offset(N, col, true) + SetPart<N>::FROM,
               SetPart<N>::LEN);
}
template <int N>
__device__ __forceinline__ const float2* rev_set(const float2* sets) {
  return sets + (SetPart<N>::SAME ? 0 : SetPart<N>::LEN);
}

// Factors rounded once from FP64, applied conjugated in inverse transforms; otherwise they
// are the products the multi-stage plans (128, 384) and the column passes of the two largest
// grids are defined with, conjugated before they are applied.
__host__ __device__ constexpr bool exact_factors(int n, bool col) {
  return n == 64 || n == 256 || n == 512 || ((n == 768 || n == 1024) && !col);
}

template <bool INV, bool EXACT>
__device__ __forceinline__ float2 twiddle(float2 a, float2 w) {
  if constexpr (EXACT) return INV ? mulc(a, w) : mul(a, w);
  else return mul(a, INV ? make_float2(w.x, -w.y) : w);
}

// One super-stage on v[0 .. A B) of butterfly b: before radix A the factors ta[q * P + k]
// (P > 1 only), before radix B the factors tb[m * P A + k + q P]; output o = q1 + A q2
// belongs at (b - k) A B + k + o P.
template <int A, int B, int P, bool INV, bool EDGE, bool EXACT>
__device__ __forceinline__ void super_stage(float2* v, int k, const float2* ta, const float2* tb) {
  if constexpr (B == 1) {
    if constexpr (P > 1) {
#pragma unroll
      for (int q = 1; q < A; ++q) v[q] = twiddle<INV, EXACT>(v[q], ta[q * P + k]);
    }
    dft<A, INV, EDGE>(v);
  } else {
    float2 y[A * B];
    float2 wa[A];
    if constexpr (P > 1) {
#pragma unroll
      for (int q = 1; q < A; ++q) wa[q] = ta[q * P + k];
    }
#pragma unroll
    for (int m = 0; m < B; ++m) {
      float2 t[A];
#pragma unroll
      for (int q = 0; q < A; ++q) {
        t[q] = v[m + q * B];
        if constexpr (P > 1)
          if (q > 0) t[q] = twiddle<INV, EXACT>(t[q], wa[q]);
      }
      dft<A, INV, EDGE>(t);
#pragma unroll
      for (int q = 0; q < A; ++q) y[m * A + q] = t[q];
    }
#pragma unroll
    for (int q = 0; q < A; ++q) {
      float2 t[B];
      t[0] = y[q];
#pragma unroll
      for (int m = 1; m < B; ++m) {
        // the first super-stage's factor for q = 0 is one
        t[m] = (P == 1 && q == 0) ? y[m * A + q]
                                  : twiddle<INV, EXACT>(y[m * A + q], tb[m * P * A + k + q * P]);
      }
      dft<B, INV, false>(t);
#pragma unroll
      for (int q2 = 0; q2 < B; ++q2) v[q + A * q2] = t[q2];
    }
  }
}

// Transform of the SEQ sequences a warp holds.  On entry slot u = lane + 32 t of v holds
// x_{u / NB0}[u % NB0 + q N/R0] at v[t R0 + q], on exit X in the same form for R1 and NB1.
// Sequence r exchanges through sbuf + r * ld (PADDED values; a first super-stage writes
// R0 b + o into rows of R0 + 1 values, so that neighbouring lanes hit distinct banks).
// `set` is the part of the factor set that the plan reads (SetPart), in shared memory
// (load_sets) or in the table itself.
template <int N, bool INV, bool REV, bool EDGE>
__device__ __forceinline__ void warp_fft(float2* v, float2* sbuf, int ld, const float2* set,
                                         int lane) {
  using PL = Plan2<N, REV>;
  constexpr int R0 = PL::R0, R1 = PL::R1, NB0 = PL::NB0, NB1 = PL::NB1, SEQ = PL::SEQ;
  constexpr bool EXACT = exact_factors(N, false);
#pragma unroll
  for (int t = 0; t < PL::PER0; ++t) {
    const int u = lane + 32 * t;
    if ((SEQ * NB0) % 32 == 0 || u < SEQ * NB0) {
      super_stage<PL::A0, PL::B0, 1, INV, EDGE, EXACT>(v + t * R0, 0, nullptr,
                                                       set + SetPart<N>::AT0);
      float2* row = sbuf + (u / NB0) * ld + (u % NB0) * (R0 + 1);
#pragma unroll
      for (int o = 0; o < R0; ++o) row[o] = v[t * R0 + o];
    }
  }
  __syncwarp();
#pragma unroll
  for (int t = 0; t < PL::PER1; ++t) {
    const int u = lane + 32 * t;
    if ((SEQ * NB1) % 32 == 0 || u < SEQ * NB1) {
      const float2* row = sbuf + (u / NB1) * ld + u % NB1;
#pragma unroll
      for (int q = 0; q < R1; ++q) v[t * R1 + q] = row[q * (NB1 + 1)];
    }
  }
  __syncwarp();
#pragma unroll
  for (int t = 0; t < PL::PER1; ++t) {
    const int u = lane + 32 * t;
    if ((SEQ * NB1) % 32 == 0 || u < SEQ * NB1)
      super_stage<PL::A1, PL::B1, R0, INV, false, EXACT>(v + t * R1, u % NB1,
                                                         set + SetPart<N>::AT1,
                                                         set + SetPart<N>::AT2);
  }
}

}  // namespace pf
}  // namespace eels
