// Band-limited plane-wave multislice on the GPU (Eqs. 3, 4, MSop, MSTop).
//
// A slice step psi -> F^-1[P F[t psi]] is split into two passes over a batch of
// waves.  Between the passes every wave is kept in "row-spectrum" form: an
// array [y][kx'] of N rows by N/2 columns holding the x-DFT of the wave restricted
// to the band box |kx| < N/4 (column kx' < N/4 is frequency kx', otherwise
// kx' - N/2).  Because the propagator limits every wave to p^2 + q^2 < (N/4)^2,
// nothing outside the box is ever needed.
//
//   row pass    (one warp per 1, 2 or 4 rows y): zero-pad kx to N, inverse FFT_x, multiply
//                by t (or conj t), optionally store the even samples (the N/2
//                representation used by the S-matrices), forward FFT_x, keep the box.
//   column pass (one CTA per few columns kx'): FFT_y, keep the box, multiply by the
//                propagator table (or its conjugate), zero-pad, inverse FFT_y.
//
// Scale convention: W holds the true row spectrum; the row pass produces N times
// the true real-space wave and N times the true row spectrum, and the propagator
// table carries the 1/N^2 that restores W after the column pass.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "internal.h"
#include "plan_fft.cuh"

namespace eels {

namespace {

constexpr int kRowWarps = 4;   // warps per CTA of the row pass

// CTAs per SM the row pass is compiled for: 64 registers of data per thread leave room for
// 16 warps; more warps with fewer registers were slower at every grid (1024: 2.72 us per
// wave with 16 warps, 2.87 with 20, 3.08 with 24).
template <int N>
__host__ __device__ constexpr int row_ctas() {
  return pf::Seqs<N>::E > 16 ? 4 : 5;
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

template <int N>
struct RowSmem {
  static constexpr int BUF = pf::Seqs<N>::SEQ * pf::Seqs<N>::PADDED;   // values per warp
  static constexpr size_t BYTES = (size_t)kRowWarps * BUF * sizeof(float2) +
                                  (size_t)pf::Seqs<N>::SEQ * N * sizeof(float2) +
                                  (size_t)pf::SetPart<N>::BOTH * sizeof(float2);
};

// Inputs of the inverse x-FFT of rows y0 .. y0 + SEQ - 1 of a wave: the band box, zero-padded
// to N.  START: the wave is a plane wave, formed here instead of being read (the first slice
// of a sweep; writing plane waves out and reading them back costs a build 4 % of its time).
template <int N, bool START>
__device__ __forceinline__ void row_load(float2* v, const float2* __restrict__ W,
                                         const PlaneWaves& start, const float2* __restrict__ tw,
                                         int64_t wave, int y0, int lane) {
  constexpr int NH = N / 2, NQ = N / 4, SEQ = pf::Seqs<N>::SEQ;
  using PI = pf::Plan2<N, true>;
  int col = -1, ky = 0;   // START: the wave's box column (-1: none) and y frequency
  float2 a = make_float2(0.f, 0.f);
  if constexpr (START) {
    const int p = start.px[wave];
    if (STEM_REQUIRE(p >= -NH && p < NH)) col = p >= 0 ? p : p + NH;
    ky = start.py[wave];
    a = start.amp[wave];
  }
#pragma unroll
  for (int t = 0; t < PI::PER0; ++t) {
    const int u = lane + 32 * t;
    if ((SEQ * PI::NB0) % 32 == 0 || u < SEQ * PI::NB0) {
      const int y = y0 + u / PI::NB0, b = u % PI::NB0;
      const float2* src = W + (wave * N + y) * NH + b;
      float2 on = make_float2(0.f, 0.f);
      if constexpr (START) {
        const int m = ky * y % N;
        on = cmul(a, cconj(__ldg(tw + (m < 0 ? m + N : m))));   // exp(+2 pi i ky y / N)
      }
#pragma unroll
      for (int q = 0; q < PI::R0; ++q) {
        const int at = q * PI::NB0;
        float2 x = make_float2(0.f, 0.f);
        if (at < NQ || at >= N - NQ) {
          const int i = at < NQ ? at : at - NH;
          if constexpr (START) x = b + i == col ? on : x;
          else x = src[i];
        }
        v[t * PI::R0 + q] = x;
      }
    }
  }
}

// The row pass of one wave's rows y0 .. y0 + SEQ - 1, loaded in v (row_load), by one warp:
// trows holds their SEQ rows of t, fset and rset the factor sets of the two plans.
template <int N, bool CONJ>
__device__ __forceinline__ void row_wave(float2* v, float2* sbuf, const float2* trows,
                                         const float2* fset, const float2* rset, int64_t wave,
                                         int y0, int lane, float2* __restrict__ Phi,
                                         int store_mode, float2* __restrict__ S, int s_waves,
                                         int64_t s_stride, int fft_out) {
  constexpr int NH = N / 2, NQ = N / 4;
  constexpr int SEQ = pf::Seqs<N>::SEQ, LD = pf::Seqs<N>::PADDED;
  using PF = pf::Plan2<N, false>;   // forward transform
  pf::warp_fft<N, true, true, true>(v, sbuf, LD, rset, lane);

  // real space: slot u holds N psi(x = u % NB0 + q N/R0, y0 + u / NB0)
#pragma unroll
  for (int t = 0; t < PF::PER0; ++t) {
    const int u = lane + 32 * t;
    if ((SEQ * PF::NB0) % 32 == 0 || u < SEQ * PF::NB0) {
      const int y = y0 + u / PF::NB0, b = u % PF::NB0;
      const float2* trow = trows + (u / PF::NB0) * N + b;
      // even x only: N/R0 is even, so x has the parity of b
      const bool store = store_mode != 0 && ((y | b) & 1) == 0 && wave < s_waves;
      float2* srow = S + wave * s_stride + (int64_t)(y >> 1) * NH + (b >> 1);
#pragma unroll
      for (int q = 0; q < PF::R0; ++q) {
        const float2 before = v[t * PF::R0 + q];
        const float2 after = pf::mul_c<CONJ>(before, trow[q * PF::NB0]);
        if (store) srow[q * (PF::NB0 / 2)] = store_mode == 1 ? after : before;
        v[t * PF::R0 + q] = after;
      }
    }
  }
  if (!fft_out) return;
  pf::warp_fft<N, false, false, false>(v, sbuf, LD, fset, lane);
#pragma unroll
  for (int t = 0; t < PF::PER1; ++t) {
    const int u = lane + 32 * t;
    if ((SEQ * PF::NB1) % 32 == 0 || u < SEQ * PF::NB1) {
      float2* dst = Phi + (wave * N + y0) * NH + (u / PF::NB1) * NH + u % PF::NB1;
#pragma unroll
      for (int q = 0; q < PF::R1; ++q) {
        const int at = q * PF::NB1;
        if (at < NQ) dst[at] = v[t * PF::R1 + q];
        else if (at >= N - NQ) dst[at - NH] = v[t * PF::R1 + q];
      }
    }
  }
}

// Row pass of many waves.  A CTA takes SEQ rows y0 .. y0 + SEQ - 1 of `chunk` waves, one warp
// a wave at a time: the rows of t and the factor sets lie in shared memory for all of them
// (read per row from L2 and L1 they cost as many wavefronts and far more latency), and the
// rows of a warp's next wave are fetched to L2 while it transforms this one's.  No unit is
// saturated: of the issue slots 68 % are used (ncu, 305 waves at 1024; L1 and shared memory
// 68 %, FMA pipe 55 %, DRAM 45 %), one warp in six waits for instructions, and 16 warps are
// what the registers allow.  us per wave, rows read per wave / so: adjoint pass with the
// S_out store, 1024: 3.22 / 2.95, 768: 1.83 / 1.55, 512: 0.58 / 0.57, 384: 1.00 / 0.48 (four
// stages and three exchanges before); pass of a build, 256: 0.150 / 0.146, 128: 0.085 / 0.043,
// 64: 0.036 / 0.018.
template <int N, bool CONJ, bool START>
__global__ void __launch_bounds__(kRowWarps * 32, row_ctas<N>())
k_row_pass(const float2* __restrict__ W, const PlaneWaves start, float2* __restrict__ Phi,
           const float2* __restrict__ t_slice, int store_mode, float2* __restrict__ S,
           int s_waves, int64_t s_stride, int fft_out, const float2* __restrict__ tw,
           int n_waves, int chunk) {
  constexpr int NH = N / 2, SEQ = pf::Seqs<N>::SEQ;
  extern __shared__ float2 smem[];
  float2* trows = smem + kRowWarps * RowSmem<N>::BUF;   // [SEQ][N]
  float2* sets = trows + SEQ * N;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* sbuf = smem + warp * RowSmem<N>::BUF;
  const int y0 = blockIdx.x * SEQ;
  const int w0 = blockIdx.y * chunk + warp, w_end = min(n_waves, (int)(blockIdx.y + 1) * chunk);
  pf::load_sets<N>(sets, tw, false);
  pf::copy_async(trows, t_slice + (int64_t)y0 * N, SEQ * N);

  float2 v[pf::Seqs<N>::E];
  if (w0 < w_end) row_load<N, START>(v, W, start, tw, w0, y0, lane);
  pf::cp_async_wait();
  __syncthreads();

  for (int64_t wave = w0; wave < w_end; wave += kRowWarps) {
    if (wave != w0) row_load<N, START>(v, W, start, tw, wave, y0, lane);
    if (!START && wave + kRowWarps < w_end) {   // the next rows: SEQ * NH values, contiguous
      const float2* next = W + ((wave + kRowWarps) * N + y0) * NH;
#pragma unroll
      for (int i = lane * 16; i < SEQ * NH; i += 512) prefetch_l2(next + i);
    }
    row_wave<N, CONJ>(v, sbuf, trows, sets, pf::rev_set<N>(sets), wave, y0, lane, Phi, store_mode,
                      S, s_waves, s_stride, fft_out);
  }
}

// Row pass of few waves: a warp takes SEQ rows of one wave and the CTA's warps neighbouring
// rows; t and the factor sets are read where they lie (L2, L1) and no warp waits for another.
// k_row_pass fills shared memory before its first butterfly, which one or two waves a warp do
// not pay for, and of the 4 m + 1 beams of an aperture three warps of its last CTA have none.
// Mean row launch of a build, us, k_row_pass -> this: 512: 9 waves 16.2 -> 12.4, 37 34.7 ->
// 30.5; 256: 37 13.9 -> 12.3; 1024: 5 28.3 -> 24.5; 768: 9 28.4 -> 23.8; 128: 37 8.3 -> 8.2.
// Six CTAs per SM at 256 (80 registers): 145 waves 28.5 us, with five 30.0.
template <int N>
__host__ __device__ constexpr int few_ctas() {
  return N == 256 ? 6 : row_ctas<N>();
}
template <int N>
__global__ void __launch_bounds__(kRowWarps * 32, few_ctas<N>())
k_row_pass_few(const float2* __restrict__ W, const PlaneWaves start, float2* __restrict__ Phi,
               const float2* __restrict__ t_slice, int conj_t, int store_mode,
               float2* __restrict__ S, int s_waves, int64_t s_stride, int fft_out,
               const float2* __restrict__ tw) {
  constexpr int SEQ = pf::Seqs<N>::SEQ;
  extern __shared__ float2 smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* sbuf = smem + warp * RowSmem<N>::BUF;
  const int y0 = (blockIdx.x * kRowWarps + warp) * SEQ;
  const int64_t wave = blockIdx.y;
  const float2* fset = tw + pf::set_offset(N, false, false) + pf::SetPart<N>::FROM;
  const float2* rset = pf::SetPart<N>::SAME
                           ? fset
                           : tw + pf::set_offset(N, false, true) + pf::SetPart<N>::FROM;
  const float2* trows = t_slice + (int64_t)y0 * N;
  float2 v[pf::Seqs<N>::E];
  if (start.px) row_load<N, true>(v, W, start, tw, wave, y0, lane);
  else row_load<N, false>(v, W, start, tw, wave, y0, lane);
  if (conj_t)
    row_wave<N, true>(v, sbuf, trows, fset, rset, wave, y0, lane, Phi, store_mode, S, s_waves,
                      s_stride, fft_out);
  else
    row_wave<N, false>(v, sbuf, trows, fset, rset, wave, y0, lane, Phi, store_mode, S, s_waves,
                       s_stride, fft_out);
}

// Column pass.  A CTA takes CB neighbouring columns of `chunk` waves, a wave at a time; a
// thread holds a butterfly of one column, and the lanes of a warp run over the columns
// first, so that rows are read and written in segments of CB values straight from
// registers and shared memory carries only the exchange inside each transform.  (One warp
// per column with the tile staged in shared memory took twice the wavefronts and was bound
// by them.)  us per wave of a pass of many waves, with the staged tile / so: 1024: 2.18 /
// 1.74, 768: 1.70 / 1.06, 512: 0.468 / 0.377, 384: 0.64 / 0.26, 256: 0.109 / 0.101; the copy
// bandwidth would allow 1.23, 0.69, 0.31, 0.17 and 0.08.  CB (columns, col_pass_m) and CTAS
// (CTAs per SM) are the fastest measured; at 768 and 1024 two CTAs of 8 columns are all the
// registers that an SM has, 16 of its 64 warps.
template <int N, int COLS>
struct ColCfg {
  using PF = pf::Plan2<N, false>;
  static constexpr int CB = COLS;
  static constexpr int CTAS = N == 64 ? 8 : N == 128 || N == 256 ? 5 : N == 384 ? 3
                            : N == 1024 && CB == 16 ? 1 : 2;
  static constexpr int TPC = pf::col_threads(N), THREADS = CB * TPC;
  static constexpr int PER0 = (PF::NB0 + TPC - 1) / TPC, PER1 = (PF::NB1 + TPC - 1) / TPC;
  static constexpr int E = PER0 * PF::R0 > PER1 * PF::R1 ? PER0 * PF::R0 : PER1 * PF::R1;
  static constexpr int EX = pf::Seqs<N>::PADDED * CB;   // exchange buffer, values
  static constexpr size_t BYTES = (size_t)(EX + pf::SetPart<N>::BOTH) * sizeof(float2);
};

// MODE 0 / 1: multiply by the propagator table / its conjugate and go back to rows;
// MODE 2: multiply by the table and sum |.|^2 over the detector bins.
template <int N, int MODE, int CB>
__global__ void __launch_bounds__(ColCfg<N, CB>::THREADS, ColCfg<N, CB>::CTAS)
k_col_pass(const float2* __restrict__ Phi, float2* __restrict__ W, const float2* __restrict__ ptab,
           const uint8_t* __restrict__ det_mask, const int* __restrict__ wave_out,
           double* __restrict__ det_acc, double det_scale, const float2* __restrict__ tw,
           int n_waves, int chunk) {
  using CC = ColCfg<N, CB>;
  constexpr int NH = N / 2, NQ = N / 4;
  using PF = pf::Plan2<N, false>;
  using PI = pf::Plan2<N, true>;
  constexpr bool EXACT = pf::exact_factors(N, true);
  extern __shared__ float2 ex[];
  float2* fset = ex + CC::EX;
  const float2* rset = pf::rev_set<N>(fset);
  const int c = threadIdx.x % CB, b0 = threadIdx.x / CB;
  const int kx = blockIdx.x * CB + c;
  const int w0 = blockIdx.y * chunk, w_end = min(n_waves, (int)(blockIdx.y + 1) * chunk);
  pf::load_sets<N>(fset, tw, true);
  using SP = pf::SetPart<N>;

  for (int64_t wave = w0; wave < w_end; ++wave) {
    float2 v[CC::E];
    const float2* src = Phi + wave * N * NH + kx;
#pragma unroll
    for (int t = 0; t < CC::PER0; ++t) {
      const int b = b0 + t * CC::TPC;
      if (PF::NB0 % CC::TPC == 0 || b < PF::NB0) {
#pragma unroll
        for (int q = 0; q < PF::R0; ++q)
          v[t * PF::R0 + q] = src[(int64_t)(b + q * PF::NB0) * NH];
      }
    }
    if (N > 256 && wave + 1 < w_end) {   // the next wave's rows of these columns
      const float2* next = Phi + ((wave + 1) * N + threadIdx.x) * NH + blockIdx.x * CB;
#pragma unroll
      for (int r = 0; r < N / CC::THREADS; ++r) prefetch_l2(next + (int64_t)r * CC::THREADS * NH);
    }
    pf::cp_async_wait();
    __syncthreads();   // the factor sets are there; the last exchange has been read
#pragma unroll
    for (int t = 0; t < CC::PER0; ++t) {
      const int b = b0 + t * CC::TPC;
      if (PF::NB0 % CC::TPC == 0 || b < PF::NB0) {
        pf::super_stage<PF::A0, PF::B0, 1, false, false, EXACT>(v + t * PF::R0, 0, nullptr,
                                                                fset + SP::AT0);
        float2* dst = ex + b * (PF::R0 + 1) * CB + c;
#pragma unroll
        for (int o = 0; o < PF::R0; ++o) dst[o * CB] = v[t * PF::R0 + o];
      }
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < CC::PER1; ++t) {
      const int b = b0 + t * CC::TPC;
      if (PF::NB1 % CC::TPC == 0 || b < PF::NB1) {
        const float2* from = ex + b * CB + c;
#pragma unroll
        for (int q = 0; q < PF::R1; ++q) v[t * PF::R1 + q] = from[q * (PF::NB1 + 1) * CB];
      }
    }
    if constexpr (MODE != 2) __syncthreads();   // read before the inverse overwrites it
    float acc = 0.f;
#pragma unroll
    for (int t = 0; t < CC::PER1; ++t) {
      const int b = b0 + t * CC::TPC;
      if (PF::NB1 % CC::TPC == 0 || b < PF::NB1) {
        float2* x = v + t * PF::R1;
        pf::super_stage<PF::A1, PF::B1, PF::R0, false, false, EXACT>(x, b, fset + SP::AT1,
                                                                     fset + SP::AT2);
        // x[q] is ky = b + q NB1; the table depends on kx^2 + ky^2 only, so its rows may be
        // read along kx
#pragma unroll
        for (int q = 0; q < PF::R1; ++q) {
          const int at = q * PF::NB1;
          if (at < NQ || at >= N - NQ) {
            const int ky = b + (at < NQ ? at : at - NH);
            if constexpr (MODE != 2) {
              x[q] = pf::mul_c<MODE == 1>(x[q], __ldg(ptab + (int64_t)ky * NH + kx));
            } else if (det_mask[(int64_t)kx * NH + ky]) {
              const float2 val = pf::mul(x[q], __ldg(ptab + (int64_t)ky * NH + kx));
              acc = fmaf(val.x, val.x, fmaf(val.y, val.y, acc));
            }
          } else {
            x[q] = make_float2(0.f, 0.f);
          }
        }
        if constexpr (MODE != 2) {
          pf::super_stage<PI::A0, PI::B0, 1, true, true, EXACT>(x, 0, nullptr, rset + SP::AT0);
          float2* dst = ex + b * (PI::R0 + 1) * CB + c;
#pragma unroll
          for (int o = 0; o < PI::R0; ++o) dst[o * CB] = x[o];
        }
      }
    }
    if constexpr (MODE != 2) {
      __syncthreads();
#pragma unroll
      for (int t = 0; t < CC::PER0; ++t) {
        const int b = b0 + t * CC::TPC;
        if (PI::NB1 % CC::TPC == 0 || b < PI::NB1) {
          float2* x = v + t * PI::R1;
          const float2* from = ex + b * CB + c;
#pragma unroll
          for (int q = 0; q < PI::R1; ++q) x[q] = from[q * (PI::NB1 + 1) * CB];
          pf::super_stage<PI::A1, PI::B1, PI::R0, true, false, EXACT>(x, b, rset + SP::AT1,
                                                                      rset + SP::AT2);
          float2* dst = W + (wave * N + b) * NH + kx;
#pragma unroll
          for (int q = 0; q < PI::R1; ++q) dst[(int64_t)q * PI::NB1 * NH] = x[q];
        }
      }
    } else {
      const int out = wave_out[wave];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if ((threadIdx.x & 31) == 0 && out >= 0 && acc != 0.f)
        atomicAdd(det_acc + out, det_scale * (double)acc);
    }
  }
}

__global__ void k_transmission(const float* __restrict__ v, double sigma, float2* __restrict__ t,
                               int64_t count) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x) {
    double s, c;
    sincos(sigma * (double)v[i], &s, &c);
    t[i] = make_float2((float)c, (float)s);
  }
}

__global__ void k_propagator_table(float2* __restrict__ ptab, int n, double cell, double lam,
                                   double dz, float scale) {
  const int nh = n / 2, nq = n / 4;
  const int total = nh * nh;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int a = i / nh, b = i % nh;             // [kx'][ky']
    const int kx = a < nq ? a : a - nh;
    const int ky = b < nq ? b : b - nh;
    const int64_t k2 = (int64_t)kx * kx + (int64_t)ky * ky;
    float2 p = make_float2(0.f, 0.f);
    if (16 * k2 < (int64_t)n * n) {
      // phase = -pi * lam * dz * |k|^2, argument (in units of pi) reduced mod 2 in FP64
      double arg = lam * dz * (double)k2 / (cell * cell);
      arg -= 2.0 * floor(0.5 * arg);
      float s, c;
      sincospif(-(float)arg, &s, &c);
      p = make_float2(c * scale, s * scale);
    }
    ptab[i] = p;
  }
}

// One block writes kInitRows rows of one wave as float4 pairs of row-spectrum values
// (N/2 is even, so every row starts on a 16-byte boundary); only the thread holding
// column box(px) computes a nonzero value.
constexpr int kInitRows = 16;

__global__ void k_init_plane_waves(float2* __restrict__ W, int n, const int* __restrict__ px,
                                   const int* __restrict__ py, const float2* __restrict__ amp,
                                   const float2* __restrict__ tw) {
  const int nh = n / 2, npair = nh / 2;
  const int64_t wave = blockIdx.y;
  if (!STEM_REQUIRE(px[wave] >= -nh && px[wave] < nh)) return;   // beam column on the grid
  const int col = px[wave] >= 0 ? px[wave] : px[wave] + nh;
  const float2 a = amp[wave];
  const int q = py[wave];
  float4* base = reinterpret_cast<float4*>(W + wave * (int64_t)n * nh);
  const int y0 = blockIdx.x * kInitRows;
  for (int r = 0; r < kInitRows && y0 + r < n; ++r) {
    const int y = y0 + r;
    float4* row = base + (int64_t)y * npair;
    for (int k2 = threadIdx.x; k2 < npair; k2 += blockDim.x) {
      float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
      if (k2 == (col >> 1)) {
        int m = (int)(((int64_t)q * y) % n);
        if (m < 0) m += n;
        const float2 v = cmul(a, cconj(tw[m]));   // exp(+2 pi i q y / N)
        if (col & 1) {
          o.z = v.x;
          o.w = v.y;
        } else {
          o.x = v.x;
          o.y = v.y;
        }
      }
      row[k2] = o;
    }
  }
}

__global__ void k_probe_init(float2* __restrict__ W, int n, const double* __restrict__ rx,
                             const double* __restrict__ ry, const int* __restrict__ bp,
                             const int* __restrict__ bq, int n_beams, int f, double cell,
                             double c, const float2* __restrict__ tw) {
  extern __shared__ float2 coef[];   // [n_beams]
  const int nh = n / 2, nq = n / 4;
  const int64_t wave = blockIdx.y;
  for (int j = threadIdx.x; j < n_beams; j += blockDim.x) {
    // a_j = c exp(-2 pi i f (p Rx + q Ry) / L), phase in cycles reduced in FP64
    double cyc = (double)f * ((double)bp[j] * rx[wave] + (double)bq[j] * ry[wave]) / cell;
    cyc -= floor(cyc);
    double s, co;
    sincospi(-2.0 * cyc, &s, &co);
    coef[j] = make_float2((float)(c * co), (float)(c * s));
  }
  __syncthreads();
  const int64_t per = (int64_t)n * nh;
  float2* dst = W + wave * per;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < per;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int y = (int)(i / nh), k = (int)(i % nh);
    const int kx = k < nq ? k : k - nh;
    float2 v = make_float2(0.f, 0.f);
    for (int j = 0; j < n_beams; ++j) {
      if (f * bp[j] != kx) continue;
      int m = (int)(((int64_t)f * bq[j] * y) % n);
      if (m < 0) m += n;
      v = cadd(v, cmul(coef[j], cconj(tw[m])));
    }
    dst[i] = v;
  }
}

// One CTA per (output row y, spawn).  Writes the row-pass output form of the
// inelastic wave Interp(H . D) of Eq. Hn0Psi: only even rows y = 2m carry the
// N/2-grid row spectrum 4 * sum_u x(m,u) exp(-2 pi i kx u/(N/2)), odd rows are
// zero; the column pass only looks at the band box of the y-spectrum, where this
// equals the spectrum of the Fourier-interpolated wave.
__global__ void k_spawn(int n, const int* __restrict__ src, const int* __restrict__ site,
                        const int* __restrict__ type, int first_wave, const float2* __restrict__ D,
                        const float2* __restrict__ H, int n_types, int h_mul, int w,
                        const int* __restrict__ win_x0, const int* __restrict__ win_y0,
                        float2* __restrict__ Phi, const float2* __restrict__ tw) {
  extern __shared__ float2 sm[];
  float2* xrow = sm;                 // [w] x(m, u) = H * D
  int* gcol = (int*)(sm + w);        // [w] grid column of u
  const int nh = n / 2, nq = n / 4;
  const int y = blockIdx.x;
  const int k = blockIdx.y;
  const int s = site[k];
  if (!STEM_REQUIRE(s >= 0 && src[k] >= 0 && type[k] >= 0 && type[k] < n_types &&
                    window_ok(win_x0[s], win_y0[s], w, nh)))
    return;   // the whole block, before any barrier
  const int64_t wave = first_wave + k;
  float2* dst = Phi + (wave * n + y) * nh;
  int v = -1;
  if ((y & 1) == 0) {
    v = (y / 2 - win_y0[s]) % nh;
    if (v < 0) v += nh;
    if (v >= w) v = -1;
  }
  if (v < 0) {
    for (int i = threadIdx.x; i < nh; i += blockDim.x) dst[i] = make_float2(0.f, 0.f);
    return;
  }
  const float2* drow = D + (int64_t)src[k] * nh * nh + (int64_t)(y / 2) * nh;
  const float2* hrow = H + (((int64_t)s * h_mul * n_types + type[k]) * w + v) * w;
  for (int u = threadIdx.x; u < w; u += blockDim.x) {
    const int g = (win_x0[s] + u) % nh;
    gcol[u] = g;
    xrow[u] = cmul(hrow[u], drow[g]);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nh; i += blockDim.x) {
    const int kx = i < nq ? i : i - nh;
    float2 acc = make_float2(0.f, 0.f);
    for (int u = 0; u < w; ++u) {
      int m = (int)(((int64_t)2 * kx * gcol[u]) % n);
      if (m < 0) m += n;
      acc = cadd(acc, cmul(xrow[u], tw[m]));   // exp(-2 pi i kx g / (N/2))
    }
    dst[i] = cscale(acc, 4.f);
  }
}

// Waves per CTA: a multiple of the waves in flight in it (`width`), at most 16 of them, and
// no more than leave about kCtaRounds CTAs per resident one (`resident`: CTAs the device holds).
constexpr int kCtaRounds = 3;
int wave_chunk(int n_waves, int blocks_x, int width, int resident) {
  const int64_t items = (n_waves + width - 1) / width;
  const int64_t per = std::max<int64_t>(1, items * blocks_x / (kCtaRounds * (int64_t)resident));
  return width * (int)std::min<int64_t>(per, 16);
}

// The chunk between half and twice of `chunk` (at most 16) whose rounds of CTAs, two to an
// SM, take least, the largest of equal ones.  A last round of at most one CTA per SM, which
// then has it to itself, is counted as 0.6 of a full one (an estimate).  Pass at 512: 593
// waves in chunks of 10 leave a fourth round of 48 CTAs, in chunks of 16 two full rounds; 145
// waves 80 us with chunks of 5, 70 so, 441 waves 219 and 182; at 768 1329 waves 1441 and 1411.
int even_rounds(int n_waves, int blocks_x, int chunk) {
  const int64_t sms = sm_count();
  int best = chunk;
  double least = 0;
  for (int c = std::min(2 * chunk, 16); 2 * c >= chunk && c > 0; --c) {
    const int64_t ctas = (int64_t)((n_waves + c - 1) / c) * blocks_x, rest = ctas % (2 * sms);
    const double time = c * (double(ctas / (2 * sms)) + (rest > sms ? 1.0 : rest ? 0.6 : 0.0));
    if (least == 0 || time < least) { least = time; best = c; }
  }
  return best;
}

// Launches of up to this many row groups (SEQ rows of a wave) go to k_row_pass_few, `warps` of
// k_row_pass being resident on an SM.  Rounds of resident warps at which the two take the
// same time: 64: 4, 128: 8, 256: 10, 512: 13, 768: 18, 1024: 11 to 20, 384: about 50.
int64_t few_rows(int warps) { return 11LL * warps * sm_count(); }

template <int N, bool CONJ, bool START>
cudaError_t row_pass_c(int n_waves, const float2* W, const PlaneWaves& start, float2* Phi,
                       const float2* t, int store_mode, float2* S, int s_waves, int64_t s_stride,
                       int fft_out, const float2* tw, cudaStream_t s) {
  static std::atomic<uint64_t> attr{0};
  cudaError_t e = smem_attr_once(k_row_pass<N, CONJ, START>, RowSmem<N>::BYTES, attr);
  if (e != cudaSuccess) return e;
  const int gx = N / pf::Seqs<N>::SEQ;
  const int chunk = wave_chunk(n_waves, gx, kRowWarps, sm_count() * row_ctas<N>());
  dim3 grid(gx, (n_waves + chunk - 1) / chunk);
  k_row_pass<N, CONJ, START><<<grid, kRowWarps * 32, RowSmem<N>::BYTES, s>>>(
      W, start, Phi, t, store_mode, S, s_waves, s_stride, fft_out, tw, n_waves, chunk);
  return cudaGetLastError();
}

template <int N>
cudaError_t row_pass_n(int n_waves, const float2* W, const PlaneWaves* start, float2* Phi,
                       const float2* t, int conj_t, int store_mode, float2* S, int s_waves,
                       int64_t s_stride, int fft_out, const float2* tw, cudaStream_t s) {
  const PlaneWaves pw = start ? *start : PlaneWaves{};
  if ((int64_t)n_waves * (N / pf::Seqs<N>::SEQ) <= few_rows(kRowWarps * row_ctas<N>())) {
    static std::atomic<uint64_t> attr{0};
    constexpr size_t smem = (size_t)kRowWarps * RowSmem<N>::BUF * sizeof(float2);
    cudaError_t e = smem_attr_once(k_row_pass_few<N>, smem, attr);
    if (e != cudaSuccess) return e;
    dim3 grid(N / (kRowWarps * pf::Seqs<N>::SEQ), n_waves);
    k_row_pass_few<N><<<grid, kRowWarps * 32, smem, s>>>(W, pw, Phi, t, conj_t, store_mode, S,
                                                         s_waves, s_stride, fft_out, tw);
    return cudaGetLastError();
  }
  const auto fn = conj_t ? (start ? row_pass_c<N, true, true> : row_pass_c<N, true, false>)
                         : (start ? row_pass_c<N, false, true> : row_pass_c<N, false, false>);
  return fn(n_waves, W, pw, Phi, t, store_mode, S, s_waves, s_stride, fft_out, tw, s);
}

template <int N, int MODE, int CB>
cudaError_t col_pass_c(int n_waves, const float2* Phi, float2* W, const float2* ptab,
                       const uint8_t* det_mask, const int* wave_out, double* det_acc,
                       double det_scale, const float2* tw, cudaStream_t s) {
  using CC = ColCfg<N, CB>;
  static std::atomic<uint64_t> attr{0};
  cudaError_t e = smem_attr_once(k_col_pass<N, MODE, CB>, CC::BYTES, attr);
  if (e != cudaSuccess) return e;
  const int gx = N / 2 / CB;
  int chunk = wave_chunk(n_waves, gx, 1, sm_count() * CC::CTAS);
  if (CC::CTAS == 2) chunk = even_rounds(n_waves, gx, chunk);
  dim3 grid(gx, (n_waves + chunk - 1) / chunk);
  k_col_pass<N, MODE, CB><<<grid, CC::THREADS, CC::BYTES, s>>>(
      Phi, W, ptab, det_mask, wave_out, det_acc, det_scale, tw, n_waves, chunk);
  return cudaGetLastError();
}

// 16 columns (128-byte segments) at 512, and at 1024 for many waves: one CTA is then all that
// an SM holds, and the last rounds weigh more than the longer segments give (1024, us a pass
// with 8 and 16 columns: 317 waves 590 and 650, 1257 waves 2254 and 2237, 2801 waves 4999 and
// 4881).
template <int N, int MODE>
cudaError_t col_pass_m(int n_waves, const float2* Phi, float2* W, const float2* ptab,
                       const uint8_t* det_mask, const int* wave_out, double* det_acc,
                       double det_scale, const float2* tw, cudaStream_t s) {
  const auto fn = [&] {
    if constexpr (N == 1024) return n_waves < 1024 ? col_pass_c<N, MODE, 8> : col_pass_c<N, MODE, 16>;
    else return col_pass_c<N, MODE, N == 512 ? 16 : 8>;
  }();
  return fn(n_waves, Phi, W, ptab, det_mask, wave_out, det_acc, det_scale, tw, s);
}

template <int N>
cudaError_t col_pass_n(int n_waves, const float2* Phi, float2* W, const float2* ptab, int conj_p,
                       int mode, const uint8_t* det_mask, const int* wave_out, double* det_acc,
                       double det_scale, const float2* tw, cudaStream_t s) {
  if (mode == 1)
    return col_pass_m<N, 2>(n_waves, Phi, W, ptab, det_mask, wave_out, det_acc, det_scale, tw, s);
  return conj_p ? col_pass_m<N, 1>(n_waves, Phi, W, ptab, det_mask, wave_out, det_acc, det_scale,
                                   tw, s)
                : col_pass_m<N, 0>(n_waves, Phi, W, ptab, det_mask, wave_out, det_acc, det_scale,
                                   tw, s);
}

}  // namespace

#define EELS_FOR_EACH_N(X) X(64) X(128) X(256) X(384) X(512) X(768) X(1024)

bool grid_supported(int n) {
#define EELS_CASE(NN) if (n == NN) return true;
  EELS_FOR_EACH_N(EELS_CASE)
#undef EELS_CASE
  return false;
}

int twiddle_table_size(int n) {
  return grid_supported(n) ? pf::table_len(n) : twiddle_table_len(n);
}

namespace {

// Factors of one set of the plans of plan_fft.cuh.
void fill_plan_set(int n, bool col, bool rev, float2* h) {
  const float2* root = h;   // exp(-2 pi i k / n), k < n
  float2* set = h + pf::set_offset(n, col, rev);
  const int a0 = pf::plan_a(n, rev, 0), b0 = pf::plan_b(n, rev, 0);
  const int a1 = pf::plan_a(n, rev, 1), b1 = pf::plan_b(n, rev, 1);
  for (int i = 0; i < pf::set_len(n); ++i) set[i] = make_float2(0.f, 0.f);
  auto mul = [](float2 a, float2 b) {   // the rounding of the device's cmul
    return make_float2(std::fmaf(a.x, b.x, -(a.y * b.y)), std::fmaf(a.x, b.y, a.y * b.x));
  };
  // the radix-r factors exp(-2 pi i q ks / n), q < r: table entries, or for r > 4 products
  // of two of them
  auto factors = [&](int r, int ks, float2* w) {
    w[0] = make_float2(1.f, 0.f);
    if (r <= 4) {
      for (int q = 1; q < r; ++q) w[q] = root[(q * ks) % n];
      return;
    }
    w[1] = root[ks];
    w[2] = mul(w[1], w[1]);
    w[3] = mul(w[2], w[1]);
    w[4] = mul(w[2], w[2]);
    for (int q = 5; q < std::min(r, 8); ++q) w[q] = mul(w[4], w[q - 4]);
    float2 hi = root[(8 * ks) % n];
    const float2 w8 = hi;
    for (int a = 1; a < r / 8; ++a) {
      w[8 * a] = hi;
      for (int q = 1; q < 8; ++q) w[8 * a + q] = mul(hi, w[q]);
      hi = mul(hi, w8);
    }
  };
  float2 w[32];
  if (b0 > 1)
    for (int k = 0; k < a0; ++k) {
      factors(b0, k * (n / (a0 * b0)), w);
      for (int m = 0; m < b0; ++m) set[m * a0 + k] = w[m];
    }
  const int p = a0 * b0, p1 = p * a1;
  for (int k = 0; k < p; ++k) {
    if (pf::exact_factors(n, col))
      for (int q = 0; q < a1; ++q) w[q] = root[(q * k) % n];
    else
      factors(a1, k * (n / p1), w);
    for (int q = 0; q < a1; ++q) set[32 + q * p + k] = w[q];
  }
  if (b1 > 1)
    for (int k = 0; k < p1; ++k) {
      factors(b1, k * (n / (p1 * b1)), w);
      for (int m = 0; m < b1; ++m) set[32 + n + m * p1 + k] = w[m];
    }
}

}  // namespace

void fill_twiddle_tables(int n, float2* h) {
  auto root = [n](int64_t e) {
    const double a = 2.0 * 3.14159265358979323846 * (double)(e % n) / (double)n;
    return make_float2((float)std::cos(a), (float)-std::sin(a));
  };
  for (int k = 0; k < n; ++k) h[k] = root(k);
  for (int k = n; k < twiddle_table_len(n); ++k) h[k] = make_float2(0.f, 0.f);
  if (grid_supported(n))
    for (int i = 0; i < 4; ++i) fill_plan_set(n, i >= 2, i & 1, h);
  if (plan_len(n) != 2) return;
  // stage 1 of the two-stage plan: radix r1 after a first stage of radix r0 (r0 r1 = n)
  const int r0 = plan_radix(n, 0), r1 = plan_radix(n, 1);
  for (int q = 0; q < r1; ++q)
    for (int k = 0; k < r0; ++k) h[n + q * r0 + k] = root((int64_t)q * k);
}

cudaError_t launch_row_pass(int n, int n_waves, const float2* W, float2* Phi, const float2* t,
                            int conj_t, int store_mode, float2* S, int s_waves, int64_t s_stride,
                            int fft_out, const float2* tw, cudaStream_t s,
                            const PlaneWaves* start) {
  if (n_waves <= 0) return cudaSuccess;
#define EELS_CASE(NN) \
  if (n == NN) return row_pass_n<NN>(n_waves, W, start, Phi, t, conj_t, store_mode, S, s_waves, s_stride, fft_out, tw, s);
  EELS_FOR_EACH_N(EELS_CASE)
#undef EELS_CASE
  return cudaErrorInvalidValue;
}

cudaError_t launch_col_pass(int n, int n_waves, const float2* Phi, float2* W, const float2* ptab,
                            int conj_p, int mode, const uint8_t* det_mask, const int* wave_out,
                            double* det_acc, double det_scale, const float2* tw, cudaStream_t s) {
  if (n_waves <= 0) return cudaSuccess;
#define EELS_CASE(NN) \
  if (n == NN) return col_pass_n<NN>(n_waves, Phi, W, ptab, conj_p, mode, det_mask, wave_out, det_acc, det_scale, tw, s);
  EELS_FOR_EACH_N(EELS_CASE)
#undef EELS_CASE
  return cudaErrorInvalidValue;
}

cudaError_t launch_transmission(const float* v, double sigma, float2* t, int64_t count,
                                cudaStream_t s) {
  k_transmission<<<1184, 256, 0, s>>>(v, sigma, t, count);
  return cudaGetLastError();
}

cudaError_t launch_propagator_table(float2* ptab, int n, double cell, double lam, double dz,
                                    float scale, cudaStream_t s) {
  const int total = (n / 2) * (n / 2);
  k_propagator_table<<<(total + 255) / 256, 256, 0, s>>>(ptab, n, cell, lam, dz, scale);
  return cudaGetLastError();
}

cudaError_t launch_init_plane_waves(float2* W, int n, int n_waves, const int* px, const int* py,
                                    const float2* amp, const float2* tw, cudaStream_t s) {
  if (n_waves <= 0) return cudaSuccess;
  dim3 grid((unsigned)((n + kInitRows - 1) / kInitRows), n_waves);
  k_init_plane_waves<<<grid, 128, 0, s>>>(W, n, px, py, amp, tw);
  return cudaGetLastError();
}

cudaError_t launch_probe_init(float2* W, int n, int n_probes, const double* rx, const double* ry,
                              const int* bp, const int* bq, int n_beams, int f, double cell,
                              double c, const float2* tw, cudaStream_t s) {
  if (n_probes <= 0) return cudaSuccess;
  const int64_t per = (int64_t)n * (n / 2);
  dim3 grid((unsigned)((per + 255) / 256), n_probes);
  k_probe_init<<<grid, 256, n_beams * sizeof(float2), s>>>(W, n, rx, ry, bp, bq, n_beams, f, cell,
                                                           c, tw);
  return cudaGetLastError();
}

cudaError_t launch_spawn(int n, const SpawnList& sp, const float2* D, const float2* H, int n_types,
                         int h_mul, int w, const int* win_x0, const int* win_y0, float2* Phi,
                         const float2* tw, cudaStream_t s) {
  if (sp.count <= 0) return cudaSuccess;
  dim3 grid(n, sp.count);
  const size_t smem = (size_t)w * (sizeof(float2) + sizeof(int));
  k_spawn<<<grid, 256, smem, s>>>(n, sp.src, sp.site, sp.type, sp.first_wave, D, H, n_types,
                                  h_mul, w, win_x0, win_y0, Phi, tw);
  return cudaGetLastError();
}

EELS_CHECK_COLLECTOR(collect_checks_ms)

}  // namespace eels
