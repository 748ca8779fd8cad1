// Elastic STEM images (ADF, incoherent bright field) from the exit-surface S-matrix
// (Sec. IV D), in three passes over a batch of scan rows:
//
//   cut pass:     psi_R on its L/f cut, psi_R[y'][x'] = sum_j ax_j(Rx) ay_j(Ry)
//                 S_exit[j][(y0(R) + y') % (N/2)][(x0(R) + x') % (N/2)]; the S-matrix
//                 beams are combined with the probe coefficients of Eq. illum (Sec. III).
//   row pass:     forward DFT of every cut row (register-resident FFT).
//   column pass:  forward DFT of every cut column, then |.|^2 summed over the bins of
//                 each detector (FP64 accumulation per probe and detector).
//
// Scale: S_exit is stored N times the true decimated exit wave and the probe
// coefficients carry no c = f/sqrt(n_in); the caller applies the constant.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace eels {

namespace {

constexpr int kCutWarps = 8;      // warps per CTA of the cut pass
constexpr int kBeamChunk = 32;    // beams whose coefficients are staged at a time
constexpr int kBeamAhead = 2;     // beams whose S values a thread loads together; divides kBeamChunk
constexpr int kFftWarps = 8;

// Packed pairs of floats: one instruction for the real and imaginary part, each rounded as
// the scalar operation.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// Cut pass.  A CTA takes G consecutive probes ix0 .. of one scan row, a thread one column of
// two neighbouring cut rows (elements (row pair, column) in one list, so that no lane is
// left over at the end of a row); every S_exit value of the group's column span is loaded once
// for all its probes.  Each product is rounded and then added (six FP32 operations per
// complex product), beams in ascending order.  Bound by the FP32 pipe: coefficients lie in
// shared memory as (c.x, c.x), (c.y, c.y), so that a product is three packed instructions
// and half of the issue slots are left for the loads, and two rows share each coefficient.
// 512-grid crystal, f = 2, 32 x 32 probes, 593 beams: 4.87 -> 2.65 ms (one row per CTA with
// scalar products before); the FP32 pipe alone would take 1.57 ms for the cuts' own pixels.
template <int G>
__global__ void __launch_bounds__(kCutWarps * 32, 2)
k_exit_cut(const float2* __restrict__ S, int n_in, int nh, int m,
           const float2* __restrict__ axT, const float2* __restrict__ ayT, int n_sx, int n_sy,
           const int* __restrict__ wx, const int* __restrict__ wy, int iy0, bool from_last,
           float2* __restrict__ out) {
  __shared__ ulonglong2 coef[2][kBeamChunk][G];   // (c.x, c.x), (c.y, c.y)
  __shared__ int dx[G];
  const int ix0 = blockIdx.x * G;
  const int np = min(G, n_sx - ix0);
  const int iyl = blockIdx.z;
  const int iy = iy0 + iyl;
  // columns are counted from the first probe's origin, or the last one's (from_last)
  const int xa = wx[from_last ? ix0 + np - 1 : ix0];
  // window origins on the grid (the block's row origin and that column origin decide for
  // the whole block; a bad column origin of another probe is replaced by it)
  if (!STEM_REQUIRE(wy[iy] >= 0 && wy[iy] < nh && xa >= 0 && xa < nh)) return;
  if (threadIdx.x < G) {
    int xg = threadIdx.x < np ? wx[ix0 + threadIdx.x] : xa;
    if (!STEM_REQUIRE(xg >= 0 && xg < nh)) xg = xa;
    dx[threadIdx.x] = (xg - xa + nh) % nh;
  }
  __syncthreads();
  int span = 0;
  for (int g = 0; g < np; ++g) span = max(span, dx[g]);
  const int U = min(span + m, nh);          // columns xa .. xa + U - 1 (cyclic)
  const int first = blockIdx.y * kCutWarps * 32;   // this CTA's (row pair, column) elements
  if (first >= (m / 2) * U) return;                // the same for the whole block
  const int yp = 2 * ((first + (int)threadIdx.x) / U), u = (first + (int)threadIdx.x) % U;
  const bool active = yp < m;
  const int64_t plane = (int64_t)nh * nh;
  const int x = (xa + (active ? u : 0)) % nh, y0 = (wy[iy] + (active ? yp : 0)) % nh;
  const int y1 = y0 + 1 == nh ? 0 : y0 + 1;
  const float2* S0 = S + (int64_t)y0 * nh + x;
  const int d1 = (y1 - y0) * nh;            // the second row's offset

  // coefficients of the beams j0 .. j0 + kBeamChunk - 1 (zero past n_in and past the probes)
  auto stage = [&](int j0, int buf) {
    for (int idx = threadIdx.x; idx < kBeamChunk * G; idx += kCutWarps * 32) {
      const int jj = idx % kBeamChunk, g = idx / kBeamChunk, j = j0 + jj;
      float2 c = make_float2(0.f, 0.f);
      if (j < n_in && g < np)
        c = cmul(__ldg(axT + (int64_t)(ix0 + g) * n_in + j), __ldg(ayT + (int64_t)iy * n_in + j));
      coef[buf][jj][g] = make_ulonglong2(pack2(c.x, c.x), pack2(c.y, c.y));
    }
  };
  uint64_t acc[2][G];
#pragma unroll
  for (int g = 0; g < G; ++g) acc[0][g] = acc[1][g] = 0ull;
  // S values of the beams j .. j + kBeamAhead - 1, loaded while the ones before are used
  float2 ahead[2][kBeamAhead];
  auto load = [&](int j) {
#pragma unroll
    for (int e = 0; e < kBeamAhead; ++e) {
      const float2* p = S0 + (int64_t)(j + e) * plane;
      const bool on = active && j + e < n_in;
      ahead[0][e] = on ? __ldg(p) : make_float2(0.f, 0.f);
      ahead[1][e] = on ? __ldg(p + d1) : make_float2(0.f, 0.f);
    }
  };
  stage(0, 0);
  load(0);
  int buf = 0;
  for (int j0 = 0; j0 < n_in; j0 += kBeamChunk, buf ^= 1) {
    __syncthreads();
    if (j0 + kBeamChunk < n_in) stage(j0 + kBeamChunk, buf ^ 1);
    if (!active) continue;
    const int jc = min(kBeamChunk, n_in - j0);
    for (int jj = 0; jj < jc; jj += kBeamAhead) {
      float2 s[2][kBeamAhead];
#pragma unroll
      for (int e = 0; e < kBeamAhead; ++e) s[0][e] = ahead[0][e], s[1][e] = ahead[1][e];
      load(j0 + jj + kBeamAhead);
#pragma unroll
      for (int e = 0; e < kBeamAhead; ++e) {
        if (jj + e >= jc) break;
        uint64_t v[2], r[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          v[h] = pack2(s[h][e].x, s[h][e].y);
          r[h] = pack2(-s[h][e].y, s[h][e].x);
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
          const ulonglong2 c = coef[buf][jj + e][g];
#pragma unroll
          for (int h = 0; h < 2; ++h)
            acc[h][g] = add2(acc[h][g], fma2(c.x, v[h], mul2(c.y, r[h])));
        }
      }
    }
  }
  if (active) {
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int xp = (u - dx[g] + nh) % nh;
      if (g < np && xp < m) {
        uint64_t* dst = reinterpret_cast<uint64_t*>(
            out + (((int64_t)iyl * n_sx + ix0 + g) * m + yp) * m + xp);
        dst[0] = acc[0][g];
        dst[m] = acc[1][g];
      }
    }
  }
}

// In-place forward DFT of `rows` rows of length M (ROWS rows per warp).
template <int M>
__global__ void __launch_bounds__(kFftWarps * 32)
k_cut_rows(float2* __restrict__ X, int64_t rows, const float2* __restrict__ tw) {
  constexpr int ROWS = RegFFT<M>::ROWS;
  constexpr int LDR = spad_len(M);
  constexpr int E = RegFFT<M>::E;
  using PF = Plan<M>;
  extern __shared__ float2 smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* sbuf = smem + warp * ROWS * LDR;
  const int64_t r0 = ((int64_t)blockIdx.x * kFftWarps + warp) * ROWS;
  if (r0 >= rows) return;
  float2 v[E];
  {
    constexpr int R0 = PF::R(0), NB0 = M / R0, PER0 = PF::per(0);
#pragma unroll
    for (int t = 0; t < PER0; ++t) {
      const int u = lane + 32 * t;
      const bool live = ((ROWS * NB0) % 32 == 0 || u < ROWS * NB0) && r0 + u / NB0 < rows;
      const float2* src = X + (r0 + u / NB0) * M;
#pragma unroll
      for (int q = 0; q < R0; ++q)
        v[t * R0 + q] = live ? src[u % NB0 + q * NB0] : make_float2(0.f, 0.f);
    }
  }
  reg_fft<M>(v, sbuf, LDR, tw, lane);
  {
    constexpr int RF = PF::R(PF::NS - 1), NBF = M / RF, PERF = PF::per(PF::NS - 1);
#pragma unroll
    for (int t = 0; t < PERF; ++t) {
      const int u = lane + 32 * t;
      if (((ROWS * NBF) % 32 == 0 || u < ROWS * NBF) && r0 + u / NBF < rows) {
        float2* dst = X + (r0 + u / NBF) * M;
#pragma unroll
        for (int q = 0; q < RF; ++q) dst[u % NBF + q * NBF] = v[t * RF + q];
      }
    }
  }
}

// Forward DFT of every column of cut blockIdx.y (ROWS columns per warp), then
// sum |X|^2 over each detector's bins (bit d of mask[ky][kx]) into img[d][probe].
template <int M>
__global__ void __launch_bounds__(kFftWarps * 32)
k_cut_cols_detect(const float2* __restrict__ X, const uint8_t* __restrict__ mask, int n_det,
                  int n_sx, int iy0, int64_t img_stride, double* __restrict__ img,
                  const float2* __restrict__ tw) {
  constexpr int ROWS = RegFFT<M>::ROWS;
  constexpr int LDR = spad_len(M);
  constexpr int E = RegFFT<M>::E;
  using PF = Plan<M>;
  extern __shared__ float2 smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* sbuf = smem + warp * ROWS * LDR;
  const int c0 = (blockIdx.x * kFftWarps + warp) * ROWS;
  if (c0 >= M) return;
  const float2* cut = X + (int64_t)blockIdx.y * M * M;
  float2 v[E];
  {
    constexpr int R0 = PF::R(0), NB0 = M / R0, PER0 = PF::per(0);
#pragma unroll
    for (int t = 0; t < PER0; ++t) {
      const int u = lane + 32 * t;
      const int col = c0 + u / NB0;
      const bool live = ((ROWS * NB0) % 32 == 0 || u < ROWS * NB0) && col < M;
#pragma unroll
      for (int q = 0; q < R0; ++q)
        v[t * R0 + q] = live ? cut[(int64_t)(u % NB0 + q * NB0) * M + col] : make_float2(0.f, 0.f);
    }
  }
  reg_fft<M>(v, sbuf, LDR, tw, lane);
  float acc[kMaxDetectors];
#pragma unroll
  for (int d = 0; d < kMaxDetectors; ++d) acc[d] = 0.f;
  {
    constexpr int RF = PF::R(PF::NS - 1), NBF = M / RF, PERF = PF::per(PF::NS - 1);
#pragma unroll
    for (int t = 0; t < PERF; ++t) {
      const int u = lane + 32 * t;
      const int col = c0 + u / NBF;
      if (((ROWS * NBF) % 32 == 0 || u < ROWS * NBF) && col < M) {
#pragma unroll
        for (int q = 0; q < RF; ++q) {
          const int ky = u % NBF + q * NBF;
          const unsigned bits = mask[ky * M + col];
          if (bits) {
            const float2 z = v[t * RF + q];
            const float p = fmaf(z.x, z.x, z.y * z.y);
#pragma unroll
            for (int d = 0; d < kMaxDetectors; ++d)
              if (bits & (1u << d)) acc[d] += p;
          }
        }
      }
    }
  }
  const int cutg = blockIdx.y;
  const int64_t probe = (int64_t)iy0 * n_sx + cutg;
  for (int d = 0; d < n_det; ++d) {
    float a = acc[d];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0 && a != 0.f) atomicAdd(img + d * img_stride + probe, (double)a);
  }
}

template <int M>
cudaError_t cut_fft_detect(float2* X, int n_cut, const uint8_t* mask, int n_det, int n_sx,
                           int iy0, int64_t img_stride, double* img, const float2* tw,
                           cudaStream_t s) {
  constexpr int ROWS = RegFFT<M>::ROWS;
  const size_t smem = (size_t)kFftWarps * ROWS * spad_len(M) * sizeof(float2);
  static std::atomic<uint64_t> rows_attr{0}, cols_attr{0};
  cudaError_t e0 = smem_attr_once(k_cut_rows<M>, smem, rows_attr);
  if (e0 != cudaSuccess) return e0;
  e0 = smem_attr_once(k_cut_cols_detect<M>, smem, cols_attr);
  if (e0 != cudaSuccess) return e0;
  const int64_t rows = (int64_t)n_cut * M;
  const int64_t per_cta = (int64_t)kFftWarps * ROWS;
  k_cut_rows<M><<<(unsigned)((rows + per_cta - 1) / per_cta), kFftWarps * 32, smem, s>>>(X, rows, tw);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  dim3 g((unsigned)((M + per_cta - 1) / per_cta), (unsigned)n_cut);
  k_cut_cols_detect<M><<<g, kFftWarps * 32, smem, s>>>(X, mask, n_det, n_sx, iy0, img_stride, img, tw);
  return cudaGetLastError();
}

__global__ void k_divide(double* __restrict__ map, const double* __restrict__ bf, int n_types,
                         int64_t n_pix) {
  const int64_t total = (int64_t)n_types * n_pix;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x)
    map[i] = map[i] / bf[i % n_pix];
}

}  // namespace

cudaError_t launch_divide(double* map, const double* bf, int n_types, int64_t n_pix,
                          cudaStream_t s) {
  if (n_types <= 0 || n_pix <= 0) return cudaSuccess;
  const int64_t total = (int64_t)n_types * n_pix;
  const unsigned blocks = (unsigned)std::min<int64_t>((total + 255) / 256, 4096);
  k_divide<<<blocks, 256, 0, s>>>(map, bf, n_types, n_pix);
  return cudaGetLastError();
}

bool cut_supported(int m) {
  switch (m) {
    case 16: case 32: case 48: case 64: case 96: case 128: case 192: case 256: case 384: case 512:
      return true;
    default:
      return false;
  }
}

namespace {

template <int G>
cudaError_t exit_cut_g(const float2* S, int n_in, int nh, int m, const float2* axT,
                       const float2* ayT, int n_sx, int n_sy, const int* wx, const int* wy,
                       int iy0, int n_rows, int max_span, bool from_last, float2* out,
                       cudaStream_t s) {
  const int elements = (m / 2) * std::min(m + max_span, nh), threads = kCutWarps * 32;
  dim3 g((unsigned)((n_sx + G - 1) / G), (unsigned)((elements + threads - 1) / threads),
         (unsigned)n_rows);
  k_exit_cut<G><<<g, kCutWarps * 32, 0, s>>>(S, n_in, nh, m, axT, ayT, n_sx, n_sy, wx, wy, iy0,
                                             from_last, out);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_exit_cut(const float2* S, int n_in, int nh, int m, const float2* axT,
                            const float2* ayT, int n_sx, int n_sy, const int* wx, const int* wy,
                            int iy0, int n_rows, int max_span, bool from_last, float2* out,
                            cudaStream_t s) {
  if (n_rows <= 0) return cudaSuccess;
  // probes per CTA: 16 share each S value best; fewer where 16 would leave more than a
  // quarter of the accumulators without a probe, or half of the SMs without a CTA (64 x 64
  // cuts of 16 x 2 probes, 145 beams: 102 us a call with 16 CTAs, 75 with 64)
  const int pad16 = (n_sx + 15) / 16 * 16, pad8 = (n_sx + 7) / 8 * 8;
  const int threads = kCutWarps * 32;
  const int64_t per_group =
      (int64_t)((m / 2 * std::min(m + max_span, nh) + threads - 1) / threads) * n_rows;
  const auto fn = n_sx <= 4 || 2 * per_group * (pad8 / 8) < sm_count() ? exit_cut_g<4>
                  : 4 * (pad16 - pad8) > pad16 || 2 * per_group * (pad16 / 16) < sm_count()
                      ? exit_cut_g<8>
                      : exit_cut_g<16>;
  return fn(S, n_in, nh, m, axT, ayT, n_sx, n_sy, wx, wy, iy0, n_rows, max_span, from_last, out, s);
}

cudaError_t launch_cut_detect(int m, float2* X, int n_cut, const uint8_t* mask, int n_det,
                              int n_sx, int iy0, int64_t img_stride, double* img,
                              const float2* tw, cudaStream_t s) {
  if (n_cut <= 0) return cudaSuccess;
  switch (m) {
#define EELS_CUT_CASE(MM) \
    case MM: return cut_fft_detect<MM>(X, n_cut, mask, n_det, n_sx, iy0, img_stride, img, tw, s);
    EELS_CUT_CASE(16) EELS_CUT_CASE(32) EELS_CUT_CASE(48) EELS_CUT_CASE(64) EELS_CUT_CASE(96)
    EELS_CUT_CASE(128) EELS_CUT_CASE(192) EELS_CUT_CASE(256) EELS_CUT_CASE(384)
    EELS_CUT_CASE(512)
#undef EELS_CUT_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

EELS_CHECK_COLLECTOR(collect_checks_elastic)

}  // namespace eels
