// Inelastic contraction on CUDA cores in FP32 (Eq. SHn0 and the |.|^2 scan sum of
// the second algorithm listing of Sec. III).
//
//   GEMM 1   M_t[d][j] = sum_{p in W_s} conj(Sout[d][p]) H_t[p] Sin[j][p]
//   GEMM 2   V[d][R]   = sum_j M_t[d][j] a_j(R),  a_j(R) = axT[ix(R)][j] ayT[iy(R)][j]
//            map[type_t][R] += sum_d |V[d][R]|^2        (FP64 atomics)
//
// Sin / Sout are depth planes [beam][N/2][N/2]; the window W_s of a site is the
// periodic w x w block at (win_x0, win_y0).  R runs over the scan positions whose
// PRISM window contains the site: a product of a column list and a row list.
#include "common.cuh"
#include "internal.h"

namespace eels {

namespace {

constexpr int TK = 16;   // K values per step

__device__ __forceinline__ void cfma_conj(float2& acc, float2 a, float2 b) {
  // acc += conj(a) * b
  acc.x = fmaf(a.x, b.x, fmaf(a.y, b.y, acc.x));
  acc.y = fmaf(a.x, b.y, fmaf(-a.y, b.x, acc.y));
}
__device__ __forceinline__ void cfma(float2& acc, float2 a, float2 b) {
  acc.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, acc.x));
  acc.y = fmaf(a.x, b.y, fmaf(a.y, b.x, acc.y));
}

// 8-byte asynchronous copy to shared memory; zero where !on (gmem is not read then)
__device__ __forceinline__ void cp_async8(float2* smem, const float2* gmem, bool on) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(smem)),
               "l"(gmem), "r"(on ? 8 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}

// Both products run one loop over K: 256 threads, a 16 IM x 16 JN output tile (thread
// (tx, ty) holds rows ty + 16 i, columns tx + 16 j), K in steps of 16 in ascending order
// with one accumulator per output, so the tile shape does not change a result.  A goes to
// shared memory by cp.async two steps ahead; B is formed from two factors loaded one step
// ahead into registers.  One barrier per step.
//
// Measured against one 64 x 64 tile per transition, loaded without overlap: a 128-grid
// request 2.05 -> 1.57 ms of GEMM 1 and 0.22 -> 0.15 of GEMM 2, two 256-grid configurations
// 9.2 -> 6.23 and 2.8 -> 2.10 ms, a 64-grid map 0.156 -> 0.048 ms.  The FMA
// pipe is 63 % busy: an FMA that reads three registers runs at two thirds of the rate
// (25.6 against 38 T/s), and packed f32x2 FMAs do too; they were no faster.
template <int IM, int JN>
struct Tile {
  static constexpr int S = 3;   // shared-memory stages
  float2 As[S][TK][16 * IM + 1];
  float2 Bs[S][TK][16 * JN + 1];
};

// copy_a(it, As): issues this thread's copies of step it (element k = tid % 16 of rows
// tid / 16 + 16 i); load_b(it): loads the factors of B step it; store_b(Bs): multiplies and
// stores them.  Steps at or past `steps` copy and load nothing.
template <int IM, int JN, bool CONJ, class CopyA, class LoadB, class StoreB>
__device__ __forceinline__ void tile_loop(Tile<IM, JN>& tl, int steps, float2 (&acc)[IM][JN],
                                          CopyA copy_a, LoadB load_b, StoreB store_b) {
  constexpr int S = Tile<IM, JN>::S;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int i = 0; i < IM; ++i)
#pragma unroll
    for (int j = 0; j < JN; ++j) acc[i][j] = make_float2(0.f, 0.f);
  for (int it = 0; it < S - 1; ++it) {
    if (it < steps) copy_a(it, tl.As[it]);
    cp_async_commit();
  }
  if (steps > 0) load_b(0);
  int buf = 0;
  for (int it = 0; it < steps; ++it) {
    store_b(tl.Bs[buf]);
    cp_async_wait<S - 2>();
    __syncthreads();   // step it is there; every thread has left step it - 1
    if (it + S - 1 < steps) copy_a(it + S - 1, tl.As[buf == 0 ? S - 1 : buf - 1]);
    cp_async_commit();
    if (it + 1 < steps) load_b(it + 1);
#pragma unroll 4
    for (int k = 0; k < TK; ++k) {
      float2 a[IM], b[JN];
#pragma unroll
      for (int i = 0; i < IM; ++i) a[i] = tl.As[buf][k][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < JN; ++j) b[j] = tl.Bs[buf][k][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < IM; ++i)
#pragma unroll
        for (int j = 0; j < JN; ++j) {
          if (CONJ) cfma_conj(acc[i][j], a[i], b[j]);
          else cfma(acc[i][j], a[i], b[j]);
        }
    }
    buf = buf + 1 == S ? 0 : buf + 1;
  }
}

// GEMM 1 of the types t0 .. t0 + nt - 1 of one site per blockIdx.z: columns (t, j) of all
// types side by side (they share A), M[(slot nt + t)][d][j].
template <int IM, int JN>
__global__ void __launch_bounds__(256, IM * JN >= 14 ? 2 : 3)
k_gemm1(const float2* __restrict__ Sout, const float2* __restrict__ Sin, int nh, int n_out,
        int n_in, int w, const float2* __restrict__ H, int n_types, int h_mul,
        const int* __restrict__ sites, int t0, int nt, const int* __restrict__ win_x0,
        const int* __restrict__ win_y0, float2* __restrict__ M, int64_t m_stride) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Tile<IM, JN>& tl = *reinterpret_cast<Tile<IM, JN>*>(smem_raw);
  const int slot = blockIdx.z, s = sites[slot];
  if (!STEM_REQUIRE(s >= 0 && t0 >= 0 && t0 + nt <= n_types &&
                    window_ok(win_x0[s], win_y0[s], w, nh)))
    return;   // the whole block, before any barrier
  const int x0 = win_x0[s], y0 = win_y0[s];
  const int d0 = blockIdx.y * 16 * IM, c0 = blockIdx.x * 16 * JN;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;   // loads: tx is k, ty the row
  const int64_t plane = (int64_t)nh * nh;
  const int P = w * w;
  // this thread's columns in loads: type and beam (beam -1: past the end)
  int type[JN], beam[JN];
  const float2* Hs = H + ((int64_t)s * h_mul * n_types + t0) * P;
#pragma unroll
  for (int j = 0; j < JN; ++j) {
    const int c = c0 + ty + 16 * j;
    type[j] = c / n_in;
    beam[j] = c < nt * n_in ? c - type[j] * n_in : -1;
  }
  // window pixel of K element p = 16 it + tx, walked row by row as it grows by 16
  struct Walk {
    int x0, y0, w, nh, u, v;
    __device__ int next() {   // plane offset of the pixel, then 16 pixels on
      int gy = y0 + v, gx = x0 + u;
      if (gy >= nh) gy -= nh;
      if (gx >= nh) gx -= nh;
      u += TK;
      while (u >= w) { u -= w; ++v; }
      return gy * nh + gx;
    }
  };
  Walk wa{x0, y0, w, nh, tx % w, tx / w}, wb = wa;
  float2 h[JN], sv[JN];
  float2 acc[IM][JN];
  tile_loop<IM, JN, true>(
      tl, (P + TK - 1) / TK, acc,
      [&](int it, float2 (*As)[16 * IM + 1]) {
        const bool in = it * TK + tx < P;
        const int off = in ? wa.next() : 0;
#pragma unroll
        for (int i = 0; i < IM; ++i) {
          const int d = d0 + ty + 16 * i;
          const bool on = in && d < n_out;
          cp_async8(&As[tx][ty + 16 * i], on ? Sout + (int64_t)d * plane + off : Sout, on);
        }
      },
      [&](int it) {
        const int p = it * TK + tx;
        const bool in = p < P;
        const int off = in ? wb.next() : 0;
#pragma unroll
        for (int j = 0; j < JN; ++j) {
          const bool on = in && beam[j] >= 0;
          h[j] = on ? __ldg(Hs + ((int64_t)type[j] * P + p)) : make_float2(0.f, 0.f);
          sv[j] = on ? __ldg(Sin + ((int64_t)beam[j] * plane + off)) : make_float2(0.f, 0.f);
        }
      },
      [&](float2 (*Bs)[16 * JN + 1]) {
#pragma unroll
        for (int j = 0; j < JN; ++j) Bs[tx][ty + 16 * j] = cmul(h[j], sv[j]);
      });
#pragma unroll
  for (int j = 0; j < JN; ++j) {
    const int c = c0 + tx + 16 * j;
    if (c >= nt * n_in) continue;
    const int t = c / n_in;
    float2* Mt = M + ((int64_t)slot * nt + t) * m_stride + (c - t * n_in);
#pragma unroll
    for (int i = 0; i < IM; ++i) {
      const int d = d0 + ty + 16 * i;
      if (d < n_out) Mt[(int64_t)d * n_in] = acc[i][j];
    }
  }
}

// GEMM 2 of one site per blockIdx.z.  A row tile is G groups of 64 detector beams; the
// groups of all types are listed side by side (they share the probe columns).  |V|^2 is
// summed within a group in FP32 in a fixed order and added to the FP64 map.
template <int G, int JN>
__global__ void __launch_bounds__(256, 2)
k_gemm2_abs2(const float2* __restrict__ M, int64_t m_stride, int n_out, int n_in,
             const float2* __restrict__ axT, const float2* __restrict__ ayT, int n_sx, int n_sy,
             const int* __restrict__ sites, int t0, int nt, const int* __restrict__ xoff,
             const int* __restrict__ xcnt, const int* __restrict__ xlist,
             const int* __restrict__ yoff, const int* __restrict__ ycnt,
             const int* __restrict__ ylist, double* __restrict__ map) {
  constexpr int IM = 4 * G, TN = 16 * JN;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Tile<IM, JN>& tl = *reinterpret_cast<Tile<IM, JN>*>(smem_raw);
  __shared__ float red[G][16][TN];
  __shared__ int rix[TN], riy[TN];
  const int slot = blockIdx.z, s = sites[slot];
  const int nx = xcnt[s], nr = nx * ycnt[s];
  const int r0 = blockIdx.x * TN;
  if (r0 >= nr) return;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  if (threadIdx.x < TN) {
    const int r = r0 + threadIdx.x;
    int ix = -1, iy = -1;
    if (r < nr) {
      ix = xlist[xoff[s] + r % nx];
      iy = ylist[yoff[s] + r / nx];
      if (!STEM_REQUIRE(ix >= 0 && ix < n_sx && iy >= 0 && iy < n_sy)) ix = iy = -1;   // skipped
    }
    rix[threadIdx.x] = ix;
    riy[threadIdx.x] = iy;
  }
  __syncthreads();
  const int per_type = (n_out + 63) / 64, groups = nt * per_type;
  // M rows of this thread's loads: row ty + 16 i of the tile is beam 64 g + ty + 16 (i % 4)
  // of group blockIdx.y G + i / 4
  const float2* Mg[G];
  int dg[G];   // first beam of the group; n_out where there is no such group
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int gi = blockIdx.y * G + g, t = gi / per_type;
    dg[g] = gi < groups ? 64 * (gi - t * per_type) : n_out;
    Mg[g] = M + ((int64_t)slot * nt + (gi < groups ? t : 0)) * m_stride;
  }
  int ix[JN], iy[JN];
#pragma unroll
  for (int j = 0; j < JN; ++j) {
    ix[j] = rix[ty + 16 * j];
    iy[j] = riy[ty + 16 * j];
  }
  float2 fx[JN], fy[JN];
  float2 acc[IM][JN];
  tile_loop<IM, JN, false>(
      tl, (n_in + TK - 1) / TK, acc,
      [&](int it, float2 (*As)[16 * IM + 1]) {
        const int k = it * TK + tx;
#pragma unroll
        for (int i = 0; i < IM; ++i) {
          const int d = dg[i / 4] + ty + 16 * (i % 4);
          const bool on = k < n_in && d < n_out;
          cp_async8(&As[tx][ty + 16 * i], on ? Mg[i / 4] + (int64_t)d * n_in + k : M, on);
        }
      },
      [&](int it) {
        const int k = it * TK + tx;
#pragma unroll
        for (int j = 0; j < JN; ++j) {
          const bool on = k < n_in && ix[j] >= 0;
          fx[j] = on ? __ldg(axT + ((int64_t)ix[j] * n_in + k)) : make_float2(0.f, 0.f);
          fy[j] = on ? __ldg(ayT + ((int64_t)iy[j] * n_in + k)) : make_float2(0.f, 0.f);
        }
      },
      [&](float2 (*Bs)[16 * JN + 1]) {
#pragma unroll
        for (int j = 0; j < JN; ++j) Bs[tx][ty + 16 * j] = cmul(fx[j], fy[j]);
      });
  // |V|^2 summed over each group's rows, per scan position
#pragma unroll
  for (int g = 0; g < G; ++g)
#pragma unroll
    for (int j = 0; j < JN; ++j) {
      float sum = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 v = acc[4 * g + i][j];
        sum = fmaf(v.x, v.x, fmaf(v.y, v.y, sum));
      }
      red[g][ty][tx + 16 * j] = sum;
    }
  __syncthreads();
  for (int e = threadIdx.x; e < G * TN; e += 256) {
    const int g = e / TN, c = e % TN, gi = blockIdx.y * G + g;
    if (gi >= groups || rix[c] < 0) continue;
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) sum += red[g][i][c];
    const int64_t idx = ((int64_t)(t0 + gi / per_type) * n_sy + riy[c]) * n_sx + rix[c];
    atomicAdd(map + idx, (double)sum);
  }
}

__global__ void k_phase_table(float2* __restrict__ out, const int* __restrict__ bidx, int n_beams,
                              int f, double cell, double r0, double step, int n_pos,
                              int r_first) {
  const int total = n_beams * n_pos;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int j = i % n_beams, r = i / n_beams;
    const double R = __dadd_rn(r0, __dmul_rn((double)(r_first + r), step));
    double cyc = (double)f * (double)bidx[j] * R / cell;   // exp(-2 pi i cyc)
    cyc -= floor(cyc);
    double s, c;
    sincospi(-2.0 * cyc, &s, &c);
    out[i] = make_float2((float)c, (float)s);
  }
}

__global__ void k_accumulate(double* __restrict__ acc, const double* __restrict__ x,
                             int64_t count) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x)
    acc[i] += x[i];
}

__global__ void k_scale(double* a, int64_t count, double scale) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x)
    a[i] *= scale;
}

// a *= scale, and bit 2 of *flag set if any scaled value is not finite (NaN or Inf)
__global__ void k_scale_check(double* a, int64_t count, double scale, int* flag) {
  int bad = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double v = a[i] * scale;
    a[i] = v;
    bad |= !isfinite(v);
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 2);
}

}  // namespace

namespace {

// Estimated cycles of one K step over a whole launch with 16 im x 16 jn tiles: the CTAs of
// the busiest SM after one another, each 128 im jn cycles of FMA issue and the issue slots of
// its loads and its loop, plus the latency of a step where one CTA has an SM to itself.
double step_cost(double ctas, int im, int jn, double per_load, double fixed) {
  const double per_sm = ceil(ctas / sm_count());
  return per_sm * (128.0 * im * jn + per_load * (im + jn) + fixed) + (per_sm < 2 ? 500.0 : 0.0);
}

template <int IM, int JN>
cudaError_t gemm1_tile(const float2* Sout, const float2* Sin, int nh, int n_out, int n_in, int w,
                       const float2* H, int n_types, int h_mul, const SiteBatch& sb,
                       const int* win_x0, const int* win_y0, float2* M, int64_t m_stride,
                       cudaStream_t s) {
  static std::atomic<uint64_t> attr{0};
  cudaError_t e = smem_attr_once(k_gemm1<IM, JN>, sizeof(Tile<IM, JN>), attr);
  if (e != cudaSuccess) return e;
  dim3 grid((sb.nt * n_in + 16 * JN - 1) / (16 * JN), (n_out + 16 * IM - 1) / (16 * IM), sb.count);
  k_gemm1<IM, JN><<<grid, 256, sizeof(Tile<IM, JN>), s>>>(Sout, Sin, nh, n_out, n_in, w, H,
                                                          n_types, h_mul, sb.site, sb.t0, sb.nt,
                                                          win_x0, win_y0, M, m_stride);
  return cudaGetLastError();
}

template <int G, int JN>
cudaError_t gemm2_tile(const float2* M, int64_t m_stride, int n_out, int n_in, const float2* axT,
                       const float2* ayT, int n_sx, int n_sy, const SiteBatch& sb,
                       const WindowLists& wl, double* map, cudaStream_t s) {
  static std::atomic<uint64_t> attr{0};
  cudaError_t e = smem_attr_once(k_gemm2_abs2<G, JN>, sizeof(Tile<4 * G, JN>), attr);
  if (e != cudaSuccess) return e;
  const int groups = sb.nt * ((n_out + 63) / 64);
  dim3 grid((wl.max_nr + 16 * JN - 1) / (16 * JN), (groups + G - 1) / G, sb.count);
  k_gemm2_abs2<G, JN><<<grid, 256, sizeof(Tile<4 * G, JN>), s>>>(
      M, m_stride, n_out, n_in, axT, ayT, n_sx, n_sy, sb.site, sb.t0, sb.nt, wl.xoff, wl.xcnt,
      wl.xlist, wl.yoff, wl.ycnt, wl.ylist, map);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_gemm1_fp32(const float2* Sout, const float2* Sin, int nh, int n_out, int n_in,
                              int w, const float2* H, int n_types, int h_mul, const SiteBatch& sb,
                              const int* win_x0, const int* win_y0, float2* M, int64_t m_stride,
                              cudaStream_t s) {
  if (sb.count <= 0 || sb.nt <= 0) return cudaSuccess;
  // the tile that wastes least on the edges of n_out and nt n_in, or spreads a small
  // launch over more SMs (the 64-grid map takes 60 CTAs of 16 x 16 instead of 18 of 32 x 32:
  // 218 -> 198 us).  A load and the loop cost 68 (im + jn) + 300 issue slots a step by the
  // instruction counts.
  int im = 0, jn = 0;
  double best = 0;
  for (int i : {8, 7, 6, 5, 4, 2, 1})
    for (int j : {4, 2, 1}) {
      if (j == 1 ? i > 2 : i < 2) continue;   // not built
      const int64_t ctas = (int64_t)((sb.nt * n_in + 16 * j - 1) / (16 * j)) *
                           ((n_out + 16 * i - 1) / (16 * i)) * sb.count;
      const double c = step_cost((double)ctas, i, j, 68.0, 300.0);
      if (im == 0 || c < best) { best = c; im = i; jn = j; }
    }
#define EELS_G1(I, J)                                                                         \
  if (im == I && jn == J)                                                                     \
    return gemm1_tile<I, J>(Sout, Sin, nh, n_out, n_in, w, H, n_types, h_mul, sb, win_x0,     \
                            win_y0, M, m_stride, s);
  EELS_G1(8, 4) EELS_G1(7, 4) EELS_G1(6, 4) EELS_G1(5, 4) EELS_G1(4, 4) EELS_G1(2, 4)
  EELS_G1(8, 2) EELS_G1(7, 2) EELS_G1(6, 2) EELS_G1(5, 2) EELS_G1(4, 2) EELS_G1(2, 2)
  EELS_G1(2, 1) EELS_G1(1, 1)
#undef EELS_G1
  return cudaErrorInvalidValue;
}

cudaError_t launch_gemm2_abs2_fp32(const float2* M, int64_t m_stride, int n_out, int n_in,
                                   const float2* axT, const float2* ayT, int n_sx, int n_sy,
                                   const SiteBatch& sb, const WindowLists& wl, double* map,
                                   cudaStream_t s) {
  if (sb.count <= 0 || sb.nt <= 0 || wl.max_nr <= 0) return cudaSuccess;
  const int groups = sb.nt * ((n_out + 63) / 64);
  // positions past a site's own count cost nothing (those tiles return at once), so the
  // tiles that run are counted, not those of the largest site: 32 columns for the two
  // 256-grid configurations instead of 64, 2.46 -> 2.10 ms
  int g = 0, jn = 0;
  double best = 0;
  for (int i : {2, 1})
    for (int j : {4, 2, 1}) {
      if (i == 2 && j == 1) continue;   // not built
      const double ctas = wl.tiles[j / 2] * ((groups + i - 1) / i) * sb.count;
      const double c = step_cost(ctas, 4 * i, j, 20.0, 120.0);
      if (g == 0 || c < best) { best = c; g = i; jn = j; }
    }
#define EELS_G2(I, J)                                                                         \
  if (g == I && jn == J)                                                                      \
    return gemm2_tile<I, J>(M, m_stride, n_out, n_in, axT, ayT, n_sx, n_sy, sb, wl, map, s);
  EELS_G2(2, 4) EELS_G2(1, 4) EELS_G2(2, 2) EELS_G2(1, 2) EELS_G2(1, 1)
#undef EELS_G2
  return cudaErrorInvalidValue;
}

cudaError_t launch_phase_table(float2* out, const int* bidx, int n_beams, int f, double cell,
                               double r0, double step, int n_pos, cudaStream_t s,
                               int r_first) {
  const int total = n_beams * n_pos;
  if (total <= 0) return cudaSuccess;
  k_phase_table<<<(total + 255) / 256, 256, 0, s>>>(out, bidx, n_beams, f, cell, r0, step, n_pos,
                                                    r_first);
  return cudaGetLastError();
}

cudaError_t launch_accumulate(double* acc, const double* x, int64_t count, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  k_accumulate<<<256, 256, 0, s>>>(acc, x, count);
  return cudaGetLastError();
}

cudaError_t launch_scale_check(double* a, int64_t count, double scale, int* flag,
                               cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  k_scale_check<<<256, 256, 0, s>>>(a, count, scale, flag);
  return cudaGetLastError();
}

cudaError_t launch_scale(double* a, int64_t count, double scale, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  k_scale<<<256, 256, 0, s>>>(a, count, scale);
  return cudaGetLastError();
}

EELS_CHECK_COLLECTOR(collect_checks_fp32)

}  // namespace eels
