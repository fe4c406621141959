// Numerical monochromatisation by CGLS (Sec. 4.2, Eqs. 12-13).
//
// Broadband pattern b = C m, C = sum_j w_j T_j (w_j: spectral weight / a_j^2), where T_j samples m at
// c + (i - c) / a_j along both axes (c = M / 2, a_j = lambda_j / lambda_c) with linear interpolation
// and zero outside the grid. k CGLS steps from x_0 = 0 give the least-squares solution over the
// Krylov subspace of Eq. 13.
//
// All k steps run on chip: the search direction p (with a one-pixel zero border, so samples outside
// the grid read zeros) and the residual r live in shared memory, the step's product vector in registers,
// x in registers or (k_mono_walk) tensor memory. C^T r runs separably per wavelength, r S_j then S_j^T (.), with the coordinate formula of
// C, so the GPU's C^T is exactly the transpose of its C. Step sizes and norms are FP64 block
// reductions in a fixed order (bitwise reproducible). Two forms:
//   k_mono_walk  M = 64, 128 (one CTA per pattern) and 256 (a cluster of four): threads walk strips of
//                samples (described there)
//   k_mono_cgls  M = 8, 16, 32 (one CTA per pattern), tiles too small for the strips: C p gathers four
//                neighbours per pixel and wavelength, C^T r reads a table of the transposed
//                interpolation (at most kTapsT taps an output)
#include <cuda_runtime.h>
#include <math.h>

#include "cluster.cuh"
#include "engine.h"
#include "fused_common.cuh"

namespace ptycho {

namespace {

constexpr int kTapsT = 8;  // entries of one column of S_j (a_j <= 2.5: at most 2 a_j + 3)

template <int M>
struct MonoShape {
  static constexpr int TPB = M == 8 ? 64 : 256;
  static constexpr int PPT = M * M / TPB;  // pixels per thread
  static constexpr int LDP = M + 2;        // padded row of p
  static constexpr size_t P_BYTES = (size_t)LDP * LDP * 4;
  static constexpr int LDR = M + 1;         // padded row of r and T (conflict-free column walks)
  static constexpr size_t R_BYTES = (size_t)M * LDR * 4;
  static constexpr size_t TAB_BYTES = (size_t)M * kTapsT * 8 + (size_t)M * 4;  // taps, then counts
  static constexpr size_t RED_BYTES = (size_t)(TPB / 32 + 1) * 2 * 8;
  static constexpr size_t SPEC_BYTES = (size_t)3 * kMonoMaxJ * 4;
  static constexpr size_t ROW_BYTES = (size_t)2 * M * 8;  // C p: row samples (i0, f), two buffers
  static constexpr size_t BYTES = P_BYTES + 2 * R_BYTES + TAB_BYTES + RED_BYTES + SPEC_BYTES + ROW_BYTES;
  static_assert(M * M % TPB == 0 && TPB % M == 0, "pixel ownership");
};

// sample position of output index i under scale 1 / a: i0 in [-1, M - 1] and fraction f (zero
// weight outside the grid: i0 = -1, f = 0 reads the zero border)
__device__ __forceinline__ void interp_at(int i, float c, float inv_a, int M, int& i0, float& f) {
  const float t = fmaf((float)i - c, inv_a, c);
  if (!(t >= -1.f && t < (float)M)) {
    i0 = -1;
    f = 0.f;
    return;
  }
  const float fl = floorf(t);
  i0 = (int)fl;
  f = t - fl;
}

// FP64 sums of two per-thread values over the CTA, in a fixed order; every thread gets both. The
// warps' sums are finished by warp 0 alone (shuffle tree) and broadcast through shared memory.
template <int TPB>
__device__ __forceinline__ void block_sum2(double a, double b, double* red, double& oa, double& ob) {
  constexpr int NW = TPB / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  __syncthreads();  // red is free (previous readers are done)
  if (lane == 0) {
    red[2 * warp] = a;
    red[2 * warp + 1] = b;
  }
  __syncthreads();
  if (warp == 0) {
    double x = lane < NW ? red[2 * lane] : 0.0, y = lane < NW ? red[2 * lane + 1] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      x += __shfl_xor_sync(0xffffffffu, x, o);
      y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    if (lane == 0) {
      red[2 * NW] = x;
      red[2 * NW + 1] = y;
    }
  }
  __syncthreads();
  oa = red[2 * NW];
  ob = red[2 * NW + 1];
}

template <int M>
__global__ void __launch_bounds__(MonoShape<M>::TPB, 1) k_mono_cgls(const MonoArgs a) {
  using SH = MonoShape<M>;
  constexpr int TPB = SH::TPB, PPT = SH::PPT, LDP = SH::LDP, LDR = SH::LDR, RSTEP = TPB / M;
  extern __shared__ __align__(16) unsigned char smem[];
  float* Pp = reinterpret_cast<float*>(smem);                        // (M + 2)^2, zero border
  float* R = reinterpret_cast<float*>(smem + SH::P_BYTES);               // M x LDR
  float* T = reinterpret_cast<float*>(smem + SH::P_BYTES + SH::R_BYTES);  // M x LDR, r S_j
  // column u of S_j: its non-zero taps (weight, source index as float bits) in increasing source
  // order, zero-filled to kTapsT, and their count
  float2* tab = reinterpret_cast<float2*>(smem + SH::P_BYTES + 2 * SH::R_BYTES);
  const float4* tab4 = reinterpret_cast<const float4*>(tab);
  int* tab_n = reinterpret_cast<int*>(tab + M * kTapsT);
  double* red = reinterpret_cast<double*>(smem + SH::P_BYTES + 2 * SH::R_BYTES + SH::TAB_BYTES);
  // spectrum: 1 / a_j, a_j, w_j
  float* s_inv = reinterpret_cast<float*>(smem + SH::P_BYTES + 2 * SH::R_BYTES + SH::TAB_BYTES + SH::RED_BYTES);
  float* s_a = s_inv + kMonoMaxJ;
  float* s_w = s_a + kMonoMaxJ;
  float2* s_rt = reinterpret_cast<float2*>(smem + SH::P_BYTES + 2 * SH::R_BYTES + SH::TAB_BYTES + SH::RED_BYTES +
                                           SH::SPEC_BYTES);  // 2 x M

  const int tid = threadIdx.x;
  const int col = tid % M, row0 = tid / M;
  const float c = 0.5f * (float)M;
  const int n = blockIdx.x;
  const float* bn = a.b + (size_t)n * M * M;
  float* xn = a.x + (size_t)n * M * M;
  double* rs = a.resid ? a.resid + (size_t)n * (a.k + 1) : nullptr;

  // C^T v for the own pixels into acc, v in R (separable per wavelength, through T)
  auto adjoint = [&](float (&acc)[PPT]) {
#pragma unroll
    for (int m = 0; m < PPT; ++m) acc[m] = 0.f;
    for (int j = 0; j < a.J; ++j) {
      const float inv_a = s_inv[j], sa = s_a[j];
      // column u of S_j: the sources x with i0(x) in {u - 1, u}; weight 1 - f (i0 = u) or f (i0 = u - 1)
      // (M * kTapsT is a multiple of 32 and so is TPB: every warp runs whole iterations, and the 8
      // lanes of one column sit in one warp)
      for (int e = tid; e < M * kTapsT; e += TPB) {
        const int u = e / kTapsT, l = e % kTapsT;
        const int lo = max(0, (int)ceilf(fmaf((float)(u - 1) - c, sa, c)) - 1);
        const int hi = min(M - 1, (int)floorf(fmaf((float)(u + 1) - c, sa, c)) + 1);
        const int src = lo + l;
        float w = 0.f;
        if (src <= hi) {
          int i0;
          float f;
          interp_at(src, c, inv_a, M, i0, f);
          w = i0 == u ? 1.f - f : (i0 == u - 1 ? f : 0.f);
        }
        const unsigned nz = __ballot_sync(0xffffffffu, w != 0.f);
        const unsigned grp = (nz >> ((tid & 31) & ~(kTapsT - 1))) & ((1u << kTapsT) - 1u);
        const int cnt = __popc(grp);
        if (w != 0.f) tab[u * kTapsT + __popc(grp & ((1u << l) - 1u))] = make_float2(w, __int_as_float(src));
        if (l >= cnt) tab[u * kTapsT + l] = make_float2(0.f, __int_as_float(0));
        if (l == 0) tab_n[u] = cnt;
      }
      __syncthreads();
      // T(y, v) = sum_x S_j[x, v] R(y, x); zero-filled taps add exact zeros
      if constexpr (M >= 32) {
        // a warp walks 32 consecutive rows of one column: the column's taps are a broadcast and the
        // padded rows put the 32 loads (and the store) in 32 different banks
        const int lane = tid & 31, warp = tid >> 5;
#pragma unroll 4
        for (int m = 0; m < PPT; ++m) {
          const int unit = warp * PPT + m;
          const int v = unit % M, y = (unit / M) * 32 + lane;
          const int nt = tab_n[v];
          float s = 0.f;
#pragma unroll
          for (int h = 0; h < kTapsT / 2; ++h)
            if (2 * h < nt) {
              const float4 e = tab4[v * (kTapsT / 2) + h];
              s = fmaf(e.x, R[y * LDR + __float_as_int(e.y)], s);
              s = fmaf(e.z, R[y * LDR + __float_as_int(e.w)], s);
            }
          T[y * LDR + v] = s;
        }
      } else {
        int ci[kTapsT];
        float cw[kTapsT];
#pragma unroll
        for (int h = 0; h < kTapsT / 2; ++h) {
          const float4 e = tab4[col * (kTapsT / 2) + h];
          cw[2 * h] = e.x;
          ci[2 * h] = __float_as_int(e.y);
          cw[2 * h + 1] = e.z;
          ci[2 * h + 1] = __float_as_int(e.w);
        }
        const int nt = __reduce_max_sync(0xffffffffu, tab_n[col]);
#pragma unroll
        for (int m = 0; m < PPT; ++m) {
          const int y = row0 + m * RSTEP;
          float s = 0.f;
#pragma unroll
          for (int l = 0; l < kTapsT; ++l)
            if (l < nt) s = fmaf(cw[l], R[y * LDR + ci[l]], s);
          T[y * LDR + col] = s;
        }
      }
      __syncthreads();
      // acc(u, v) += w_j sum_y S_j[y, u] T(y, v)
      const float wj = s_w[j];
#pragma unroll
      for (int m = 0; m < PPT; ++m) {
        const int u = row0 + m * RSTEP;
        const int nh = (__reduce_max_sync(0xffffffffu, tab_n[u]) + 1) / 2;
        float s = 0.f;
#pragma unroll
        for (int h = 0; h < kTapsT / 2; ++h)
          if (h < nh) {
            const float4 e = tab4[u * (kTapsT / 2) + h];
            s = fmaf(e.x, T[__float_as_int(e.y) * LDR + col], s);
            s = fmaf(e.z, T[__float_as_int(e.w) * LDR + col], s);
          }
        acc[m] = fmaf(wj, s, acc[m]);
      }
      __syncthreads();  // the table and T are rebuilt for the next wavelength
    }
  };

  // C p for the own pixels into acc, p in Pp. The row samples of a wavelength are the same for a
  // whole row of pixels: a table per wavelength (two buffers: the barrier that publishes table j
  // also ends every read of table j - 2)
  auto forward = [&](float (&acc)[PPT]) {
#pragma unroll
    for (int m = 0; m < PPT; ++m) acc[m] = 0.f;
    for (int j = 0; j < a.J; ++j) {
      const float inv_a = s_inv[j], wj = s_w[j];
      float2* rt = s_rt + (j & 1) * M;
      for (int i = tid; i < M; i += TPB) {
        int i0;
        float f;
        interp_at(i, c, inv_a, M, i0, f);
        rt[i] = make_float2(__int_as_float(i0), f);
      }
      __syncthreads();
      int x0;
      float fx;
      interp_at(col, c, inv_a, M, x0, fx);
      const float gx = 1.f - fx;
#pragma unroll
      for (int m = 0; m < PPT; ++m) {
        const float2 ry = rt[row0 + m * RSTEP];
        const int y0 = __float_as_int(ry.x);
        const float fy = ry.y;
        const float* p0 = Pp + (y0 + 1) * LDP + (x0 + 1);
        const float top = fmaf(fx, p0[1], gx * p0[0]);
        const float bot = fmaf(fx, p0[LDP + 1], gx * p0[LDP]);
        acc[m] = fmaf(wj, fmaf(fy, bot, (1.f - fy) * top), acc[m]);
      }
    }
  };

  // ---- start: spectrum to shared memory, zero border of p, r = b, x = 0
  for (int i = tid; i < a.J; i += TPB) {
    s_inv[i] = a.inv_a[i];
    s_a[i] = a.a[i];
    s_w[i] = a.w[i];
  }
  for (int i = tid; i < LDP * LDP; i += TPB) Pp[i] = 0.f;
  float xk[PPT], acc[PPT];
  float rr = 0.f;  // per-thread partial sums in FP32 (PPT terms), CTA sums in FP64
#pragma unroll
  for (int m = 0; m < PPT; ++m) {
    const int y = row0 + m * RSTEP;
    const float v = bn[y * M + col];
    R[y * LDR + col] = v;
    rr = fmaf(v, v, rr);
    xk[m] = 0.f;
  }
  __syncthreads();
  adjoint(acc);  // s_0 = C^T b
  double gamma = 0.0, rr_all = 0.0;
  {
    float g = 0.f;
#pragma unroll
    for (int m = 0; m < PPT; ++m) g = fmaf(acc[m], acc[m], g);
    block_sum2<TPB>(g, rr, red, gamma, rr_all);
  }
  if (rs && tid == 0) rs[0] = sqrt(rr_all);
#pragma unroll
  for (int m = 0; m < PPT; ++m) Pp[(row0 + m * RSTEP + 1) * LDP + col + 1] = acc[m];
  __syncthreads();

  for (int it = 0; it < a.k; ++it) {
    if (!(gamma > 0.0)) {  // C^T r = 0: x is the least-squares solution already
      if (rs && tid == 0) rs[it + 1] = sqrt(rr_all);
      continue;
    }
    forward(acc);  // q = C p
    double qq = 0.0;
    {
      float l = 0.f;
#pragma unroll
      for (int m = 0; m < PPT; ++m) l = fmaf(acc[m], acc[m], l);
      double unused;
      block_sum2<TPB>(l, 0.0, red, qq, unused);
    }
    if (!(qq > 0.0)) {
      if (rs && tid == 0) rs[it + 1] = sqrt(rr_all);
      continue;
    }
    const float alpha = (float)(gamma / qq);
    rr = 0.f;
#pragma unroll
    for (int m = 0; m < PPT; ++m) {
      const int y = row0 + m * RSTEP;
      xk[m] = fmaf(alpha, Pp[(y + 1) * LDP + col + 1], xk[m]);
      const float r = fmaf(-alpha, acc[m], R[y * LDR + col]);
      R[y * LDR + col] = r;
      rr = fmaf(r, r, rr);
    }
    __syncthreads();
    adjoint(acc);  // s = C^T r
    double gnew = 0.0;
    {
      float g = 0.f;
#pragma unroll
      for (int m = 0; m < PPT; ++m) g = fmaf(acc[m], acc[m], g);
      block_sum2<TPB>(g, rr, red, gnew, rr_all);
    }
    if (rs && tid == 0) rs[it + 1] = sqrt(rr_all);
    const float beta = (float)(gnew / gamma);
    gamma = gnew;
#pragma unroll
    for (int m = 0; m < PPT; ++m) {
      float* pp = Pp + (row0 + m * RSTEP + 1) * LDP + col + 1;
      *pp = fmaf(beta, *pp, acc[m]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int m = 0; m < PPT; ++m) {
    const float v = xk[m];
    xn[(row0 + m * RSTEP) * M + col] = a.clamp ? fmaxf(v, 0.f) : v;
  }
}

__device__ __forceinline__ double ld_cluster_f64(uint32_t addr) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void st_cluster_f64(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

// ---- M = 64, 128 and 256: strips of 16 outputs of two lines per thread.
//
// Both operators walk a line of samples in increasing order, so what neighbouring outputs share is
// loaded once and stays in registers:
//   C p     lanes = columns, a thread walks 16 rows of two columns. The row sample index i0 advances
//           by 0 or 1 from row to row for a_j >= 1, so the x-interpolated rows i0 and i0 + 1 are
//           kept and only the row that is new is interpolated (2 / a_j loads an output, not 4).
//   C^T r   the sources of one axis form consecutive groups G_u = {y : i0(y) = u}; with B_u = sum_{G_u}
//           f r and A_u = sum_{G_u} (1 - f) r the transposed interpolation is A_u + B_{u-1}, every
//           source read once. Pass 1 runs it along the rows (lanes = rows) into T, pass 2 along the
//           columns.
// What a walk cannot compute as it goes is, per wavelength and axis, where each strip starts and which
// steps advance: 16 bytes a strip, built once per launch. The fractions f come from a table where one of
// every wavelength fits beside the rest (FT), else from the running index (three more instructions per
// source of two lines: 7.17 against 6.82 ms for 900 patterns of 128^2, J = 32, k = 10).
//
// TILE x TILE outputs per CTA. M = TILE: one CTA per pattern. M = 2 TILE (QUAD): a cluster of four,
// one quadrant each. Sampling about the centre c = M / 2 never crosses it (t(i) < c for i < c, t(i) >= c
// for i >= c), so a quadrant reads its own samples and one halo row and column of p, and adds to its own
// outputs and one halo row and column of C^T r: the only data that leaves a CTA, once per product.
//
// Bound: instruction issue; shared-memory wavefronts (2 / a_j per warp of outputs and wavelength for C,
// 2 a_j + 1 for C^T) are about half of it.
template <int TILE_, bool QUAD_>
struct WalkShape {
  static constexpr int TILE = TILE_, STRIP = 16, AXES = QUAD_ ? 2 : 1;
  static constexpr int TPB = TILE * TILE / (2 * STRIP);
  static constexpr int CG = TILE / 64;        // warps side by side over one half of the lanes' lines
  static constexpr int LDP = TILE + 2;         // p with a one-sample border
  static constexpr int LDR = TILE + 1;         // r and T (odd: walks along rows are conflict-free)
  static constexpr int MIN_BLOCKS = TILE == 64 ? 4 : 1;
  static constexpr size_t align16(size_t v) { return (v + 15) / 16 * 16; }
  static constexpr size_t P_BYTES = align16((size_t)LDP * LDP * 4);
  static constexpr size_t R_BYTES = align16((size_t)TILE * LDR * 4);
  static constexpr size_t RED_BYTES = (size_t)(TPB / 32 + 1) * 2 * 8 + 4 * 2 * 8;
  static constexpr size_t SPEC_BYTES = (size_t)3 * kMonoMaxJ * 4;
  static constexpr size_t HALO_BYTES = (size_t)(2 * TILE + 8) * 4;  // and the tensor-memory address
  // x lives in tensor memory (2 STRIP columns of each thread's lane): it is touched once a step, and the
  // registers it would take are what the walks need to keep loads in flight
  static constexpr uint32_t TMEM_COLS = TPB / 128 * 2 * STRIP;
  // of one wavelength: a record per strip and axis; QUAD: the group starts of the row axis as well
  static constexpr size_t TAB_S = (size_t)TILE / STRIP * 16;
  static constexpr size_t TAB = AXES * TAB_S + (QUAD_ ? align16((size_t)TILE + 2) : 0);
  static constexpr size_t FIXED = P_BYTES + 2 * R_BYTES + RED_BYTES + SPEC_BYTES + HALO_BYTES;
  static constexpr size_t TAB_F = (size_t)AXES * TILE * 4;
  // (16 bytes behind the tables: a walk loads one source ahead)
  static constexpr size_t bytes(int J, bool ft) { return FIXED + (size_t)J * (TAB + (ft ? TAB_F : 0)) + 16; }
  static constexpr size_t LIMIT = MIN_BLOCKS == 1 ? 232448 : 233472 / MIN_BLOCKS - 1024;  // of one CTA
  static_assert(TILE % 64 == 0 && TPB % 32 == 0 && TPB > TILE, "strips, a thread per halo element");
  static_assert(bytes(kMonoMaxJ, false) <= LIMIT, "the largest spectrum without fraction tables fits");
};

// a value that is the same in all lanes, marked so for the compiler (uniform registers and branches)
__device__ __forceinline__ int warp_uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }

// the samples of one axis under scale 1 / a: position of index i is fma(i - c, inv_a, c)
struct WalkAxis {
  float inv_a, c;
  int o;           // the tile's origin
  const float* f;  // fractions of the tile's samples (with tables)
};

// walks the sources of two lines in order, each loaded one step before it is used (the uniform branches
// of a walk keep the compiler from moving a load ahead of the one that decides about it)
template <int ES, int LINE2, bool FT>
struct Sources {
  const unsigned char* line;
  const WalkAxis& x;
  int k;       // the next source (tile frame)
  float kc;    // its index - c
  float f, r[2];
  __device__ __forceinline__ Sources(const unsigned char* l, const WalkAxis& ax, int first)
      : line(l), x(ax), k(first), kc((float)(ax.o + first) - ax.c) {
    load();
  }
  // (the load after a line's last source reads the padding behind it and is not used)
  __device__ __forceinline__ void load() {
    if constexpr (FT) f = x.f[k];
#pragma unroll
    for (int h = 0; h < 2; ++h) r[h] = *reinterpret_cast<const float*>(line + k * ES + h * LINE2);
  }
  // the next source, of the group of output u: v += (1 - f) r, b += f r with f = its position - u, from
  // the table x.f (FT) or the running index
  __device__ __forceinline__ void take(float u, float (&v)[2], float (&b)[2]) {
    const float ft = FT ? f : fmaf(kc, x.inv_a, x.c) - u, g = 1.f - ft;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      v[h] = fmaf(g, r[h], v[h]);
      b[h] = fmaf(ft, r[h], b[h]);
    }
    ++k;
    kc += 1.f;
    load();
  }
};

// the transposed interpolation of one strip of two lines, outputs u0 .. (ES bytes between samples, the
// second line LINE2 bytes after the first), groups of at most GM sources. st = (., ., first source of the
// group before the strip | its count << 8 | (groups of 3) << 16, (groups of >= 1) | (groups of >= 2) << 16);
// sink(i, v) takes output i of both lines, last = what the last group adds to the output after them
template <int GM, int ES, int LINE2, int STRIP, bool FT, class Sink>
__device__ __forceinline__ void adjoint_walk(const unsigned char* line, const WalkAxis& x, int u0, int4 st,
                                             float (&last)[2], Sink sink) {
  const int z = warp_uniform(st.z), w = warp_uniform(st.w);
  const int before = (z >> 8) & 3;
  Sources<ES, LINE2, FT> src(line, x, z & 0xff);
  const float uf = (float)(x.o + u0);
  float prev[2] = {0.f, 0.f};
  {
    float unused[2] = {0.f, 0.f};
#pragma unroll
    for (int l = 0; l < GM; ++l)
      if (before > l) src.take(uf - 1.f, unused, prev);
  }
#pragma unroll
  for (int i = 0; i < STRIP; ++i) {
    float v[2] = {prev[0], prev[1]};
    prev[0] = prev[1] = 0.f;
    const float u = uf + (float)i;
    if (w & (1 << i)) src.take(u, v, prev);
    if (GM > 1 && (w & (1 << (16 + i)))) src.take(u, v, prev);
    if (GM > 2 && (z & (1 << (16 + i)))) src.take(u, v, prev);
    sink(i, v);
  }
  last[0] = prev[0];
  last[1] = prev[1];
}

template <int TILE, bool QUAD, bool FT>
__global__ void __launch_bounds__(WalkShape<TILE, QUAD>::TPB, WalkShape<TILE, QUAD>::MIN_BLOCKS)
    k_mono_walk(const MonoArgs a) {
  using SH = WalkShape<TILE, QUAD>;
  constexpr int M = QUAD ? 2 * TILE : TILE;
  constexpr int TPB = SH::TPB, STRIP = SH::STRIP, CG = SH::CG, LDP = SH::LDP, LDR = SH::LDR, HALF = TILE / 2;
  extern __shared__ __align__(16) unsigned char smem[];
  float* Pp = reinterpret_cast<float*>(smem);                  // (TILE + 2)^2, border of zeros or halo
  float* R = reinterpret_cast<float*>(smem + SH::P_BYTES);     // TILE x LDR
  unsigned char* Tb = smem + SH::P_BYTES + SH::R_BYTES;
  float* T = reinterpret_cast<float*>(Tb);                     // TILE x LDR: r S_j, column TILE its halo
  double* red = reinterpret_cast<double*>(Tb + SH::R_BYTES);
  double* slots = red + 2 * (TPB / 32 + 1);                    // 4 x 2 CTA sums (used in rank 0)
  float* s_inv = reinterpret_cast<float*>(Tb + SH::R_BYTES + SH::RED_BYTES);
  float* s_a = s_inv + kMonoMaxJ;
  float* s_w = s_a + kMonoMaxJ;
  float* h_col = s_w + kMonoMaxJ;                              // QUAD: received halo column, row, corner
  float* h_row = h_col + TILE;
  float* h_cor = h_row + TILE;
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(h_cor + 4);
  unsigned char* tabs = smem + SH::FIXED;                      // [wavelength][axis: rows, columns]

  const int tid = threadIdx.x, lane = tid & 31, warp = warp_uniform(tid >> 5);
  const int l0 = (warp % CG) * 32 + lane;      // the two lines of this thread: l0 and l0 + HALF
  const int strip = warp / CG, u0 = strip * STRIP;
  const int rank = QUAD ? (int)cluster_ctarank() : 0;
  const int oy = QUAD ? (rank >> 1) * TILE : 0, ox = QUAD ? (rank & 1) * TILE : 0;
  const float c = 0.5f * (float)M;
  const int n = QUAD ? blockIdx.x / 4 : blockIdx.x;
  const float* bn = a.b + (size_t)n * M * M;
  float* xn = a.x + (size_t)n * M * M;
  double* rs = a.resid && rank == 0 ? a.resid + (size_t)n * (a.k + 1) : nullptr;
  // fractions (FT) and strip records of wavelength j on an axis (0: rows, 1: columns)
  float* s_f = reinterpret_cast<float*>(tabs + (size_t)a.J * SH::TAB);
  auto tab_f = [&](int j, int axis) { return FT ? s_f + (j * SH::AXES + (QUAD ? axis : 0)) * TILE : nullptr; };
  auto tab_s = [&](int j, int axis) {
    return reinterpret_cast<const int4*>(tabs + (size_t)j * SH::TAB + (QUAD ? axis : 0) * SH::TAB_S);
  };

  auto sum2 = [&](double x, double y, double& gx, double& gy) {
    if constexpr (!QUAD) {
      block_sum2<TPB>(x, y, red, gx, gy);
    } else {
      double cx, cy;
      block_sum2<TPB>(x, y, red, cx, cy);
      const uint32_t slots_s = smem_addr(slots);
      cluster_sync_all();  // the slots are free (every rank read the previous sums)
      if (tid == 0) {
        st_cluster_f64(map_rank(slots_s + 16u * rank, 0), cx);
        st_cluster_f64(map_rank(slots_s + 16u * rank + 8u, 0), cy);
      }
      cluster_sync_all();
      gx = gy = 0.0;
      for (int q = 0; q < 4; ++q) {
        gx += ld_cluster_f64(map_rank(slots_s + 16u * q, 0));
        gy += ld_cluster_f64(map_rank(slots_s + 16u * q + 8u, 0));
      }
    }
  };

  // the records of every wavelength: one warp per 32 samples of a (wavelength, axis), which are 32
  // consecutive outputs of C and groups of C^T
  auto build = [&]() {
    for (int e = warp; e < a.J * SH::AXES * (TILE / 32); e += TPB / 32) {
      const int ja = e / (TILE / 32), y = (e % (TILE / 32)) * 32 + lane;
      const int j = ja / SH::AXES, axis = ja % SH::AXES, o = axis ? ox : oy;
      const float inv_a = s_inv[j], sa = s_a[j];
      unsigned char* base = tabs + (size_t)j * SH::TAB;
      // C: sample row of output o + y; outside the grid the row before the tile's first
      int i0, ip;
      float f, fp;
      interp_at(o + y, c, inv_a, M, i0, f);
      interp_at(o + y - 1, c, inv_a, M, ip, fp);
      if (i0 == -1 && f == 0.f) i0 = o - 1;
      if (ip == -1 && fp == 0.f) ip = o - 1;
      if constexpr (FT) tab_f(j, axis)[y] = f;
      const bool head = y % STRIP == 0;
      const unsigned adv = __ballot_sync(0xffffffffu, head || i0 != ip);
      const unsigned both = __ballot_sync(0xffffffffu, head || (i0 != ip && i0 != ip + 1));
      // C^T: group u is the run of sources with sample position in [u, u + 1), found among the six
      // about c + (u - c) a_j; a run starts where the ones before it end. The first source at or after
      // the group before this warp's 32 by a search (the same in all lanes).
      auto at = [&](int src) { return fmaf((float)src - c, inv_a, c); };
      auto count = [&](int u) {
        const int lo = (int)fminf(fmaxf(ceilf(fmaf((float)u - c, sa, c)), (float)o), (float)(o + TILE)) - 1;
        int cnt = 0;
#pragma unroll
        for (int l = 0; l < 6; ++l) {
          const float t = at(lo + l);
          cnt += (lo + l >= o && lo + l < o + TILE && t >= (float)u && t < (float)(u + 1)) ? 1 : 0;
        }
        return cnt;
      };
      const int ub = o + y - lane - 1;  // the group before the warp's first
      int sb = (int)fminf(fmaxf(ceilf(fmaf((float)ub - c, sa, c)), (float)o), (float)(o + TILE));
      while (sb > o && at(sb - 1) >= (float)ub) --sb;
      while (sb < o + TILE && !(at(sb) >= (float)ub)) ++sb;
      const int cb = count(ub), cnt = count(o + y);
      int run = cnt;  // inclusive prefix sum
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, run, d);
        if (lane >= d) run += v;
      }
      const int s0 = sb - o + cb + run - cnt;  // this group's first source
      const int cp = __shfl_up_sync(0xffffffffu, cnt, 1), before = lane == 0 ? cb : cp;
      if (QUAD && axis == 0) {
        unsigned char* gs = base + 2 * SH::TAB_S;
        gs[y + 1] = (unsigned char)s0;
        if (y == 0) gs[0] = (unsigned char)(s0 - before);
        if (y == TILE - 1) gs[TILE + 1] = (unsigned char)(s0 + cnt);
      }
      const unsigned ge1 = __ballot_sync(0xffffffffu, cnt >= 1), ge2 = __ballot_sync(0xffffffffu, cnt >= 2);
      const unsigned ge3 = __ballot_sync(0xffffffffu, cnt >= 3);
      if (head) {
        const int sh = lane & 16;
        reinterpret_cast<int4*>(base + axis * SH::TAB_S)[y / STRIP] = make_int4(
            i0 + 1 - o, (int)(((adv >> sh) & 0xffffu) | ((both >> sh) << 16)),
            (int)((unsigned)(s0 - before) | ((unsigned)before << 8) | ((ge3 >> sh) << 16)),
            (int)(((ge1 >> sh) & 0xffffu) | ((ge2 >> sh) << 16)));
      }
    }
  };

  float ex = 0.f, hx[2] = {0.f, 0.f};  // QUAD: this thread's share of the halo column and row

  // C^T v for the own pixels into acc (two columns x STRIP rows), v in R
  auto adjoint = [&](float (&acc)[2][STRIP]) {
#pragma unroll
    for (int i = 0; i < STRIP; ++i) acc[0][i] = acc[1][i] = 0.f;
    ex = hx[0] = hx[1] = 0.f;
    for (int j = 0; j < a.J; ++j) {
      const float wj = s_w[j], aj = s_a[j], inv_a = s_inv[j];
      // the largest group of scale a holds ceil(a) sources (one for a <= 1); a margin covers the
      // rounding of the sample positions
      const int gm = (aj == 1.f || aj < 0.999f) ? 1 : aj < 1.999f ? 2 : 3;
      // pass 1: T(y, v) = sum_x S_j[x, v] R(y, x)
      {
        const unsigned char* line = reinterpret_cast<const unsigned char*>(R + l0 * LDR);
        const WalkAxis x{inv_a, c, ox, tab_f(j, 1)};
        const int4 st = tab_s(j, 1)[strip];
        float* t0 = T + l0 * LDR + u0;
        float last[2];
        auto sink = [&](int i, const float (&v)[2]) {
          t0[i] = v[0];
          t0[HALF * LDR + i] = v[1];
        };
        if (gm == 2) adjoint_walk<2, 4, 4 * HALF * LDR, STRIP, FT>(line, x, u0, st, last, sink);
        else if (gm == 1) adjoint_walk<1, 4, 4 * HALF * LDR, STRIP, FT>(line, x, u0, st, last, sink);
        else adjoint_walk<3, 4, 4 * HALF * LDR, STRIP, FT>(line, x, u0, st, last, sink);
        if (QUAD && u0 == TILE - STRIP) {
          t0[STRIP] = last[0];
          t0[HALF * LDR + STRIP] = last[1];
        }
      }
      __syncthreads();  // T is complete
      // pass 2: acc(u, v) += w_j sum_y S_j[y, u] T(y, v)
      {
        const unsigned char* line = reinterpret_cast<const unsigned char*>(T + l0);
        const WalkAxis x{inv_a, c, oy, tab_f(j, 0)};
        const int4 st = tab_s(j, 0)[strip];
        float last[2];
        auto sink = [&](int i, const float (&v)[2]) {
          acc[0][i] = fmaf(wj, v[0], acc[0][i]);
          acc[1][i] = fmaf(wj, v[1], acc[1][i]);
        };
        if (gm == 2) adjoint_walk<2, 4 * LDR, 4 * HALF, STRIP, FT>(line, x, u0, st, last, sink);
        else if (gm == 1) adjoint_walk<1, 4 * LDR, 4 * HALF, STRIP, FT>(line, x, u0, st, last, sink);
        else adjoint_walk<3, 4 * LDR, 4 * HALF, STRIP, FT>(line, x, u0, st, last, sink);
        if constexpr (QUAD) {
          if (u0 == TILE - STRIP) {
            hx[0] = fmaf(wj, last[0], hx[0]);
            hx[1] = fmaf(wj, last[1], hx[1]);
          }
          if ((rank & 1) == 0 && tid <= TILE) {  // the halo column (v = TILE), output u = tid
            const unsigned char* gs = reinterpret_cast<const unsigned char*>(tab_s(j, 0)) + 2 * SH::TAB_S;
            const int sb = gs[tid], s0 = gs[tid + 1], s1 = tid < TILE ? gs[tid + 2] : s0;
            const float u = (float)(oy + tid);
            float v = 0.f;
            for (int q = sb; q < s1; ++q) {  // group u - 1 with f, group u with 1 - f
              const float t = fmaf((float)(oy + q) - c, inv_a, c);
              v = fmaf(q < s0 ? t - (u - 1.f) : 1.f - (t - u), T[q * LDR + TILE], v);
            }
            ex = fmaf(wj, v, ex);
          }
        }
      }
      __syncthreads();  // T is free
    }
    if constexpr (QUAD) {
      // halo shares to their owners: the column to the right, the row below, the corner across
      if ((rank & 1) == 0 && tid <= TILE) {
        if (tid < TILE) st_cluster_f32(map_rank(smem_addr(h_col + tid), (unsigned)(rank + 1)), ex);
        else if (rank == 0) st_cluster_f32(map_rank(smem_addr(h_cor), 3u), ex);
      }
      if (rank < 2 && u0 == TILE - STRIP) {
        st_cluster_f32(map_rank(smem_addr(h_row + l0), (unsigned)(rank + 2)), hx[0]);
        st_cluster_f32(map_rank(smem_addr(h_row + l0 + HALF), (unsigned)(rank + 2)), hx[1]);
      }
      cluster_sync_all();
      if (rank >= 2 && u0 == 0) {
        acc[0][0] += h_row[l0];
        acc[1][0] += h_row[l0 + HALF];
      }
      if ((rank & 1) && l0 == 0) {
#pragma unroll
        for (int i = 0; i < STRIP; ++i) acc[0][i] += h_col[u0 + i];
        if (rank == 3 && u0 == 0) acc[0][0] += h_cor[0];
      }
    }
  };

  // C p for the own pixels into acc, p in Pp
  auto forward = [&](float (&acc)[2][STRIP]) {
#pragma unroll
    for (int i = 0; i < STRIP; ++i) acc[0][i] = acc[1][i] = 0.f;
    for (int j = 0; j < a.J; ++j) {
      const float inv_a = s_inv[j], wj = s_w[j];
      const bool inside = FT || inv_a <= 1.f;  // no sample leaves the grid
      const int4 st = tab_s(j, 0)[strip];
      const unsigned char* q[2];
      const int mask = warp_uniform(st.y), x = warp_uniform(st.x);
      int off = (x - 1) * (LDP * 4);  // of row i0 - 1, i0 the sample row
      float yc = (float)(oy + u0) - c, i0f = (float)(oy + x - 2);
      float fx[2], gx[2], top[2] = {0.f, 0.f}, bot[2] = {0.f, 0.f}, nx[2][2] = {};
      const float4* f4 = reinterpret_cast<const float4*>(tab_f(j, 0) + (FT ? u0 : 0));
      float4 fr = make_float4(0.f, 0.f, 0.f, 0.f);
      // the two columns' samples; w_j goes into their weights
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        int x0;
        interp_at(ox + l0 + h * HALF, c, inv_a, M, x0, fx[h]);
        gx[h] = wj * (1.f - fx[h]);
        if (x0 == -1 && fx[h] == 0.f) gx[h] = 0.f, x0 = ox - 1;  // outside the grid: no weight
        fx[h] *= wj;
        q[h] = reinterpret_cast<const unsigned char*>(Pp + (x0 + 1 - ox));
      }
#pragma unroll
      for (int i = 0; i < STRIP; ++i) {
        if (mask & (1 << i)) {
          off += LDP * 4;
          i0f += 1.f;
          top[0] = bot[0];
          top[1] = bot[1];
          if (mask & (1 << (16 + i))) {
            if (i > 0) {  // i0 advanced by more than one: its row from the samples
              int ia, ib;
              float fa;
              interp_at(oy + u0 + i, c, inv_a, M, ia, fa);
              if (ia == -1 && fa == 0.f) ia = oy - 1;
              interp_at(oy + u0 + i - 1, c, inv_a, M, ib, fa);
              if (ib == -1 && fa == 0.f) ib = oy - 1;
              off += warp_uniform((ia - ib - 1) * LDP * 4);
              i0f += (float)(ia - ib - 1);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const float* p = reinterpret_cast<const float*>(q[h] + off);
              top[h] = fmaf(fx[h], p[1], gx[h] * p[0]);
              nx[h][0] = p[LDP];
              nx[h][1] = p[LDP + 1];
            }
          }
          // the row after next is loaded one step ahead of its use (past the tile's last row it reads
          // what lies behind p and is not used)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float* p = reinterpret_cast<const float*>(q[h] + off) + 2 * LDP;
            bot[h] = fmaf(fx[h], nx[h][1], gx[h] * nx[h][0]);
            nx[h][0] = p[0];
            nx[h][1] = p[1];
          }
        }
        if (FT && i % 4 == 0) fr = f4[i / 4];
        float f = FT ? (i % 4 == 0 ? fr.x : i % 4 == 1 ? fr.y : i % 4 == 2 ? fr.z : fr.w)
                     : fmaf(yc + (float)i, inv_a, c) - i0f;
        if (!inside) {
          int ia;
          interp_at(oy + u0 + i, c, inv_a, M, ia, f);  // 0 outside the grid (the zero row before the tile's)
        }
        const float g = 1.f - f;
#pragma unroll
        for (int h = 0; h < 2; ++h) acc[h][i] = fmaf(f, bot[h], fmaf(g, top[h], acc[h][i]));
      }
    }
  };

  // ---- start: spectrum to shared memory, zero border of p, r = b, x = 0
  for (int i = tid; i < a.J; i += TPB) {
    s_inv[i] = a.inv_a[i];
    s_a[i] = a.a[i];
    s_w[i] = a.w[i];
  }
  for (int i = tid; i < LDP * LDP; i += TPB) Pp[i] = 0.f;
  if (warp == 0) tmem_alloc(smem_addr(s_tmem), SH::TMEM_COLS);
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  const uint32_t tx = *s_tmem + ((uint32_t)(32 * (warp % 4)) << 16) + (uint32_t)(warp / 4 * 2 * STRIP);
  static_assert(STRIP == 16, "x: one 16-column access per column of pixels");
  float acc[2][STRIP];
  float rr = 0.f;  // per-thread partial sums in FP32, CTA sums in FP64
#pragma unroll
  for (int i = 0; i < STRIP; ++i)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float v = bn[(size_t)(oy + u0 + i) * M + ox + l0 + h * HALF];
      R[(u0 + i) * LDR + l0 + h * HALF] = v;
      rr = fmaf(v, v, rr);
      acc[h][i] = 0.f;
    }
#pragma unroll
  for (int h = 0; h < 2; ++h) tmem_st16(tx + 16 * h, acc[h]);  // x = 0
  tmem_wait_st();
  if constexpr (QUAD) cluster_sync_all();  // every rank's p border is zero before a neighbour writes its halo
  else __syncthreads();
  build();
  __syncthreads();
  // p <- acc + beta p on the own pixels (first: p <- acc), and its halo copies in the other quadrants
  auto store_p = [&](float beta, bool first) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int i = 0; i < STRIP; ++i) {
        float* q = Pp + (u0 + i + 1) * LDP + l0 + h * HALF + 1;
        const float v = first ? acc[h][i] : fmaf(beta, *q, acc[h][i]);
        *q = v;
        if constexpr (QUAD) {
          const bool r0 = u0 + i == 0 && rank >= 2, c0 = l0 + h * HALF == 0 && (rank & 1);
          const int col = l0 + h * HALF, row = u0 + i;
          if (r0) st_cluster_f32(map_rank(smem_addr(Pp + (TILE + 1) * LDP + col + 1), (unsigned)(rank - 2)), v);
          if (c0) st_cluster_f32(map_rank(smem_addr(Pp + (row + 1) * LDP + TILE + 1), (unsigned)(rank - 1)), v);
          if (r0 && c0) st_cluster_f32(map_rank(smem_addr(Pp + (TILE + 1) * LDP + TILE + 1), 0u), v);
        }
      }
    if constexpr (QUAD) cluster_sync_all();
    else __syncthreads();
  };
  adjoint(acc);  // s_0 = C^T b
  double gamma = 0.0, rr_all = 0.0;
  auto norm = [&]() {
    float s = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int i = 0; i < STRIP; ++i) s = fmaf(acc[h][i], acc[h][i], s);
    return s;
  };
  sum2(norm(), rr, gamma, rr_all);
  if (rs && tid == 0) rs[0] = sqrt(rr_all);
  store_p(0.f, true);

  for (int it = 0; it < a.k; ++it) {
    if (!(gamma > 0.0)) {  // C^T r = 0: x is the least-squares solution already
      if (rs && tid == 0) rs[it + 1] = sqrt(rr_all);
      continue;
    }
    forward(acc);  // q = C p
    double qq = 0.0, unused;
    sum2(norm(), 0.0, qq, unused);
    if (!(qq > 0.0)) {
      if (rs && tid == 0) rs[it + 1] = sqrt(rr_all);
      continue;
    }
    const float alpha = (float)(gamma / qq);
    rr = 0.f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float xk[STRIP];
      tmem_ld16(tx + 16 * h, xk);
      tmem_wait_ld();
#pragma unroll
      for (int i = 0; i < STRIP; ++i) {
        const int y = u0 + i, x = l0 + h * HALF;
        xk[i] = fmaf(alpha, Pp[(y + 1) * LDP + x + 1], xk[i]);
        const float r = fmaf(-alpha, acc[h][i], R[y * LDR + x]);
        R[y * LDR + x] = r;
        rr = fmaf(r, r, rr);
      }
      tmem_st16(tx + 16 * h, xk);
    }
    tmem_wait_st();
    __syncthreads();
    adjoint(acc);  // s = C^T r
    double gnew = 0.0;
    sum2(norm(), rr, gnew, rr_all);
    if (rs && tid == 0) rs[it + 1] = sqrt(rr_all);
    const float beta = (float)(gnew / gamma);
    gamma = gnew;
    store_p(beta, false);
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float xk[STRIP];
    tmem_ld16(tx + 16 * h, xk);
    tmem_wait_ld();
#pragma unroll
    for (int i = 0; i < STRIP; ++i)
      xn[(size_t)(oy + u0 + i) * M + ox + l0 + h * HALF] = a.clamp ? fmaxf(xk[i], 0.f) : xk[i];
  }
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  if (warp == 0) tmem_dealloc(*s_tmem, SH::TMEM_COLS);
  if constexpr (QUAD) cluster_sync_all();  // no rank exits while another may still read its shared memory
}

template <int TILE, bool QUAD, bool FT>
cudaError_t launch_walk_t(const MonoArgs& a, cudaStream_t s) {
  using SH = WalkShape<TILE, QUAD>;
  auto kern = k_mono_walk<TILE, QUAD, FT>;
  const size_t bytes = SH::bytes(a.J, FT);
  // (the largest any call takes, so that calls of several threads never lower it under one another)
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::LIMIT);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(QUAD ? a.N * 4 : a.N));
  cfg.blockDim = dim3(SH::TPB);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = QUAD ? 4 : 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

template <int TILE, bool QUAD>
cudaError_t launch_walk(const MonoArgs& a, cudaStream_t s) {
  using SH = WalkShape<TILE, QUAD>;
  return SH::bytes(a.J, true) <= SH::LIMIT ? launch_walk_t<TILE, QUAD, true>(a, s)
                                           : launch_walk_t<TILE, QUAD, false>(a, s);
}

template <int M>
cudaError_t launch_mono_t(const MonoArgs& a, cudaStream_t s) {
  using SH = MonoShape<M>;
  auto kern = k_mono_cgls<M>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::BYTES);
  if (e != cudaSuccess) return e;
  kern<<<a.N, SH::TPB, SH::BYTES, s>>>(a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_mono(const MonoArgs& a, cudaStream_t s) {
  if (a.N == 0) return cudaSuccess;
  switch (a.M) {
    case 8: return launch_mono_t<8>(a, s);
    case 16: return launch_mono_t<16>(a, s);
    case 32: return launch_mono_t<32>(a, s);
    case 64: return launch_walk<64, false>(a, s);
    case 128: return launch_walk<128, false>(a, s);
    case 256: return launch_walk<128, true>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ptycho
