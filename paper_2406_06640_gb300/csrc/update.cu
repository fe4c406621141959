// Atomic-free simultaneous object / probe update of the data-parallel engine.
//
//   N_O(r) = sum_n c_n(r - r_n),            c_n = sum_k conj(P_k) dpsi_{n,k}
//   D_O(r) = sum_n sum_k |P_k(r - r_n)|^2
//   O     += beta_O N_O / (D_O + delta_O max D_O)           (pixels with D_O = 0 unchanged)
//   N_P,k  = sum_n conj(o_n) dpsi_{n,k},   D_P = sum_n |o_n|^2
//   P_k   += beta_P N_P,k / (D_P + delta_P max D_P)         (pixels with D_P = 0 unchanged)
//
// The paper's engines (ePIE, rPIE, DM, LSQML; Sec. 1 and Sec. 4.5) all move
// the object and probe with conj(P) dpsi / |P|^2 style steps; this is the
// simultaneous form of that step. Every sum runs in a fixed order (per-tile
// position lists in increasing n, per-slot partials in slot order), so an
// iteration is bitwise reproducible.
//
// The intensity error of Sec. 4.2, E = sqrt(sum (Ihat - I)^2 / sum I^2), is
// finished here in FP64 from the per-slot partials of the fused kernel.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "constraint.cuh"
#include "engine.h"
#include "cluster.cuh"
#include "fft.cuh"

namespace ptycho {

// ------------------------------------------------------------------ plan-time sums: sum I, sum I^2, bad values
__global__ void k_intensity_sums(const float* __restrict__ I, size_t count, double* __restrict__ partials) {
  __shared__ double s1[256], s2[256], s3[256];
  double a = 0.0, b = 0.0, bad = 0.0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
    const float v = I[i];
    if (!isfinite(v)) bad += 1e30;
    else if (v < 0.f) bad += 1.0;
    else {
      a += (double)v;
      b += (double)v * (double)v;
    }
  }
  s1[threadIdx.x] = a;
  s2[threadIdx.x] = b;
  s3[threadIdx.x] = bad;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      s1[threadIdx.x] += s1[threadIdx.x + w];
      s2[threadIdx.x] += s2[threadIdx.x + w];
      s3[threadIdx.x] += s3[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    partials[3 * blockIdx.x + 0] = s1[0];
    partials[3 * blockIdx.x + 1] = s2[0];
    partials[3 * blockIdx.x + 2] = s3[0];
  }
}

__global__ void k_finish_sums(const double* __restrict__ partials, int nblocks, double* __restrict__ out) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    double a = 0.0, b = 0.0, c = 0.0;
    for (int i = 0; i < nblocks; ++i) {
      a += partials[3 * i];
      b += partials[3 * i + 1];
      c += partials[3 * i + 2];
    }
    out[0] = a;
    out[1] = b;
    out[2] = c;
  }
}

__global__ void k_sqrt(const float* __restrict__ I, float* __restrict__ out, size_t count) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
    out[i] = sqrtf(I[i]);
}

cudaError_t launch_sqrt(const float* I, float* out, size_t count, cudaStream_t s) {
  const int nb = (int)std::min<size_t>(4096, (count + 255) / 256);
  k_sqrt<<<nb, 256, 0, s>>>(I, out, count);
  return cudaGetLastError();
}

cudaError_t launch_intensity_sums(const float* I, size_t count, double* partials, int nblocks, cudaStream_t s) {
  k_intensity_sums<<<nblocks, 256, 0, s>>>(I, count, partials);
  return cudaGetLastError();
}
cudaError_t launch_finish_sums(const double* partials, int nblocks, double* out, cudaStream_t s) {
  k_finish_sums<<<1, 32, 0, s>>>(partials, nblocks, out);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ |P|^2 map
// sum_k |P_k|^2 per probe pixel, and the maxima of D_O and D_P cleared for this update's gather (staged and
// queued plans; the fused kernels of single plans make both, probe_map)
__global__ void __launch_bounds__(256) k_p2(const UpdateArgs u) {
  const int MM = u.M * u.M;
  const int p = blockIdx.x * 256 + threadIdx.x;
  if (p < 2) u.dmax[p] = 0;
  if (p >= MM) return;
  float s = 0.f;
  for (int k = 0; k < u.K; ++k) s += cabs2(u.P[(size_t)k * MM + p]);
  u.p2[p] = s;
}

// ------------------------------------------------------------------ pc-DM probe partials
// After the object step: slot s sums, over positions n = s, s + slots, ..., conj(o'_n)(psi_n,k - P_k o'_n)
// into pacc[s][k] and |o'_n|^2 into dacc[s] (o'_n: the new object under position n). Inside a
// complex-constraint window the states first move with their boxes, psi_n,k += P_k (o'_n - o''_n),
// o''_n the object before the constraint. grid (ceil(M^2 / 512), slots); one thread per two neighbouring
// probe pixels and every mode (KT >= K), so o'_n is read once. Bound by reading the state (N K M^2 complex):
// 16-byte loads, two positions in flight
template <int KT>
__global__ void __launch_bounds__(256) k_dm_probe_partials(const UpdateArgs u) {
  const int MM = u.M * u.M;
  const int p = (blockIdx.x * 256 + threadIdx.x) * 2;
  if (p >= MM) return;
  const int s = blockIdx.y, K = u.K;
  const int row = p / u.M, col = p % u.M;
  float2 pk[KT][2], acc[KT][2];
#pragma unroll
  for (int k = 0; k < KT; ++k)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      pk[k][h] = k < K ? u.P[(size_t)k * MM + p + h] : make_float2(0.f, 0.f);
      acc[k][h] = make_float2(0.f, 0.f);
    }
  float d[2] = {0.f, 0.f};
#pragma unroll 2
  for (int n = s; n < u.N; n += u.slots) {
    const int2 r = u.pos[n];
    const size_t q = (size_t)(r.x + row) * u.obj_w + r.y + col;
    float4* ps = reinterpret_cast<float4*>(u.dm_psi + (size_t)n * K * MM + p);
    const float2 o[2] = {u.O[q], u.O[q + 1]};
    float4 st[KT];
#pragma unroll
    for (int k = 0; k < KT; ++k)
      if (k < K) st[k] = ps[(size_t)k * (MM / 2)];
    float2 dlt[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    if (u.dm_obj_prev) {
      dlt[0] = csub(o[0], u.dm_obj_prev[q]);
      dlt[1] = csub(o[1], u.dm_obj_prev[q + 1]);
    }
    d[0] += cabs2(o[0]);
    d[1] += cabs2(o[1]);
#pragma unroll
    for (int k = 0; k < KT; ++k)
      if (k < K) {
        float2 w[2] = {make_float2(st[k].x, st[k].y), make_float2(st[k].z, st[k].w)};
        if (u.dm_obj_prev) {
          w[0] = cadd(w[0], cmul(pk[k][0], dlt[0]));
          w[1] = cadd(w[1], cmul(pk[k][1], dlt[1]));
          ps[(size_t)k * (MM / 2)] = make_float4(w[0].x, w[0].y, w[1].x, w[1].y);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
          acc[k][h] = cadd(acc[k][h], cconjmul(o[h], csub(w[h], cmul(pk[k][h], o[h]))));
      }
  }
#pragma unroll
  for (int k = 0; k < KT; ++k)
    if (k < K)
      *reinterpret_cast<float4*>(const_cast<float2*>(u.pacc) + ((size_t)s * K + k) * MM + p) =
          make_float4(acc[k][0].x, acc[k][0].y, acc[k][1].x, acc[k][1].y);
  *reinterpret_cast<float2*>(const_cast<float*>(u.dacc) + (size_t)s * MM + p) = make_float2(d[0], d[1]);
}

static void launch_dm_probe_partials(const UpdateArgs& u, cudaStream_t s) {
  const dim3 grid((unsigned)((u.M * u.M / 2 + 255) / 256), (unsigned)u.slots);
  if (u.K == 1) k_dm_probe_partials<1><<<grid, 256, 0, s>>>(u);
  else if (u.K == 2) k_dm_probe_partials<2><<<grid, 256, 0, s>>>(u);
  else if (u.K <= 4) k_dm_probe_partials<4><<<grid, 256, 0, s>>>(u);
  else k_dm_probe_partials<8><<<grid, 256, 0, s>>>(u);
}

// ------------------------------------------------------------------ gather: N_O, D_O and N_P, D_P
// One launch sums both sides. A unit of work is 256 PX values, PX per thread: part of a 32 x 32 object tile
// (its positions' contributions and |P|^2 under their boxes), or probe pixels of one mode or of D_P (their
// per-slot partials). Every sum has a fixed order.
//   SPLIT = 8: a unit is a whole tile (PX = 4) shared by a cluster of eight blocks. Block `rank` takes terms
//     rank, rank + 8, ..., and the ranks' sums are added in rank order through distributed shared memory. For
//     long lists: a tile in the middle of a dense scan holds hundreds of positions.
//   SPLIT = 1: a unit is 8 rows of a tile (PX = 1) and one block, whose threads hold the eight sums themselves. For
//     short lists (mini-batches, small scans), where the blocks of a cluster would mostly start, meet and end.
// Both forms add the same terms in the same order, so their results are the same bits: eight sums of every eighth
// term, then those in order (a chain of all terms loses three bits more on a scan of hundreds).
// Bound by the latency of the term loads: four (SPLIT = 8) or eight positions of PX pixels and their |P|^2 in flight
// per thread. The line between the forms is 24 terms on average, where small scans cross: iterations of one mode,
// SPLIT = 8 against 1, 100 positions of 64^2: 31 / 33 us at 22 terms, 31 / 35 at 29, 31 / 37 at 49; of 128^2: 59 / 52
// at 18, 57 / 55 at 25, 54 / 58 at 45; 400 of 32^2: 43 / 41 at 7, 38 / 39 at 30, 35 / 47 at 86. Scans of more tiles
// than the GPU has blocks cross later (400 of 128^2: 159 / 131 at 12, 149 / 131 at 25, 133 / 133 at 65, 129 / 138
// at 96; 256^2 near 100). The probe side follows the object's form; with many slots and few probe pixels the split
// would be faster for short lists too (900 positions of 8^2: 38 / 46). (Clusters of 8-row bands: 104 us against 77 us
// for 900 positions of 128^2 on 640^2, most blocks of the border tiles being overhead.)
// The maxima of D_O and D_P are integer atomics on the float bits (non-negative: the order of the bits),
// so they do not depend on the order either.
template <int SPLIT>
__global__ void __launch_bounds__(256, 3) k_gather(const UpdateArgs u, int units_o) {
  static_assert(SPLIT == 1 || SPLIT == 8, "cluster size");
  constexpr int PX = SPLIT == 8 ? 4 : 1, VALUES = 256 * PX, BANDS = 4 / PX;  // units per tile
  constexpr int U = SPLIT == 8 ? 4 : 8;                                      // positions in flight
  constexpr int SUMS = 8 / SPLIT;                                            // of this thread, per value
  __shared__ float2 s_acc[SPLIT > 1 ? VALUES : 1];
  __shared__ float s_den[SPLIT > 1 ? VALUES : 1];
  const int unit = blockIdx.x / SPLIT, rank = SPLIT > 1 ? (int)cluster_ctarank() : 0;
  const int tid = threadIdx.x;
  const int M = u.M, MM = M * M;
  const bool obj = unit < units_o;
  const int tile = unit / BANDS, X0 = tile % u.tiles_x * kObjTile;
  const int Y0 = tile / u.tiles_x * kObjTile + unit % BANDS * (kObjTile / BANDS);
  const int pu = (MM + VALUES - 1) / VALUES, k = obj ? 0 : (unit - units_o) / pu;  // k == K: D_P
  const int P0 = obj ? 0 : (unit - units_o) % pu * VALUES;
  // output of value t of the unit (object: row-major in the tile part; 64 bits, an object may hold 2^31 pixels
  // and more), -1: outside
  auto output = [&](int t) -> long long {
    if (!obj) return P0 + t < MM ? P0 + t : -1;
    const int X = X0 + t % kObjTile, Y = Y0 + t / kObjTile;
    return X < u.obj_w && Y < u.obj_h ? (long long)Y * u.obj_w + X : -1;
  };
  float m = 0.f;
  auto store = [&](int t, float2 a, float d) {
    const long long at = output(t);
    if (at < 0) return;
    if (obj) {
      u.no_part[at] = a;
      u.do_part[at] = d;
      m = fmaxf(m, d);
    } else if (k < u.K) {
      u.np_sum[(size_t)k * MM + at] = a;
    } else {
      u.dp_sum[at] = d;
      m = fmaxf(m, d);
    }
  };
  constexpr int RPR = VALUES / SPLIT;  // values a rank finishes
  float2 acc[SUMS][PX];
  float den[SUMS][PX];
#pragma unroll
  for (int r = 0; r < SUMS; ++r)
#pragma unroll
    for (int i = 0; i < PX; ++i) {
      acc[r][i] = make_float2(0.f, 0.f);
      den[r][i] = 0.f;
    }
  if (obj) {
    const int s0 = u.tile_start[tile], s1 = u.tile_start[tile + 1];
    if (s0 == s1) {  // no position (the same in every rank)
      for (int t = tid; t < RPR; t += 256) store(rank * RPR + t, make_float2(0.f, 0.f), 0.f);
      return;
    }
    const int X = X0 + (tid & 31), Y = Y0 + (tid >> 5);
    for (int base = s0 + rank; base < s1; base += U * SPLIT) {
      float2 cv[U][PX];
      float dv[U][PX];
#pragma unroll
      for (int r = 0; r < U; ++r) {
        const int idx = base + r * SPLIT;
        const int4 ent = idx < s1 ? u.tile_pos[idx] : make_int4(0, 0, -(1 << 20), 0);  // (n, row, col)
        const int cx = X - ent.z;
        const bool inx = cx >= 0 && cx < M;
        const float2* cn = u.cn + (size_t)ent.x * MM;
#pragma unroll
        for (int i = 0; i < PX; ++i) {
          const int cy = Y + 8 * i - ent.y;
          const bool in = inx && cy >= 0 && cy < M;
          cv[r][i] = in ? cn[cy * M + cx] : make_float2(0.f, 0.f);
          dv[r][i] = in ? u.p2[cy * M + cx] : 0.f;
        }
      }
#pragma unroll
      for (int r = 0; r < U; ++r)
#pragma unroll
        for (int i = 0; i < PX; ++i) {
          acc[r % SUMS][i] = cadd(acc[r % SUMS][i], cv[r][i]);
          den[r % SUMS][i] += dv[r][i];
        }
    }
  } else if (k < u.K) {
    const float2* part[PX];  // (past the last pixel: that pixel again, not stored)
#pragma unroll
    for (int i = 0; i < PX; ++i) part[i] = u.pacc + (size_t)k * MM + min(P0 + tid + 256 * i, MM - 1);
    // rounds of eight partials, sixteen loads in flight: no branch between the loads of a round
    int s = 0;
#pragma unroll SPLIT == 1 ? 2 : 4
    for (; s + 8 <= u.slots; s += 8)
#pragma unroll
      for (int r = 0; r < SUMS; ++r)
#pragma unroll
        for (int i = 0; i < PX; ++i) acc[r][i] = cadd(acc[r][i], part[i][(size_t)(s + rank + r) * u.K * MM]);
#pragma unroll
    for (int r = 0; r < SUMS; ++r)
      if (s + rank + r < u.slots)
#pragma unroll
        for (int i = 0; i < PX; ++i) acc[r][i] = cadd(acc[r][i], part[i][(size_t)(s + rank + r) * u.K * MM]);
  } else {
    const float* part[PX];
#pragma unroll
    for (int i = 0; i < PX; ++i) part[i] = u.dacc + min(P0 + tid + 256 * i, MM - 1);
    int s = 0;
#pragma unroll SPLIT == 1 ? 2 : 4
    for (; s + 8 <= u.slots; s += 8)
#pragma unroll
      for (int r = 0; r < SUMS; ++r)
#pragma unroll
        for (int i = 0; i < PX; ++i) den[r][i] += part[i][(size_t)(s + rank + r) * MM];
#pragma unroll
    for (int r = 0; r < SUMS; ++r)
      if (s + rank + r < u.slots)
#pragma unroll
        for (int i = 0; i < PX; ++i) den[r][i] += part[i][(size_t)(s + rank + r) * MM];
  }
  // (thread tid's values are tid, tid + 256, ...: rows tid / 32 + 8 i of a tile)
  if constexpr (SPLIT == 1) {
    float2 a = make_float2(0.f, 0.f);
    float d = 0.f;
#pragma unroll
    for (int r = 0; r < SUMS; ++r) {
      a = cadd(a, acc[r][0]);
      d += den[r][0];
    }
    store(tid, a, d);
  } else {
#pragma unroll
    for (int i = 0; i < PX; ++i) {
      s_acc[tid + 256 * i] = acc[0][i];
      s_den[tid + 256 * i] = den[0][i];
    }
    cluster_sync_all();  // every rank's sums are complete
    if (tid < RPR) {
      const int t = rank * RPR + tid;
      const uint32_t oa = smem_addr(&s_acc[t]), od = smem_addr(&s_den[t]);
      float2 a = make_float2(0.f, 0.f);
      float d = 0.f;
#pragma unroll
      for (int q = 0; q < SPLIT; ++q) {
        a = cadd(a, ld_cluster_f2(map_rank(oa, (unsigned)q)));
        d += ld_cluster_f32(map_rank(od, (unsigned)q));
      }
      store(t, a, d);
    }
    cluster_sync_all();  // no rank exits while another may still read its sums
  }
  const int wm = __reduce_max_sync(0xffffffffu, __float_as_int(m));
  if ((tid & 31) == 0 && wm > 0) atomicMax(&u.dmax[obj ? 0 : 1], wm);
}

// E of run r into the ring, the run counter and (where there is one) the host-visible copy
__device__ __forceinline__ void finish_error(const UpdateArgs& u, double E, unsigned long long r) {
  u.errhist[r % kErrHistory] = E;
  *u.run_counter = r + 1;
  if (u.host) {
    u.host->err = E;
    u.host->run = r + 1;
  }
}

// ------------------------------------------------------------------ apply
// Blocks 0 .. rows - 1 (rows = obj_h or 0) take one object row each: O += beta N_O / (c_d D_O + c_max max
// D_O). CC: inside a complex-constraint window the row's prefix sums of the new object follow at once
// (constraint.cu's row pass, without another launch and read of O). The next pblocks blocks take 256 probe
// pixels of a mode each; the first of them also finishes the FP64 error.
template <bool CC>
__global__ void __launch_bounds__(256) k_apply(const UpdateArgs u, const ConstraintArgs c, int rows) {
  if ((int)blockIdx.x < rows) {
    const float floor_d = u.cmax_obj * __int_as_float(u.dmax[0]);
    const size_t row = (size_t)blockIdx.x * u.obj_w;
    auto step = [&](int x) {
      const size_t q = row + x;
      const float d = u.do_part[q];
      float2 o = u.O[q];
      if (d > 0.f) {
        const float w = u.beta_obj / fmaf(u.cd_obj, d, floor_d);
        const float2 num = u.no_part[q];
        o.x = fmaf(w, num.x, o.x);
        o.y = fmaf(w, num.y, o.y);
        u.O[q] = o;
      }
      return o;
    };
    if constexpr (CC) {
      constraint_row(c, (int)blockIdx.x, step);
    } else {
      for (int x = threadIdx.x; x < u.obj_w; x += 256) step(x);
    }
    return;
  }
  const int b = (int)blockIdx.x - rows, pb = u.probe_blocks;
  if (b == 0) {
    // error numerator: strided partial sums, then a fixed tree (every load in flight at once)
    __shared__ double s_e[256];
    double e = 0.0;
    for (int s = threadIdx.x; s < u.nerr; s += 256) e += u.errpart[s];
    s_e[threadIdx.x] = e;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
      if ((int)threadIdx.x < w) s_e[threadIdx.x] += s_e[threadIdx.x + w];
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      e = s_e[0];
      if (u.err_mode != 0) e += *u.err_acc;
      if (u.err_mode == 1) {
        *u.err_acc = e;
      } else {
        const unsigned long long r = *u.run_counter;
        finish_error(u, sqrt(e / u.errden), r);
        if (u.err_mode == 2) *u.err_acc = 0.0;
      }
    }
  }
  if (!u.update_probe) return;
  const int MM = u.M * u.M;
  const int k = b / pb, p = (b % pb) * 256 + threadIdx.x;
  if (p >= MM) return;
  const float d = u.dp_sum[p];
  if (d > 0.f) {
    const float w = u.beta_probe / fmaf(u.cd_probe, d, u.cmax_probe * __int_as_float(u.dmax[1]));
    const size_t q = (size_t)k * MM + p;
    const float2 num = u.np_sum[q];
    float2 pr = u.P[q];
    pr.x = fmaf(w, num.x, pr.x);
    pr.y = fmaf(w, num.y, pr.y);
    u.P[q] = pr;
  }
}

static cudaError_t launch_p2(const UpdateArgs& u, cudaStream_t s) {
  k_p2<<<u.probe_blocks, 256, 0, s>>>(u);
  return cudaGetLastError();
}

// object and / or probe side of the gather
static cudaError_t launch_gather(const UpdateArgs& u, bool obj, bool probe, cudaStream_t s) {
  const int px = u.split_lists ? 4 : 1, MM = u.M * u.M;
  const int units_o = obj ? u.tiles_x * u.tiles_y * (4 / px) : 0;
  const int units = units_o + (probe ? (MM + 256 * px - 1) / (256 * px) * (u.K + 1) : 0);
  if (!u.split_lists) {
    k_gather<1><<<units, 256, 0, s>>>(u, units_o);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)units * 8);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 8;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_gather<8>, u, units_o);
}

// object and / or probe side of the apply; c: the row pass of the complex constraint with the object side
static cudaError_t launch_apply(const UpdateArgs& u, const ConstraintArgs* c, bool obj, bool probe, cudaStream_t s) {
  const int rows = obj ? u.obj_h : 0;
  const int blocks = rows + (probe ? u.probe_blocks * u.K : 0);
  if (c && obj) k_apply<true><<<blocks, 256, 0, s>>>(u, *c, rows);
  else k_apply<false><<<blocks, 256, 0, s>>>(u, ConstraintArgs{}, rows);
  return cudaGetLastError();
}

cudaError_t launch_update_object(const UpdateArgs& u, const ConstraintArgs* c, bool with_p2, cudaStream_t s) {
  cudaError_t e = with_p2 ? launch_p2(u, s) : cudaSuccess;
  if (e == cudaSuccess) e = launch_gather(u, true, false, s);
  if (e == cudaSuccess) e = launch_apply(u, c, true, false, s);
  return e;
}

cudaError_t launch_update_probe_dm(const UpdateArgs& u, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  if (u.update_probe || u.dm_obj_prev) {
    launch_dm_probe_partials(u, s);
    e = cudaGetLastError();
    if (e == cudaSuccess && u.update_probe) e = launch_gather(u, false, true, s);
  }
  return e == cudaSuccess ? launch_apply(u, nullptr, false, true, s) : e;
}

cudaError_t launch_update(const UpdateArgs& u, const ConstraintArgs* c, bool with_p2, bool one_apply,
                          cudaStream_t s) {
  cudaError_t e = with_p2 ? launch_p2(u, s) : cudaSuccess;
  if (e == cudaSuccess) e = launch_gather(u, true, true, s);
  if (e == cudaSuccess) e = launch_apply(u, c, true, one_apply, s);
  if (e == cudaSuccess && !one_apply) e = launch_apply(u, nullptr, false, true, s);
  return e;
}

// E of a mini-batch iteration whose batches all added their partials to *err_acc (err_mode 1): the
// same sum as a last batch in err_mode 2, so the result does not depend on which form ran
__global__ void k_err_finish(const UpdateArgs u) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const double e = *u.err_acc;
  const unsigned long long r = *u.run_counter;
  finish_error(u, sqrt(e / u.errden), r);
  *u.err_acc = 0.0;
}

cudaError_t launch_err_finish(const UpdateArgs& u, cudaStream_t s) {
  if (!u.err_acc) return cudaErrorInvalidValue;
  k_err_finish<<<1, 32, 0, s>>>(u);
  return cudaGetLastError();
}

}  // namespace ptycho
