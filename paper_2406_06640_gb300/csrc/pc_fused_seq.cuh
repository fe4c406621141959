// Fused per-position pc-engine kernel, one CTA per scan position with the K probe modes in
// sequence. Everything between the object gather and the per-position contributions stays on
// the SM; no CTA exchanges data with another, so no cluster barrier and no distributed shared
// memory is involved, and every SM of the GPU takes positions.
//
//   o_n     = O[y_n : y_n + M, x_n : x_n + M]                (Fig. 1: object box) -> TMEM
//   pass 1, k = 0 .. K-1:
//     psi_k = P_k o_n                                         (Eq. 1, mixed-state modes)
//     Psi_k = centred FFT2 (far field, checkerboard trick)    (Eq. 1)
//           | IFFT2(FFT2(psi_k) H) (near field, Fresnel transfer function)
//     S    += |Psi_k|^2   (shared memory, each thread its own detector pixels)
//     Psi_{K-1} is kept in TMEM for pass 2
//   A^G     = sqrt(S) (x) g   (Eq. 6)  or  I_m = S (x) g  (Eq. 2), g of Eq. 7 normalised,
//             separable, zero padded
//   R       = sqrt(I_n) / (A^G + eps)  or  sqrt(I_n) / sqrt(I_m + eps^2)     (Fig. 1 box 1)
//   error  += sum (Ihat - I_n)^2 with Ihat = (A^G)^2 or I_m; SINGLE: I_n = (sqrt I_n)^2, of one read
//   pass 2, k = K-1, 0, 1, .. K-2 (mode K-1 from TMEM, the others propagated again):
//     Psi'_k = R Psi_k;  psi'_k = inverse propagation;  dpsi_k = psi'_k - P_k o_n
//     c_n   += conj(P_k) dpsi_k                 (TMEM; written once per position)
//     pacc_k += conj(o_n) dpsi_k, dacc += |o_n|^2   (per-slot partials: reductions at L2 into
//                                                  the slot's own array, each element always
//                                                  added to by the same thread, so in a fixed order)
//
// Cost against the cluster form: one more forward propagation for each of K - 1 modes (cheaper on
// this GPU than a store and a load of their detector fields through L2 and HBM), in exchange for no
// exchanges and all SMs busy. Persistent: CTA `slot` takes positions slot,
// slot + slots, ... and owns partial `slot`, so every sum is taken in a fixed order and the
// iteration is bitwise reproducible.
//
// Storage per CTA (M = 128): the FFT exchange buffer (132 KB of shared memory; the blur's
// intermediate aliases it), S and then R (66 KB), twiddles and taps; in tensor memory, per
// thread, its 32 object-box values and its 32 contribution accumulators (512 columns). Probe
// modes and partials are read from L2.
#pragma once
#include <cuda_runtime.h>

#include "cluster.cuh"
#include "engine.h"
#include "fft.cuh"
#include "fft3.cuh"
#include "fused_common.cuh"

namespace ptycho {

// L2 eviction policies: the per-slot probe partials are added to once per position and mode and
// must survive in L2 between those visits; the streamed data (sqrt I, c_n) must not push them out
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
// stores of the partials, which this kernel never reads back: no memory clobber, so the compiler may
// move later loads above them
__device__ __forceinline__ void st_part(float2* a, float2 v, uint64_t pol) {
  asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(a), "f"(v.x), "f"(v.y), "l"(pol));
}
__device__ __forceinline__ void st_part(float* a, float v, uint64_t pol) {
  asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(a), "f"(v), "l"(pol));
}
// fire-and-forget add at L2. A partial element is only ever added to by one thread of one CTA, and
// reductions of one thread to one address take effect in program order, so the sums keep their order
// (position by position) and stay bitwise reproducible; no register waits for the old value
__device__ __forceinline__ void red_hint(float2* a, float2 v, uint64_t pol) {
  asm volatile("red.global.add.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(a), "f"(v.x), "f"(v.y), "l"(pol));
}
__device__ __forceinline__ void red_hint(float* a, float v, uint64_t pol) {
  asm volatile("red.global.add.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(a), "f"(v), "l"(pol));
}
// bring `bytes` (a multiple of 16, 16-byte aligned) into L2 ahead of use
__device__ __forceinline__ void prefetch_l2(const void* a, uint32_t bytes, uint64_t pol) {
  asm volatile("cp.async.bulk.prefetch.L2.global.L2::cache_hint [%0], %1, %2;" ::"l"(a), "r"(bytes), "l"(pol)
               : "memory");
}

template <int M>
struct SeqShape {
  using TL = Tile<M>;
  static constexpr int V = M == 128 ? 2 : 1;  // lines per thread (M = 128: 512 threads x 2 lines)
  static constexpr int TR = TL::T / V;        // threads per CTA
  // TMEM holds the object box and the contributions (V E complex values each per thread) when the
  // CTA has whole groups of 4 warps; smaller tiles keep them in registers
  static constexpr bool TMEM = TR % 128 == 0;
  static constexpr int COLS_PER_THREAD = 4 * V * TL::E;
  static constexpr int TMEM_COLS = TMEM ? (TR / 128) * COLS_PER_THREAD : 0;
  static_assert(!TMEM || (TMEM_COLS >= 32 && TMEM_COLS <= 512 && (TMEM_COLS & (TMEM_COLS - 1)) == 0),
                "TMEM allocation must be a power of two in [32, 512] columns");
  static constexpr int MIN_BLOCKS = M == 64 ? 2 : 1;
};

template <int M>
struct SeqSmem {
  static constexpr int LD = M + 1;  // padded row stride of the f32 detector buffers
  static constexpr size_t kX = ExchangeBytes<M>::value;  // FFT exchange buffer
  static constexpr size_t kB = (size_t)M * LD * 4;         // one f32 detector buffer
  static constexpr size_t CBUF = ((kX > kB ? kX : kB) + 15) / 16 * 16;
  static constexpr size_t ZBUF = (kB + 15) / 16 * 16;      // S, then R
  static constexpr size_t TWT = ((size_t)Tile<M>::G * Tile<M>::LDW * 8 + 15) / 16 * 16;
  static constexpr size_t TW2 = (M >= 64 ? M : 0) * 8;  // second twiddles of fft3.cuh (Tile3::TW2)
  static constexpr size_t HQ = (size_t)M * 8;
  static constexpr size_t TAPS = 2 * kMaxTaps * 4 + 8;  // taps, TMEM address
  static constexpr size_t BYTES = CBUF + ZBUF + TWT + TW2 + HQ + TAPS;
  // queued launches: the current problem's arguments and the chunk index
  static constexpr size_t DESC = (sizeof(FusedArgs) + 15) / 16 * 16 + 16;
  static constexpr size_t bytes(int mode) { return BYTES + (mode == QUEUED ? DESC : 0); }
  static_assert(BYTES % 16 == 0 && BYTES + DESC <= 232448, "shared memory budget of one CTA");
  static_assert((size_t)SeqShape<M>::TR * 8 <= CBUF, "error reduction buffer");
};

template <int M, bool NEAR, int KH, int MODE>
__global__ void __launch_bounds__(SeqShape<M>::TR, SeqShape<M>::MIN_BLOCKS) pc_seq_kernel(const FusedArgs a_in) {
  using TL = Tile<M>;
  using SM = SeqSmem<M>;
  constexpr int E = TL::E, G = TL::G, LD = SM::LD;
  constexpr int V = SeqShape<M>::V, TR = SeqShape<M>::TR;
  constexpr int NB = E > 8 ? 8 : E;  // outputs per blur strip
  constexpr bool TM = SeqShape<M>::TMEM;
  extern __shared__ __align__(16) unsigned char smem[];
  float2* cbuf = reinterpret_cast<float2*>(smem);
  float* X = reinterpret_cast<float*>(smem);               // x-blurred S (aliases the exchange buffer)
  float* Z = reinterpret_cast<float*>(smem + SM::CBUF);    // S during pass 1, then R
  float2* s_tw = reinterpret_cast<float2*>(smem + SM::CBUF + SM::ZBUF);
  float2* s_tw2 = reinterpret_cast<float2*>(smem + SM::CBUF + SM::ZBUF + SM::TWT);
  float2* s_h = s_tw2 + SM::TW2 / 8;
  float* s_gx = reinterpret_cast<float*>(s_h + M);
  float* s_gy = s_gx + kMaxTaps;
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(s_gy + kMaxTaps);

  const int tid = threadIdx.x;
  const int K = a_in.K;
  const float inv_m2 = 1.0f / (float)(M * M);

  for (int i = tid; i < G * TL::LDW; i += TR) {
    const int t = i / TL::LDW, k2 = i % TL::LDW;
    s_tw[i] = k2 < E ? a_in.tw[(t * k2) % M] : make_float2(0.f, 0.f);
  }
  // M >= 64: the three-pass transform (fft3.cuh)
  constexpr bool F3 = M >= 64;
  if constexpr (F3)
    for (int i = tid; i < Tile3<M>::TW2; i += TR) s_tw2[i] = a_in.tw[Tile3<M>::tw2_exp(i)];
  // per problem: Fresnel factors and taps (between CTA barriers)
  auto setup = [&](const FusedArgs& a) {
    if constexpr (NEAR)
      for (int i = tid; i < M; i += TR) s_h[i] = a.hq[i];
    for (int i = tid; i < 2 * KH + 1; i += TR) {
      const int d = i - KH;
      const bool in = d >= -a.kh && d <= a.kh;
      s_gx[i] = in ? a.gx[d + a.kh] : 0.f;
      s_gy[i] = in ? a.gy[d + a.kh] : 0.f;
    }
  };
  if constexpr (MODE != QUEUED) setup(a_in);
  if constexpr (MODE != QUEUED) probe_map<M>(a_in, TR);
  int line[V], tp[V];
#pragma unroll
  for (int v = 0; v < V; ++v) {
    line[v] = (tid + v * TR) / G;
    tp[v] = (tid + v * TR) % G;
  }
  // ---- TMEM: columns [colO, colO + 2 V E) hold the object box, [colC, colC + 2 V E) the
  // contributions (and, between the passes, Psi_{K-1})
  uint32_t t_lane = 0, colO = 0, colC = 0;
  if constexpr (TM) {
    const int warp = tid / 32;
    if (warp == 0) tmem_alloc(smem_addr(s_tmem), SeqShape<M>::TMEM_COLS);
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    t_lane = *s_tmem + ((uint32_t)(32 * (warp % 4)) << 16);
    colO = (uint32_t)((warp / 4) * SeqShape<M>::COLS_PER_THREAD);
    colC = colO + 2 * V * E;
  } else {
    __syncthreads();
  }
  // register storage of the small tiles (unused with TMEM)
  float2 o_r[V][E], c_r[V][E], st_r[V][E];
  float err_s = 0.f, err_c = 0.f;  // compensated per-thread sum of (Ihat - I)^2
  const uint64_t keep = policy_evict_last(), stream = policy_evict_first();

  // one scan position n of problem a; `first` starts the probe partials pacc, dacc
  auto run_position = [&](const FusedArgs& a, int n, bool first, float2* pacc, float* dacc) {
    const int2 pn = a.pos[n];
    const float2* On = a.O + (size_t)pn.x * a.obj_w + pn.y;
    const float* Qn = a.sqrtI + (size_t)n * M * M;
    const float* In = a.I + (size_t)n * M * M;  // QUEUED, DM: the counts themselves, for the error
    // sqrt(I_n) is read once, by the modulus step (and I_n, by the error): start moving it into L2 now
    if (tid == 0) prefetch_l2(Qn, (uint32_t)(M * M * 4), stream);
    if (MODE != SINGLE && tid == 0) prefetch_l2(In, (uint32_t)(M * M * 4), stream);
    float2 v[V][E];

    // ---- the object box in ROW layout into TMEM (every load in flight at once)
#pragma unroll
    for (int q = 0; q < V; ++q)
#pragma unroll
      for (int j = 0; j < E; ++j) v[q][j] = On[(size_t)line[q] * a.obj_w + tp[q] + G * j];
    if constexpr (TM) {
#pragma unroll
      for (int q = 0; q < V; ++q)
#pragma unroll
        for (int h = 0; h < E / 8; ++h) {
          float pr[16];
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) {
            pr[2 * jj] = v[q][8 * h + jj].x;
            pr[2 * jj + 1] = v[q][8 * h + jj].y;
          }
          tmem_st16(t_lane + colO + 2 * (q * E + 8 * h), pr);
        }
      tmem_wait_st();
    } else {
#pragma unroll
      for (int q = 0; q < V; ++q)
#pragma unroll
        for (int j = 0; j < E; ++j) o_r[q][j] = v[q][j];
    }

    // pc-DM: the exit-wave state of this position, K x M x M
    float2* Sn = MODE == DM ? a.psi + (size_t)n * K * M * M : nullptr;
    const bool dm_init = MODE == DM && a.dm_init;
    // ---- exit wave P_k o_n in ROW layout, or (pc-DM, CHI) the reflected wave 2 P_k o_n - psi_n,k; far
    // field: times (-1)^(y + x), which centres the transform
    auto exit_wave = [&](int k, auto chi_c) {
      constexpr bool CHI = decltype(chi_c)::value != 0;
      const float2* Pk = a.P + (size_t)k * M * M;
#pragma unroll
      for (int q = 0; q < V; ++q)
#pragma unroll
        for (int j = 0; j < E; ++j) v[q][j] = __ldg(&Pk[line[q] * M + tp[q] + G * j]);
#pragma unroll
      for (int q = 0; q < V; ++q) {
        float2 o[E];
        if constexpr (TM) {
#pragma unroll
          for (int h = 0; h < E / 8; ++h) {
            float pr[16];
            tmem_ld16(t_lane + colO + 2 * (q * E + 8 * h), pr);
            tmem_wait_ld();
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) o[8 * h + jj] = make_float2(pr[2 * jj], pr[2 * jj + 1]);
          }
        } else {
#pragma unroll
          for (int j = 0; j < E; ++j) o[j] = o_r[q][j];
        }
#pragma unroll
        for (int j = 0; j < E; ++j) {
          float2 psi = cmul(v[q][j], o[j]);
          if constexpr (CHI) {
            const float2 st = dm_init ? psi : Sn[((size_t)k * M + line[q]) * M + tp[q] + G * j];
            psi = make_float2(2.f * psi.x - st.x, 2.f * psi.y - st.y);
          }
          if (!NEAR && ((line[q] + tp[q] + G * j) & 1)) psi = make_float2(-psi.x, -psi.y);
          v[q][j] = psi;
        }
      }
    };
    using EstC = IntC<0>;
    using WaveC = IntC<MODE == DM ? 1 : 0>;  // the wave that carries the modulus step
    // ---- 2-D transforms between the ROW layout and the frequency layout (row, col) = freq(q, r)
    auto transform = [&](auto inv_c) {
      constexpr bool INV = decltype(inv_c)::value != 0;
      if constexpr (F3) {
        if constexpr (INV) fft3_inverse<M>(v, cbuf, s_tw, s_tw2, tid);
        else fft3_forward<M>(v, cbuf, s_tw, s_tw2, tid);
      } else {
        if constexpr (INV) fft2_inverse<M, V>(v, cbuf, s_tw, tid);
        else fft2_forward<M, V>(v, cbuf, s_tw, tid);
      }
    };
    auto freq = [&](int q, int r, int& row, int& col) {
      if constexpr (F3) {
        row = Tile3<M>::freq_row(tid, q, r);
        col = Tile3<M>::freq_col(tid);
      } else {
        det_coords<M, false>(tid + q * TR, r, row, col);
      }
    };
    // detector pixel of a register: the near field ends in the ROW layout, the far field in frequencies
    auto pixel = [&](int q, int r, int& row, int& col) {
      if constexpr (NEAR) det_coords<M, true>(tid + q * TR, r, row, col);
      else freq(q, r, row, col);
    };
    // ---- forward propagation to the detector (far: frequency layout; near: ROW layout, scaled)
    auto forward = [&]() {
      transform(IntC<0>{});
      if constexpr (NEAR) {
#pragma unroll
        for (int q = 0; q < V; ++q)
#pragma unroll
          for (int r = 0; r < E; ++r) {
            int fu, fv;
            freq(q, r, fu, fv);
            v[q][r] = cmul(v[q][r], cmul(s_h[fu], s_h[fv]));
          }
        transform(IntC<1>{});
#pragma unroll
        for (int q = 0; q < V; ++q)
#pragma unroll
          for (int j = 0; j < E; ++j) v[q][j] = cscale(v[q][j], inv_m2);
      }
    };

    // ---- pass 1: S = sum_k |Psi_k|^2 in Z, each thread on its own detector pixels; the last
    // mode's sum is turned into the blur's input (sqrt for the amplitude model) in place
    auto detect = [&](auto chi_c) {
      for (int k = 0; k < K; ++k) {
        // pc-DM: the next mode's state on its way into L2 while this mode is transformed
        if (MODE == DM && !dm_init && tid == 0 && (decltype(chi_c)::value == 0 ? k == K - 1 : k + 1 < K))
          prefetch_l2(Sn + (size_t)(decltype(chi_c)::value == 0 ? 0 : k + 1) * M * M, (uint32_t)(M * M * 8), keep);
        exit_wave(k, chi_c);
        forward();
        const bool last = k == K - 1;
#pragma unroll
        for (int q = 0; q < V; ++q)
#pragma unroll
          for (int r = 0; r < E; ++r) {
            int row, col;
            pixel(q, r, row, col);
            float s = cabs2(v[q][r]);
            if (k > 0) s += Z[row * LD + col];
            if (last && !a.blur_intensity) s = sqrtf(s);
            Z[row * LD + col] = s;
          }
      }
    };
    // ---- the pc intensity model of the S in Z: blur along x (columns, sigma_1) into X, then along y
    // (rows, sigma_2). PS bit 0: the error of the model intensity; bit 1: the modulus ratio R into Z
    auto model = [&](auto ps_c) {
      constexpr int PS = decltype(ps_c)::value;
      __syncthreads();  // Z complete; the exchange buffer is free (forward ended with a barrier)
      for (int w = tid; w < M * (M / NB); w += TR) {
        const int row = w % M, c0 = (w / M) * NB;
        float out[NB];
        blur_strip<NB, KH>(Z, row * LD, 1, c0, 0, M, s_gx, a.kh, out);
#pragma unroll
        for (int o = 0; o < NB; ++o) X[row * LD + c0 + o] = out[o];
      }
      __syncthreads();
      for (int w = tid; w < M * (M / NB); w += TR) {
        const int col = w % M, rs = (w / M) * NB;
        constexpr bool ROOT = MODE == SINGLE || (PS & 2) != 0, COUNTS = MODE != SINGLE && (PS & 1) != 0;
        float sq[NB], in[NB];
#pragma unroll
        for (int o = 0; o < NB; ++o) {
          if constexpr (ROOT) sq[o] = __ldcs(&Qn[(rs + o) * M + col]);
          if constexpr (COUNTS) in[o] = __ldcs(&In[(rs + o) * M + col]);
        }
        float out[NB];
        blur_strip<NB, KH>(X, col, LD, rs, 0, M, s_gy, a.kh, out);
#pragma unroll
        for (int o = 0; o < NB; ++o) {
          const float acc = out[o];
          if constexpr ((PS & 1) != 0) {
            float im;
            if constexpr (COUNTS) im = in[o];
            else im = sq[o] * sq[o];
            const float ihat = a.blur_intensity ? acc : acc * acc;
            const float d = ihat - im;
            const float y = fmaf(d, d, -err_c);
            const float tt = err_s + y;
            err_c = (tt - err_s) - y;
            err_s = tt;
          }
          if constexpr ((PS & 2) != 0)
            Z[(rs + o) * LD + col] =
                a.blur_intensity ? sq[o] * rsqrtf(acc + a.eps * a.eps) : __fdividef(sq[o], acc + a.eps);
        }
      }
      __syncthreads();
    };
    if constexpr (MODE == DM) {
      detect(EstC{});  // the estimate P o_n: its model error is E
      model(IntC<1>{});
    }
    detect(WaveC{});
    // Psi_{K-1} waits in the contribution columns (registers for the small tiles)
    if constexpr (TM) {
#pragma unroll
      for (int q = 0; q < V; ++q)
#pragma unroll
        for (int h = 0; h < E / 8; ++h) {
          float pr[16];
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) {
            pr[2 * jj] = v[q][8 * h + jj].x;
            pr[2 * jj + 1] = v[q][8 * h + jj].y;
          }
          tmem_st16(t_lane + colC + 2 * (q * E + 8 * h), pr);
        }
      tmem_wait_st();
    } else {
#pragma unroll
      for (int q = 0; q < V; ++q)
#pragma unroll
        for (int j = 0; j < E; ++j) st_r[q][j] = v[q][j];
    }
    model(IntC<(MODE == DM ? 2 : 3)>{});

    // ---- pass 2: mode K-1 from storage, then modes 0 .. K-2 propagated again
    for (int i = 0; i < K; ++i) {
      const int k = i == 0 ? K - 1 : i - 1;
      if (i == 0) {
        if constexpr (TM) {
#pragma unroll
          for (int q = 0; q < V; ++q)
#pragma unroll
            for (int h = 0; h < E / 8; ++h) {
              float pr[16];
              tmem_ld16(t_lane + colC + 2 * (q * E + 8 * h), pr);
              tmem_wait_ld();
#pragma unroll
              for (int jj = 0; jj < 8; ++jj) v[q][8 * h + jj] = make_float2(pr[2 * jj], pr[2 * jj + 1]);
            }
        } else {
#pragma unroll
          for (int q = 0; q < V; ++q)
#pragma unroll
            for (int j = 0; j < E; ++j) v[q][j] = st_r[q][j];
        }
      } else {
        exit_wave(k, WaveC{});
        forward();
      }
      // Psi' = R Psi
#pragma unroll
      for (int q = 0; q < V; ++q)
#pragma unroll
        for (int r = 0; r < E; ++r) {
          int row, col;
          pixel(q, r, row, col);
          v[q][r] = cscale(v[q][r], Z[row * LD + col]);
        }
      // back-propagation to ROW layout (times M^2)
      if constexpr (NEAR) {
        transform(IntC<0>{});
#pragma unroll
        for (int q = 0; q < V; ++q)
#pragma unroll
          for (int r = 0; r < E; ++r) {
            int fu, fv;
            freq(q, r, fu, fv);
            v[q][r] = cmulc(v[q][r], cmul(s_h[fu], s_h[fv]));
          }
      }
      transform(IntC<1>{});
      // dpsi = psi' - P_k o_n; contributions, probe partials
      const float2* Pk = a.P + (size_t)k * M * M;
      float2* pk = MODE == DM ? Sn + (size_t)k * M * M : pacc + (size_t)k * M * M;  // (pc-DM: the mode's state)
      float* dk = dacc;
      // groups of four values; the next group's probe values are loaded before this group's work (the
      // tensor-memory waits are compiler barriers: loads behind them would each expose an L2 round trip)
      float2 pn[4];
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) pn[jj] = __ldg(&Pk[line[0] * M + tp[0] + G * jj]);
#pragma unroll
      for (int q = 0; q < V; ++q) {
        const int ln = line[q];
#pragma unroll
        for (int h = 0; h < E / 4; ++h) {
          float2 p[4];
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) p[jj] = pn[jj];
          if (h + 1 < E / 4 || q + 1 < V) {
            const int q2 = h + 1 < E / 4 ? q : q + 1 < V ? q + 1 : q, h2 = h + 1 < E / 4 ? h + 1 : 0;
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) pn[jj] = __ldg(&Pk[line[q2] * M + tp[q2] + G * (4 * h2 + jj)]);
          }
          float2 st[4];
          if constexpr (MODE == DM) {
#pragma unroll
            for (int jj = 0; jj < 4; ++jj)
              st[jj] = dm_init ? make_float2(0.f, 0.f) : pk[ln * M + tp[q] + G * (4 * h + jj)];
          }
          float2 o[4], c[4];
          if constexpr (TM) {
            float pr[8], ac[8];
            tmem_ld8(t_lane + colO + 2 * (q * E + 4 * h), pr);
            if (i > 0) tmem_ld8(t_lane + colC + 2 * (q * E + 4 * h), ac);
            tmem_wait_ld();
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
              o[jj] = make_float2(pr[2 * jj], pr[2 * jj + 1]);
              c[jj] = i > 0 ? make_float2(ac[2 * jj], ac[2 * jj + 1]) : make_float2(0.f, 0.f);
            }
          } else {
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
              o[jj] = o_r[q][4 * h + jj];
              c[jj] = i > 0 ? c_r[q][4 * h + jj] : make_float2(0.f, 0.f);
            }
          }
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            const int j = 4 * h + jj;
            const int x = tp[q] + G * j;
            float2 psi_new = cscale(v[q][j], inv_m2);
            if (!NEAR && ((ln + x) & 1)) psi_new = make_float2(-psi_new.x, -psi_new.y);
            const float2 ov = cmul(p[jj], o[jj]);
            float2 dpsi = csub(psi_new, ov);
            if constexpr (MODE == DM) {
              // psi_n <- psi_n + Pi_F(chi) - P o_n, and the overlap step takes psi_n - P o_n (its probe
              // sums follow the object step)
              st[jj] = cadd(dm_init ? ov : st[jj], dpsi);
              pk[ln * M + x] = st[jj];
              dpsi = csub(st[jj], ov);
            }
            c[jj] = cadd(c[jj], cconjmul(p[jj], dpsi));
            if constexpr (MODE != DM) {
              // the first position of a partial sets it, the later ones add to it
              const float2 dp = cconjmul(o[jj], dpsi);
              if (first) {
                st_part(&pk[ln * M + x], dp, keep);
                if (i == 0) st_part(&dk[ln * M + x], cabs2(o[jj]), keep);
              } else {
                red_hint(&pk[ln * M + x], dp, keep);
                if (i == 0) red_hint(&dk[ln * M + x], cabs2(o[jj]), keep);
              }
            }
          }
          if constexpr (TM) {
            float ac[8];
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
              ac[2 * jj] = c[jj].x;
              ac[2 * jj + 1] = c[jj].y;
            }
            tmem_st8(t_lane + colC + 2 * (q * E + 4 * h), ac);
          } else {
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) c_r[q][4 * h + jj] = c[jj];
          }
        }
      }
      if constexpr (TM) tmem_wait_st();
    }
    // ---- c_n, written once (streaming: the object gather reads it after this launch)
    float2* cn = a.cn + (size_t)n * M * M;
#pragma unroll
    for (int q = 0; q < V; ++q) {
      float2 c[E];
      if constexpr (TM) {
#pragma unroll
        for (int h = 0; h < E / 8; ++h) {
          float ac[16];
          tmem_ld16(t_lane + colC + 2 * (q * E + 8 * h), ac);
          tmem_wait_ld();
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) c[8 * h + jj] = make_float2(ac[2 * jj], ac[2 * jj + 1]);
        }
      } else {
#pragma unroll
        for (int j = 0; j < E; ++j) c[j] = c_r[q][j];
      }
#pragma unroll
      for (int j = 0; j < E; ++j) __stcs(&cn[line[q] * M + tp[q] + G * j], c[j]);
    }
    // the next position's pass 1 rewrites Z, which other threads read above
    __syncthreads();
  };

  // ---- FP64 error numerator of partial `part` (the compensated FP32 thread sums, added in a fixed tree);
  // its other K - 1 entries are zero (the error is per position, not per mode)
  auto finish = [&](const FusedArgs& a, int part) {
    double* red = reinterpret_cast<double*>(smem);
    red[tid] = (double)err_s - (double)err_c;
    __syncthreads();
    for (int w = TR / 2; w > 0; w >>= 1) {
      if (tid < w) red[tid] += red[tid + w];
      __syncthreads();
    }
    for (int k = tid; k < K; k += TR) a.errpart[(size_t)part * K + k] = k == 0 ? red[0] : 0.0;
    err_s = 0.f;
    err_c = 0.f;
  };

  if constexpr (MODE == QUEUED) {
    // chunk (problem, first position, end, partial): thread 0 takes the next index
    FusedArgs* s_desc = reinterpret_cast<FusedArgs*>(smem + SM::BYTES);
    int* s_item = reinterpret_cast<int*>(smem + SM::BYTES + SM::DESC - 16);
    for (;;) {
      __syncthreads();  // the previous chunk's arguments, item and reduction buffer are read
      if (tid == 0) *s_item = atomicAdd(a_in.queue, 1);
      __syncthreads();
      const int c = *s_item;
      if (c >= a_in.nchunks) break;
      const int4 ch = a_in.chunks[c];
      const int* src = reinterpret_cast<const int*>(a_in.probs + ch.x);
      for (int i = tid; i < (int)(sizeof(FusedArgs) / 4); i += TR) reinterpret_cast<int*>(s_desc)[i] = src[i];
      __syncthreads();
      setup(*s_desc);
      __syncthreads();
      float2* pacc = s_desc->pacc + (size_t)ch.w * K * M * M;
      float* dacc = s_desc->dacc + (size_t)ch.w * M * M;
      for (int n = ch.y; n < ch.z; ++n) run_position(*s_desc, n, n == ch.y, pacc, dacc);
      finish(*s_desc, ch.w);
    }
  } else {
    // CTA `slot` takes positions slot, slot + slots, ... and owns partial `slot`
    const int slot = blockIdx.x, nslots = gridDim.x;
    float2* pacc = MODE == DM ? nullptr : a_in.pacc + (size_t)slot * K * M * M;
    float* dacc = MODE == DM ? nullptr : a_in.dacc + (size_t)slot * M * M;
    for (int n = slot; n < a_in.N; n += nslots) run_position(a_in, n, n == slot, pacc, dacc);
    finish(a_in, slot);
  }
  if constexpr (TM) {
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    if (tid / 32 == 0) tmem_dealloc(*s_tmem, SeqShape<M>::TMEM_COLS);
  }
}

// ------------------------------------------------------------------ launches
template <int M, bool NEAR, int KH, int MODE>
static cudaError_t launch_seq_kh(const FusedArgs& a, int slots, cudaStream_t s) {
  auto kern = pc_seq_kernel<M, NEAR, KH, MODE>;
  constexpr size_t bytes = SeqSmem<M>::bytes(MODE);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e != cudaSuccess) return e;
  kern<<<slots, SeqShape<M>::TR, bytes, s>>>(a);
  return cudaGetLastError();
}

// the paper's 11 x 11 kernel (Sec. 3.1) has its own instantiation; any other odd size up to 31
// runs with the taps zero-padded to 31
template <int M, int MODE>
static cudaError_t launch_seq_t(const FusedArgs& a, int slots, cudaStream_t s) {
  if (a.near_field)
    return a.kh == 5 ? launch_seq_kh<M, true, 5, MODE>(a, slots, s) : launch_seq_kh<M, true, 15, MODE>(a, slots, s);
  return a.kh == 5 ? launch_seq_kh<M, false, 5, MODE>(a, slots, s) : launch_seq_kh<M, false, 15, MODE>(a, slots, s);
}

template <int MODE>
static cudaError_t launch_seq(int M, const FusedArgs& a, int slots, cudaStream_t s) {
  switch (M) {
    case 8: return launch_seq_t<8, MODE>(a, slots, s);
    case 16: return launch_seq_t<16, MODE>(a, slots, s);
    case 32: return launch_seq_t<32, MODE>(a, slots, s);
    case 64: return launch_seq_t<64, MODE>(a, slots, s);
    case 128: return launch_seq_t<128, MODE>(a, slots, s);
    default: return cudaErrorInvalidValue;
  }
}

// co-resident CTAs over the whole GPU, the smallest count over the instantiations; CTAs on one SM
// must not ask for more than its 512 TMEM columns together (tcgen05.alloc would wait for columns
// that a persistent CTA never frees), which the shared-memory and register budgets guarantee
template <int M, int MODE>
static cudaError_t seq_slots_t(int* slots) {
  int dev = 0, sms = 0, best = 1 << 30;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  constexpr size_t bytes = SeqSmem<M>::bytes(MODE);
  const void* kerns[4] = {(const void*)pc_seq_kernel<M, false, 5, MODE>, (const void*)pc_seq_kernel<M, false, 15, MODE>,
                          (const void*)pc_seq_kernel<M, true, 5, MODE>, (const void*)pc_seq_kernel<M, true, 15, MODE>};
  for (const void* k : kerns) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, SeqShape<M>::TR, bytes);
    if (e != cudaSuccess) return e;
    if (SeqShape<M>::TMEM && per_sm * SeqShape<M>::TMEM_COLS > 512) return cudaErrorInvalidConfiguration;
    best = per_sm < best ? per_sm : best;
  }
  *slots = best * sms;
  return cudaSuccess;
}

template <int MODE>
static cudaError_t seq_slots(int M, int* slots) {
  switch (M) {
    case 8: return seq_slots_t<8, MODE>(slots);
    case 16: return seq_slots_t<16, MODE>(slots);
    case 32: return seq_slots_t<32, MODE>(slots);
    case 64: return seq_slots_t<64, MODE>(slots);
    case 128: return seq_slots_t<128, MODE>(slots);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ptycho
