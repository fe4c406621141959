// Staged path for probe sizes whose M x M complex tile exceeds one SM's
// shared memory (M = 256). Same iteration as the fused kernel (Eqs. 1, 2, 6, 7,
// Fig. 1 box 1), split into passes over an L2-sized scratch W that holds a
// chunk of C positions x K modes:
//
//   far field:  rows(exit wave, DFT) -> cols(DFT: S) -> modulus (R) -> cols(DFT, R x, IDFT)
//               -> rows(IDFT, dpsi, contributions)
//   near field: rows(exit wave, DFT) -> cols(DFT, x H, IDFT) -> rows(IDFT: S)
//               -> modulus (R) -> rows(IDFT, R x, DFT) -> cols(DFT, x conj H, IDFT)
//               -> rows(IDFT, dpsi, contributions)
//
// The pass that reaches the detector field walks the K modes in order and writes S = sum_k |Psi_k|^2 only; the
// pass after the modulus repeats that line transform on its way back. So W is written once less (it
// streams through HBM for large chunks, and the passes run at its rate), and the modulus pass reads one
// float per pixel instead of K complex values (with halo rows).
//
// A length-256 line is transformed by 16 threads: a radix-16 pass in
// registers over x = t + 16 j, the twiddle W_256^(t k2), a warp-local swap in
// shared memory, and a second radix-16 pass; thread t then holds frequencies
// t + 16 k1. The inverse consumes that layout and returns x = t + 16 j.
// All sums that cross CTAs are written to per-(slot, mode) or per-(position,
// row-block) partials and added in a fixed order, as on the fused path.
#include <cuda_runtime.h>

#include "big_line.cuh"
#include "engine.h"
#include "fft.cuh"
#include "fused_common.cuh"

namespace ptycho {

namespace {

constexpr int RB = 16;   // rows per modulus block

// twiddles W_BL^(t k2) for t < 16 and the k2 of the first pass, from the host table W_BL^m
template <int BL>
__device__ __forceinline__ void load_tw(float2* s_tw, const float2* tw) {
  constexpr int TWS = BigShape<BL>::TWS, K2 = BigShape<BL>::E;
  for (int i = threadIdx.x; i < BigShape<BL>::TWN; i += blockDim.x) {
    const int t = i / TWS, k2 = i % TWS;
    s_tw[i] = k2 < K2 ? tw[(t * k2) % BL] : make_float2(0.f, 0.f);
  }
}

}  // namespace

// ---- row passes. mode 0: exit wave + forward DFT; 1: inverse DFT, R x (row), forward DFT in place
template <int BL, int MODE, bool NEAR>
__global__ void __launch_bounds__(BigShape<BL>::LROW * BT) k_big_rows(const BigArgs b) {
  constexpr int E = BigShape<BL>::E, LROW = BigShape<BL>::LROW;
  __shared__ float2 s_tw[BigShape<BL>::TWN];
  __shared__ float2 s_sw[LROW][BigShape<BL>::SWN];
  load_tw<BL>(s_tw, b.tw);
  __syncthreads();
  const int li = threadIdx.x / BT, t = threadIdx.x % BT;
  const int y = blockIdx.x * LROW + li;
  const int k = blockIdx.y, c = blockIdx.z;
  const int n = b.n0 + c;
  const size_t MM = (size_t)BL * BL;
  float2* row = b.W + ((size_t)c * b.K + k) * MM + (size_t)y * BL;
  float2 a[E];
  if constexpr (MODE == 0) {
    const int2 pn = b.pos[n];
    const float2* Pk = b.P + (size_t)k * MM + (size_t)y * BL;
    const float2* On = b.O + (size_t)(pn.x + y) * b.obj_w + pn.y;
    // pc-DM second sweep: the reflected wave chi = 2 P o_n - psi_n
    const float2* St = b.dm_pass == 2 ? b.psi + ((size_t)n * b.K + k) * MM + (size_t)y * BL : nullptr;
#pragma unroll
    for (int j = 0; j < E; ++j) {
      const int x = t + 16 * j;
      float2 psi = cmul(Pk[x], On[x]);
      if (St) {
        const float2 st = b.dm_init ? psi : St[x];
        psi = make_float2(2.f * psi.x - st.x, 2.f * psi.y - st.y);
      }
      if (!NEAR && ((y + x) & 1)) psi = make_float2(-psi.x, -psi.y);
      a[j] = psi;
    }
  } else {
    // Psi' = R Psi (the modulus ratio of this position)
    const float* Rr = b.R + (size_t)c * MM + (size_t)y * BL;
    float R[E];
#pragma unroll
    for (int r = 0; r < E; ++r) a[r] = row[line_freq<BL>(t, r)];
#pragma unroll
    for (int j = 0; j < E; ++j) R[j] = Rr[t + 16 * j];
    line_fft<BL, true>(a, s_sw[li], s_tw, t);
    const float s = 1.0f / (float)(BL * BL);
#pragma unroll
    for (int j = 0; j < E; ++j) a[j] = cscale(cscale(a[j], s), R[j]);
  }
  line_fft<BL, false>(a, s_sw[li], s_tw, t);
#pragma unroll
  for (int r = 0; r < E; ++r) row[line_freq<BL>(t, r)] = a[r];
}

// near field: S = sum_k |Psi_k|^2 of the inverse row DFTs / M^2
template <int BL>
__global__ void __launch_bounds__(BigShape<BL>::LROW * BT) k_big_rows_detector(const BigArgs b) {
  constexpr int E = BigShape<BL>::E, LROW = BigShape<BL>::LROW;
  __shared__ float2 s_tw[BigShape<BL>::TWN];
  __shared__ float2 s_sw[LROW][BigShape<BL>::SWN];
  load_tw<BL>(s_tw, b.tw);
  __syncthreads();
  const int li = threadIdx.x / BT, t = threadIdx.x % BT;
  const int y = blockIdx.x * LROW + li, c = blockIdx.y;
  const size_t MM = (size_t)BL * BL;
  const float s = 1.0f / (float)(BL * BL);
  float sum[E];
#pragma unroll
  for (int j = 0; j < E; ++j) sum[j] = 0.f;
  for (int k = 0; k < b.K; ++k) {
    const float2* row = b.W + ((size_t)c * b.K + k) * MM + (size_t)y * BL;
    float2 a[E];
#pragma unroll
    for (int r = 0; r < E; ++r) a[r] = row[line_freq<BL>(t, r)];
    line_fft<BL, true>(a, s_sw[li], s_tw, t);
#pragma unroll
    for (int j = 0; j < E; ++j) sum[j] += cabs2(cscale(a[j], s));
  }
  float* S = b.S + (size_t)c * MM + (size_t)y * BL;
#pragma unroll
  for (int j = 0; j < E; ++j) S[t + 16 * j] = sum[j];
}

// ---- column passes on a BL x LINES tile staged through shared memory; the line swaps use the tile's own
// column (its values are in registers then), so a CTA takes half the shared memory of a separate swap
// buffer and four to eight CTAs overlap their loads, transforms and stores on an SM (with one CTA of 32
// lines per SM the three phases ran one after the other: 112 us for 32 positions x 8 modes of 256^2).
// op 0: S of the forward DFTs of every mode (far forward); 1: DFT, R x, IDFT (far backward);
// 2: DFT, x H, IDFT (near forward); 3: DFT, x conj H, IDFT (near backward)
template <int BL, int OP>
__global__ void __launch_bounds__(BigShape<BL>::LINES * BT, BL == 256 ? (OP < 2 ? 3 : 4) : 2) k_big_cols(const BigArgs b) {
  constexpr int E = BigShape<BL>::E, LINES = BigShape<BL>::LINES;
  constexpr int TP = LINES + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* tile = reinterpret_cast<float2*>(smem_raw);  // [SWN][TP], rows 0 .. BL - 1 staged
  float2* s_tw = tile + BigShape<BL>::SWN * TP;
  float2* s_h = s_tw + BigShape<BL>::TWN;                  // OP >= 2: BL
  float* s_r = reinterpret_cast<float*>(s_h);              // OP == 1: BL x TP
  load_tw<BL>(s_tw, b.tw);
  if constexpr (OP >= 2)
    for (int i = threadIdx.x; i < BL; i += blockDim.x) s_h[i] = b.hq[i];
  const int x0 = blockIdx.x * LINES, c = OP == 0 ? blockIdx.y : blockIdx.z;
  const size_t MM = (size_t)BL * BL;
  const int cl = threadIdx.x / BT, t = threadIdx.x % BT;
  const ColumnSwap<BL, TP> sw{tile + cl};
  float sum[OP == 0 ? E : 1];
  if constexpr (OP == 0)
#pragma unroll
    for (int r = 0; r < E; ++r) sum[r] = 0.f;
  constexpr int UL = OP == 0 ? 4 : BL / BT;  // tile loads in flight per thread (the sums take registers)
  const int k_lo = OP == 0 ? 0 : blockIdx.y, k_hi = OP == 0 ? b.K : k_lo + 1;
  for (int k = k_lo; k < k_hi; ++k) {
    float2* Wk = b.W + ((size_t)c * b.K + k) * MM;
    // coalesced tile load: LINES consecutive columns per row; the far-field backward pass stages the
    // modulus ratio of this position beside it
    const float* Rc = b.R + (size_t)c * MM;
#pragma unroll UL
    for (int i = threadIdx.x; i < BL * LINES; i += LINES * BT) {
      const int yy = i / LINES, xx = i % LINES;
      tile[yy * TP + xx] = Wk[(size_t)yy * BL + x0 + xx];
      if constexpr (OP == 1) s_r[yy * TP + xx] = Rc[(size_t)yy * BL + x0 + xx];
    }
    __syncthreads();
    float2 a[E];
#pragma unroll
    for (int j = 0; j < E; ++j) a[j] = tile[(t + 16 * j) * TP + cl];
    __syncwarp();  // the line's values are in registers: its column is the swap buffer now
    line_fft_swap<BL, false>(a, sw, s_tw, t);  // a[r] = column spectrum at u = line_freq(t, r)
    if constexpr (OP == 0) {
#pragma unroll
      for (int r = 0; r < E; ++r) sum[r] += cabs2(a[r]);
      __syncthreads();  // the next mode's load, or S, rewrites the tile
      continue;
    } else if constexpr (OP == 1) {
#pragma unroll
      for (int r = 0; r < E; ++r) a[r] = cscale(a[r], s_r[line_freq<BL>(t, r) * TP + cl]);  // Psi' = R Psi
    } else {
      const float2 hv = s_h[x0 + cl];  // H(u, v) = h[u] h[v], v = this column's frequency
#pragma unroll
      for (int r = 0; r < E; ++r) {
        const float2 hh = cmul(s_h[line_freq<BL>(t, r)], hv);
        a[r] = OP == 2 ? cmul(a[r], hh) : cmulc(a[r], hh);
      }
    }
    line_fft_swap<BL, true>(a, sw, s_tw, t);
    // (a line's transform ends with a warp barrier after its last read of the swap)
#pragma unroll
    for (int j = 0; j < E; ++j) tile[(t + 16 * j) * TP + cl] = a[j];
    __syncthreads();
#pragma unroll 4
    for (int i = threadIdx.x; i < BL * LINES; i += LINES * BT) {
      const int yy = i / LINES, xx = i % LINES;
      Wk[(size_t)yy * BL + x0 + xx] = tile[yy * TP + xx];
    }
  }
  if constexpr (OP == 0) {
#pragma unroll
    for (int r = 0; r < E; ++r) tile[line_freq<BL>(t, r) * TP + cl].x = sum[r];
    __syncthreads();
    float* S = b.S + (size_t)c * MM;
#pragma unroll 4
    for (int i = threadIdx.x; i < BL * LINES; i += LINES * BT) {
      const int yy = i / LINES, xx = i % LINES;
      S[(size_t)yy * BL + x0 + xx] = tile[yy * TP + xx].x;
    }
  }
}

// ---- modulus: rows [y0, y0 + RB) of one position from S, with KH halo rows for the y blur. Writes the ratio
// R to its own buffer; the next pass applies Psi' = R Psi as it loads W. Each blur keeps a window of samples
// in registers for eight outputs (blur_strip), lanes along the other axis of an odd-stride buffer.
template <int BL>
constexpr int kModTpb = BL == 256 ? 256 : 512;
// CTAs that the shared memory lets on an SM, asked for in registers as well (KH = 5 at 512 columns with 79 registers
// and one CTA instead of 64 and two: 49 positions of 512^2, two modes, 886 against 812 us an iteration)
template <int BL, int KH>
constexpr int kModCtas = (BL == 256 ? 2 : 1) * (KH == 5 ? 2 : 1);

template <int BL, int KH>
__global__ void __launch_bounds__(kModTpb<BL>, kModCtas<BL, KH>) k_big_modulus(const BigArgs b) {
  constexpr int TPB = kModTpb<BL>;
  constexpr int HR = RB + 2 * KH;  // rows held
  constexpr int LD = BL + 1, NB = 8;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* sA = reinterpret_cast<float*>(smem_raw);  // HR x LD
  float* sB = sA + HR * LD;                        // HR x LD
  __shared__ float s_gx[2 * KH + 1], s_gy[2 * KH + 1];
  __shared__ double s_red[TPB];
  for (int i = threadIdx.x; i < 2 * KH + 1; i += blockDim.x) {
    const int d = i - KH;
    const bool in = d >= -b.kh && d <= b.kh;
    s_gx[i] = in ? b.gx[d + b.kh] : 0.f;
    s_gy[i] = in ? b.gy[d + b.kh] : 0.f;
  }
  const int y0 = blockIdx.x * RB, c = blockIdx.y;
  const int n = b.n0 + c;
  const size_t MM = (size_t)BL * BL;
  // amplitude or intensity of the mode sum; rows outside the pattern are zero
  const float* Sc = b.S + (size_t)c * MM;
#pragma unroll 4
  for (int i = threadIdx.x; i < HR * BL; i += TPB) {
    const int r = i / BL, x = i % BL, yy = y0 - KH + r;
    const float s = yy >= 0 && yy < BL ? Sc[(size_t)yy * BL + x] : 0.f;
    sA[r * LD + x] = b.blur_intensity ? s : sqrtf(s);
  }
  __syncthreads();
  // blur along x (columns, sigma_1), zero padded
  for (int w = threadIdx.x; w < HR * (BL / NB); w += TPB) {
    const int r = w % HR, c0 = (w / HR) * NB;
    float out[NB];
    blur_strip<NB, KH>(sA, r * LD, 1, c0, 0, BL, s_gx, b.kh, out);
#pragma unroll
    for (int o = 0; o < NB; ++o) sB[r * LD + c0 + o] = out[o];
  }
  __syncthreads();
  // blur along y (rows, sigma_2) for the own rows, ratio, error
  const float eps = b.eps;
  float es = 0.f, ec = 0.f;
  // the ratio takes sqrt(I), the error the counts I as they were given (their rounded roots squared are off by
  // more than an ulp); pc-DM: each sweep needs one of the two
  const float* Sn = b.sqrtI + (size_t)n * MM;
  const float* In = b.I + (size_t)n * MM;
  const bool ratio = b.dm_pass != 1, error = b.dm_pass != 2;
  for (int w = threadIdx.x; w < BL * (RB / NB); w += TPB) {
    const int x = w % BL, rs = (w / BL) * NB;
    float sq[NB], im[NB], out[NB];
#pragma unroll
    for (int o = 0; o < NB; ++o) {
      sq[o] = ratio ? __ldcs(&Sn[(size_t)(y0 + rs + o) * BL + x]) : 0.f;
      im[o] = error ? __ldcs(&In[(size_t)(y0 + rs + o) * BL + x]) : 0.f;
    }
    blur_strip<NB, KH>(sB, x, LD, rs + KH, 0, HR, s_gy, b.kh, out);
#pragma unroll
    for (int o = 0; o < NB; ++o) {
      const float acc = out[o];
      float ihat, R;
      if (b.blur_intensity) {
        ihat = acc;
        R = sq[o] * rsqrtf(acc + eps * eps);
      } else {
        ihat = acc * acc;
        R = __fdividef(sq[o], acc + eps);
      }
      const float dd = ihat - im[o];
      const float yv = fmaf(dd, dd, -ec);
      const float tt = es + yv;
      ec = (tt - es) - yv;
      es = tt;
      if (ratio) b.R[(size_t)c * MM + (size_t)(y0 + rs + o) * BL + x] = R;
    }
  }
  if (!error) return;  // pc-DM: the error is the estimate's (first sweep); uniform per block
  s_red[threadIdx.x] = (double)es - (double)ec;
  __syncthreads();
  for (int w = TPB / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) s_red[threadIdx.x] += s_red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) b.errpart[(size_t)n * (BL / RB) + blockIdx.x] = s_red[0];
}

// fire-and-forget adds at L2 for the probe partials: within one launch every element is added to by
// one thread only, and launches are ordered, so each sum keeps its position order (bitwise
// reproducible) while no thread waits for the old value
__device__ __forceinline__ void red_add(float2* a, float2 v) {
  asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(a), "f"(v.x), "f"(v.y));
}
__device__ __forceinline__ void red_add(float* a, float v) {
  asm volatile("red.global.add.f32 [%0], %1;" ::"l"(a), "f"(v));
}

// ---- final inverse row DFT of every mode, dpsi, contributions. A CTA owns FR rows of the tile and walks the
// positions g, g + groups, ... of the chunk (g = blockIdx.y) and their modes.
// ACC: the launch's probe sums of (group, mode, rows) stay in shared memory, every element touched by one thread,
// and are added to the group's partial once per launch (a sum of sums: one chain over all chunks' positions
// would be several times longer than the partials per position of a chunk that it replaces). Otherwise (partials of K modes too large for three CTAs on an
// SM) one group per position and L2 reductions into its partial. pc-DM (b.psi) has no probe partials here.
template <int BL>
struct FinalShape {
  static constexpr int FR = 4, TPB = FR * BT;
  static constexpr size_t ACC_MAX = 72 * 1024;  // three CTAs on an SM
  static constexpr size_t acc_bytes(int K) { return (size_t)K * FR * BL * sizeof(float2); }
  static constexpr bool accumulates(int K) { return acc_bytes(K) <= ACC_MAX; }
};

template <int BL, bool NEAR, bool ACC>
__global__ void __launch_bounds__(FinalShape<BL>::TPB) k_big_final(const BigArgs b, int nc) {
  constexpr int E = BigShape<BL>::E, FR = FinalShape<BL>::FR;
  constexpr bool AHEAD = BL == 256;  // registers for the next mode's line and this one's probe values
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* s_p = reinterpret_cast<float2*>(smem_raw);  // ACC: K x FR x BL
  __shared__ float2 s_tw[BigShape<BL>::TWN];
  __shared__ float2 s_sw[FR][BigShape<BL>::SWN];
  load_tw<BL>(s_tw, b.tw);
  __syncthreads();
  const int li = threadIdx.x / BT, t = threadIdx.x % BT;
  const int y = blockIdx.x * FR + li;
  const int g = blockIdx.y, G = gridDim.y, K = b.K;
  if (g >= nc) return;  // (a short last chunk: the group's partial stays as it is)
  const bool start = b.n0 == b.n_first;  // this launch starts the partials
  const size_t MM = (size_t)BL * BL, yo = (size_t)y * BL;
  const float s = 1.0f / (float)(BL * BL);
  float2* pacc = b.pacc + (size_t)g * K * MM + yo;
  float* dacc = b.dacc + (size_t)g * MM + yo;
  float dsum[E];
#pragma unroll
  for (int j = 0; j < E; ++j) dsum[j] = 0.f;
  auto line = [&](int c, int k, float2 (&a)[E]) {
    const float2* row = b.W + ((size_t)c * K + k) * MM + yo;
#pragma unroll
    for (int r = 0; r < E; ++r) a[r] = row[line_freq<BL>(t, r)];
  };
  float2 nx[AHEAD ? E : 1];
  if constexpr (AHEAD) line(g, 0, nx);
  for (int c = g; c < nc; c += G) {
    const int n = b.n0 + c;
    const bool first = c == g && (ACC || start);
    const int2 pn = b.pos[n];
    const float2* On = b.O + (size_t)(pn.x + y) * b.obj_w + pn.y;
    float2 cacc[E], ov[AHEAD ? E : 1];
#pragma unroll
    for (int j = 0; j < E; ++j) {
      cacc[j] = make_float2(0.f, 0.f);
      const float2 o = On[t + 16 * j];
      dsum[j] += cabs2(o);
      if constexpr (AHEAD) ov[j] = o;
    }
    for (int k = 0; k < K; ++k) {
      const float2* Pk = b.P + (size_t)k * MM + yo;
      float2 a[E], pv[AHEAD ? E : 1];
      if constexpr (AHEAD) {
#pragma unroll
        for (int r = 0; r < E; ++r) a[r] = nx[r];
#pragma unroll
        for (int j = 0; j < E; ++j) pv[j] = Pk[t + 16 * j];
        if (k + 1 < K) line(c, k + 1, nx);
        else if (c + G < nc) line(c + G, 0, nx);
      } else {
        line(c, k, a);
      }
      line_fft<BL, true>(a, s_sw[li], s_tw, t);
      // pc-DM: psi_n <- psi_n + Pi_F(chi) - P o_n, the overlap step takes psi_n - P o_n (its probe
      // sums follow the object step)
      float2* St = b.psi ? b.psi + ((size_t)n * K + k) * MM + yo : nullptr;
#pragma unroll
      for (int j = 0; j < E; ++j) {
        const int x = t + 16 * j;
        float2 psi_new = cscale(a[j], s);
        if (!NEAR && ((y + x) & 1)) psi_new = make_float2(-psi_new.x, -psi_new.y);
        const float2 p = AHEAD ? pv[AHEAD ? j : 0] : Pk[x], o = AHEAD ? ov[AHEAD ? j : 0] : On[x];
        const float2 po = cmul(p, o);
        float2 dpsi = csub(psi_new, po);
        if (St) {
          const float2 st = cadd(b.dm_init ? po : St[x], dpsi);
          St[x] = st;
          dpsi = csub(st, po);
        }
        cacc[j] = cadd(cacc[j], cconjmul(p, dpsi));
        const float2 pc = cconjmul(o, dpsi);
        if constexpr (ACC) {
          float2& q = s_p[(k * FR + li) * BL + x];
          q = first ? pc : cadd(q, pc);
        } else if (!St) {
          if (first) pacc[(size_t)k * MM + x] = pc;
          else red_add(&pacc[(size_t)k * MM + x], pc);
        }
      }
    }
    float2* cn = b.cn + (size_t)n * MM + yo;
#pragma unroll
    for (int j = 0; j < E; ++j) cn[t + 16 * j] = cacc[j];
  }
  if (b.psi) return;
#pragma unroll
  for (int j = 0; j < E; ++j) dacc[t + 16 * j] = start ? dsum[j] : dacc[t + 16 * j] + dsum[j];
  if constexpr (ACC)
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int j = 0; j < E; ++j) {
        float2& q = pacc[(size_t)k * MM + t + 16 * j];
        const float2 v = s_p[(k * FR + li) * BL + t + 16 * j];
        q = start ? v : cadd(q, v);
      }
}

template <int BL, int OP>
constexpr size_t big_cols_smem() {
  return sizeof(float2) * ((size_t)BigShape<BL>::SWN * (BigShape<BL>::LINES + 1) + BigShape<BL>::TWN) +
         (OP >= 2 ? sizeof(float2) * BL : OP == 1 ? sizeof(float) * BL * (BigShape<BL>::LINES + 1) : 0);
}

int big_row_blocks(int M) { return M / RB; }

// groups of the final pass (probe partials of an accumulation that starts with nc positions): as many as
// are co-resident, so that no second wave is nearly empty; one per position without accumulators
template <int BL>
static cudaError_t final_groups(int K, int nc, int* out) {
  using FS = FinalShape<BL>;
  int dev = 0, sms = 0, most = 1 << 30;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  for (auto kern : {k_big_final<BL, false, true>, k_big_final<BL, true, true>}) {
    int per_sm = 0;
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FS::ACC_MAX);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, FS::TPB, FS::acc_bytes(K));
    most = per_sm < most ? per_sm : most;
  }
  if (e != cudaSuccess) return e;
  const int g = most * sms / (BL / FS::FR);
  *out = g < 1 ? 1 : g < nc ? g : nc;
  return cudaSuccess;
}
cudaError_t big_groups(int M, int K, bool dm, int nc, int* out) {
  *out = nc;
  if (dm) return cudaSuccess;
  if (M == 256 && FinalShape<256>::accumulates(K)) return final_groups<256>(K, nc, out);
  if (M == 512 && FinalShape<512>::accumulates(K)) return final_groups<512>(K, nc, out);
  return cudaSuccess;
}

template <int BL, int KH>
constexpr size_t big_mod_smem() { return sizeof(float) * 2 * (size_t)(RB + 2 * KH) * (BL + 1); }

template <int BL, bool NEAR>
static cudaError_t big_final(const BigArgs& b, int nc, cudaStream_t s) {
  using FS = FinalShape<BL>;
  if (FS::accumulates(b.K) && !b.psi) {
    const dim3 grid(BL / FS::FR, b.groups);
    const size_t bytes = FS::acc_bytes(b.K);
    cudaError_t e = cudaFuncSetAttribute(k_big_final<BL, NEAR, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)FS::ACC_MAX);
    if (e != cudaSuccess) return e;
    k_big_final<BL, NEAR, true><<<grid, FS::TPB, bytes, s>>>(b, nc);
  } else {
    k_big_final<BL, NEAR, false><<<dim3(BL / FS::FR, nc), FS::TPB, 0, s>>>(b, nc);
  }
  return cudaGetLastError();
}

// the passes of one chunk; `full` false stops after the modulus pass (pc-DM first sweep)
template <int BL>
static cudaError_t big_passes(const BigArgs& b, int nc, bool full, cudaStream_t s) {
  constexpr int LINES = BigShape<BL>::LINES, LROW = BigShape<BL>::LROW;
  const dim3 blk(LINES * BT), rblk(LROW * BT);
  const dim3 grow(BL / LROW, b.K, nc), gdet(BL / LROW, nc), gcol(BL / LINES, b.K, nc), gcol0(BL / LINES, nc);
  const dim3 gmod(BL / RB, nc);
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(k_big_cols<BL, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)big_cols_smem<BL, 0>())) != cudaSuccess ||
      (e = cudaFuncSetAttribute(k_big_cols<BL, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)big_cols_smem<BL, 1>())) != cudaSuccess ||
      (e = cudaFuncSetAttribute(k_big_cols<BL, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)big_cols_smem<BL, 2>())) != cudaSuccess ||
      (e = cudaFuncSetAttribute(k_big_cols<BL, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)big_cols_smem<BL, 3>())) != cudaSuccess)
    return e;
  if ((e = cudaFuncSetAttribute(k_big_modulus<BL, 5>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)big_mod_smem<BL, 5>())) != cudaSuccess)
    return e;
  if ((e = cudaFuncSetAttribute(k_big_modulus<BL, 15>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)big_mod_smem<BL, 15>())) != cudaSuccess)
    return e;
  if (b.near_field) {
    k_big_rows<BL, 0, true><<<grow, rblk, 0, s>>>(b);
    k_big_cols<BL, 2><<<gcol, blk, big_cols_smem<BL, 2>(), s>>>(b);
    k_big_rows_detector<BL><<<gdet, rblk, 0, s>>>(b);
  } else {
    k_big_rows<BL, 0, false><<<grow, rblk, 0, s>>>(b);
    k_big_cols<BL, 0><<<gcol0, blk, big_cols_smem<BL, 0>(), s>>>(b);
  }
  if (b.kh == 5) k_big_modulus<BL, 5><<<gmod, kModTpb<BL>, big_mod_smem<BL, 5>(), s>>>(b);
  else k_big_modulus<BL, 15><<<gmod, kModTpb<BL>, big_mod_smem<BL, 15>(), s>>>(b);
  if (!full) return cudaGetLastError();
  if (b.near_field) {
    k_big_rows<BL, 1, true><<<grow, rblk, 0, s>>>(b);
    k_big_cols<BL, 3><<<gcol, blk, big_cols_smem<BL, 3>(), s>>>(b);
    return big_final<BL, true>(b, nc, s);
  }
  k_big_cols<BL, 1><<<gcol, blk, big_cols_smem<BL, 1>(), s>>>(b);
  return big_final<BL, false>(b, nc, s);
}

static cudaError_t big_dispatch(const BigArgs& b, int nc, bool full, cudaStream_t s) {
  if (b.M == 256) return big_passes<256>(b, nc, full, s);
  if (b.M == 512) return big_passes<512>(b, nc, full, s);
  return cudaErrorInvalidValue;
}

cudaError_t launch_big_chunk(const BigArgs& b, int nc, cudaStream_t s) { return big_dispatch(b, nc, true, s); }

cudaError_t launch_big_chunk_dm(const BigArgs& b, int nc, cudaStream_t s) {
  if (!b.psi) return cudaErrorInvalidValue;
  BigArgs e = b;
  e.dm_pass = 1;  // the estimate P o_n through the propagation and the model, for the error only
  cudaError_t err = big_dispatch(e, nc, false, s);
  if (err != cudaSuccess) return err;
  e.dm_pass = 2;  // chi = 2 P o_n - psi_n: its modulus ratio, back-propagation, state update
  return big_dispatch(e, nc, true, s);
}

}  // namespace ptycho
