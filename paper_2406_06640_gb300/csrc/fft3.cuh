// 2-D transform of an M x M tile (M = 64, 128) in three register passes with two exchanges.
//
// The row / transpose / column form of fft.cuh moves the tile through shared memory three times (two
// line-internal swaps and the transpose), which bounds it: at M = 128 a transform takes 4.7 us on an SM,
// 3.0 of them shared-memory wavefronts. With 16 S values per thread (S = M / 64) the 2 log2 M index bits
// need only three passes, so two exchanges; decimation in frequency along both axes at once:
//   ROW layout     thread tid = NT yl + t, NT = M / 16: register a[s][j] holds line yl + 64 s, x = t + NT j (the
//                  ROW layout of fft.cuh)
//   pass A         DFT-16 over j -> k2, DFT-S over s -> frequency bit s of y; twiddle W_M^(t k2)
//   exchange 1     slot tid + k2 L1 + s 16 L1: consecutive threads write consecutive slots; the reader of
//                  (s, k2, yb) takes its NT values of t as 16-byte pairs for yl = yb + 16 ya (L1 even, L1 / 2 odd:
//                  eight lanes of neighbouring k2 fall into the eight 16-byte banks)
//   pass B         thread (k2, yb, s) = (tid % 16, tid / 16 % 16, tid / 256): DFT-4 over ya -> ka, DFT-NT over
//                  t -> k1. The twiddle of line yl = yb + 16 ya for bit s is split: W_8^(ya s) in front of
//                  the DFT-4 (no table; s is uniform over a warp), W_M^(yb s) together with W_64^(yb ka)
//                  behind it: one multiplication fewer per value than W_M^(yl s) in pass A. The DFT-4 comes
//                  first for the rounding: a model whose dark pixels amplify it (200 counts per pattern, flat
//                  start, 12 global phases of the probe) deviates from FP64 by 6.9e-5 in the median and
//                  8.8e-5 at most, against 8.9e-5 and 1.3e-4 with the DFT-NT in front (7.0e-5 and 1.1e-4 for
//                  the row / transpose / column form).
//   exchange 2     slot col + M (ka + 4 yb + 64 s), col = k2 + 16 k1: both sides run along col
//   pass C         thread (col, ka) = (tid % M, tid / M): DFT-16 over yb -> kb
//   FREQ layout    register a[s][kb] holds frequency row s + S (ka + 4 kb), column col
// The inverse runs the steps mirrored and returns to the ROW layout (unscaled: times M^2); its pass B takes the
// DFT-4 first as well, right behind the twiddles (632 -> 628 us an iteration of 900 x 128^2, four modes; dark
// pixels do not see the inverse's rounding: the deviations above are the same).
// (The slots of both exchanges are bijections onto [0, 16 S L1) and [0, M^2); conflict-free throughout.)
#pragma once
#include <cuda_runtime.h>

#include "fft.cuh"

namespace ptycho {

template <int M_>
struct Tile3 {
  static constexpr int M = M_, S = M / 64, NT = M / 16, THREADS = 4 * M;
  static constexpr int L1 = THREADS + 2;
  static constexpr int SMEM = 16 * S * L1;  // float2 slots (>= M * M)
  static constexpr int TW2 = 64 * S;        // W_M^(yb (S ka + s)) at (s * 16 + yb) * 4 + ka
  // exponent e of the table entry i: W_M^e
  __host__ __device__ static constexpr int tw2_exp(int i) { return i / 4 % 16 * (S * (i % 4) + i / 64) % M; }
  static_assert((M == 64 || M == 128) && SMEM >= M * M, "M = 64 or 128");
  __device__ __forceinline__ static int freq_row(int tid, int s, int kb) { return s + S * (tid / M + 4 * kb); }
  __device__ __forceinline__ static int freq_col(int tid) { return tid % M; }
};

// exchange buffer of a fused kernel's 2-D transform: this file's for M = 64 and 128, fft.cuh's below
template <int M, bool F3 = (M >= 64)>
struct ExchangeBytes {
  static constexpr size_t value = (size_t)Tile<M>::SMEM * 8;
};
template <int M>
struct ExchangeBytes<M, true> {
  static constexpr size_t value = (size_t)Tile3<M>::SMEM * 8;
};

// tw[t * 17 + k2] = W_M^(t k2), tw2 the table described at Tile3::TW2.
// The shared buffer must be free on entry; it is free again on return.
template <int M>
__device__ __forceinline__ void fft3_forward(float2 (&a)[Tile3<M>::S][16], float2* sm, const float2* tw,
                                             const float2* tw2, int tid) {
  using T = Tile3<M>;
  constexpr int S = T::S, NT = T::NT, L1 = T::L1;
  // ---- pass A
  const float2* twt = tw + tid % NT * 17;
#pragma unroll
  for (int s = 0; s < S; ++s) dft<16, false>(a[s]);
#pragma unroll
  for (int k2 = 0; k2 < 16; ++k2) {
    if constexpr (S == 2) {
      const float2 d = csub(a[0][k2], a[S - 1][k2]);
      a[0][k2] = cadd(a[0][k2], a[S - 1][k2]);
      a[S - 1][k2] = d;
    }
    if (k2 > 0) {
      const float2 w = twt[k2];
#pragma unroll
      for (int s = 0; s < S; ++s) a[s][k2] = cmul(a[s][k2], w);
    }
#pragma unroll
    for (int s = 0; s < S; ++s) sm[tid + k2 * L1 + s * 16 * L1] = a[s][k2];
  }
  __syncthreads();
  // ---- pass B
  const int k2 = tid % 16, yb = tid / 16 % 16, sb = tid / 256;
  float2 b[4][NT];
  {
    const float2* q = sm + sb * 16 * L1 + k2 * L1 + yb * NT;
#pragma unroll
    for (int ya = 0; ya < 4; ++ya)
#pragma unroll
      for (int t = 0; t < NT; t += 2) {
        const float4 v = *reinterpret_cast<const float4*>(q + ya * 16 * NT + t);
        b[ya][t] = make_float2(v.x, v.y);
        b[ya][t + 1] = make_float2(v.z, v.w);
      }
  }
  if (S == 2 && sb) {
#pragma unroll
    for (int k1 = 0; k1 < NT; ++k1) {
      b[1][k1] = mul_w16<false, 2>(b[1][k1]);
      b[2][k1] = mul_w16<false, 4>(b[2][k1]);
      b[3][k1] = mul_w16<false, 6>(b[3][k1]);
    }
  }
#pragma unroll
  for (int k1 = 0; k1 < NT; ++k1) dft4<false>(b[0][k1], b[1][k1], b[2][k1], b[3][k1]);
#pragma unroll
  for (int ya = 0; ya < 4; ++ya) dft<NT, false>(b[ya]);
#pragma unroll
  for (int ka = 0; ka < 4; ++ka) {
    if (ka == 0 && !(S == 2 && sb)) continue;
    const float2 w = tw2[(sb * 16 + yb) * 4 + ka];
#pragma unroll
    for (int k1 = 0; k1 < NT; ++k1) b[ka][k1] = cmul(b[ka][k1], w);
  }
  __syncthreads();
  {
    float2* q = sm + k2 + M * (4 * yb + 64 * sb);
#pragma unroll
    for (int ka = 0; ka < 4; ++ka)
#pragma unroll
      for (int k1 = 0; k1 < NT; ++k1) q[16 * k1 + M * ka] = b[ka][k1];
  }
  __syncthreads();
  // ---- pass C
  const float2* q = sm + tid % M + M * (tid / M);
#pragma unroll
  for (int s = 0; s < S; ++s) {
#pragma unroll
    for (int i = 0; i < 16; ++i) a[s][i] = q[M * (4 * i + 64 * s)];
    dft<16, false>(a[s]);
  }
  __syncthreads();
}

template <int M>
__device__ __forceinline__ void fft3_inverse(float2 (&a)[Tile3<M>::S][16], float2* sm, const float2* tw,
                                             const float2* tw2, int tid) {
  using T = Tile3<M>;
  constexpr int S = T::S, NT = T::NT, L1 = T::L1;
  {
    float2* q = sm + tid % M + M * (tid / M);
#pragma unroll
    for (int s = 0; s < S; ++s) {
      dft<16, true>(a[s]);
#pragma unroll
      for (int i = 0; i < 16; ++i) q[M * (4 * i + 64 * s)] = a[s][i];
    }
  }
  __syncthreads();
  const int k2 = tid % 16, yb = tid / 16 % 16, sb = tid / 256;
  float2 b[4][NT];
  {
    const float2* q = sm + k2 + M * (4 * yb + 64 * sb);
#pragma unroll
    for (int ka = 0; ka < 4; ++ka) {
      const float2 w = tw2[(sb * 16 + yb) * 4 + ka];
#pragma unroll
      for (int k1 = 0; k1 < NT; ++k1) {
        b[ka][k1] = q[16 * k1 + M * ka];
        if (ka > 0 || (S == 2 && sb)) b[ka][k1] = cmulc(b[ka][k1], w);
      }
    }
  }
#pragma unroll
  for (int k1 = 0; k1 < NT; ++k1) dft4<true>(b[0][k1], b[1][k1], b[2][k1], b[3][k1]);
  if (S == 2 && sb) {
#pragma unroll
    for (int k1 = 0; k1 < NT; ++k1) {
      b[1][k1] = mul_w16<true, 2>(b[1][k1]);
      b[2][k1] = mul_w16<true, 4>(b[2][k1]);
      b[3][k1] = mul_w16<true, 6>(b[3][k1]);
    }
  }
#pragma unroll
  for (int ya = 0; ya < 4; ++ya) dft<NT, true>(b[ya]);
  __syncthreads();
  {
    float2* q = sm + sb * 16 * L1 + k2 * L1 + yb * NT;
#pragma unroll
    for (int ya = 0; ya < 4; ++ya)
#pragma unroll
      for (int t = 0; t < NT; t += 2)
        *reinterpret_cast<float4*>(q + ya * 16 * NT + t) =
            make_float4(b[ya][t].x, b[ya][t].y, b[ya][t + 1].x, b[ya][t + 1].y);
  }
  __syncthreads();
  const float2* twt = tw + tid % NT * 17;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
#pragma unroll
    for (int s = 0; s < S; ++s) a[s][i] = sm[tid + i * L1 + s * 16 * L1];
    if (i > 0) {
      const float2 w = twt[i];
#pragma unroll
      for (int s = 0; s < S; ++s) a[s][i] = cmulc(a[s][i], w);
    }
    if constexpr (S == 2) {
      const float2 d = a[S - 1][i];
      a[S - 1][i] = csub(a[0][i], d);
      a[0][i] = cadd(a[0][i], d);
    }
  }
#pragma unroll
  for (int s = 0; s < S; ++s) dft<16, true>(a[s]);
  __syncthreads();
}

}  // namespace ptycho
