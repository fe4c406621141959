// Host run of the three-pass 2-D transform of csrc/fft3.cuh, as tests/fft_host_emu.cpp runs fft.cuh: one
// std::thread per CUDA thread, a std::barrier for __syncthreads. Besides the transforms it checks that
// every slot of both exchanges stays inside the buffer (a guard zone behind it stays untouched).
// Usage: fft3_host_emu M -> "forward <rel L2>  roundtrip <rel L2>  guard <0 or 1>"
#include <barrier>
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <thread>
#include <vector>

static std::barrier<>* g_bar;
#define __syncthreads() g_bar->arrive_and_wait()
#define __syncwarp() g_bar->arrive_and_wait()
#include "fft3.cuh"

using namespace ptycho;
using cd = std::complex<double>;

template <int M>
static int run() {
  using T = Tile3<M>;
  constexpr int S = T::S, NT = T::NT, TR = T::THREADS;
  std::mt19937 rng(M);
  std::normal_distribution<double> nd;
  std::vector<cd> A(M * M);
  for (auto& z : A) z = cd(nd(rng), nd(rng));
  auto W = [](long e) {
    const double t = -2.0 * M_PI * (double)(((e % M) + M) % M) / M;
    return cd(std::cos(t), std::sin(t));
  };
  auto f2 = [](cd z) { return make_float2((float)z.real(), (float)z.imag()); };
  // 16-byte aligned buffer with a guard zone
  std::vector<float4> store(T::SMEM / 2 + 64);
  float2* sm = reinterpret_cast<float2*>(store.data());
  for (int i = 0; i < 128; ++i) sm[T::SMEM + i] = make_float2(12345.f, -1.f);
  std::vector<float2> tw(NT * 17), tw2(T::TW2);
  for (int t = 0; t < NT; ++t)
    for (int k = 0; k < 16; ++k) tw[t * 17 + k] = f2(W((long)t * k));
  for (int i = 0; i < T::TW2; ++i) tw2[i] = f2(W(T::tw2_exp(i)));
  std::vector<cd> F(M * M), B(M * M);
  std::barrier<> bar(TR);
  g_bar = &bar;
  std::vector<std::thread> th;
  for (int tid = 0; tid < TR; ++tid)
    th.emplace_back([&, tid] {
      float2 a[S][16];
      const int yl = tid / NT, t = tid % NT;
      for (int s = 0; s < S; ++s)
        for (int j = 0; j < 16; ++j) a[s][j] = f2(A[(yl + 64 * s) * M + t + NT * j]);
      fft3_forward<M>(a, sm, tw.data(), tw2.data(), tid);
      for (int s = 0; s < S; ++s)
        for (int r = 0; r < 16; ++r) F[T::freq_row(tid, s, r) * M + T::freq_col(tid)] = cd(a[s][r].x, a[s][r].y);
      fft3_inverse<M>(a, sm, tw.data(), tw2.data(), tid);
      for (int s = 0; s < S; ++s)
        for (int j = 0; j < 16; ++j) B[(yl + 64 * s) * M + t + NT * j] = cd(a[s][j].x, a[s][j].y);
    });
  for (auto& t : th) t.join();
  std::vector<cd> R(M * M), Y(M * M);
  for (int y = 0; y < M; ++y)
    for (int v = 0; v < M; ++v) {
      cd s = 0;
      for (int x = 0; x < M; ++x) s += A[y * M + x] * W((long)v * x);
      R[y * M + v] = s;
    }
  for (int u = 0; u < M; ++u)
    for (int v = 0; v < M; ++v) {
      cd s = 0;
      for (int y = 0; y < M; ++y) s += R[y * M + v] * W((long)u * y);
      Y[u * M + v] = s;
    }
  double e1 = 0, n1 = 0, e2 = 0, n2 = 0;
  for (int i = 0; i < M * M; ++i) {
    e1 += std::norm(F[i] - Y[i]);
    n1 += std::norm(Y[i]);
    e2 += std::norm(B[i] / (double)(M * M) - A[i]);
    n2 += std::norm(A[i]);
  }
  int guard = 1;
  for (int i = 0; i < 128; ++i) guard &= sm[T::SMEM + i].x == 12345.f && sm[T::SMEM + i].y == -1.f;
  std::printf("forward %.3e roundtrip %.3e guard %d\n", std::sqrt(e1 / n1), std::sqrt(e2 / n2), guard);
  return 0;
}

int main(int argc, char** argv) {
  if (argc != 2) return 2;
  const int M = std::atoi(argv[1]);
  return M == 64 ? run<64>() : M == 128 ? run<128>() : 2;
}
