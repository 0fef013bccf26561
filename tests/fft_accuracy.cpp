// The double-precision register FFT of the step kernels (fft_block.cuh), run on
// the CPU with a thread per GPU thread, against a long double DFT: prints the
// relative rms error of the forward and inverse transform for each length.
#include <cuda_runtime.h>

#include <barrier>
#include <cmath>
#include <cstdio>
#include <random>
#include <thread>
#include <vector>

static inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static inline double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
static inline void __syncthreads() {}
template <class T> T __ldg(const T* p) { return *p; }
#include "fft_block.cuh"

struct Sync {
  std::barrier<>* b;
  void operator()() const { b->arrive_and_wait(); }
};

int main() {
  using namespace shf;
  const long double pi2 = 2 * acosl(-1.0L);
  std::vector<double2> table(stage_table_len());
  for (int a = 1; a < LOG2_NMAX; ++a)
    for (int lr = 1; lr <= 3 && a + lr <= LOG2_NMAX; ++lr)
      for (int j = 0; j < 2 << a; ++j) {
        const long double th = pi2 * j / (1 << (a + lr));
        table[2 * stage_table_offset(a, lr) + j] = {(double)cosl(th), (double)sinl(th)};
      }
  std::mt19937_64 gen(7);
  std::normal_distribution<double> noise;
  for (int ln : {4, 5, 6, 7, 8, 9, 10}) {
    const int N = 1 << ln, T = N / kP, trials = ln <= 6 ? 64 : ln <= 8 ? 16 : 4;
    std::vector<double2> tws(2 * compact_stage_pairs(LOG2_NMAX, kLogP));
    stage_tables_to_smem(tws.data(), table.data(), ln, kLogP, 0, 1);
    std::vector<long double> c(N), s(N);
    for (int k = 0; k < N; ++k) c[k] = cosl(pi2 * k / N), s[k] = sinl(pi2 * k / N);
    long double err[2] = {};
    for (int trial = 0; trial < trials; ++trial) {
      std::vector<double2> x(N), got[2], buf[2];
      for (auto& v : x) v = {noise(gen), noise(gen)};
      for (int d = 0; d < 2; ++d) got[d].resize(N), buf[d].resize(padded_len(N));
      std::barrier<> bar(T);
      std::vector<std::thread> threads;
      for (int t = 0; t < T; ++t)
        threads.emplace_back([&, t] {
          const Sync sync{&bar};
          for (int d = 0; d < 2; ++d) {
            double2 v[kP];
            for (int q = 0; q < kP; ++q) v[q] = x[t + q * T];
            if (d) fft_reg<true>(v, ln, t, buf[d].data(), tws.data(), sync);
            else fft_reg<false>(v, ln, t, buf[d].data(), tws.data(), sync);
            for (int q = 0; q < kP; ++q) got[d][t + q * T] = v[q];
          }
        });
      for (auto& t : threads) t.join();
      for (int d = 0; d < 2; ++d) {
        long double e2 = 0, n2 = 0;
        for (int k = 0; k < N; ++k) {
          long double re = 0, im = 0;
          for (int i = 0; i < N; ++i) {
            const int p = (int)((long)i * k % N);
            const long double sp = d ? s[p] : -s[p];
            re += x[i].x * c[p] - x[i].y * sp;
            im += x[i].x * sp + x[i].y * c[p];
          }
          const long double dr = got[d][k].x - re, di = got[d][k].y - im;
          e2 += dr * dr + di * di;
          n2 += re * re + im * im;
        }
        err[d] += e2 / n2;
      }
    }
    std::printf("%d %.4Le %.4Le\n", N, sqrtl(err[0] / trials), sqrtl(err[1] / trials));
  }
}
