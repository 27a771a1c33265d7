// Runs fp_decide (fp_stop.cuh) for one block on host threads, with a status word that another
// block changes after `n` of this block's reads of it.  Prints, per n, how many threads returned
// true, how many false, and how many took part in the sum.
#include <atomic>
#include <barrier>
#include <cmath>
#include <cstdio>
#include <functional>
#include <thread>
#include <vector>

struct Idx { unsigned x; };
static thread_local Idx threadIdx;
static thread_local Idx blockIdx{1};
static std::barrier<>* g_bar;
static void sync_threads() { g_bar->arrive_and_wait(); }
#define __CUDACC__
#define __device__
#define __forceinline__ inline
#define __shared__ static
#define __syncthreads sync_threads
using std::isfinite;
using std::sqrt;
#include "fp_stop.cuh"

struct Word {   // a scalar that other blocks may change between two reads
  double before = 0.0, after = 0.0;
  int n = 1 << 30;
  std::atomic<int> reads{0};
};
struct Ref {
  Word* w;
  operator double() const { return w->reads++ < w->n ? w->before : w->after; }
  void operator=(double v) const { w->before = w->after = v; }
};
struct Scalars {
  Word* w;
  Ref operator[](int q) const { return Ref{w + q}; }
};

int main() {
  constexpr int kThreads = 64;
  for (double stop : {1.0, 3.0})
    for (int n = 0; n <= kThreads + 2; ++n) {
      Word sc[16];
      // block 0 stops the loop: converged (1), or at the iteration limit (3)
      sc[afc::F_THRESH].before = sc[afc::F_THRESH].after = stop == 1.0 ? 10.0 : 1e-3;
      sc[afc::F_MAXIT].before = sc[afc::F_MAXIT].after = 5.0;
      sc[afc::F_CORR].before = sc[afc::F_CORR].after = stop == 1.0 ? 2.0 : 5.0;
      sc[afc::F_STATUS].after = stop;
      sc[afc::F_STATUS].n = n;
      std::barrier<> bar(kThreads);
      g_bar = &bar;
      std::atomic<int> yes{0}, no{0}, summed{0};
      std::vector<std::thread> ts;
      for (unsigned t = 0; t < kThreads; ++t)
        ts.emplace_back([&, t] {
          threadIdx.x = t;
          const bool go = afc::fp_decide(
              Scalars{sc},
              [&] {
                ++summed;
                sync_threads();
                sync_threads();
                return 1.0;
              },
              [](bool) {});
          ++(go ? yes : no);
          bar.arrive_and_drop();   // a thread that left no longer meets the others
        });
      for (auto& t : ts) t.join();
      std::printf("%g %d %d %d %d\n", stop, n, yes.load(), no.load(), summed.load());
    }
}
