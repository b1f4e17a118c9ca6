// Host check of gj_block.cuh: 256 threads, one running at a time from barrier to barrier, in several orders of the
// threads (any order is allowed between two barriers). Whatever the order, the result has to be the inverse.
#include <algorithm>
#include <cmath>
#include <complex>
#include <condition_variable>
#include <cstdio>
#include <mutex>
#include <numeric>
#include <random>
#include <thread>
#include <vector>

#include "gj_block.cuh"

struct Cplx {
  using S = std::complex<double>;
  static S zero() { return 0.0; }
  static S neg(S a) { return -a; }
  static bool is_zero(S a) { return a == S(0.0); }
  static S inv(S a) { return 1.0 / a; }
  static S fma2(S a, S x, S y) { return a + x * y; }
};

constexpr int T = 256;

// Baton scheduler: the first thread in `order` that does not wait at a barrier runs next. A block barrier opens
// when every thread that has not finished is at it, a warp barrier when the 32 threads of the warp are.
struct Sched {
  enum { RUN, WARP, BLOCK, DONE };
  std::mutex m;
  std::condition_variable cv[T];
  std::vector<int> order, state = std::vector<int>(T, RUN);
  int current = -1;
  void open() {
    int live = 0, at = 0;
    for (int s : state) {
      live += s != DONE;
      at += s == BLOCK;
    }
    if (live && at == live)
      for (int& s : state)
        if (s == BLOCK) s = RUN;
    for (int w = 0; w < T; w += 32)
      if (std::all_of(state.begin() + w, state.begin() + w + 32, [](int s) { return s == WARP; }))
        std::fill(state.begin() + w, state.begin() + w + 32, (int)RUN);
  }
  void next() {
    open();
    current = -1;
    for (int t : order)
      if (state[t] == RUN) {
        current = t;
        cv[t].notify_one();
        return;
      }
  }
  void stop(int t, int s) {  // thread t reaches a barrier or its end
    std::unique_lock<std::mutex> l(m);
    state[t] = s;
    next();
    if (s != DONE) cv[t].wait(l, [&] { return current == t; });
  }
  void start(int t) {
    std::unique_lock<std::mutex> l(m);
    cv[t].wait(l, [&] { return current == t; });
  }
};

struct Sync {
  Sched* s;
  int t;
  void block() const { s->stop(t, Sched::BLOCK); }
  void warp() const { s->stop(t, Sched::WARP); }
};

int main() {
  using S = Cplx::S;
  std::mt19937 gen(3);
  std::normal_distribution<double> nd;
  std::vector<S> A(32 * 32);
  for (int i = 0; i < 32; ++i)
    for (int j = 0; j < 32; ++j) A[32 * i + j] = S(nd(gen), nd(gen)) * 0.05 + (i == j ? S(2.0) : S(0.0));
  int bad = 0;
  for (int o = 0; o < 4; ++o) {
    Sched sc;
    sc.order.resize(T);
    std::iota(sc.order.begin(), sc.order.end(), 0);
    if (o == 1) std::reverse(sc.order.begin(), sc.order.end());
    if (o > 1) std::shuffle(sc.order.begin(), sc.order.end(), gen);
    std::vector<S> B = A, fcol(32), prow(32), rowj(32);
    std::vector<int> rc(T, -2);
    std::vector<std::thread> th;
    for (int t = 0; t < T; ++t)
      th.emplace_back([&, t] {
        sc.start(t);
        const int tx = t & 15, ty = t >> 4;
        S x[2][2];
        for (int a = 0; a < 2; ++a)
          for (int b = 0; b < 2; ++b) x[a][b] = B[32 * (ty + 16 * a) + tx + 16 * b];
        rc[t] = gwi::gj_invert32<Cplx>(x, fcol.data(), prow.data(), rowj.data(), t, Sync{&sc, t});
        for (int a = 0; a < 2; ++a)
          for (int b = 0; b < 2; ++b) B[32 * (ty + 16 * a) + tx + 16 * b] = x[a][b];
        sc.stop(t, Sched::DONE);
      });
    {
      std::lock_guard<std::mutex> l(sc.m);
      sc.next();
    }
    for (auto& t : th) t.join();
    double err = 0.0;
    for (int i = 0; i < 32; ++i)
      for (int j = 0; j < 32; ++j) {
        S s = i == j ? -1.0 : 0.0;
        for (int k = 0; k < 32; ++k) s += A[32 * i + k] * B[32 * k + j];
        err = std::max(err, std::abs(s));
      }
    const bool ok = err < 1e-13 && std::all_of(rc.begin(), rc.end(), [](int r) { return r == -1; });
    bad += !ok;
    std::printf("order %d: |A A^-1 - 1| = %.1e%s\n", o, err, ok ? "" : "  WRONG");
  }
  std::printf("%d orders wrong\n", bad);
  return bad != 0;
}
