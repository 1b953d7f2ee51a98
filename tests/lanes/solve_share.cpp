// The elimination of the double-float parameter families (TermBlock::solve_share):
// every access to the rows in shared memory is ordered.
#include "lanes.h"

#include "term_block.cuh"

template <int N, int NW>
int check(unsigned seed) {
  using B = hc::TermBlock<N, NW>;
  std::vector<double> store(B::acc_bytes() / 8 + 2, 0.0);
  unsigned char* acc = reinterpret_cast<unsigned char*>(store.data() + ((uintptr_t)store.data() / 8 & 1));
  lanes::m().watched.clear();
  lanes::watch(acc, B::acc_bytes());
  auto* A = reinterpret_cast<hc::cx<hc::df>*>(acc);
  uint64_t r = seed + 17;
  double a[N][N + 1][2];
  for (int i = 0; i < N; ++i)
    for (int j = 0; j <= N; ++j)
      for (int c = 0; c < 2; ++c) {
        r = r * 6364136223846793005ull + 1442695040888963407ull;
        a[i][j][c] = (double)(int64_t)r / 9.3e18;
      }
  for (int j = 0; j <= N; ++j)
    for (int i = 0; i < N; ++i)
      A[B::LR * j + i] = hc::to_cxdf(hc::mk<double>(a[i][j][0], a[i][j][1]));
  double x[N][2];
  bool ok = true;
  const int races = lanes::run(32 * NW, seed, [&] {
    const hc::Group g = hc::make_group<32>();
    B h{nullptr, 0, g, nullptr, nullptr, nullptr, acc};
    hc::cx<hc::df> dinv;
    int col;
    const bool fine = h.solve_share(N + 1, dinv, col);
    if (!fine) ok = false;
    if (threadIdx.x < 32 && col >= 0) {
      const hc::cx<hc::df> v = A[N * B::LR + (g.wl & (B::LR - 1))] * dinv;
      x[col][0] = (double)hc::re_of(v);
      x[col][1] = (double)hc::im_of(v);
    }
  });
  double worst = 0.0;
  for (int i = 0; i < N; ++i) {
    double re = -a[i][N][0], im = -a[i][N][1];
    for (int j = 0; j < N; ++j) {
      re += a[i][j][0] * x[j][0] - a[i][j][1] * x[j][1];
      im += a[i][j][0] * x[j][1] + a[i][j][1] * x[j][0];
    }
    worst = std::max(worst, std::fabs(re) + std::fabs(im));
  }
  // residual of a backward stable elimination in 48 bits, |A| |x| up to a few hundred
  if (!ok || !(worst < 1e-9)) {
    std::printf("N %d, %d warps: residual %g\n", N, NW, worst);
    return races + 1;
  }
  return races;
}

int main() {
  int bad = 0;
  for (unsigned seed = 0; seed < 3; ++seed)
    bad += check<1, 1>(seed) + check<3, 1>(seed) + check<4, 1>(seed) + check<7, 1>(seed) +
           check<8, 2>(seed) + check<12, 4>(seed) + check<18, 4>(seed) + check<18, 1>(seed);
  return bad != 0;
}
