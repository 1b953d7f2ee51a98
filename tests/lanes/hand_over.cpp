// The two loops of the mixed tracking kernels (run_tracker): what the first loop
// hands over is ordered before the second loop's reads, and every path is finished
// once -- or, under a step budget, as many as it allows.  The problem: x_i' = 1 from
// 1 + i at t = 0, an identity Jacobian.
#include "lanes.h"

#include "tracker.cuh"

template <int N, int L>
struct Straight {
  static constexpr int PARTS = 1, ROWL = L, WARPS = 1;
  static constexpr bool kCoop = false;
  hc::GroupMem sm;
  __device__ void init(const hc::Group&) const {}
  __device__ hc::cx<double> start(int64_t path, int i) const {
    return hc::mk<double>(1.0 + i, (double)path);
  }
  template <class R>
  __device__ void eval(const hc::cx<R> (&)[N], int i, R t, R, hc::cx<R> (&row)[N + 1],
                       hc::cx<R>& H, hc::cx<R>& Ht) const {
    const int ii = i < N ? i : 0;
    for (int j = 0; j < N; ++j) row[j] = hc::mk<R>(R(j == ii), R(0));
    const hc::cx<float> x = sm.vf[ii];
    H = hc::mk<R>(R(x.re) - R(1 + ii) - t, R(0));
    Ht = hc::mk<R>(R(-1), R(0));
  }
  template <bool SCALE>
  __device__ void residual_df(const hc::cdf* xs, int i, double t, hc::cx<float>& H,
                              float& sc) const {
    const int ii = i < N ? i : 0;
    H = hc::mk<float>((float)((double)xs[ii].re() - 1.0 - ii - t), 0.f);
    sc = 4.f;
  }
  template <bool SCALE>
  __device__ void residual64(const hc::cx<double>* xs, int i, double t, double,
                             hc::cx<double>& H, double& sc) const {
    const int ii = i < N ? i : 0;
    H = hc::mk<double>(xs[ii].re - 1.0 - ii - t, 0.0);
    sc = 4.0;
  }
};
template <int N, int L>
struct StraightProblem {
  hc::GroupMem sm;
  __device__ Straight<N, L> hom(int64_t) const { return {sm}; }
};

template <int N, int L>
int check(unsigned seed, int warps, int items, int max_steps_fp32, unsigned long long budget) {
  std::vector<double> smem(hc::block_smem_bytes(L, 0, 0, 32 * warps) / 8 + 2, 0.0);
  unsigned char* mem =
      reinterpret_cast<unsigned char*>(smem.data() + ((uintptr_t)smem.data() / 8 & 1));
  std::vector<double> x(2 * N * items, 0.0);
  std::vector<uint8_t> status(items, 0);
  std::vector<int32_t> steps(3 * items, 0);
  std::vector<unsigned long long> link(items, ~0ull), ctl(4, 0);
  hc::LaunchCommon c;
  std::memset(&c, 0, sizeof c);
  hc::DevSettings& s = c.s;
  s.dt_min = 1e-8, s.dt_max = 0.1, s.dt_init = 0.05, s.newton_tol = 1e-10;
  s.newton_tol_fp32 = 1e-5, s.max_first_corr = 0.1, s.max_first_corr_fp32 = 0.1;
  s.refine_tol = 1e-12, s.r_inf = 1e6, s.finite_tol = 1e-6, s.real_tol = 1e-8;
  s.singular_cond = 1e12, s.t_endgame = 0.9, s.dt_min_fp32 = 1e-4;
  s.max_newton = s.max_newton_ir = 3, s.max_steps = 1000, s.grow_after = 2;
  s.refine_iters = 3, s.max_steps_fp32 = max_steps_fp32;
  c.n_items = c.paths = items;
  c.queue = &ctl[0];
  c.step_total = &ctl[1];
  c.step_budget = budget;
  c.x_out = x.data();
  c.status_out = status.data();
  c.steps_out = steps.data();
  c.hand_list = link.data();
  c.items_step = 1;
  lanes::m().watched.clear();
  lanes::m().atomics.clear();
  lanes::watch(mem, hc::block_smem_bytes(L, 0, 0, 32 * warps));
  lanes::watch(x.data(), 8 * x.size());
  lanes::watch(status.data(), status.size(), 1);
  lanes::watch(steps.data(), 4 * steps.size());
  lanes::watch(link.data(), 8 * link.size());
  lanes::watch(ctl.data(), 8 * ctl.size());
  lanes::atomic_word(&ctl[0]);
  lanes::atomic_word(&ctl[1]);
  lanes::atomic_word(mem + hc::group_smem_bytes(L, 0) - 16);
  int bad = lanes::run(32 * warps, seed, [&] {
    const hc::Group g = hc::make_group<L, true>();
    const hc::GroupMem sm = hc::make_group_mem<L>(mem, 0);
    const StraightProblem<N, L> prob{sm};
    if (budget)
      hc::run_tracker<N, L, true, StraightProblem<N, L>, double, hc::F_BUDGET>(prob, c, g, sm);
    else
      hc::run_tracker<N, L, true, StraightProblem<N, L>>(prob, c, g, sm);
  });
  int begun = 0;
  for (int k = 0; k < items; ++k) begun += steps[3 * k] != 0;
  const int groups = 32 / L * warps;
  // a path takes 10 steps at least: three finished ones exceed 26
  if (budget == 26 && begun > groups + 2) {
    std::printf("%d paths begun by %d groups under a budget of two paths\n", begun, groups);
    return bad + 1;
  }
  for (int k = 0; k < items; ++k)
    if ((status[k] & 0x7f) != 1 || std::fabs(x[2 * N * k] - 2.0) > 1e-10 || steps[3 * k] < 10) {
      if (budget && !status[k]) continue;
      std::printf("path %d: status %d x %.12g steps %d\n", k, status[k], x[2 * N * k], steps[3 * k]);
      return bad + 1;
    }
  return bad;
}

int main() {
  int bad = 0;
  for (unsigned seed = 0; seed < 3; ++seed)
    bad += check<2, 4>(seed, 1, 20, 1000, 0) + check<3, 8>(seed, 2, 30, 1000, 0) +
           check<3, 16>(seed, 3, 17, 3, 0) + check<2, 8>(seed, 2, 9, 1, 0) +
           check<2, 8>(seed, 2, 60, 1, 26) + check<2, 8>(seed, 2, 20, 5, 1ull << 40);
  return bad != 0;
}
