// Whole tracking kernels on the CPU (term tables and dense tables, every precision):
// every access to shared data is ordered and every path ends.
#include "lanes.h"

#include "dense_kernel.cuh"
#include "term_block.cuh"
#include "term_param.cuh"

static hc::DevSettings settings() {
  hc::DevSettings s;
  std::memset(&s, 0, sizeof s);
  s.dt_min = 1e-3, s.dt_max = 0.25, s.dt_init = 0.25, s.newton_tol = 1e-9;
  s.newton_tol_fp32 = 1e-5, s.max_first_corr = 0.5, s.max_first_corr_fp32 = 0.5;
  s.refine_tol = 1e-10, s.r_inf = 1e6, s.finite_tol = 1e-3, s.real_tol = 1e-8;
  s.singular_cond = 1e12, s.t_endgame = 0.9, s.dt_min_fp32 = 1e-2;
  s.max_newton = s.max_newton_ir = 4, s.max_steps = 40, s.grow_after = 2;
  s.refine_iters = 3, s.max_steps_fp32 = 20;
  return s;
}

struct Outputs {
  std::vector<double> x;
  std::vector<uint8_t> status;
  std::vector<int32_t> steps;
  std::vector<unsigned long long> link, ctl;
  void bind(hc::LaunchCommon& c, int n, int items) {
    x.assign(2 * n * items, 0.0);
    status.assign(items, 0);
    steps.assign(3 * items, 0);
    link.assign(items, 0);
    ctl.assign(4, 0);
    std::memset(&c, 0, sizeof c);
    c.s = settings();
    c.n_items = c.paths = items;
    c.queue = &ctl[0];
    c.step_total = &ctl[1];
    c.x_out = x.data();
    c.status_out = status.data();
    c.steps_out = steps.data();
    c.hand_list = link.data();
    c.items_step = 1;
    lanes::m().watched.clear();
    lanes::m().atomics.clear();
    lanes::watch(x.data(), 8 * x.size());
    lanes::watch(status.data(), status.size(), 1);
    lanes::watch(steps.data(), 4 * steps.size());
    lanes::watch(link.data(), 8 * link.size());
    lanes::watch(ctl.data(), 8 * ctl.size());
    lanes::atomic_word(&ctl[0]);
    lanes::atomic_word(&ctl[1]);
  }
  int ended() const {
    int k = 0;
    for (uint8_t s : status) k += s != 0;
    return k;
  }
};
struct Block {  // a block's dynamic shared memory
  std::vector<double> store;
  unsigned char* mem;
  explicit Block(size_t bytes) : store(bytes / 8 + 2, 0.0) {
    mem = reinterpret_cast<unsigned char*>(store.data() + ((uintptr_t)store.data() / 8 & 1));
    lanes::watch(mem, bytes);
  }
};

// Rows x_i x_i' - p x_i' - 2 x_i + 2 p, i' = i + 1 mod N, slightly scaled from row to
// row, from p = 1 to p = 1.1 + 0.2 i: the root x = p is followed.
template <int N, class RUN>
int family(unsigned seed, int L, int warps, int items, size_t smem, int head, RUN run) {
  const int TT = 4, LS = L, P = 1;
  std::vector<hc::TermRec> rec(TT * LS);
  std::vector<double2> s64(TT * LS, make_double2(0, 0));
  std::vector<hc::cdf> sdf(TT * LS);
  const double coef[4] = {1, -1, -2, 2};
  for (int k = 0; k < TT; ++k)
    for (int i = 0; i < LS; ++i) {
      hc::TermRec& r = rec[k * LS + i];
      std::memset(&r, 0, sizeof r);
      for (int f = 0; f < hc::kMaxTermFactors; ++f) r.idx[f] = (uint8_t)LS, r.tgt[f] = 255;
      r.d = k == 0 || k == 1 ? 2 : 1;
      if (i >= N) continue;
      const int j = (i + 1) % N;
      auto put = [&](int f, int v, int t) { r.idx[f] = (uint8_t)v, r.tgt[f] = (uint8_t)t; };
      if (k == 0) put(0, i, i), put(1, j, j);
      if (k == 1) put(0, LS + 1, N), put(1, j, j);
      if (k == 2) put(0, i, i);
      if (k == 3) put(0, LS + 1, N);
      const double c = coef[k] * (1.0 + 0.01 * i);
      r.s = make_float2((float)c, 0.f);
      s64[k * LS + i] = make_double2(c, 0.0);
      sdf[k * LS + i] = hc::split_cdf_host(c, 0.0);
    }
  // the summation lists, as the library builds them
  auto lists = [&](int nw, std::vector<int32_t>& ptr, std::vector<uint32_t>& ent) {
    const int NT = 32 * nw, CH = hc::term_df_slots(N, nw);
    ptr.assign(1, 0);
    ent.clear();
    for (int k0 = 0; k0 < TT; k0 += CH)
      for (int e = 0; e < N * N + N; ++e) {
        const int i = e < N * N ? e % N : e - N * N, target = e < N * N ? e / N : N;
        for (int kk = 0; kk < CH && k0 + kk < TT; ++kk) {
          const hc::TermRec& r = rec[(k0 + kk) * LS + i];
          for (int f = r.d - 1; f >= 0; --f)
            if (r.tgt[f] == target)
              ent.push_back((uint32_t)(f * NT + kk * N + i) |
                            (target == N ? (uint32_t)(r.idx[f] + P) << 16 : 0u));
        }
        ptr.push_back((int32_t)ent.size());
      }
    ent.push_back(0);
  };
  std::vector<int32_t> ptr[2];
  std::vector<uint32_t> ent[2];
  lists(1, ptr[0], ent[0]);
  lists(std::max(warps, 2), ptr[1], ent[1]);
  std::vector<double2> p0{make_double2(1, 0)}, p1{make_double2(1.1, 0.2)}, start(N * items);
  for (int k = 0; k < items; ++k)
    for (int i = 0; i < N; ++i) start[k * N + i] = make_double2(1.0 + 1e-3 * k, 0);
  hc::TermArgs a;
  std::memset(&a, 0, sizeof a);
  Outputs o;
  o.bind(a.c, N, items);
  a.rec = rec.data(), a.s64 = s64.data(), a.sdf = sdf.data();
  for (int v = 0; v < 2; ++v) a.sum_ptr[v] = ptr[v].data(), a.sum_ent[v] = ent[v].data();
  a.TT = TT, a.P = P, a.ls = LS, a.extra = 1 + 3 * P;
  a.p0 = p0.data(), a.p1 = p1.data(), a.start = start.data();
  Block b(smem);
  if (head) lanes::atomic_word(b.mem + head);
  const int bad = run(a, b.mem);
  if (o.ended() != items) {
    std::printf("N %d: %d of %d paths ended\n", N, o.ended(), items);
    return bad + 1;
  }
  return bad;
}

template <int N, int NW>
int family_df(unsigned seed, int items) {
  using B = hc::TermBlock<N, NW>;
  constexpr int L = N <= 4 ? 4 : N <= 8 ? 8 : N <= 16 ? 16 : 32;
  const int threads = NW == 1 ? 64 : 32 * NW;
  const size_t smem = hc::block_smem_bytes(32, 4, B::acc_bytes(), threads,
                                           hc::endgame_smem_bytes(32, false), 1, NW);
  return family<N>(seed, L, NW, items, smem, 0, [&](hc::TermArgs& a, unsigned char* mem) {
    return lanes::run(threads, seed, [&] {
      const hc::Group g = hc::make_group<32>();
      const hc::GroupMem sm = hc::make_group_mem<32>(mem, a.extra, B::acc_bytes(),
                                                     hc::endgame_smem_bytes(32, false), 1, NW);
      hc::TermBlockProblem<N, NW> prob{&a, g, sm};
      if (NW == 1 || threadIdx.x < 32) {
        hc::run_tracker<N, 32, false, hc::TermBlockProblem<N, NW>, hc::df>(prob, a.c, g, sm);
        if constexpr (NW > 1) prob.hom(0).post(B::OP_EXIT, 0.0, 0);
      } else {
        B h = prob.hom(0);
        h.serve();
      }
    });
  });
}

template <int N, int L, bool MIXED>
int family_rows(unsigned seed, int items) {
  constexpr int LS = N <= 4 ? 4 : N <= 8 ? 8 : N <= 16 ? 16 : 32;
  const int threads = 64, acc = hc::term_acc_bytes<N, MIXED, L>();
  const int eg = hc::endgame_smem_bytes(L, MIXED);
  const size_t smem = hc::block_smem_bytes(L, 4, acc, threads, eg);
  return family<N>(seed, LS, 1, items, smem, hc::group_smem_bytes(L, 4, acc, eg) - 16,
                   [&](hc::TermArgs& a, unsigned char* mem) {
    return lanes::run(threads, seed, [&] {
      const hc::Group g = hc::make_group<L, hc::groups_meet(L, MIXED)>();
      const hc::GroupMem sm = hc::make_group_mem<L>(mem, a.extra, acc, eg);
      hc::TermProblem<N, L, MIXED> prob{&a, g, sm};
      hc::run_tracker<N, L, MIXED, hc::TermProblem<N, L, MIXED>, double>(prob, a.c, g, sm);
    });
  });
}

// Dense kernels on random tables: most steps are rejected, which reaches every phase.
template <int N, int DEG, int PREC, int L>
int dense(unsigned seed, int items) {
  using S = hc::DenseShape<N, DEG>;
  constexpr bool MIXED = PREC == HC_PREC_MIXED, XDF = PREC == HC_PREC_DF;
  using RE = typename std::conditional<XDF, hc::df, double>::type;
  const int threads = 64, acc = hc::dense_acc_bytes<N, PREC>();
  const int eg = hc::endgame_smem_bytes(L, MIXED);
  std::vector<double> table(1 << 16);
  uint64_t r = seed + 1;
  for (size_t k = 0; k < table.size(); ++k) {
    r = r * 6364136223846793005ull + 1442695040888963407ull;
    const float f = (float)((double)(int64_t)r / 9.3e18);
    const float two[2] = {f, f * 0.5f};
    std::memcpy(&table[k], two, 8);
  }
  std::vector<double> real(1 << 16);
  for (size_t k = 0; k < real.size(); ++k) real[k] = std::sin(0.7 * k + seed);
  hc::DenseArgs a;
  std::memset(&a, 0, sizeof a);
  Outputs o;
  o.bind(a.c, N, items);
  a.D32 = (const hc::cx<float>*)table.data(), a.Ddf = (const hc::cx<hc::df>*)table.data();
  a.Edf = (const hc::cdf*)table.data();
  a.D64 = (const hc::cx<double>*)real.data(), a.E = (const hc::cx<double>*)real.data();
  a.gamma = hc::cx<double>{0.6, 0.8};
  a.gamma32 = hc::cx<float>{0.6f, 0.8f};
  a.gammadf = hc::split_cdf_host(0.6, 0.8);
  Block b(hc::block_smem_bytes(L, S::EXTRA, acc, threads, eg, XDF));
  lanes::atomic_word(b.mem + hc::group_smem_bytes(L, S::EXTRA, acc, eg, XDF) - 16);
  const int bad = lanes::run(threads, seed, [&] {
    const hc::Group g = hc::make_group<L, hc::groups_meet(L, MIXED)>();
    const hc::GroupMem sm = hc::make_group_mem<L>(b.mem, S::EXTRA, acc, eg, XDF ? 1 : 0);
    hc::DenseProblem<N, DEG, L> prob{&a, sm, g.meet};
    hc::run_tracker<N, L, MIXED, hc::DenseProblem<N, DEG, L>, RE>(prob, a.c, g, sm);
  });
  if (o.ended() != items) {
    std::printf("dense %d %d: %d of %d paths ended\n", N, DEG, o.ended(), items);
    return bad + 1;
  }
  return bad;
}

int main() {
  int bad = 0;
#define RUN(...) { const int n_ = __VA_ARGS__; if (n_) std::printf("^ " #__VA_ARGS__ "\n"); bad += n_; }
  for (unsigned seed = 0; seed < 2; ++seed) {
    RUN(family_df<3, 1>(seed, 3))
    RUN(family_df<6, 2>(seed, 2))
    RUN(family_df<9, 4>(seed, 2))
    RUN((family_rows<3, 4, true>(seed, 20)))
    RUN((family_rows<6, 8, false>(seed, 6)))
    RUN((family_rows<9, 16, true>(seed, 6)))
    RUN((family_rows<9, 16, false>(seed, 3)))
    RUN((family_rows<5, 32, true>(seed, 3)))
    RUN((dense<3, 2, HC_PREC_MIXED, 4>(seed, 20)))
    RUN((dense<5, 3, HC_PREC_MIXED, 8>(seed, 9)))
    RUN((dense<9, 2, HC_PREC_FP64, 16>(seed, 4)))
    RUN((dense<5, 2, HC_PREC_FP64, 8>(seed, 6)))
    RUN((dense<5, 3, HC_PREC_DF, 32>(seed, 2)))
    RUN((dense<9, 2, HC_PREC_DF, 32>(seed, 2)))
    RUN((dense<6, 2, HC_PREC_FP64, 32>(seed, 2)))
    RUN((dense<6, 2, HC_PREC_MIXED, 32>(seed, 2)))
  }
  return bad != 0;
}
