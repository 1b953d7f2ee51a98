// The double-float evaluator of parameter homotopies (precision DF, the last
// re-tracking tier of the mixed pipeline): one path per NW warps.
//
// What bounds these launches is the latency of a few hard paths -- thousands of
// steps, each a chain of evaluations and solves -- at about four cycles an
// instruction with one warp per scheduler.  One row per lane (TermEval) gives a
// lane all terms of its row one after the other and leaves 32 - n lanes idle.
// Here the terms are the unit of work: each thread forms the products of one
// term at a time (the term and its derivatives, prefix and suffix products as in
// TermEval) and leaves them in shared memory; then each entry of the row
// (dH_i/dx_j, dH_i/dt, H_i) is summed by one thread, in the order of the terms,
// so that every sum has the bits of the one-row-per-lane form.  The solve's
// columns are split over the warps, one barrier per pivot.
//
// The first warp runs the tracker; the others wait at a barrier for its
// commands (evaluate, residual, solve, exit).
//
// Measured against one row per lane (unrolled, 265 to 405 KB of code), ms: the
// re-tracking tiers of trifocal (4 scenes, at most 800 steps) 600 -> 219, of 4-view
// triangulation (600) 179 -> 85, of P3P (3000) 16.3 -> 7.0; precision DF on the
// same (at most 300 steps) 1200 -> 413, 4471 -> 3321, 35 -> 20.  Warps per path: four
// above 8 unknowns (before the summation lists, trifocal tiers 774 / 470 / 326 / 319
// with 1 / 2 / 4 / 8 warps, precision DF 1478 / 714 / 583 / 753), one up to 4, where
// the items of a precision DF batch fill the warps (P3P 33 / 55 / 85 with 1 / 2 / 4).
#pragma once

#include "kernels.cuh"
#include "tracker.cuh"

namespace hc {

template <int N, int NW>
struct TermBlock {
  // lanes per row replica in the solve: a warp holds the rows 32 / LR times,
  // each replica with its own columns
  static constexpr int LR = N <= 4 ? 4 : N <= 8 ? 8 : N <= 16 ? 16 : 32;
  static constexpr int PP = 32 / LR, OWN = PP * NW;  // replicas per warp, per path
  static constexpr int PARTS = 1, ROWL = LR, WARPS = NW;
  static constexpr int NT = 32 * NW;   // threads of a path
  static constexpr int CH = term_df_slots(N, NW);  // term slots per round: one term per thread
  static constexpr bool kCoop = false;
  enum : int { OP_EXIT = 0, OP_EVAL = 1, OP_RESIDUAL = 2, OP_SOLVE = 3 };
  struct Cmd {
    long long inst;
    double t;
    int op, arg;
  };
  enum : int { WANT_HT = 1, WANT_H = 2 };  // what an evaluation returns beside the rows

  const TermArgs* a;
  int64_t inst;
  Group g;
  cx<float>* Vf;
  cx<double>* Vd;
  cx<df>* Vx;
  unsigned char* acc;

  // shared memory behind acc: the matrix [A | b] or [A | I] (entry j of row i at
  // LR j + i), the terms' products, H, the command
  static constexpr int C0 = LR * (2 * N);
  __host__ __device__ static constexpr int acc_bytes() {
    return 16 * (C0 + (kMaxTermFactors + 1) * NT + 32) + 32;
  }
  __device__ __forceinline__ cx<df>* A() const { return reinterpret_cast<cx<df>*>(acc); }
  __device__ __forceinline__ cx<df>* C() const { return A() + C0; }
  __device__ __forceinline__ cx<df>* Hs() const { return C() + (kMaxTermFactors + 1) * NT; }
  __device__ __forceinline__ Cmd* cmd() const { return reinterpret_cast<Cmd*>(Hs() + 32); }

  __device__ __forceinline__ static int tid() { return NW == 1 ? threadIdx.x & 31 : threadIdx.x; }
  __device__ __forceinline__ static void sync() {
    if constexpr (NW == 1)
      __syncwarp();
    else
      asm volatile("barrier.sync 1, %0;" ::"n"(NT) : "memory");
  }
  // first warp: start an operation on all warps of the path
  __device__ __forceinline__ void post(int op, double t, int arg) const {
    if constexpr (NW > 1) {
      if (g.gl == 0) {
        cmd()->inst = inst;
        cmd()->t = t;
        cmd()->op = op;
        cmd()->arg = arg;
      }
    }
    sync();
  }
  // the other warps
  __device__ __forceinline__ void serve() {
    for (;;) {
      sync();
      const int op = cmd()->op;
      if (op == OP_EXIT) break;
      inst = cmd()->inst;
      const double t = cmd()->t;
      if (op == OP_EVAL) {
        eval_share((df)t, cmd()->arg);
      } else if (op == OP_RESIDUAL) {
        cx<double> h;
        float sc;
        residual_share<false>(t, h, sc);
      } else {
        cx<df> dinv;
        int col;
        solve_share(cmd()->arg, dinv, col);
      }
    }
  }

  __device__ __forceinline__ void init(const Group&) const {
    const int P = a->P, LS = a->ls;
    const double2* p1 = a->p1 + inst * P;
    if (g.gl == 0) {
      Vd[LS] = mk<double>(1.0, 0.0);
      Vx[LS] = mk<df>(df(1), df(0));
    }
    for (int l = g.gl; l < P; l += 32) {
      const cx<double> d = mk<double>(p1[l].x - a->p0[l].x, p1[l].y - a->p0[l].y);
      Vx[LS + 1 + P + l] = to_cxdf(d);
      Vx[LS + 1 + 2 * P + l] = to_cxdf(mk<double>(a->p0[l].x, a->p0[l].y));
    }
  }

  __device__ __forceinline__ cx<double> start(int64_t path, int i) const {
    const double2 v = a->start[path * N + i];
    return mk<double>(v.x, v.y);
  }

  // coefficient of record r at time t and its t-derivative
  __device__ __forceinline__ void coef(int64_t r, df t, cx<df>& s, cx<df>& dcr) const {
    if (a->coef_mode) {
      dcr = to_cxdf(a->dcdf[inst * (int64_t)a->TT * a->ls + r]);
      s = to_cxdf(a->c0df[r]) + t * dcr;
    } else {
      s = to_cxdf(a->sdf[r]);
    }
  }

  // The evaluation at the point Vd and time t, every thread its share.
  __device__ __noinline__ void eval_share(df t, int want) const {
    const int P = a->P, LS = a->ls, TT = a->TT, id = tid();
    cx<df>* M = A();
    if (id < N) Vx[id] = to_cxdf(Vd[id]);
    for (int l = id; l < P; l += NT) Vx[LS + 1 + l] = Vx[LS + 1 + 2 * P + l] + t * Vx[LS + 1 + P + l];
    for (int e = id; e < LR * (N + 1); e += NT) M[e] = czero<df>();
    if (id < 32) Hs()[id] = czero<df>();
    sync();
#pragma unroll 1
    for (int k0 = 0; k0 < TT; k0 += CH) {
      const int nk = min(CH, TT - k0);
      if (id < nk * N) {  // one term: its factors' product, then every derivative
        const int kk = id / N, i = id - kk * N;
        const int64_t r = (int64_t)(k0 + kk) * LS + i;
        const TermRec* rc = a->rec + r;
        const unsigned long long idx = *reinterpret_cast<const unsigned long long*>(rc->idx);
        const int d = rc->d;
        cx<df> s, dcr;
        coef(r, t, s, dcr);
        cx<df>* c = C() + id;
        cx<df> run = mk<df>(df(1), df(0));
#pragma unroll 1
        for (int f = 0; f < d; ++f) {
          c[f * NT] = run;
          run = run * Vx[(int)(idx >> (8 * f)) & 255];
        }
        c[kMaxTermFactors * NT] = run;
        cx<df> suf = s;
#pragma unroll 1
        for (int f = d - 1; f >= 0; --f) {
          const cx<df> dv = c[f * NT] * suf;
          suf = suf * Vx[(int)(idx >> (8 * f)) & 255];
          c[f * NT] = dv;
        }
      }
      sync();
      // Every entry of the rows adds its products in the order of the terms,
      // inside a term from the last factor to the first, from the round's lists
      // (trifocal, thousand cycles an evaluation: a search of the records 25, the
      // lists 9, the products 8).  The long chains, dH_i/dt (every parameter factor) and H_i
      // (every term), are the last entries, in a warp of their own.
      constexpr int E0 = (N * N + 31) & ~31, E = N * N + N;
      const int32_t* ptr = a->sum_ptr[NW > 1] + (int64_t)(k0 / CH) * E;
      const uint32_t* ent = a->sum_ent[NW > 1];
#pragma unroll 1
      for (int e = id; e < E0 + N; e += NT) {
        if (e >= N * N && e < E0) continue;
        if (e < N * N) {
          const int q = e / N, i = e - q * N;
          int m = ptr[e];
          const int end = ptr[e + 1];
          if (m == end) continue;
          cx<df> v = M[q * LR + i];
          uint32_t w = ent[m];
#pragma unroll 1
          while (m < end) {
            const uint32_t next = ent[++m];  // (one entry of padding behind the last)
            v = v + C()[w & 0xffffu];
            w = next;
          }
          M[q * LR + i] = v;
          continue;
        }
        const int i = e - E0;
        if (want & WANT_HT) {
          cx<df> v = M[N * LR + i];
          if (a->coef_mode) {
#pragma unroll 1
            for (int kk = 0; kk < nk; ++kk) {
              cx<df> s, dcr;
              coef((int64_t)(k0 + kk) * LS + i, t, s, dcr);
              v = cfma(dcr, C()[kMaxTermFactors * NT + kk * N + i], v);
            }
          } else {
            int m = ptr[N * N + i];
            const int end = ptr[N * N + i + 1];
            uint32_t w = ent[m];
#pragma unroll 1
            while (m < end) {
              const uint32_t next = ent[++m];
              v = cfma(C()[w & 0xffffu], Vx[w >> 16], v);
              w = next;
            }
          }
          M[N * LR + i] = v;
        }
        if (want & WANT_H) {
          cx<df> v = Hs()[i];
#pragma unroll 1
          for (int kk = 0; kk < nk; ++kk) {
            cx<df> s, dcr;
            coef((int64_t)(k0 + kk) * LS + i, t, s, dcr);
            v = cfma(s, C()[kMaxTermFactors * NT + kk * N + i], v);
          }
          Hs()[i] = v;
        }
      }
      sync();
    }
  }

  __device__ __forceinline__ void eval_rows(int i, df t, df, cx<df>& H, cx<df>& Ht,
                                            int want) const {
    post(OP_EVAL, (double)t, want);
    eval_share(t, want);
    H = Hs()[i];
    Ht = A()[LR * N + (i & (LR - 1))];
    __syncwarp();  // the first replica's lanes put the right-hand side in its place
  }

  template <class R>
  __device__ __forceinline__ void eval(const cx<R> (&)[N], int i, R t, R omt, cx<R> (&row)[N + 1],
                                       cx<R>& H, cx<R>& Ht) const {
    eval_rows(i, t, omt, H, Ht, WANT_HT | WANT_H);
#pragma unroll
    for (int j = 0; j < N; ++j) row[j] = A()[LR * j + (i & (LR - 1))];
  }

  // FP64 residual: the terms' products over the threads, the sums by the first
  // warp's lanes in the order of the terms
  template <bool SCALE>
  __device__ __noinline__ void residual_share(double t, cx<double>& H, float& sc) const {
    const int P = a->P, LS = a->ls, TT = a->TT, id = tid();
    const double2* p1 = a->p1 + inst * P;
    cx<double>* c = reinterpret_cast<cx<double>*>(C());
    for (int l = id; l < P; l += NT) {
      const double2 q0 = a->p0[l], q1 = p1[l];
      Vd[LS + 1 + l] = mk<double>((1.0 - t) * q0.x + t * q1.x, (1.0 - t) * q0.y + t * q1.y);
    }
    sync();
    cx<double> h = czero<double>();
    float s_abs = 0.f;
#pragma unroll 1
    for (int k0 = 0; k0 < TT; k0 += CH) {
      const int nk = min(CH, TT - k0);
      if (id < nk * N) {
        const int kk = id / N, i = id - kk * N;
        const TermRec* rc = a->rec + (int64_t)(k0 + kk) * LS + i;
        const unsigned long long idx = *reinterpret_cast<const unsigned long long*>(rc->idx);
        const int d = rc->d;
        cx<double> prod = Vd[(int)idx & 255];
#pragma unroll 1
        for (int f = 1; f < d; ++f) prod = prod * Vd[(int)(idx >> (8 * f)) & 255];
        c[id] = prod;
      }
      sync();
      if (id < N) {
#pragma unroll 1
        for (int kk = 0; kk < nk; ++kk) {
          const int64_t r = (int64_t)(k0 + kk) * LS + id;
          const cx<double> prod = c[kk * N + id];
          cx<double> s;
          if (a->coef_mode) {
            const double2 c0 = a->c0[r], dc = a->dc[inst * (int64_t)TT * LS + r];
            s = cfma(mk<double>(t, 0.0), mk<double>(dc.x, dc.y), mk<double>(c0.x, c0.y));
          } else {
            s = mk<double>(a->s64[r].x, a->s64[r].y);
          }
          h = cfma(s, prod, h);
          if (SCALE) s_abs += cabs2(cvt<float>(s)) * cabs2(cvt<float>(prod));
        }
      }
      sync();
    }
    H = h;
    sc = s_abs;
  }
  template <bool SCALE>
  __device__ __forceinline__ void residual64(const cx<double>*, int, double t, double,
                                             cx<double>& H, double& sc) const {
    float s_abs;
    post(OP_RESIDUAL, t, 0);
    residual_share<SCALE>(t, H, s_abs);
    sc = SCALE ? (double)s_abs : 0.0;
  }

  // Gauss-Jordan as gj_solve_df on the first W columns: replica o of the rows
  // (OWN in all) updates the columns j with j mod OWN = o, which no other replica
  // reads before they are pivot columns.  The warp that holds column k + 1 updates
  // it first, searches its pivot and publishes row and reciprocal (the longest
  // chain of a pivot step), and comes to its other columns behind the barrier,
  // when the next column's warp is already at its search: one barrier per pivot
  // (n = 18 with 4 warps: 22.3 -> 21.5 thousand cycles a solve).  The pivot row's
  // entries are read where they lie.  Returns whether every pivot was nonzero and
  // finite; the lanes of the first replica hold 1 / pivot of their row and the
  // column it pivoted on (-1: none).
  struct Pivot {
    cx<df> inv;
    unsigned key;
  };
  __device__ __noinline__ bool solve_share(int W, cx<df>& dinv, int& col) const {
    constexpr int UNROLL = 3;
    cx<df>* M = A();
    Pivot* pivot = reinterpret_cast<Pivot*>(C());  // two, by parity of the column
    const int r = g.wl & (LR - 1), w = NW == 1 ? 0 : (int)threadIdx.x >> 5;
    const int own = w * PP + g.wl / LR;
    bool used = r >= N;
    unsigned lo = 0xffffffffu, hi = 0u;
    dinv = mk<df>(df(1), df(0));
    col = -1;
    auto row_of = [](unsigned key) { return min(31 - (int)(key & 31u), LR - 1); };
    auto search = [&](int k) {
      const cx<df> ak = M[LR * k + r];
      const unsigned key = used ? 0u : ((__float_as_uint(cabs1(ak)) & ~31u) | (unsigned)(31 - r));
      const unsigned kmax = __reduce_max_sync(0xffffffffu, key);
      const cx<df> inv = crecip(ak);
      if (g.wl == row_of(kmax)) {
        pivot[k & 1].inv = inv;
        pivot[k & 1].key = kmax;
      }
    };
    if (w == 0) search(0);
    sync();
#pragma unroll 1
    for (int k = 0; k < N; ++k) {
      const unsigned kmax = pivot[k & 1].key;
      const cx<df> inv = pivot[k & 1].inv;
      lo = min(lo, kmax);
      hi = max(hi, kmax);
      const int rp = row_of(kmax);
      const bool me = r == rp;
      if (me) {
        used = true;
        dinv = inv;
        col = k;
      }
      const cx<df> l = me ? czero<df>() : M[LR * k + r] * inv;
      const cx<df> lr = neg(re_re(l)), li = neg(nim_im(l));
      int j = k + 1 + ((own - (k + 1)) & (OWN - 1));  // this lane's first column
      const bool ahead = k + 1 < N && ((k + 1) & (OWN - 1)) / PP == w;
      if (ahead) {
        const bool first = j == k + 1;
        cx<df> v = czero<df>();
        if (first) {
          const cx<df> p = M[LR * j + rp];
          v = dot2p(M[LR * j + r], lr, p, li, im_re(p));
        }
        __syncwarp();  // the pivot row's entry is read before its lane stores it
        if (first) M[LR * j + r] = v;
        __syncwarp();
        search(k + 1);
        if (first) j += OWN;
        sync();
      }
#pragma unroll 1
      for (; __any_sync(0xffffffffu, j < W); j += UNROLL * OWN) {
        cx<df> v[UNROLL];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
          // (behind the last column: column k, which nobody writes now)
          const int ju = LR * (j + u * OWN < W ? j + u * OWN : k);
          const cx<df> p = M[ju + rp];
          v[u] = dot2p(M[ju + r], lr, p, li, im_re(p));
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < UNROLL; ++u)
          if (j + u * OWN < W) M[LR * (j + u * OWN) + r] = v[u];
      }
      // the next step's lanes read other lanes' entries of these columns (a vote
      // orders no memory)
      if (ahead)
        __syncwarp();
      else
        sync();
    }
    if (g.wl >= LR || r >= N) col = -1;
    return (lo & ~31u) != 0u && (hi & ~31u) < 0x7f800000u;
  }
  template <bool MEET>
  __device__ __forceinline__ bool solve(const Group&, cx<df>*, cx<df>*, int W, cx<df>& dinv,
                                        int& col) const {
    post(OP_SOLVE, 0.0, W);
    return solve_share(W, dinv, col);
  }
};

template <int N, int NW>
struct TermBlockProblem {
  const TermArgs* a;
  Group g;
  GroupMem sm;
  __device__ __forceinline__ TermBlock<N, NW> hom(int64_t inst) const {
    return TermBlock<N, NW>{a, inst, g, sm.vf, sm.vd, sm.vx, sm.acc};
  }
};

// NW = 1: any block of whole warps, one path each; otherwise blocks of NW warps.
template <int N, int NW>
__global__ void __launch_bounds__(NW == 1 ? kBlock : 32 * NW)
    term_df_kernel(const __grid_constant__ TermArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const Group g = make_group<32>();
  const GroupMem sm = make_group_mem<32>(smem, a.extra, TermBlock<N, NW>::acc_bytes(),
                                         endgame_smem_bytes(32, false), 1, NW);
  TermBlockProblem<N, NW> prob{&a, g, sm};
  if (NW == 1 || threadIdx.x < 32) {
    run_tracker<N, 32, false, TermBlockProblem<N, NW>, df>(prob, a.c, g, sm);
    if constexpr (NW > 1) prob.hom(0).post(TermBlock<N, NW>::OP_EXIT, 0.0, 0);
  } else {
    TermBlock<N, NW> h = prob.hom(0);
    h.serve();
  }
}

template <int N, int NW>
KernelRef term_df_ref() {
  return KernelRef{reinterpret_cast<const void*>(&term_df_kernel<N, NW>), 32, 0,
                   TermBlock<N, NW>::acc_bytes(), endgame_smem_bytes(32, false), 1, NW};
}

}  // namespace hc
