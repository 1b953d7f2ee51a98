// Runs device code on the CPU, one coroutine per thread of a block, and reports
// accesses to shared data that no synchronisation orders.
//
// The device headers are compiled as they are, with -fsanitize=thread: the
// compiler then calls __tsan_read / __tsan_write for every access, and this file
// provides those calls instead of the sanitizer's library.  Every thread has a
// vector clock; __syncwarp and the block barriers join the clocks of those that
// meet, an atomic operation passes on what a fence before it released to a fence
// behind it, and shuffles, votes and reductions exchange values but order
// nothing -- the guarantees that CUDA gives, not what a warp happens to do.
#pragma once

#include <ucontext.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <limits>
#include <map>
#include <set>
#include <string>
#include <type_traits>
#include <vector>

#include <cuda_runtime.h>

#define LANES_RAW __attribute__((no_sanitize("thread")))

namespace lanes {

using Clock = std::vector<uint32_t>;

struct Thread {
  ucontext_t ctx;
  std::vector<char> stack;
  dim3 tid;
  bool done = false;
  int waits = 0;          // 0 runnable, else the kind of meeting
  unsigned mask = 0;      // of the meeting
  uint64_t value = 0;     // exchanged at it
  Clock vc, released, pending;
};

struct Word {  // per 4 bytes of a watched range
  int writer = -1;
  uint32_t at = 0;
  std::map<int, uint32_t> reads;
};

struct Machine {
  std::vector<Thread> th;
  ucontext_t main;
  int cur = -1;
  std::map<uintptr_t, size_t> watched;  // begin -> bytes
  std::map<uintptr_t, Word> words;
  std::map<uintptr_t, Clock> atomics;   // words accessed by atomics: their clocks
  std::set<std::string> races;
  std::function<void()> body;
};
inline Machine* machine = new Machine;
inline bool checking = false;  // the containers used by a check are instrumented too
LANES_RAW inline Machine& m() { return *machine; }
LANES_RAW inline Thread& me() { return m().th[m().cur]; }

LANES_RAW inline void join(Clock& a, const Clock& b) {
  for (size_t k = 0; k < a.size(); ++k) a[k] = std::max(a[k], b[k]);
}

// An access of the running thread.
LANES_RAW inline void check(const void* p, size_t bytes, bool write) {
  Machine& M = m();
  const uintptr_t a = (uintptr_t)p;
  auto it = M.watched.upper_bound(a);
  if (it == M.watched.begin()) return;
  --it;
  if (a >= it->first + it->second) return;
  if (a + bytes > it->first + it->second) M.races.insert("access past the end of a buffer");
  Thread& t = me();
  if (auto at = M.atomics.find(a); at != M.atomics.end()) {
    join(t.pending, at->second);
    return;
  }
  for (uintptr_t w = a & ~(uintptr_t)3; w < a + bytes; w += 4) {
    Word& x = M.words[w];
    char msg[160];
    auto race = [&](const char* what, int other) {
      std::snprintf(msg, sizeof msg, "%s of thread %d, not ordered with a %s of thread %d, offset %zu",
                    write ? "write" : "read", M.cur, what, other, (size_t)(w - it->first));
      if (M.races.size() < 20) M.races.insert(msg);
    };
    if (x.writer >= 0 && x.writer != M.cur && x.at > t.vc[x.writer]) race("write", x.writer);
    if (write) {
      for (auto& r : x.reads)
        if (r.first != M.cur && r.second > t.vc[r.first]) race("read", r.first);
      x.writer = M.cur;
      x.at = t.vc[M.cur];
      x.reads.clear();
    } else {
      x.reads[M.cur] = t.vc[M.cur];
    }
  }
}

LANES_RAW inline void access(const void* p, size_t bytes, bool write) {
  if (checking || !machine || machine->cur < 0) return;
  checking = true;
  check(p, bytes, write);
  checking = false;
}

LANES_RAW inline void yield() {
  const int c = m().cur;
  swapcontext(&m().th[c].ctx, &m().main);
}

enum : int { ORDERED = 1, EXCHANGE = 2, BLOCK = 3 };
// Meets the threads of mask in this warp (kind BLOCK: all that are not done) and
// returns the values they brought, by lane.
LANES_RAW inline std::vector<uint64_t> meet(int kind, unsigned mask, uint64_t value) {
  Thread& t = me();
  t.waits = kind;
  t.mask = mask;
  t.value = value;
  while (t.waits) yield();
  std::vector<uint64_t> got(32, 0);
  const int w0 = m().cur & ~31;
  for (int k = 0; k < 32 && w0 + k < (int)m().th.size(); ++k) got[k] = m().th[w0 + k].value;
  if (kind == EXCHANGE) {  // everyone has read before anyone goes on
    t.waits = kind;
    while (t.waits) yield();
  }
  return got;
}

// Lets those go on whose meeting is complete.
LANES_RAW inline bool release() {
  Machine& M = m();
  bool any = false;
  const int n = (int)M.th.size();
  for (int k = 0; k < n; ++k) {
    Thread& t = M.th[k];
    if (t.done || !t.waits) continue;
    std::vector<int> all;
    bool complete = true;
    if (t.waits == BLOCK) {
      for (int j = 0; j < n; ++j)
        if (!M.th[j].done) {
          all.push_back(j);
          complete = complete && M.th[j].waits == BLOCK;
        }
    } else {
      for (int j = 0; j < 32; ++j)
        if (t.mask >> j & 1u) {
          const int o = (k & ~31) + j;
          all.push_back(o);
          complete = complete && !M.th[o].done && M.th[o].waits == t.waits && M.th[o].mask == t.mask;
        }
    }
    if (!complete) continue;
    if (t.waits != EXCHANGE) {
      Clock joint(n, 0);
      for (int j : all) join(joint, M.th[j].vc);
      for (int j : all) {
        M.th[j].vc = joint;
        ++M.th[j].vc[j];
      }
    }
    for (int j : all) M.th[j].waits = 0;
    any = true;
  }
  return any;
}

LANES_RAW inline void entry() {
  m().body();
  me().done = true;
  yield();
}

// Runs body on `threads` threads; the threads advance in an order that `seed`
// picks.  Returns the number of distinct races found (printed).
LANES_RAW inline int run(int threads, unsigned seed, std::function<void()> body) {
  Machine& M = m();
  M.th.clear();
  M.th.resize(threads);
  M.words.clear();
  M.races.clear();
  M.body = body;
  for (int k = 0; k < threads; ++k) {
    Thread& t = M.th[k];
    t.tid = dim3(k, 0, 0);
    t.vc.assign(threads, 0);
    t.vc[k] = 1;
    t.released.assign(threads, 0);
    t.pending.assign(threads, 0);
    t.stack.resize(256 << 10);
    getcontext(&t.ctx);
    t.ctx.uc_stack.ss_sp = t.stack.data();
    t.ctx.uc_stack.ss_size = t.stack.size();
    t.ctx.uc_link = &M.main;
    makecontext(&t.ctx, entry, 0);
  }
  for (auto& a : M.atomics) a.second.assign(threads, 0);
  uint64_t rng = 0x9e3779b97f4a7c15ull * (seed + 1);
  std::vector<int> order(threads);
  for (int k = 0; k < threads; ++k) order[k] = k;
  for (;;) {
    bool ran = false, left = false;
    for (int k = threads - 1; k > 0; --k) {
      rng = rng * 6364136223846793005ull + 1442695040888963407ull;
      std::swap(order[k], order[(rng >> 33) % (k + 1)]);
    }
    for (int k : order) {
      Thread& t = M.th[k];
      left = left || !t.done;
      if (t.done || t.waits) continue;
      M.cur = k;
      swapcontext(&M.main, &t.ctx);
      M.cur = -1;
      ran = true;
    }
    if (!left) break;
    if (!release() && !ran) {
      M.races.insert("threads wait for one another");
      break;
    }
  }
  for (auto& r : M.races) std::printf("%s\n", r.c_str());
  return (int)M.races.size();
}

template <class T>
LANES_RAW inline uint64_t pack(T v) {
  uint64_t u = 0;
  static_assert(sizeof(T) <= 8, "one word");
  std::memcpy(&u, &v, sizeof v);
  return u;
}
template <class T>
LANES_RAW inline T unpack(uint64_t u) {
  T v;
  std::memcpy(&v, &u, sizeof v);
  return v;
}
LANES_RAW inline void fence() {
  Thread& t = me();
  join(t.vc, t.pending);
  t.released = t.vc;
  ++t.vc[m().cur];
}
template <class T, class F>
LANES_RAW inline T rmw(T* p, F f) {
  Clock& c = m().atomics[(uintptr_t)p];
  if (c.empty()) c.assign(m().th.size(), 0);
  join(me().pending, c);
  join(c, me().released);
  const T old = *p;
  *p = f(old);
  return old;
}
LANES_RAW inline void watch(const void* p, size_t bytes) { m().watched[(uintptr_t)p] = bytes; }
LANES_RAW inline void atomic_word(const void* p) { m().atomics[(uintptr_t)p]; }

inline float reciprocal(const char* text, float v) {
  if (!std::strstr(text, "rcp.approx")) std::abort();
  return 1.0f / v;
}
inline void asm_text(const char* text) {
  if (std::strstr(text, "barrier.sync")) {
    meet(BLOCK, 0, 0);
  } else {
    std::printf("inline assembly without a host form: %s\n", text);
    std::abort();
  }
}

}  // namespace lanes

// ------------------------------------------------------- what the compiler calls
extern "C" {
void __tsan_init() {}
void __tsan_func_entry(void*) {}
void __tsan_func_exit() {}
#define LANES_ACCESS(n)                                                                   \
  LANES_RAW void __tsan_read##n(void* p) { lanes::access(p, n, false); }          \
  LANES_RAW void __tsan_write##n(void* p) { lanes::access(p, n, true); }          \
  LANES_RAW void __tsan_unaligned_read##n(void* p) { lanes::access(p, n, false); } \
  LANES_RAW void __tsan_unaligned_write##n(void* p) { lanes::access(p, n, true); } \
  LANES_RAW void __tsan_volatile_read##n(void* p) { lanes::access(p, n, false); }  \
  LANES_RAW void __tsan_volatile_write##n(void* p) { lanes::access(p, n, true); }
LANES_ACCESS(1)
LANES_ACCESS(2)
LANES_ACCESS(4)
LANES_ACCESS(8)
LANES_ACCESS(16)
LANES_RAW void __tsan_read_range(void* p, size_t n) { lanes::access(p, n, false); }
LANES_RAW void __tsan_write_range(void* p, size_t n) { lanes::access(p, n, true); }
LANES_RAW void __tsan_vptr_update(void**, void*) {}
LANES_RAW void __tsan_vptr_read(void**) {}
}

// ------------------------------------------------------------- device built-ins
#define threadIdx (lanes::me().tid)
static const dim3 blockIdx(0, 0, 0), gridDim(1, 1, 1);
#define blockDim (dim3((unsigned)lanes::m().th.size(), 1, 1))

LANES_RAW inline void __syncwarp(unsigned mask = 0xffffffffu) { lanes::meet(lanes::ORDERED, mask, 0); }
LANES_RAW inline void __syncthreads() { lanes::meet(lanes::BLOCK, 0, 0); }
inline void __threadfence_block() { lanes::fence(); }
inline void __threadfence() { lanes::fence(); }
inline void __threadfence_system() { lanes::fence(); }
template <class T>
LANES_RAW inline T __shfl_sync(unsigned mask, T v, int src, int = 32) {
  return lanes::unpack<T>(lanes::meet(lanes::EXCHANGE, mask, lanes::pack(v))[src & 31]);
}
template <class T>
LANES_RAW inline T __shfl_xor_sync(unsigned mask, T v, int o, int = 32) {
  const int lane = lanes::m().cur & 31;
  return lanes::unpack<T>(lanes::meet(lanes::EXCHANGE, mask, lanes::pack(v))[(lane ^ o) & 31]);
}
template <class F>
LANES_RAW inline unsigned lanes_reduce(unsigned mask, unsigned v, F f) {
  const auto got = lanes::meet(lanes::EXCHANGE, mask, v);
  bool first = true;
  unsigned r = 0;
  for (int k = 0; k < 32; ++k)
    if (mask >> k & 1u) {
      r = first ? (unsigned)got[k] : f(r, (unsigned)got[k]);
      first = false;
    }
  return r;
}
inline unsigned __reduce_max_sync(unsigned mask, unsigned v) {
  return lanes_reduce(mask, v, [](unsigned a, unsigned b) { return std::max(a, b); });
}
inline unsigned __reduce_or_sync(unsigned mask, unsigned v) {
  return lanes_reduce(mask, v, [](unsigned a, unsigned b) { return a | b; });
}
inline int __any_sync(unsigned mask, int p) { return __reduce_or_sync(mask, p != 0) != 0; }
LANES_RAW inline unsigned __ballot_sync(unsigned mask, int p) {
  const auto got = lanes::meet(lanes::EXCHANGE, mask, p != 0);
  unsigned r = 0;
  for (int k = 0; k < 32; ++k)
    if (mask >> k & 1u) r |= (unsigned)(got[k] & 1u) << k;
  return r;
}
template <class T>
inline T __ldcg(const T* p) { return *p; }
template <class T>
inline void __stcg(T* p, T v) { *p = v; }
template <class T>
LANES_RAW inline T atomicAdd(T* p, T v) {
  return lanes::rmw(p, [&](T o) { return (T)(o + v); });
}
template <class T>
LANES_RAW inline T atomicCAS(T* p, T is, T v) {
  return lanes::rmw(p, [&](T o) { return o == is ? v : o; });
}
template <class T>
LANES_RAW inline T atomicExch(T* p, T v) {
  return lanes::rmw(p, [&](T) { return v; });
}
inline void __nanosleep(unsigned) {}

inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
inline float __frcp_rn(float a) { return 1.0f / a; }
inline float __fdividef(float a, float b) { return a / b; }
inline float __double2float_rn(double a) { return (float)a; }
inline float2 __fadd2_rn(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
inline float2 __fmul2_rn(float2 a, float2 b) { return make_float2(a.x * b.x, a.y * b.y); }
inline float2 __ffma2_rn(float2 a, float2 b, float2 c) {
  return make_float2(std::fmaf(a.x, b.x, c.x), std::fmaf(a.y, b.y, c.y));
}
inline unsigned __float_as_uint(float f) { return lanes::unpack<unsigned>(lanes::pack(f)); }
inline float __uint_as_float(unsigned u) { return lanes::unpack<float>(lanes::pack(u)); }
inline float __int_as_float(int u) { return lanes::unpack<float>(lanes::pack(u)); }
inline int __ffs(unsigned v) { return __builtin_ffs((int)v); }
inline float rsqrtf(float a) { return 1.0f / std::sqrt(a); }
inline double __drcp_rn(double a) { return 1.0 / a; }
inline void sincospi(double a, double* s, double* c) {
  *s = std::sin(M_PI * a);
  *c = std::cos(M_PI * a);
}
using std::isfinite;
using std::isnan;
using std::max;
using std::min;

// Inline assembly: by its text.  The one statement with operands is the FP32
// reciprocal, whose variables are r and v.
inline void LANES_ASM(const char* text) { lanes::asm_text(text); }
#define LANES_ASM(...) (r = lanes::reciprocal(#__VA_ARGS__, v))
#define asm LANES_ASM
#define volatile(...) (#__VA_ARGS__)
#undef __launch_bounds__
#define __launch_bounds__(...)
#undef __grid_constant__
#define __grid_constant__
#undef __noinline__
#define __noinline__ __attribute__((noinline))
