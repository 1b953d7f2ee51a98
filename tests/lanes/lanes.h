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

constexpr int kMost = 128;  // threads of a block
struct Clock {
  uint32_t at[kMost];
  LANES_RAW Clock() {
    for (uint32_t& v : at) v = 0;
  }
  LANES_RAW uint32_t& operator[](int k) { return at[k]; }
  LANES_RAW const uint32_t& operator[](int k) const { return at[k]; }
};

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

struct Word {
  int writer = -1;
  uint32_t at = 0;
  bool read = false;
  Clock reads;
};
struct Range {  // shared data, checked by words of `grain` bytes
  uintptr_t begin;
  size_t bytes, grain;
  std::vector<Word> words;
  Word* table;
};

struct Machine {
  Thread* threads = nullptr;
  int count = 0;
  uint32_t joint[kMost];
  Range* ranges = nullptr;
  int range_count = 0;
  ucontext_t main;
  int cur = -1;
  std::vector<Range> watched;
  std::map<uintptr_t, Clock> atomics;   // words accessed by atomics: their clocks
  std::set<std::string> races;
  std::function<void()> body;
};
inline Machine* machine = new Machine;
inline bool checking = false;  // the containers used by a check are instrumented too
LANES_RAW inline Machine& m() { return *machine; }
LANES_RAW inline Thread& me() { return m().threads[m().cur]; }

LANES_RAW inline void join(Clock& a, const Clock& b) {
  for (int k = 0; k < kMost; ++k) a[k] = a[k] > b[k] ? a[k] : b[k];
}

LANES_RAW inline void check(const void* p, size_t bytes, bool write) {
  Machine& M = m();
  const uintptr_t a = (uintptr_t)p;
  Range* r = nullptr;
  for (int k = 0; k < M.range_count; ++k)
    if (a - M.ranges[k].begin < M.ranges[k].bytes) r = M.ranges + k;
  if (!r) return;
  if (a + bytes > r->begin + r->bytes) {
    M.races.insert("access past the end of a buffer");
    return;
  }
  Thread& t = me();
  auto at = M.atomics.find(a);
  if (at != M.atomics.end()) {
    join(t.pending, at->second);
    return;
  }
  for (size_t w = (a - r->begin) / r->grain; w * r->grain < a + bytes - r->begin; ++w) {
    Word& x = r->table[w];
    auto race = [&](const char* what, int other) {
      char msg[160];
      std::snprintf(msg, sizeof msg,
                    "buffer %d, offset %zu: %s of thread %d, not ordered with a %s of thread %d",
                    (int)(r - M.ranges), w * r->grain, write ? "write" : "read", M.cur,
                    what, other);
      if (M.races.size() < 20) M.races.insert(msg);
    };
    if (x.writer >= 0 && x.writer != M.cur && x.at > t.vc[x.writer]) race("write", x.writer);
    if (write) {
      if (x.read)
        for (int k = 0; k < M.count; ++k)
          if (k != M.cur && x.reads[k] > t.vc[k]) race("read", k);
      x.writer = M.cur;
      x.at = t.vc[M.cur];
      x.read = false;
    } else {
      if (!x.read) x.reads = Clock();
      x.read = true;
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
  swapcontext(&m().threads[c].ctx, &m().main);
}

enum : int { ORDERED = 1, EXCHANGE = 2, BLOCK = 3 };
// Meets the threads of mask in this warp (kind BLOCK: all that are not done).  An
// exchange leaves the values that the lanes brought in got[32].
LANES_RAW inline void meet(int kind, unsigned mask, uint64_t value, uint64_t* got = nullptr) {
  Machine& M = m();
  Thread* th = M.threads;
  Thread& t = th[M.cur];
  t.waits = kind;
  t.mask = mask;
  t.value = value;
  while (t.waits) yield();
  if (!got) return;
  const int w0 = M.cur & ~31;
  for (int k = 0; k < 32; ++k) got[k] = mask >> k & 1u ? th[w0 + k].value : 0;
  t.waits = kind;  // everyone has read before anyone goes on
  while (t.waits) yield();
}

// Lets those go on whose meeting is complete.
LANES_RAW inline bool release() {
  Machine& M = m();
  Thread* th = M.threads;
  const int n = M.count;
  bool any = false;
  for (int k = 0; k < n; ++k) {
    Thread& t = th[k];
    if (t.done || !t.waits) continue;
    const int kind = t.waits, from = kind == BLOCK ? 0 : k & ~31, to = kind == BLOCK ? n : from + 32;
    auto in = [&](int j) LANES_RAW { return kind == BLOCK ? !th[j].done : (t.mask >> (j & 31) & 1u) != 0; };
    bool complete = true;
    for (int j = from; j < to && complete; ++j)
      if (in(j))
        complete = !th[j].done && th[j].waits == kind && (kind == BLOCK || th[j].mask == t.mask);
    if (!complete) continue;
    if (kind != EXCHANGE) {
      uint32_t* joint = M.joint;
      for (int c = 0; c < n; ++c) joint[c] = 0;
      for (int j = from; j < to; ++j)
        if (in(j))
          for (int c = 0; c < n; ++c) joint[c] = th[j].vc[c] > joint[c] ? th[j].vc[c] : joint[c];
      for (int j = from; j < to; ++j)
        if (in(j)) {
          for (int c = 0; c < n; ++c) th[j].vc[c] = joint[c];
          ++th[j].vc[j];
        }
    }
    for (int j = from; j < to; ++j)
      if (in(j)) th[j].waits = 0;
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
  std::vector<Thread> store(threads);
  M.threads = store.data();
  M.count = threads;
  for (Range& r : M.watched) {
    r.words.assign(r.bytes / r.grain + 1, Word());
    r.table = r.words.data();
  }
  M.ranges = M.watched.data();
  M.range_count = (int)M.watched.size();
  M.races.clear();
  M.body = body;
  for (int k = 0; k < threads; ++k) {
    Thread& t = M.threads[k];
    t.tid = dim3(k, 0, 0);
    t.vc[k] = 1;
    t.stack.resize(256 << 10);
    getcontext(&t.ctx);
    t.ctx.uc_stack.ss_sp = t.stack.data();
    t.ctx.uc_stack.ss_size = t.stack.size();
    t.ctx.uc_link = &M.main;
    makecontext(&t.ctx, entry, 0);
  }
  for (auto& a : M.atomics) a.second = Clock();
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
      Thread& t = M.threads[k];
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
  join(me().pending, c);
  join(c, me().released);
  const T old = *p;
  *p = f(old);
  return old;
}
LANES_RAW inline void watch(const void* p, size_t bytes, size_t grain = 4) {
  m().watched.push_back({(uintptr_t)p, bytes, grain, {}, nullptr});
}
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
#define blockDim (dim3((unsigned)lanes::m().count, 1, 1))

LANES_RAW inline void __syncwarp(unsigned mask = 0xffffffffu) { lanes::meet(lanes::ORDERED, mask, 0); }
LANES_RAW inline void __syncthreads() { lanes::meet(lanes::BLOCK, 0, 0); }
inline void __threadfence_block() { lanes::fence(); }
inline void __threadfence() { lanes::fence(); }
inline void __threadfence_system() { lanes::fence(); }
template <class T>
LANES_RAW inline T __shfl_sync(unsigned mask, T v, int src, int = 32) {
  uint64_t got[32];
  lanes::meet(lanes::EXCHANGE, mask, lanes::pack(v), got);
  return lanes::unpack<T>(got[src & 31]);
}
template <class T>
LANES_RAW inline T __shfl_xor_sync(unsigned mask, T v, int o, int = 32) {
  const int lane = lanes::m().cur & 31;
  uint64_t got[32];
  lanes::meet(lanes::EXCHANGE, mask, lanes::pack(v), got);
  return lanes::unpack<T>(got[(lane ^ o) & 31]);
}
template <class F>
LANES_RAW inline unsigned lanes_reduce(unsigned mask, unsigned v, F f) {
  uint64_t got[32];
  lanes::meet(lanes::EXCHANGE, mask, v, got);
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
  uint64_t got[32];
  lanes::meet(lanes::EXCHANGE, mask, p != 0, got);
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
inline int __popc(unsigned v) { return __builtin_popcount(v); }
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
