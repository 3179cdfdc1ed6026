// The bit-sliced X-drop kernel (csrc/xdrop_bits.cuh, csrc/xdrop_bits_run.cuh) run on the CPU: 32 lanes as
// fibers that meet at every warp intrinsic.  Built and driven by
// tests/test_bits_emulation.py; no GPU, no CUDA headers.
#include <ucontext.h>

#include <algorithm>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <vector>

#define __device__
#define __host__
#define __forceinline__ inline
#define __restrict__
#define XDROP_BITS_EMULATE 1
using std::max;
using std::min;

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kStack = 1 << 17;

struct Fiber {
  ucontext_t ctx;
  std::vector<char> stack;
  uint64_t in = 0;
  int src = 0;
  bool done = false;
};
Fiber g_fib[32];
ucontext_t g_main;
int g_lane = 0;
uint64_t g_snap[32];  // what every lane brought to the current meeting point

uint64_t meet(uint64_t v) {  // all 32 lanes arrive, then all continue
  g_fib[g_lane].in = v;
  const int me = g_lane;
  swapcontext(&g_fib[me].ctx, &g_main);
  return 0;
}
unsigned __ballot_sync(unsigned, bool p) {
  meet(p ? 1 : 0);
  unsigned r = 0;
  for (int i = 0; i < 32; ++i) r |= (unsigned)(g_snap[i] & 1) << i;
  return r;
}
bool __any_sync(unsigned m, bool p) { return __ballot_sync(m, p) != 0; }
bool __all_sync(unsigned m, bool p) { return __ballot_sync(m, p) == kFull; }
template <typename T>
T lane_value(T v, int from) {
  uint64_t u = 0;
  memcpy(&u, &v, sizeof(T));
  meet(u);
  T r;
  memcpy(&r, &g_snap[from], sizeof(T));
  return r;
}
template <typename T>
T __shfl_sync(unsigned, T v, int src, int w = 32) { return lane_value(v, (g_lane & ~(w - 1)) | (src & (w - 1))); }
template <typename T>
T __shfl_down_sync(unsigned, T v, int d, int w = 32) {
  return lane_value(v, (g_lane & (w - 1)) + d < w ? g_lane + d : g_lane);
}
template <typename T>
T __shfl_up_sync(unsigned, T v, int d, int w = 32) {
  return lane_value(v, (g_lane & (w - 1)) - d >= 0 ? g_lane - d : g_lane);
}
template <typename T>
T __shfl_xor_sync(unsigned, T v, int x, int w = 32) {
  (void)w;
  return lane_value(v, g_lane ^ x);
}
int __reduce_add_sync(unsigned, int v) {
  meet((uint64_t)(uint32_t)v);
  int r = 0;
  for (int i = 0; i < 32; ++i) r += (int)(uint32_t)g_snap[i];
  return r;
}
int __reduce_min_sync(unsigned, int v) {
  meet((uint64_t)(uint32_t)v);
  int r = INT32_MAX;
  for (int i = 0; i < 32; ++i) r = std::min(r, (int)(uint32_t)g_snap[i]);
  return r;
}
uint32_t __reduce_or_sync(unsigned, uint32_t v) {
  meet(v);
  uint32_t r = 0;
  for (int i = 0; i < 32; ++i) r |= (uint32_t)g_snap[i];
  return r;
}
void __syncwarp() { meet(0); }
uint32_t __funnelshift_r(uint32_t lo, uint32_t hi, unsigned s) {
  return (uint32_t)(((((uint64_t)hi) << 32) | lo) >> (s & 31));
}
uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, unsigned s) {
  return (uint32_t)((((((uint64_t)hi) << 32) | lo) << (s & 31)) >> 32);
}
uint32_t __funnelshift_rc(uint32_t lo, uint32_t hi, unsigned s) {
  return s >= 32 ? hi : __funnelshift_r(lo, hi, s);
}
uint32_t __funnelshift_lc(uint32_t lo, uint32_t hi, unsigned s) {
  return s >= 32 ? lo : __funnelshift_l(lo, hi, s);
}
uint32_t __byte_perm(uint32_t a, uint32_t b, uint32_t sel) {
  const uint64_t v = ((uint64_t)b << 32) | a;
  uint32_t r = 0;
  for (int i = 0; i < 4; ++i) r |= (uint32_t)((v >> (8 * ((sel >> (4 * i)) & 7))) & 255) << (8 * i);
  return r;
}
int __clz(int x) { return x ? __builtin_clz((unsigned)x) : 32; }
int __ffs(int x) { return __builtin_ffs(x); }
int __popc(unsigned x) { return __builtin_popcount(x); }
template <typename T, typename U>
T atomicAdd(T* p, U v) {
  const T old = *p;
  *p = (T)(old + (T)v);
  return old;
}
template <typename T, typename U>
T atomicExch(T* p, U v) {
  const T old = *p;
  *p = (T)v;
  return old;
}
template <typename T>
T atomicCAS(T* p, T expect, T v) {
  const T old = *p;
  if (old == expect) *p = v;
  return old;
}
template <typename T>
T __ldcg(const T* p) { return *p; }
void __threadfence() {}
struct { struct { operator unsigned() const { return (unsigned)g_lane; } } x; } threadIdx;

struct Item { long long a0, b0; int m, n, tag, pad; };
struct ExtOut { int best, i_end, j_end, status; long long cells; };
struct Counters { unsigned tail[16], head[16], stat[8], pool; unsigned long long cells[8]; };
struct Scoring { int M, S, G, X; };
struct ExtendParams {
  const uint32_t* words;
  const Item* items;
  ExtOut* ext;
  Counters* cnt;
  const int* wide_q;
  int wide_q_id;
  int* esc_q;
  int esc_q_id, cells_idx, bits_esc_stat, reserve, young, max_groups;
  int* res_q;
  int res_q_id;
  long long res_cap;
  uint32_t* pool;
  unsigned pool_words;
  long long q_cap;
  Scoring sc;
};

// Store words are read only inside the store: an index outside is a failure of the test.
long long g_words = 0, g_bad_reads = 0;
uint32_t ldg_word(const uint32_t* words, long long w) {
  if (w < 0 || w >= g_words) {
    ++g_bad_reads;
    return 0;
  }
  return words[w];
}
#define DIBELLA_IN_BOUNDS(v, lim, code) ((v) >= 0 && (long long)(v) < (long long)(lim) ? true : (++g_bad_reads, false))

unsigned pop_warp(Counters* cnt, int q) {
  unsigned idx = 0;
  if (g_lane == 0) idx = atomicAdd(&cnt->head[q], 1u);
  return __shfl_sync(kFull, idx, 0);
}

#include "../paper_2001_10049_gb300/csrc/xdrop_bits.cuh"
#include "../paper_2001_10049_gb300/csrc/xdrop_bits_run.cuh"

ExtendParams g_p;
int g_form = 0;

int g_map[32];

void lane_main() {
  switch (g_form) {
    case 4: bits_shared_run<4>(g_p, g_map); break;
    case 5: bits_shared_run<5>(g_p, g_map); break;
    case 6: bits_shared_run<6>(g_p, g_map); break;
    case 44: bits_warp_run<4, 4>(g_p); break;
    case 54: bits_warp_run<5, 4>(g_p); break;
    case 64: bits_warp_run<6, 4>(g_p); break;
    default: break;
  }
  g_fib[g_lane].done = true;
  swapcontext(&g_fib[g_lane].ctx, &g_main);
}

}  // namespace

// form: planes of the shared-lane form (then its suspended extensions that need
// a whole warp go on in the whole-warp form of 4 words), or 10 x planes + words of
// the whole-warp form alone.  Runs one warp over n_items extensions.  out:
// n_items x {best, i, j, cells}; a handed-on extension gets best = -1.  stats:
// queued suspensions, extensions handed to the 4-word form, items pushed beyond
// it, all suspensions.  Returns the out-of-store reads and out-of-range indices seen (0
// expected), or -1 if the lanes fell out of step.
static int run_warp(int form) {
  g_form = form;
  for (int i = 0; i < 32; ++i) {
    Fiber& f = g_fib[i];
    f.done = false;
    f.stack.resize(kStack);
    getcontext(&f.ctx);
    f.ctx.uc_stack.ss_sp = f.stack.data();
    f.ctx.uc_stack.ss_size = f.stack.size();
    f.ctx.uc_link = &g_main;
    makecontext(&f.ctx, lane_main, 0);
  }
  for (;;) {
    int n_done = 0;
    for (g_lane = 0; g_lane < 32; ++g_lane) {
      if (!g_fib[g_lane].done) swapcontext(&g_main, &g_fib[g_lane].ctx);
      n_done += g_fib[g_lane].done;
    }
    if (n_done == 32) return 0;
    if (n_done != 0) return -1;
    for (int i = 0; i < 32; ++i) g_snap[i] = g_fib[i].in;
  }
}

extern "C" long long bits_emulate(int form, const uint32_t* words, long long n_words, const long long* a0,
                                  const long long* b0, const int* m, const int* n, int n_items, int X,
                                  int reserve, int young, int max_groups, int pool_words, int res_cap, long long* out,
                                  long long* stats) {
  std::vector<Item> items(n_items);
  std::vector<ExtOut> ext(n_items);
  std::vector<int> q(n_items), res(res_cap, -1), esc(n_items, -1), last(n_items, -1);
  std::vector<uint32_t> pool(pool_words + 1);
  for (int i = 0; i < n_items; ++i) {
    items[i] = Item{a0[i], b0[i], m[i], n[i], 0, 0};
    ext[i].best = -1;
    q[i] = form >= 10 ? -2 - i : i;
  }
  Counters cnt;
  memset(&cnt, 0, sizeof(cnt));
  cnt.tail[0] = (unsigned)n_items;
  ExtendParams p{words, items.data(), ext.data(), &cnt, q.data(), 0, esc.data(), 1, 1, 2, reserve, young,
                 max_groups, res.data(), 2, res_cap, pool.data(), (unsigned)pool_words, n_items, {1, -1, -1, X}};
  g_words = n_words;
  g_bad_reads = 0;
  g_p = p;
  int rc = run_warp(form);
  if (rc == 0 && form < 10) {
    p.wide_q = esc.data();
    p.wide_q_id = 1;
    p.esc_q = last.data();
    p.esc_q_id = 3;
    g_p = p;
    rc = run_warp(10 * form + 4);
  }
  if (rc) return rc;
  for (int i = 0; i < n_items; ++i) {
    out[4 * i] = ext[i].best;
    out[4 * i + 1] = ext[i].i_end;
    out[4 * i + 2] = ext[i].j_end;
    out[4 * i + 3] = ext[i].cells;
  }
  stats[0] = cnt.tail[2];
  stats[1] = cnt.tail[1];
  stats[2] = cnt.tail[3];
  stats[3] = cnt.stat[2];
  return g_bad_reads;
}
