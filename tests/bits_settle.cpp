// bits_settle of csrc/xdrop_bits_run.cuh on the CPU emulation of bits_emulation.cpp:
// the cells that the lanes of equal groups have counted, summed per group.  Built
// and driven by tests/test_bits_settle.py.
#include "bits_emulation.cpp"

namespace {

uint32_t g_counts[32];
long long g_sums[32];
int g_len;

void settle_lane() {
  BitLane<6, 1> L;
  BitForm<6, 1>::clear(L);
  L.cells = g_counts[g_lane];
  BitTask t;
  memset(&t, 0, sizeof(t));
  t.cells = 7;
  const int first = g_lane / g_len * g_len;
  bits_settle<6, 1>(L, t, g_lane, first, g_len, group_masks(g_lane, first, g_len));
  g_sums[g_lane] = t.cells;
  g_fib[g_lane].done = true;
  swapcontext(&g_fib[g_lane].ctx, &g_main);
}

}  // namespace

extern "C" void settle_sums(const uint32_t* counts, int len, long long* sums) {
  memcpy(g_counts, counts, sizeof(g_counts));
  g_len = len;
  for (int i = 0; i < 32; ++i) {
    Fiber& f = g_fib[i];
    f.done = false;
    f.stack.resize(kStack);
    getcontext(&f.ctx);
    f.ctx.uc_stack.ss_sp = f.stack.data();
    f.ctx.uc_stack.ss_size = f.stack.size();
    f.ctx.uc_link = &g_main;
    makecontext(&f.ctx, settle_lane, 0);
  }
  for (int n_done = 0; n_done < 32;) {
    n_done = 0;
    for (g_lane = 0; g_lane < 32; ++g_lane) {
      if (!g_fib[g_lane].done) swapcontext(&g_main, &g_fib[g_lane].ctx);
      n_done += g_fib[g_lane].done;
    }
    for (int i = 0; i < 32; ++i) g_snap[i] = g_fib[i].in;
  }
  memcpy(sums, g_sums, sizeof(g_sums));
}
