// The batch's bit-sliced kernels (see xdrop_bits.cuh): the shared-lane form, the
// whole-warp form, and the pool of suspended extensions.  Included by
// dibella_xdrop.cu inside its anonymous namespace after xdrop_bits.cuh.

// What a group of lanes works on (the same in all its lanes).
struct BitTask {
  int item, m, n;
  int f0;        // the window's lowest place on antidiagonal d is i = f0 + (d + 1) / 2
  int bi, bj;    // cell of the best score
  long long a0, b0, cells;
  bool active;
  int restarts;  // times it has started over in the shared-lane form, as the pool was full
  __device__ __forceinline__ int window(int d) const { return f0 + ((d + 1) >> 1); }
};

__device__ __forceinline__ void bits_finish(const ExtendParams& p, const BitTask& t, int best) {
  ExtOut o;
  o.best = best; o.i_end = t.bi; o.j_end = t.bj; o.status = 0; o.cells = t.cells;
  p.ext[t.item] = o;
  atomicAdd(&p.cnt->cells[p.cells_idx], (unsigned long long)t.cells);
}
// A suspended extension in the pool: kDumpHead words (item, d, f0, best, bi, bj,
// r1 and r2, words held, cells, window), then its words plane by plane: both
// rows' planes and the dead mask.  It was suspended because its band needs
// another window, so it says which: `want` words from place `shift` of the one
// held on.  A queue entry is the pool offset (a multiple of 32)
// plus want - 1 (of at most 32 words), or -2 - item for an extension that starts
// over because the pool was full; -1 is a slot that is not written yet.
//
// The pool is not given back within a launch, and once a request has found it
// full it stays full.  From then on what is suspended starts over, so that has to
// end: an extension starts over at most kMaxRestarts times in the shared-lane form
// (counted in its result's status until then) and goes on to the whole-warp launch,
// and the whole-warp form keeps one whose band has become narrow instead of handing
// it back.  (Bounded by the queue's slots alone, 6,000 bases of AC against as many
// of A at X = 25 were started 202 times with 100 slots.)
constexpr int kDumpHead = 16;
// (1.7 M E. coli-sized seeds at X = 25, whose 734,000 suspensions run out of pool:
// 1,098 / 987 / 950 ms with 2 / 4 / 8 where no limit took 946, and 939 with 16 where
// no limit took 938.  What is passed on has a warp of 4 words a lane to itself:
// 4.9 / 1.4 / 0.15 / 0.003% of the cells, in 335 / 95 / 13 / 6 ms.)
constexpr int kMaxRestarts = 16;
template <int NB>
__device__ __forceinline__ unsigned dump_words(int len) {
  return (unsigned)(kDumpHead + (2 * NB + 1) * len + 31) & ~31u;
}

// Writes the extension of lanes first .. first + len - 1 (W words each) to the
// pool and its entry to `queue` (null: none).  Every lane of the warp calls it;
// `mine` says whose group it is.  Returns the entry; with `keep`, -1 and nothing
// done if the pool is full.
template <int NB, int W>
__device__ __forceinline__ int bits_suspend(const ExtendParams& p, const BitLane<NB, W>& L, const BitTask& t, bool mine,
                                             int lane, int first, int len, int shift, int want, int* queue,
                                             int q_id, bool keep = false) {
  const bool leader = mine && lane == first;
  const unsigned size = dump_words<NB>(W * len);
  int off = -1;
  if (leader && *((volatile unsigned*)&p.cnt->pool) < p.pool_words) {
    const unsigned at = atomicAdd(&p.cnt->pool, size);
    if (at + size <= p.pool_words) off = (int)at;
  }
  off = __shfl_sync(kFull, off, first);
  if (keep && off < 0) return -1;
  if (mine && off >= 0) {
    uint32_t* o = p.pool + off;
    if (leader) {
      o[0] = (uint32_t)t.item;
      o[1] = (uint32_t)L.d;
      o[2] = (uint32_t)t.f0;
      o[3] = (uint32_t)L.best;
      o[4] = (uint32_t)t.bi;
      o[5] = (uint32_t)t.bj;
      o[6] = L.r1;
      o[7] = L.r2;
      o[8] = (uint32_t)(W * len);
      o[9] = (uint32_t)t.cells;
      o[10] = (uint32_t)(t.cells >> 32);
      o[11] = (uint32_t)shift;
    }
    o += kDumpHead + W * (lane - first);
#pragma unroll
    for (int w = 0; w < W; ++w) {
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        o[(2 * k) * (W * len) + w] = L.r[0][w][k];
        o[(2 * k + 1) * (W * len) + w] = L.r[1][w][k];
      }
      o[2 * NB * (W * len) + w] = L.dead[w];
    }
  }
  __threadfence();
  __syncwarp();
  const int entry = off >= 0 ? off + min(want, 32) - 1 : -2 - t.item;
  if (leader) {
    if (off < 0) {
      atomicAdd(&p.cnt->cells[7], (unsigned long long)t.cells);
      if (queue == p.res_q) {
        if (t.restarts < kMaxRestarts) {
          p.ext[t.item].status = t.restarts + 1;
          __threadfence();
        } else {
          queue = p.esc_q;
          q_id = p.esc_q_id;
        }
      }
    }
    atomicAdd(&p.cnt->stat[p.bits_esc_stat], 1u);
  }
  if (leader && queue != nullptr) {
    unsigned s = atomicAdd(&p.cnt->tail[q_id], 1u);
    // An extension may be suspended any number of times, but it enters esc_q
    // only once: that is where it goes when its own queue has no slot left.
    if (queue != p.esc_q && (long long)s >= p.res_cap) {
      queue = p.esc_q;
      s = atomicAdd(&p.cnt->tail[p.esc_q_id], 1u);
    }
    if (DIBELLA_IN_BOUNDS(s, queue == p.esc_q ? p.q_cap : p.res_cap, 2)) atomicExch(&queue[s], entry);
  }
  return __shfl_sync(kFull, entry, first);
}

// The task of queue entry v (>= 0: suspended, else -2 - item: from the start,
// its window's lowest place `start_f0`); true if suspended.
__device__ __forceinline__ bool bits_task(const ExtendParams& p, BitTask& t, int v, int start_f0) {
  const bool held = v >= 0;
  const uint32_t* o = p.pool + (v & ~31);
  t.item = held ? (int)__ldcg(o) : -2 - v;
  t.restarts = 0;
  t.active = DIBELLA_IN_BOUNDS(t.item, p.q_cap, 3);  // (debug build: a bad item is dropped)
  if (!t.active) return false;
  const Item it = p.items[t.item];
  t.m = it.m;
  t.n = it.n;
  t.a0 = it.a0;
  t.b0 = it.b0;
  t.f0 = held ? (int)__ldcg(o + 2) : start_f0;
  t.bi = held ? (int)__ldcg(o + 4) : 0;
  t.bj = held ? (int)__ldcg(o + 5) : 0;
  t.cells = held ? (long long)(__ldcg(o + 9) | ((unsigned long long)__ldcg(o + 10) << 32)) : 0;
  return held;
}

// The rows of a suspended extension: this lane's words begin at place `bit` of
// the window it held (places outside it are dead).  W > 1: at a whole word.
template <int NB, int W>
__device__ __forceinline__ void bits_load(const ExtendParams& p, BitLane<NB, W>& L, int v, int bit) {
  const uint32_t* o = p.pool + (v & ~31);
  BitForm<NB, W>::init(L, -1);
  L.d = (int)__ldcg(o + 1);
  L.best = (int)__ldcg(o + 3);
  L.r1 = __ldcg(o + 6);
  L.r2 = __ldcg(o + 7);
  const int len = (int)__ldcg(o + 8);
  const unsigned r = (unsigned)bit & 31u;
  o += kDumpHead;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const int x = (bit >> 5) + w;
    const bool in = x >= 0 && x < len, in1 = x + 1 >= 0 && x + 1 < len;
#pragma unroll
    for (int v2 = 0; v2 <= 2 * NB; ++v2) {  // the planes in the order of bits_suspend, then the dead mask
      const uint32_t fill = v2 < 2 * NB ? BitForm<NB, W>::dead_plane(v2 >> 1) : 0xFFFFFFFFu;
      uint32_t y = in ? __ldcg(o + v2 * len + x) : fill;
      if (W == 1) y = __funnelshift_r(y, in1 ? __ldcg(o + v2 * len + x + 1) : fill, r);
      if (v2 < 2 * NB)
        L.r[v2 & 1][w][v2 >> 1 < NB ? v2 >> 1 : 0] = y;
      else
        L.dead[w] = y;
    }
  }
}

// Brings the group's cell count and best cell up to date (before its layout changes or it ends).
template <int NB, int W>
__device__ __forceinline__ void bits_settle(BitLane<NB, W>& L, BitTask& t, int lane, int first, int len,
                                            const GroupMasks& gm) {
  // Inclusive scan within the group, in 64 bits: a layout lasts as long as the band
  // keeps its place, and 2^25 antidiagonals of a steady band are beyond 32 bits in
  // the group (in a lane they stay below: 32 W cells each, W up to 4).
  unsigned long long s = L.cells;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long v = __shfl_up_sync(kFull, s, o);
    if (lane - o >= first) s += v;
  }
  t.cells += (long long)__shfl_sync(kFull, s, first + len - 1);
  L.cells = 0;
  int lo, hi;
  group_ends<W>(L.imp, lane, first, gm.grp, lo, hi);
  if (L.imp_d >= 0) {
    t.bi = t.window(L.imp_d) + lo;
    t.bj = L.imp_d - t.bi;
  }
  L.imp_d = -1;
#pragma unroll
  for (int w = 0; w < W; ++w) L.imp[w] = 0;
}

constexpr int kCheck = 16;
constexpr int kMarginTrig = kCheck / 2 + 1;  // places of the window that a band may cross until the next look
constexpr int kMarginNew = 12;               // kept free at both ends of a window that is laid out anew (10 to 16: the same)
constexpr int kMarginKeep = 20;              // ... and of one that gives lanes back
constexpr int kInitLanes = 2;
// Lanes beyond its own that a suspended extension waits for before it joins
// others: without, two extensions can suspend each other every few looks (150,000
// seeds at X = 15 with 3 lanes counted for each: 194 ms, 44 with 4 spare lanes; with
// the 4 lanes that the rule below counts, 38 either way).
constexpr int kResumeSlack = 4;
constexpr int kNoRoom = INT32_MIN;           // (no queue entry: see bits_suspend)
#ifndef XDROP_BITS_SHARED_MAX  // (the CPU test lowers it, to reach the whole-warp form with short sequences)
#define XDROP_BITS_SHARED_MAX 32
#endif
constexpr int kSharedMax = XDROP_BITS_SHARED_MAX;  // lanes that one extension may take
constexpr int kNarrowAgain = 24 * kSharedMax;      // live cells below which the whole-warp form gives one back

// Whole-warp form: the extension of queue entry v by all 32 lanes, W words
// each, for a band that outgrows one word a lane.  With BACK it is suspended to
// the shared-lane form again once its band has become narrow, while the pool has
// room; a band that outgrows this form too goes to esc_q (from W = 4 on: to the
// forms that hold scores, from the start).
template <int NB, int W, bool BACK>
__device__ __forceinline__ void bits_warp_one(const ExtendParams& p, int v, const uint32_t (&kx)[NB]) {
  using F = BitForm<NB, W>;
  constexpr int kWin = 32 * 32 * W;
  constexpr int kMargin = 17;  // 32 antidiagonals between looks: at most 16 places either way
  const int lane = threadIdx.x & 31;
  const GroupMasks gm = group_masks(lane, 0, 32);
  const uint32_t* __restrict__ words = p.words;
  BitTask t;
  typename F::Lane L;
  F::clear(L);
  if (bits_task(p, t, v, -kWin / 2)) {  // its words go to the middle of the window
    const int off = (32 * W - (int)__ldcg(p.pool + (v & ~31) + 8)) / 2;
    bits_load<NB, W>(p, L, v, 32 * (W * lane - off));
    t.f0 -= 32 * off;
  } else {
    if (!t.active) return;
    F::init(L, kWin / 2 - 32 * W * lane);
  }
  F::load_window(L, words, t.a0, t.b0, t.m, t.n, t.window(L.d) + 32 * W * lane, L.d);
  bool back = BACK;
  for (;;) {
    F::load_feed(L, words, t.a0, t.b0, t.m, t.n, t.window(L.d) + 32 * W * lane, L.d);
    F::template steps<32, true>(L, kx, gm);
    uint32_t live[W];
#pragma unroll
    for (int w = 0; w < W; ++w) live[w] = ~L.dead[w];
    int lo, hi;
    group_ends<W>(live, lane, 0, kFull, lo, hi);
    const bool narrow = back && lo >= 0 && hi - lo < kNarrowAgain;
    const bool inside = lo >= kMargin && hi <= kWin - 1 - kMargin;
    if (inside && !narrow) continue;
    bits_settle<NB, W>(L, t, lane, 0, 32, gm);
    if (lo < 0) {  // ended
      if (lane == 0) bits_finish(p, t, L.best);
      break;
    }
    if (narrow) {
      const int want = (hi - lo + 1 + 2 * kMarginNew + 31) >> 5;
      if (bits_suspend<NB, W>(p, L, t, true, lane, 0, 32, lo - ((32 * want - (hi - lo + 1)) >> 1), want, p.res_q,
                              p.res_q_id, true) != -1)
        break;
      back = false;
      if (inside) continue;
    }
    // Move the window by whole lanes to bring the band to its middle.
    const int by = ((lo + hi) / 2 - kWin / 2 + (lo < kMargin ? -16 * W : 16 * W)) / (32 * W);
    const int nlo = lo - by * 32 * W, nhi = hi - by * 32 * W;
    if (nlo < kMargin || nhi > kWin - 1 - kMargin) {
      if (W < 4) {
        bits_suspend<NB, W>(p, L, t, true, lane, 0, 32, 0, 32 * W, p.esc_q, p.esc_q_id);
      } else if (lane == 0) {
        const unsigned s = atomicAdd(&p.cnt->tail[p.esc_q_id], 1u);
        if (DIBELLA_IN_BOUNDS(s, p.q_cap, 2)) p.esc_q[s] = t.item;
        atomicAdd(&p.cnt->stat[p.bits_esc_stat], 1u);
        atomicAdd(&p.cnt->cells[7], (unsigned long long)t.cells);
      }
      break;
    }
    const int src = lane + by;
    const bool held = src >= 0 && src < 32;
#pragma unroll
    for (int w = 0; w < W; ++w) {
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        const uint32_t x = __shfl_sync(kFull, L.r[0][w][k], src & 31), y = __shfl_sync(kFull, L.r[1][w][k], src & 31);
        L.r[0][w][k] = held ? x : F::dead_plane(k);
        L.r[1][w][k] = held ? y : F::dead_plane(k);
      }
      const uint32_t dd = __shfl_sync(kFull, L.dead[w], src & 31);
      L.dead[w] = held ? dd : 0xFFFFFFFFu;
    }
    t.f0 += by * 32 * W;
    F::load_window(L, words, t.a0, t.b0, t.m, t.n, t.window(L.d) + 32 * W * lane, L.d);
  }
  __syncwarp();
}

// The extensions of the queue one by one (persistent).
template <int NB, int W>
__device__ __forceinline__ void bits_warp_run(const ExtendParams& p) {
  uint32_t kx[NB];
  bits_threshold<NB>(p.sc.X, kx);
  const unsigned tail = *((volatile unsigned*)&p.cnt->tail[p.wide_q_id]);
  for (;;) {
    const unsigned q = pop_warp(p.cnt, p.wide_q_id);
    if (q >= tail) break;
    bits_warp_one<NB, W, false>(p, p.wide_q[q], kx);
  }
}

// Shared-lane form (persistent): a warp's 32 lanes, one word of 32 cells each,
// are dealt out to as many extensions as their bands leave room for, so that a
// band of 24 cells takes two lanes and one of 130 cells six.  Every kCheck
// antidiagonals each group looks whether its band has come near an end of its
// window; if one has (or has ended), the whole warp's layout is redone: ended
// groups write their result, bands get the lanes they need, free lanes are
// given to the next extensions of the queue, and all rows move to their new
// lanes by shuffles.  An extension that has run for fewer than p.young
// antidiagonals, or whose band takes more than half of them, counts for
// p.reserve lanes (the band that an extension of two unrelated sequences grows
// and keeps), and at most p.max_groups share a warp.
// If the bands outgrow the warp, the extension that has come least far is
// suspended to the pool, from where any warp with room takes it up again; a band
// too wide for 32 lanes goes on in the whole-warp form.
template <int NB>
__device__ __forceinline__ void bits_shared_run(const ExtendParams& p, int* map) {
  using F = BitForm<NB, 1>;
  const int lane = threadIdx.x & 31;
  uint32_t kx[NB];
  bits_threshold<NB>(p.sc.X, kx);
  const unsigned tail = *((volatile unsigned*)&p.cnt->tail[p.wide_q_id]);
  const uint32_t* __restrict__ words = p.words;
  typename F::Lane L;
  F::clear(L);
  BitTask t;
  t.item = t.m = t.n = t.f0 = t.bi = t.bj = 0;
  t.a0 = t.b0 = t.cells = 0;
  t.restarts = 0;
  t.active = false;
  int first = lane, len = 1;  // this lane's group; a lane without work is a group of its own
  GroupMasks gm = group_masks(lane, first, len);
  bool exhausted = false;
  for (;;) {
    // ---- layout ----
    bits_settle<NB, 1>(L, t, lane, first, len, gm);
    const uint32_t live[1] = {~L.dead[0]};
    int lo, hi;
    group_ends<1>(live, lane, first, gm.grp, lo, hi);
    if (t.active && lo < 0) {
      if (lane == first) bits_finish(p, t, L.best);
      t.active = false;
    }
    // Lanes wanted, from place b of the present window on (the band in the
    // middle); a window that the band neither nears nor leaves lanes of stays.
    const bool trig = lo < kMarginTrig || hi > 32 * len - 1 - kMarginTrig;
    const int width = hi - lo + 1;
    const int fit = (width + 2 * (trig ? kMarginNew : kMarginKeep) + 31) >> 5;
    const int need = trig || fit < len ? fit : len;
    const int b = trig || fit < len ? lo - ((32 * need - width) >> 1) : 0;
    int want = t.active && lane == first ? need : 0;
    int total = __reduce_add_sync(kFull, want);
    // A band that needs more than 32 lanes: the warp suspends all others and
    // goes on with it in the whole-warp form.  Else, if the bands need more than
    // 32 lanes together, those that have come least far are suspended.
    const unsigned wide = __ballot_sync(kFull, want > kSharedMax);
    int alone = -1;
    while (wide ? total > 0 : total > 32) {
      const int key = want > kSharedMax ? lane : (want ? (L.d + 1) * 32 + lane : INT32_MAX);
      const int who = __reduce_min_sync(kFull, key) & 31;
      const bool take = alone == -1 && ((wide >> who) & 1u);
      const int v = bits_suspend<NB, 1>(p, L, t, first == who && t.active, lane, who, __shfl_sync(kFull, len, who), b,
                                        want, take ? nullptr : ((wide >> who) & 1u) ? p.esc_q : p.res_q,
                                        ((wide >> who) & 1u) ? p.esc_q_id : p.res_q_id);
      if (take) alone = v;
      if (lane == who) want = 0;
      total = __reduce_add_sync(kFull, want);
    }
    if (alone != -1) {
      bits_warp_one<NB, 2, true>(p, alone, kx);
      t.active = false;
      F::clear(L);
      first = lane;
      len = 1;
      gm = group_masks(lane, first, len);
      continue;
    }
    t.active = __shfl_sync(kFull, want, first) > 0;
    // Extensions for the lanes that are left: suspended ones first.  A warp that
    // suspends one looks here again before it ends, so none is left behind.
    int room = 32 - __reduce_add_sync(kFull, L.d < p.young || (2 * want > p.reserve && want > kInitLanes) ? max(want, want > 0 ? p.reserve : 0)
                                                                                    : want);
    int groups = __popc(__ballot_sync(kFull, want > 0)), used = total;
    int entry = -1, efirst = 0, elen = 0;  // what this lane's new group takes up
    bool over = false;
    bool waiting = false;  // a suspended one waits for more lanes: no new ones, or they would crowd it out for good
    while (groups < p.max_groups) {
      int v = -1;
      if (lane == 0) {
        for (;;) {
          const unsigned h = *((volatile unsigned*)&p.cnt->head[p.res_q_id]);
          if ((long long)h >= p.res_cap || h >= *((volatile unsigned*)&p.cnt->tail[p.res_q_id])) break;
          const int c = *((volatile int*)&p.res_q[h]);
          if (c == -1) break;
          if ((c >= 0 ? (c & 31) + 1 + (groups > 0 ? kResumeSlack : 0) : max(kInitLanes, p.reserve)) > room) {
            v = kNoRoom;
            break;
          }
          if (atomicCAS(&p.cnt->head[p.res_q_id], h, h + 1) == h) {
            v = c;
            break;
          }
        }
      }
      v = __shfl_sync(kFull, v, 0);
      if (v == kNoRoom) waiting = true;
      if (v == -1 || v == kNoRoom) break;
      __threadfence();  // its words were written before its queue entry
      const int l = v >= 0 ? (v & 31) + 1 : kInitLanes;
      if (lane >= used && lane < used + l) {
        entry = v;
        over = v < 0;
        efirst = used;
        elen = l;
      }
      used += l;
      room -= v >= 0 ? l : max(kInitLanes, p.reserve);
      ++groups;
    }
    int n_new = exhausted || waiting ? 0 : min(room / p.reserve, p.max_groups - groups);
    if (n_new > 0) {
      unsigned base = 0;
      if (lane == 0) base = atomicAdd(&p.cnt->head[p.wide_q_id], (unsigned)n_new);
      base = __shfl_sync(kFull, base, 0);
      const int got = base < tail ? (int)min((unsigned)n_new, tail - base) : 0;
      exhausted = got < n_new;
      if (lane >= used && lane < used + kInitLanes * got) {
        const int j = (lane - used) / kInitLanes;
        entry = -2 - p.wide_q[base + (unsigned)j];
        efirst = used + j * kInitLanes;
        elen = kInitLanes;
      }
      used += kInitLanes * got;
    }
    if (used == 0) break;
    // new first lanes: the kept groups in their order, then the new ones
    int s = want;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(kFull, s, o);
      if (lane >= o) s += v;
    }
    const int at = s - want;  // (leaders)
    uint32_t starts = __reduce_or_sync(kFull, want > 0 ? 1u << at : 0u);
    if (want > 0) map[at] = lane;
    __syncwarp();
    const int nfirst = lane < total ? 31 - __clz((int)(starts & ((2u << lane) - 1u))) : lane;
    const int from = lane < total ? map[nfirst] : lane;  // the group's old leader
    __syncwarp();
    const int old_len = __shfl_sync(kFull, len, from), old_want = __shfl_sync(kFull, want, from);
    const int shift = __shfl_sync(kFull, b, from);
    const int place = shift + 32 * (lane - nfirst);
    const unsigned bit = (unsigned)place & 31u;
    const int src = from + (place >> 5);
    const bool held = lane < total && src >= from && src < from + old_len;
    const bool held1 = lane < total && src + 1 >= from && src + 1 < from + old_len;
#pragma unroll
    for (int v = 0; v <= 2 * NB; ++v) {  // every plane of both rows, then the dead mask
      const uint32_t fill = v < 2 * NB ? F::dead_plane(v % NB) : 0xFFFFFFFFu;
      const uint32_t old = v < 2 * NB ? L.r[v / NB < 2 ? v / NB : 0][0][v % NB] : L.dead[0];
      const uint32_t x = __shfl_sync(kFull, old, src & 31), y = __shfl_sync(kFull, old, (src + 1) & 31);
      const uint32_t z = __funnelshift_r(held ? x : fill, held1 ? y : fill, bit);
      if (v < 2 * NB)
        L.r[v / NB < 2 ? v / NB : 0][0][v % NB] = z;
      else
        L.dead[0] = z;
    }
    L.r1 = __shfl_sync(kFull, L.r1, from);
    L.r2 = __shfl_sync(kFull, L.r2, from);
    L.d = __shfl_sync(kFull, L.d, from);
    L.best = __shfl_sync(kFull, L.best, from);
    t.item = __shfl_sync(kFull, t.item, from);
    t.m = __shfl_sync(kFull, t.m, from);
    t.n = __shfl_sync(kFull, t.n, from);
    t.f0 = __shfl_sync(kFull, t.f0, from) + shift;
    t.bi = __shfl_sync(kFull, t.bi, from);
    t.bj = __shfl_sync(kFull, t.bj, from);
    t.a0 = __shfl_sync(kFull, t.a0, from);
    t.b0 = __shfl_sync(kFull, t.b0, from);
    t.cells = __shfl_sync(kFull, t.cells, from);
    t.restarts = __shfl_sync(kFull, t.restarts, from);
    t.active = lane < total;
    first = nfirst;
    len = old_want;
    if (elen > 0) {
      first = efirst;
      len = elen;
      if (bits_task(p, t, entry, -16 * kInitLanes)) {
        const int place = (int)__ldcg(p.pool + (entry & ~31) + 11);
        t.f0 += place;
        bits_load<NB, 1>(p, L, entry, place + 32 * (lane - first));
      } else {
        F::init(L, 16 * kInitLanes - 32 * (lane - first));
        if (over) t.restarts = __ldcg(&p.ext[t.item].status);
      }
    }
    if (!t.active) {
      F::clear(L);
      first = lane;
      len = 1;
    }
    if (!__any_sync(kFull, t.active)) continue;  // (debug build: only bad items)
    gm = group_masks(lane, first, len);
    if (t.active) F::load_window(L, words, t.a0, t.b0, t.m, t.n, t.window(L.d) + 32 * (lane - first), L.d);
    // ---- antidiagonals, until a band comes near an end of its window ----
    const uint32_t near_end = (gm.end_lo & ((1u << kMarginTrig) - 1u)) | (gm.end_hi & ~((1u << (32 - kMarginTrig)) - 1u));
    for (;;) {
      if (t.active) F::load_feed(L, words, t.a0, t.b0, t.m, t.n, t.window(L.d) + 32 * (lane - first), L.d);
      // (a lane without work is never clipped: its planes stay 0 and its band empty)
      const bool clip = __any_sync(kFull, t.active && F::clipped(L));
      bool look = false;
#pragma unroll 1
      for (int h = 0; h < 32 && !look; h += kCheck) {
        if (clip)
          F::template steps<kCheck, true>(L, kx, gm);
        else
          F::template steps<kCheck, false>(L, kx, gm);
        const uint32_t any = __ballot_sync(kFull, L.dead[0] != 0xFFFFFFFFu);
        look = __any_sync(kFull, t.active && ((any & gm.grp) == 0 || (~L.dead[0] & near_end) != 0));
      }
      if (look) break;
    }
  }
}

