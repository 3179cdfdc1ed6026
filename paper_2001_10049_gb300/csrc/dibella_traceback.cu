// Traceback of seeded X-drop alignments: the edits of each seed's best
// alignment as run-length encoded columns (diBELLA Sec. 1: an alignment is
// the list of edits that makes two overlapping regions identical; Sec. 2: an
// alignment's columns pair two characters, or a character with a gap).
//
// The extension is the one dibella_xdrop_batch computes (band of antidiagonal
// d from the live cells of d-1 widened by one, live iff H >= best(<d) - X,
// strict improvement with the smallest i on ties, both extensions from the
// seed); each evaluated cell also keeps the move that gave its value, taking
// the diagonal first, then the step in A, then the step in B' on equal
// values.  The walk from the best cell back to the seed follows those moves.
//
// A warp per seed re-runs both extensions with the band's cells across its
// lanes.  Its scratch (a slot of the caller's workspace per warp) holds three
// rows of H indexed by the position in A, read and written coalesced, and a
// stream of 32-bit words with, per evaluated antidiagonal, two header words
// (the band's first i and its width), the band's moves at 2 bits per cell
// (packed by warp reductions), and a trailer word (the width again), so that
// lane 0 can walk back one antidiagonal at a time from the best cell.
//
// With unit scores and X <= 59 the extension runs in the bit-sliced form
// (xdrop_bits.cuh) with one word of cells a lane: the comparisons that choose a
// cell's value are its move, two planes of 32 cells a lane, so recording costs a
// store and a few counts.  Both extensions run at once, 16 lanes each, where
// their bands and move words allow.  The walk back is done by the lanes
// together: each holds the move words of one or two of the next 32
// antidiagonals, and a run of diagonal steps is one look-up.  Bands beyond 990
// cells take the general form above.
// 2,000 accepted overlaps of E. coli-sized reads at X = 25 take 13.5 to 18.2 ms (the
// general form, bound by its rows in memory and one lane's walk, 50 to 73), by the
// longest overlap among them: a serial chain of some 70,000 antidiagonals, about a
// third of its time the walk.

#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/dibella.h"

namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;
__device__ __forceinline__ uint32_t ldg_word(const uint32_t* __restrict__ words, long long w) { return __ldg(words + w); }

#include "xdrop_bits.cuh"

constexpr int kTbThreads = 128;
constexpr int32_t kDead = INT32_MIN / 2;  // dead, or outside its antidiagonal's band
constexpr uint32_t kMoveNone = 0, kMoveDiag = 1, kMoveA = 2, kMoveB = 3;
constexpr uint32_t kOpEq = DIBELLA_OP_EQ, kOpX = DIBELLA_OP_DIFF, kOpIns = DIBELLA_OP_INS, kOpDel = DIBELLA_OP_DEL;

struct TbArgs {
  const uint32_t* words;
  const int64_t* word_offsets;
  const int32_t* lengths;
  long long n_reads;
  const dibella_pair_t* pairs;
  long long n_pairs;
  int k, M, S, G, X;
  int max_len;
  dibella_result_t* results;
  uint32_t* ops;
  int ops_per_seed;
  int32_t* n_ops;
  long long n_lanes;
  long long moves_words;
  char* workspace;
  long long lane_bytes;
};

__host__ __device__ inline long long tb_copy_words(long long len) { return ((len + 15) / 16 + 3) / 4 * 4; }

// Base q of the copy whose first base is base index `start` of the store.
__host__ __device__ inline uint32_t tb_base(const uint32_t* words, long long start, long long q) {
  const long long g = start + q;
  return (words[g >> 4] >> (2 * (g & 15))) & 3u;
}

// One extension's sequences: a(i) = base a0 + sa * i of the store (sa = +1 or
// -1), likewise b(j); m and n characters.
struct TbSeq {
  long long a0, b0;
  int sa, sb;
  int m, n;
};

struct TbExt {
  int best, i_end, j_end;
  long long cells;
  long long best_rec;  // stream index of the best antidiagonal's header (-1: the origin)
  bool recorded;       // every antidiagonal up to the best one fit the stream
};

// The X-drop extension from the origin, run by the 32 lanes of a warp (every
// lane calls it; lane l computes cell i = i0 + l of each 32-cell chunk of the
// band), recording moves into mv (capacity cap words) while they fit.  The
// rows r0..r2 (antidiagonals d, d-1, d-2, indexed by i) live in the warp's
// workspace slot, read and written coalesced.  Each chunk's 2-bit moves are
// packed 16 cells to a word by two warp OR-reductions; lane 0 writes the
// stream, so its format is the one tb_walk reads.  All lanes return the same
// result.
__device__ TbExt tb_extend_warp(const TbArgs& p, const TbSeq& s, int32_t* r0, int32_t* r1, int32_t* r2,
                                uint32_t* mv, long long cap) {
  constexpr unsigned kAll = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31;
  TbExt e{0, 0, 0, 0, -1, true};
  int lo2 = 1, hi2 = 0, lo1 = 0, hi1 = 0;
  if (lane == 0) r1[0] = 0;
  __syncwarp();
  int live_lo = 0, live_hi = 0;
  int best = 0;
  long long w = 0;
  bool streaming = true;
  const int last_d = s.m + s.n;
  for (int d = 1; d <= last_d; ++d) {
    int lo = live_lo > d - s.n ? live_lo : d - s.n;
    if (lo < 0) lo = 0;
    int hi = live_hi + 1 < d ? live_hi + 1 : d;
    if (hi > s.m) hi = s.m;
    if (lo > hi) break;
    const int width = hi - lo + 1;
    const long long rec = w;
    const bool keep = streaming && w + 3 + (width + 15) / 16 <= cap;
    streaming = keep;
    if (keep && lane == 0) {
      mv[w] = (uint32_t)lo;
      mv[w + 1] = (uint32_t)width;
    }
    if (keep) w += 2;
    const int threshold = best - p.X;
    int row_best = kDead, row_best_i = -1, new_lo = -1, new_hi = -1;
    for (int i0 = lo; i0 <= hi; i0 += 32) {
      const int i = i0 + lane;
      const int j = d - i;
      int h = kDead;
      uint32_t from = kMoveNone;
      bool live = false;
      if (i <= hi) {
        if (i >= 1 && j >= 1 && i - 1 >= lo2 && i - 1 <= hi2 && r2[i - 1] != kDead) {
          const uint32_t x = tb_base(p.words, s.a0, (long long)s.sa * (i - 1));
          const uint32_t y = tb_base(p.words, s.b0, (long long)s.sb * (j - 1));
          const int v = r2[i - 1] + (x == y ? p.M : p.S);
          if (v > h) {
            h = v;
            from = kMoveDiag;
          }
        }
        if (i >= 1 && i - 1 >= lo1 && i - 1 <= hi1 && r1[i - 1] != kDead && r1[i - 1] + p.G > h) {
          h = r1[i - 1] + p.G;
          from = kMoveA;
        }
        if (j >= 1 && i >= lo1 && i <= hi1 && r1[i] != kDead && r1[i] + p.G > h) {
          h = r1[i] + p.G;
          from = kMoveB;
        }
        live = h != kDead && h >= threshold;
        r0[i] = live ? h : kDead;
      }
      const uint32_t bits = live ? from : kMoveNone;
      const uint32_t wlo = __reduce_or_sync(kAll, lane < 16 ? bits << (2 * lane) : 0u);
      const uint32_t whi = __reduce_or_sync(kAll, lane >= 16 ? bits << (2 * (lane - 16)) : 0u);
      const int c0 = i0 - lo;  // cell offset of the chunk; a multiple of 32
      if (keep && lane == 0) {
        mv[w + c0 / 16] = wlo;
        if (c0 + 16 < width) mv[w + c0 / 16 + 1] = whi;
      }
      const unsigned bl = __ballot_sync(kAll, live);
      if (bl) {
        if (new_lo < 0) new_lo = i0 + __ffs(bl) - 1;
        new_hi = i0 + 31 - __clz(bl);
        const int cmax = __reduce_max_sync(kAll, live ? h : kDead);
        if (cmax > row_best) {  // strictly larger: an earlier chunk (smaller i) keeps a tie
          row_best = cmax;
          row_best_i = i0 + __ffs(__ballot_sync(kAll, live && h == cmax)) - 1;
        }
      }
    }
    e.cells += width;
    if (keep) {
      w += (width + 15) / 16;
      if (lane == 0) mv[w] = (uint32_t)width;
      w += 1;
    }
    __syncwarp();  // the row of d is complete before any lane reads it as d-1
    if (new_lo < 0) break;
    if (row_best > best) {
      best = row_best;
      e.best = best;
      e.i_end = row_best_i;
      e.j_end = d - row_best_i;
      e.best_rec = rec;
      e.recorded = keep;
    }
    live_lo = new_lo;
    live_hi = new_hi;
    int32_t* t = r2;  // rotate: d-1 -> d-2, d -> d-1
    r2 = r1;
    r1 = r0;
    r0 = t;
    lo2 = lo1;
    hi2 = hi1;
    lo1 = lo;
    hi1 = hi;
  }
  return e;
}

// Run-length writer over one seed's op words.
struct TbRuns {
  uint32_t* out;
  int cap;
  int n;       // runs written
  bool full;   // more runs than cap were needed
  uint32_t op;  // pending run
  uint32_t len;
  __host__ __device__ void push(uint32_t o) { push_run(o, 1); }
  __host__ __device__ void push_run(uint32_t o, uint32_t l) {
    if (len && o == op) {
      len += l;
      return;
    }
    flush();
    op = o;
    len = l;
  }
  __host__ __device__ void flush() {
    if (!len) return;
    if (n < cap)
      out[n] = (len << 4) | op;
    else
      full = true;
    ++n;
    len = 0;
  }
};

// Walks back from the extension's best cell to the origin, pushing each
// column's op.  Returns false if a visited cell lies outside its recorded
// band or has no move.
__host__ __device__ bool tb_walk(const TbArgs& p, const TbSeq& s, const TbExt& e, const uint32_t* mv, TbRuns* runs) {
  int i = e.i_end, j = e.j_end;
  long long rec = e.best_rec;
  while (i > 0 || j > 0) {
    if (rec < 0) return false;
    const int lo = (int)mv[rec], width = (int)mv[rec + 1];
    const int c = i - lo;
    if (c < 0 || c >= width) return false;
    const uint32_t move = (mv[rec + 2 + c / 16] >> (2 * (c & 15))) & 3u;
    int steps;  // antidiagonals stepped back
    if (move == kMoveDiag) {
      const uint32_t x = tb_base(p.words, s.a0, (long long)s.sa * (i - 1));
      const uint32_t y = tb_base(p.words, s.b0, (long long)s.sb * (j - 1));
      runs->push(x == y ? kOpEq : kOpX);
      --i;
      --j;
      steps = 2;
    } else if (move == kMoveA) {
      runs->push(kOpDel);
      --i;
      steps = 1;
    } else if (move == kMoveB) {
      runs->push(kOpIns);
      --j;
      steps = 1;
    } else {
      return false;
    }
    if (i == 0 && j == 0) break;
    for (int t = 0; t < steps; ++t) {  // the record before starts after its trailer
      if (rec < 1) return false;
      const long long prev_width = mv[rec - 1];
      rec -= 3 + (prev_width + 15) / 16;
    }
  }
  return true;
}

// ---- bit-sliced form ---------------------------------------------------------
// Its slot: a word for each antidiagonal (lanes that hold its band | place of
// the first one's lowest cell / 32, see below), where the general form has its
// rows, and the move words: two (hi, lo) of each such lane, antidiagonal after
// antidiagonal.  Those take no more words than the general form's records
// (2 T <= 3 + ceil(width / 16) for a band of any width over T words), so what
// fits is decided by the general form's count.  The window moves by whole words,
// so that the lowest cell of a lane's word is i = (d + 1) / 2 + 32 q.
constexpr int kTbWin = 1024;

struct TbBits {
  int best, i_end, j_end;
  long long cells;
  long long best_off;  // the best antidiagonal's first move word
  bool recorded;       // every antidiagonal up to the best one fit
};

// The extension of a (ascending from a0) and b (descending from b0) by the
// whole warp; false if its band outgrew the window.
template <int NB>
__device__ bool tb_extend_bits(const TbArgs& p, long long a0, long long b0, int m, int n, const uint32_t (&kx)[NB],
                               uint32_t* head, uint32_t* moves, TbBits& e) {
  using F = BitForm<NB, 1>;
  constexpr int kMargin = 17;  // 32 antidiagonals between looks: at most 16 places either way
  const int lane = threadIdx.x & 31;
  const GroupMasks gm = group_masks(lane, 0, 32);
  typename F::Lane L;
  F::clear(L);
  F::init(L, kTbWin / 2 - 32 * lane);
  int f0 = -kTbWin / 2;
  long long off = 0, used = 0, imp_off = 0;
  bool keep = true, imp_keep = true;
  e.i_end = e.j_end = 0;
  e.cells = 0;
  auto record = [&](const BitMoves<1>& mv) {
    const unsigned bal = __ballot_sync(kFull, mv.band[0] != 0);
    if (bal == 0) return;
    const int width = __reduce_add_sync(kFull, __popc(mv.band[0]));
    const int t = __popc(bal), first = __ffs((int)bal) - 1;
    e.cells += width;
    const int rec = 3 + ((width + 15) >> 4);
    keep = keep && used + rec <= p.moves_words;
    if (L.imp_d == L.d) {
      imp_off = off;
      imp_keep = keep;
    }
    if (!keep) return;
    used += rec;
    if (lane == 0) head[L.d] = (uint32_t)t | ((uint32_t)((f0 >> 5) + first) << 6);
    if (mv.band[0] != 0) *(uint2*)(moves + off + 2 * (lane - first)) = make_uint2(mv.hi[0], mv.lo[0]);
    off += 2 * t;
  };
  F::load_window(L, p.words, a0, b0, m, n, f0 + 32 * lane, 0);
  for (;;) {
    F::load_feed(L, p.words, a0, b0, m, n, f0 + ((L.d + 1) >> 1) + 32 * lane, L.d);
#pragma unroll 1
    for (int k = 0; k < 32; k += 2) {
      BitMoves<1> mv;
      F::template step<true, true>(L, L.r[0], L.r[1], kx, gm, &mv);
      record(mv);
      F::template step<false, true>(L, L.r[1], L.r[0], kx, gm, &mv);
      record(mv);
    }
    const uint32_t live[1] = {~L.dead[0]};
    int lo, hi;
    group_ends<1>(live, lane, 0, kFull, lo, hi);
    if (lo >= kMargin && hi <= kTbWin - 1 - kMargin) continue;
    int at, at_hi;
    group_ends<1>(L.imp, lane, 0, kFull, at, at_hi);
    if (L.imp_d >= 0) {
      e.i_end = f0 + ((L.imp_d + 1) >> 1) + at;
      e.j_end = L.imp_d - e.i_end;
    }
    L.imp_d = -1;
    if (lo < 0) break;
    const int by = ((lo + hi) / 2 - kTbWin / 2 + (lo < kMargin ? -16 : 16)) / 32;
    if (lo - 32 * by < kMargin || hi - 32 * by > kTbWin - 1 - kMargin) return false;
    const int src = lane + by;
    const bool held = src >= 0 && src < 32;
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      const uint32_t x = __shfl_sync(kFull, L.r[0][0][k], src & 31), y = __shfl_sync(kFull, L.r[1][0][k], src & 31);
      L.r[0][0][k] = held ? x : F::dead_plane(k);
      L.r[1][0][k] = held ? y : F::dead_plane(k);
    }
    const uint32_t dd = __shfl_sync(kFull, L.dead[0], src & 31);
    L.dead[0] = held ? dd : 0xFFFFFFFFu;
    f0 += 32 * by;
    F::load_window(L, p.words, a0, b0, m, n, f0 + ((L.d + 1) >> 1) + 32 * lane, L.d);
  }
  e.best = L.best;
  e.best_off = imp_off;
  e.recorded = imp_keep;
  __syncwarp();  // the records are read by other lanes
  return true;
}

// A run-length writer whose state all lanes of a group hold; its first lane
// writes, run x to out[step * x].
struct TbWarpRuns {
  uint32_t* out;
  long long cap;
  int step;
  bool writer;
  int n;
  uint32_t op, len;
  __device__ void push(uint32_t o, uint32_t l) {
    if (len && o == op) {
      len += l;
      return;
    }
    flush();
    op = o;
    len = l;
  }
  __device__ void flush() {
    if (!len) return;
    if (writer && n < cap) out[(long long)step * n] = (len << 4) | op;
    ++n;
    len = 0;
  }
};

// The columns from cell (i, j), whose antidiagonal's move words start at off,
// back to the origin.  A group is G lanes (16: two walks at once, or 32); lane l
// of it takes the antidiagonals d - l (and d - l - 16) of the next 32 and loads
// the two words that the path can meet there, so that a column is a look-up of
// every lane and one shuffle.  The words of a downward stream lie below `moves`.
template <int G>
__device__ void tb_walk_bits(const uint32_t* head, const uint32_t* moves, bool down, int i, int j, long long off,
                             TbWarpRuns& runs) {
  constexpr int U = 32 / G;
  const int gl = threadIdx.x & (G - 1);
  int d = i + j;
  while (__any_sync(kFull, d > 0)) {
    const int d0 = d;
    int i0[U], w[U], before = 0;
    long long mine[U];
    uint2 top[U], low[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int dl = d - gl - G * u;
      const uint32_t h = dl >= 1 ? head[dl] : 0u;
      const int t = (int)(h & 63u);
      int s = t;  // words of the antidiagonals from d down to this one
#pragma unroll
      for (int o = 1; o < G; o <<= 1) {
        const int v = __shfl_up_sync(kFull, s, o, G);
        if (gl >= o) s += v;
      }
      s += before;
      before = __shfl_sync(kFull, s, G - 1, G);
      if (u == 0) off += 2 * __shfl_sync(kFull, t, 0, G);
      mine[u] = off - 2ll * s;
      i0[u] = ((dl + 1) >> 1) + 32 * ((int)h >> 6);
      w[u] = (i - i0[u]) >> 5;  // the path meets [i - 31, i]: words w and w - 1
      const uint2 zero = make_uint2(0, 0);
      const long long at = mine[u] + 2 * w[u];
      top[u] = w[u] >= 0 && w[u] < t ? *(const uint2*)(moves + (down ? -2 - at : at)) : zero;
      low[u] = w[u] >= 1 && w[u] - 1 < t ? *(const uint2*)(moves + (down ? -at : at - 2)) : zero;
    }
    // From the present cell (antidiagonal d0 - x) every lane looks up the move of
    // the cell that a run of diagonal steps would reach on its antidiagonal (the
    // diagonal keeps to every other one): the lowest of them with another move
    // ends the run, and that move follows it.
    while (__any_sync(kFull, d > 0 && d > d0 - 30)) {
      const int x = d0 - d;
      uint32_t gap = 0, eq = 0;  // bit l: antidiagonal d0 - l
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int pos = i - ((gl + G * u - x) >> 1) - i0[u];
        const bool at_top = (pos >> 5) == w[u];
        const uint32_t hi = at_top ? top[u].x : low[u].x, lo = at_top ? top[u].y : low[u].y;
        const unsigned bh = __ballot_sync(kFull, (hi >> (pos & 31)) & 1u), bl = __ballot_sync(kFull, (lo >> (pos & 31)) & 1u);
        if (G == 32) {
          gap = bh;
          eq = bl;
        } else {
          gap |= ((bh >> (threadIdx.x & 16)) & 0xFFFFu) << (G * u);
          eq |= ((bl >> (threadIdx.x & 16)) & 0xFFFFu) << (G * u);
        }
      }
      if (d > 0 && d > d0 - 30) {
        const int stop = min(30 + (x & 1), d0);
        const uint32_t ends = gap & (0x55555555u << (x & 1)) & (0xFFFFFFFFu << x);
        const int at = ends ? __ffs((int)ends) - 1 : 32;
        int r = (min(at, stop) - x) >> 1;  // diagonal steps
        i -= r;
        j -= r;
        uint32_t same = (eq >> x) & 0x55555555u;
        while (r > 0) {
          const bool is = same & 1u;
          const uint32_t other = is ? ~same & 0x55555555u : same;
          const int c = min(r, other ? (__ffs((int)other) - 1) >> 1 : 16);
          runs.push(is ? kOpEq : kOpX, (uint32_t)c);
          same = shr_clamp(same, 2u * (uint32_t)c);
          r -= c;
        }
        if (at < stop) {
          const bool in_b = (eq >> at) & 1u;
          runs.push(in_b ? kOpIns : kOpDel, 1);
          i -= !in_b;
          j -= in_b;
        }
        d = i + j;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const long long v = __shfl_sync(kFull, mine[u], (d0 - d) & (G - 1), G);
      off = (d0 - d) / G == u ? v : off;
    }
  }
}

// Left (lanes 0-15) and right extension (lanes 16-31) of a seed at once, 16
// words of cells each: both share the slot, the left one's move words growing up
// from `moves`, the right one's down from `end`, and head (the right one's
// antidiagonals after the left one's).  Whether everything fits is decided on an
// upper bound of the general form's count; false if that or a window does not do
// (the caller then takes the extensions one after the other).
template <int NB>
__device__ bool tb_extend_both(const TbArgs& p, long long a0, long long b0, int m, int n, const uint32_t (&kx)[NB],
                               uint32_t* head, uint32_t* moves, uint32_t* end, TbBits& e) {
  using F = BitForm<NB, 1>;
  constexpr int kMargin = 17, kWin = 512;
  const int lane = threadIdx.x & 31, first = lane & 16, gl = lane & 15;
  const bool down = first != 0;
  const GroupMasks gm = group_masks(lane, first, 16);
  typename F::Lane L;
  F::clear(L);
  F::init(L, kWin / 2 - 32 * gl);
  int f0 = -kWin / 2;
  int off = 0, imp_off = 0;
  e.i_end = e.j_end = 0;
  uint2* const base = (uint2*)(down ? end - 2 : moves);
  const long long room = end - moves < (1ll << 30) ? end - moves : (1ll << 30);
  auto record = [&](const BitMoves<1>& mv) {
    const unsigned bal = __ballot_sync(kFull, mv.band[0] != 0) & gm.grp;
    const int t = __popc(bal), at = __ffs((int)bal) - 1;
    imp_off = L.imp_d == L.d ? off : imp_off;
    if (bal && gl == 0) head[L.d] = (uint32_t)t | ((uint32_t)((f0 >> 5) + at - first) << 6);
    const int o = off + lane - at;
    if (mv.band[0] != 0) base[down ? -o : o] = make_uint2(mv.hi[0], mv.lo[0]);
    off += t;
  };
  F::load_window(L, p.words, a0, b0, m, n, f0 + 32 * gl, 0);
  for (;;) {
    // Room for 32 antidiagonals of 16 words on both sides.
    const int other = __shfl_xor_sync(kFull, off, 16);
    if (__any_sync(kFull, 2ll * (off + other + 2 * 32 * 16) > room ||
                              2ll * (off + 32 * 16) + 3ll * (L.d + 32) > p.moves_words))
      return false;
    F::load_feed(L, p.words, a0, b0, m, n, f0 + ((L.d + 1) >> 1) + 32 * gl, L.d);
#pragma unroll 1
    for (int k = 0; k < 32; k += 2) {
      BitMoves<1> mv;
      F::template step<true, true>(L, L.r[0], L.r[1], kx, gm, &mv);
      record(mv);
      F::template step<false, true>(L, L.r[1], L.r[0], kx, gm, &mv);
      record(mv);
    }
    const uint32_t live[1] = {~L.dead[0]};
    int lo, hi;
    group_ends<1>(live, lane, first, gm.grp, lo, hi);
    const bool done = lo < 0, near_end = !done && (lo < kMargin || hi > kWin - 1 - kMargin);
    if (__any_sync(kFull, near_end) || __all_sync(kFull, done)) {
      int at, at_hi;
      group_ends<1>(L.imp, lane, first, gm.grp, at, at_hi);
      if (L.imp_d >= 0) {
        e.i_end = f0 + ((L.imp_d + 1) >> 1) + at;
        e.j_end = L.imp_d - e.i_end;
      }
      L.imp_d = -1;
      L.imp[0] = 0;
      if (__all_sync(kFull, done)) break;
      const int by = near_end ? ((lo + hi) / 2 - kWin / 2 + (lo < kMargin ? -16 : 16)) / 32 : 0;
      if (__any_sync(kFull, near_end && (lo - 32 * by < kMargin || hi - 32 * by > kWin - 1 - kMargin))) return false;
      const int src = gl + by;
      const bool held = src >= 0 && src < 16;
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        const uint32_t x = __shfl_sync(kFull, L.r[0][0][k], src & 15, 16), y = __shfl_sync(kFull, L.r[1][0][k], src & 15, 16);
        L.r[0][0][k] = held ? x : F::dead_plane(k);
        L.r[1][0][k] = held ? y : F::dead_plane(k);
      }
      const uint32_t dd = __shfl_sync(kFull, L.dead[0], src & 15, 16);
      L.dead[0] = held ? dd : 0xFFFFFFFFu;
      f0 += 32 * by;
      F::load_window(L, p.words, a0, b0, m, n, f0 + ((L.d + 1) >> 1) + 32 * gl, L.d);
    }
  }
  long long cells = L.cells;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) cells += __shfl_xor_sync(kFull, cells, o);
  e.cells = cells;
  e.best = L.best;
  e.best_off = 2ll * imp_off;
  e.recorded = true;
  __syncwarp();  // the records are read by other lanes
  return true;
}

__device__ __forceinline__ TbBits tb_from_lane(const TbBits& e, int lane) {
  TbBits r;
  r.best = __shfl_sync(kFull, e.best, lane);
  r.i_end = __shfl_sync(kFull, e.i_end, lane);
  r.j_end = __shfl_sync(kFull, e.j_end, lane);
  r.cells = __shfl_sync(kFull, e.cells, lane);
  r.best_off = __shfl_sync(kFull, e.best_off, lane);
  r.recorded = true;
  return r;
}

// Seed t as tb_seed does it, in the bit-sliced form; false (results to be
// written by tb_seed) if a band outgrew its window.  The seed is valid.
template <int NB>
__device__ bool tb_seed_bits(const TbArgs& p, long long t, char* scratch, const dibella_pair_t& pr, long long lenA,
                             long long lenB) {
  const int lane = threadIdx.x & 31;
  const int k = p.k;
  uint32_t kx[NB];
  bits_threshold<NB>(p.X, kx);
  uint32_t* head = (uint32_t*)scratch;
  uint32_t* moves = head + ((2ll * p.max_len + 5) & ~1ll);
  const long long fA = p.word_offsets[pr.read_a] * 16, rA = fA + tb_copy_words(lenA) * 16;
  const long long fB = p.word_offsets[pr.read_b] * 16, rB = fB + tb_copy_words(lenB) * 16;
  const long long bp0 = pr.strand ? rB : fB;  // B', and its reverse complement
  const long long bc0 = pr.strand ? fB : rB;
  const long long pa = pr.pos_a;
  const long long pb = pr.strand ? lenB - pr.pos_b - k : (long long)pr.pos_b;
  const bool eq = lane < k && tb_base(p.words, fA, pa + lane) == tb_base(p.words, bp0, pb + lane);
  const unsigned seed_eq = __ballot_sync(kFull, eq);
  const int n_eq = __popc(seed_eq);
  // Left: a(x) = A[pa-1-x] from A's reverse complement, b(y) = B'[pb-1-y];
  // right: a(x) = A[pa+k+x], b(y) = B'[pb+k+y] from the other copy.
  const long long la = rA + (lenA - pa), lb = bp0 + pb - 1, ra = fA + pa + k, rb = bc0 + (lenB - 1 - pb - k);
  const int lm = (int)pa, ln = (int)pb, rm = (int)(lenA - pa - k), rn = (int)(lenB - pb - k);
  uint32_t* ops = p.ops + t * (long long)p.ops_per_seed;
  TbWarpRuns runs{ops, p.ops_per_seed, 1, lane == 0, 0, 0, 0};
  TbWarpRuns back{nullptr, 0, -1, lane == 0, 0, 0, 0};
  const uint32_t* back_last = nullptr;  // the right walk's last run; the others follow it, last to first
  TbBits el, er;
  bool ok = true;
  auto seed_columns = [&]() {
    for (int q = 0; q < k; ++q) runs.push((seed_eq >> q) & 1u ? kOpEq : kOpX, 1);
  };
  // The walk of the right extension writes its run x to its head[d - x], an
  // antidiagonal that it has left (a run is a column at least).
  const bool rt = lane >= 16;
  TbBits e;
  uint32_t* own = head + (rt ? lm + ln + 1 : 0);
  uint32_t* end = (uint32_t*)(scratch + 12ll * (p.max_len + 2) + 4 * p.moves_words);
  end -= (end - head) & 1;
  if (tb_extend_both<NB>(p, rt ? ra : la, rt ? rb : lb, rt ? rm : lm, rt ? rn : ln, kx, own, moves, end, e)) {
    const int d = e.i_end + e.j_end;
    TbWarpRuns both{rt ? own + d : ops, rt ? (long long)d : (long long)p.ops_per_seed, rt ? -1 : 1, (lane & 15) == 0,
                    0, 0, 0};
    tb_walk_bits<16>(own, rt ? end : moves, rt, e.i_end, e.j_end, e.best_off, both);
    if (rt) both.flush();
    __syncwarp();
    el = tb_from_lane(e, 0);
    er = tb_from_lane(e, 16);
    runs.n = __shfl_sync(kFull, both.n, 0);
    runs.op = __shfl_sync(kFull, both.op, 0);
    runs.len = __shfl_sync(kFull, both.len, 0);
    back.n = __shfl_sync(kFull, both.n, 16);
    back_last = head + (lm + ln + 1) + er.i_end + er.j_end - back.n + 1;
    seed_columns();
  } else {
    if (!tb_extend_bits<NB>(p, la, lb, lm, ln, kx, head, moves, el)) return false;
    ok = el.recorded;
    if (ok) {
      tb_walk_bits<32>(head, moves, false, el.i_end, el.j_end, el.best_off, runs);
      seed_columns();
    }
    __syncwarp();  // the left walk has read the records before the right extension rewrites them
    if (!tb_extend_bits<NB>(p, ra, rb, rm, rn, kx, head, moves, er)) return false;
    if (ok) ok = er.recorded;
    if (ok) {
      const int d = er.i_end + er.j_end;
      back.out = head + d;
      back.cap = d;
      tb_walk_bits<32>(head, moves, false, er.i_end, er.j_end, er.best_off, back);
      back.flush();
      __syncwarp();
      back_last = head + d - back.n + 1;
    }
  }
  if (back.n > 0) {  // the first may join the seed's last run; the others follow as they are
    const uint32_t w = back_last[0];
    runs.push(w & 15u, w >> 4);
    runs.flush();
    for (int x = lane; x < back.n - 1; x += 32)
      if (runs.n + x < runs.cap) runs.out[runs.n + x] = back_last[1 + x];
    runs.n += back.n - 1;
  }
  runs.flush();
  if (lane == 0) {
    dibella_result_t r;
    r.score_left = el.best;
    r.score_right = er.best;
    r.score = n_eq * p.M + (k - n_eq) * p.S + el.best + er.best;
    r.begin_a = (uint32_t)(pa - el.i_end);
    r.end_a = (uint32_t)(pa + k + er.i_end);
    const long long bb = pb - el.j_end, eb = pb + k + er.j_end;
    r.begin_b = (uint32_t)(pr.strand ? lenB - eb : bb);
    r.end_b = (uint32_t)(pr.strand ? lenB - bb : eb);
    r.status = n_eq == k ? 0 : DIBELLA_RES_SEED_MISMATCH;
    r.cells = el.cells + er.cells;
    p.results[t] = r;
    p.n_ops[t] = !ok ? -2 : (runs.n > runs.cap ? -1 : runs.n);
  }
  __syncwarp();
  return true;
}

// Everything for seed t with one warp and its workspace slot: the result
// record (as dibella_xdrop_batch writes it, without the best-of-pair flag) and
// the run-length encoded columns from (begin_a, begin_b') to (end_a, end_b').
// Every lane runs both extensions; lane 0 walks back and writes.  NB > 0: in the
// bit-sliced form where its window holds the bands.
template <int NB>
__device__ void tb_seed(const TbArgs& p, long long t, char* scratch) {
  const int lane = threadIdx.x & 31;
  const dibella_pair_t pr = p.pairs[t];
  dibella_result_t r;
  r.score = r.score_left = r.score_right = 0;
  r.begin_a = r.end_a = r.begin_b = r.end_b = 0;
  r.status = 0;
  r.cells = 0;
  const int k = p.k;
  bool valid = (long long)pr.read_a < p.n_reads && (long long)pr.read_b < p.n_reads && pr.strand <= 1;
  long long lenA = 0, lenB = 0;
  if (valid) {
    lenA = p.lengths[pr.read_a];
    lenB = p.lengths[pr.read_b];
    valid = (long long)pr.pos_a + k <= lenA && (long long)pr.pos_b + k <= lenB;
  }
  if (!valid) {
    r.status = DIBELLA_RES_INVALID_SEED;
    if (lane == 0) {
      p.results[t] = r;
      p.n_ops[t] = 0;
    }
    return;
  }
  if (lenA > p.max_len || lenB > p.max_len) {  // the H rows would not hold the band
    r.status = DIBELLA_RES_BAND_OVERFLOW;
    if (lane == 0) {
      p.results[t] = r;
      p.n_ops[t] = -3;
    }
    return;
  }
  if (NB > 0 && tb_seed_bits<(NB > 0 ? NB : 4)>(p, t, scratch, pr, lenA, lenB)) return;
  const long long fA = p.word_offsets[pr.read_a] * 16;
  const long long fB = p.word_offsets[pr.read_b] * 16;
  const long long bp0 = pr.strand ? fB + tb_copy_words(lenB) * 16 : fB;  // B': forward or reverse-complement copy
  const long long pa = pr.pos_a;
  const long long pb = pr.strand ? lenB - pr.pos_b - k : (long long)pr.pos_b;
  int seed = 0;
  bool exact = true;
  for (int q = 0; q < k; ++q) {
    const bool eq = tb_base(p.words, fA, pa + q) == tb_base(p.words, bp0, pb + q);
    seed += eq ? p.M : p.S;
    exact = exact && eq;
  }
  const long long hw = (long long)p.max_len + 2;
  int32_t* rows = (int32_t*)scratch;
  uint32_t* mv = (uint32_t*)(scratch + 3 * hw * 4);
  // Left: a(i) = A[pa-1-i], b(j) = B'[pb-1-j]; right: a(i) = A[pa+k+i], b(j) = B'[pb+k+j].
  const TbSeq L{fA + pa - 1, bp0 + pb - 1, -1, -1, (int)pa, (int)pb};
  const TbSeq R{fA + pa + k, bp0 + pb + k, 1, 1, (int)(lenA - pa - k), (int)(lenB - pb - k)};
  TbRuns runs{p.ops + t * (long long)p.ops_per_seed, p.ops_per_seed, 0, false, 0, 0};
  bool ok = true;
  // The left walk runs from its best cell (the alignment's start) toward the
  // seed: its columns come out in alignment order.
  const TbExt el = tb_extend_warp(p, L, rows, rows + hw, rows + 2 * hw, mv, p.moves_words);
  if (lane == 0) {
    ok = el.recorded && tb_walk(p, L, el, mv, &runs);
    for (int q = 0; q < k && ok; ++q)
      runs.push(tb_base(p.words, fA, pa + q) == tb_base(p.words, bp0, pb + q) ? kOpEq : kOpX);
  }
  __syncwarp();  // the left walk has read the stream before the right extension rewrites it
  // The right walk yields its columns last to first: its runs go to the H
  // rows (free once the extension is done; at most m + n runs fit there),
  // then into the seed's runs in reverse order.
  const TbExt er = tb_extend_warp(p, R, rows, rows + hw, rows + 2 * hw, mv, p.moves_words);
  if (lane == 0) {
    if (ok) {
      TbRuns back{(uint32_t*)rows, (int)(3 * hw < 0x7FFFFFFF ? 3 * hw : 0x7FFFFFFF), 0, false, 0, 0};
      ok = er.recorded && tb_walk(p, R, er, mv, &back);
      back.flush();
      ok = ok && !back.full;
      for (int x = back.n - 1; x >= 0 && ok; --x) runs.push_run(back.out[x] & 15u, back.out[x] >> 4);
    }
    runs.flush();
  }
  r.score = seed + el.best + er.best;
  r.score_left = el.best;
  r.score_right = er.best;
  r.begin_a = (uint32_t)(pa - el.i_end);
  r.end_a = (uint32_t)(pa + k + er.i_end);
  const long long bb = pb - el.j_end, eb = pb + k + er.j_end;
  r.begin_b = (uint32_t)(pr.strand ? lenB - eb : bb);
  r.end_b = (uint32_t)(pr.strand ? lenB - bb : eb);
  r.status = exact ? 0 : DIBELLA_RES_SEED_MISMATCH;
  r.cells = el.cells + er.cells;
  if (lane == 0) {
    p.results[t] = r;
    p.n_ops[t] = !ok ? -2 : (runs.full ? -1 : runs.n);
  }
  __syncwarp();  // lane 0's use of the rows ends before the next seed
}

// A warp per seed: warp w (of n_lanes warps, one workspace slot each) takes
// seeds w, w + n_lanes, ...
template <int NB>
__global__ void __launch_bounds__(kTbThreads) traceback_kernel(TbArgs p) {
  const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  if (warp >= p.n_lanes) return;
  char* scratch = p.workspace + warp * p.lane_bytes;
  for (long long t = warp; t < p.n_pairs; t += p.n_lanes) tb_seed<NB>(p, t, scratch);
}

long long tb_lane_bytes(long long max_len, long long moves_words) {
  const long long b = 3 * (max_len + 2) * 4 + moves_words * 4;
  return (b + 255) / 256 * 256;
}

}  // namespace

extern "C" {

int dibella_traceback_workspace_bytes(int64_t n_lanes, int32_t max_read_len, int64_t moves_words,
                                      int64_t* bytes_out) {
  if (!bytes_out || n_lanes < 1 || n_lanes > (1ll << 24) || max_read_len < 0 ||
      max_read_len > DIBELLA_MAX_READ_LEN || moves_words < 2 || moves_words > (1ll << 34))
    return DIBELLA_EINVAL;
  *bytes_out = (int64_t)(n_lanes * tb_lane_bytes(max_read_len, moves_words));
  return DIBELLA_OK;
}

int dibella_xdrop_traceback(const uint32_t* packed_words, const int64_t* read_word_offsets,
                            const int32_t* read_lengths, int64_t n_reads, int32_t max_read_len,
                            const dibella_pair_t* pairs, int64_t n_pairs, int32_t k, dibella_scoring_t scoring,
                            dibella_result_t* results, uint32_t* ops, int32_t ops_per_seed, int32_t* n_ops,
                            int64_t n_lanes, int64_t moves_words, void* workspace, int64_t workspace_bytes,
                            void* stream) {
  if (n_reads < 0 || n_pairs < 0 || n_pairs > (1ll << 29) || k < 1 || k > DIBELLA_MAX_K) return DIBELLA_EINVAL;
  if (scoring.match <= 0 || scoring.match > DIBELLA_MAX_SCORE || scoring.mismatch > 0 ||
      scoring.mismatch < -DIBELLA_MAX_SCORE || scoring.gap >= 0 || scoring.gap < -DIBELLA_MAX_SCORE ||
      scoring.xdrop < 0 || scoring.xdrop > DIBELLA_XDROP_INF)
    return DIBELLA_EINVAL;
  if (ops_per_seed < 1 || max_read_len < 0 || max_read_len > DIBELLA_MAX_READ_LEN) return DIBELLA_EINVAL;
  int64_t need = 0;
  if (dibella_traceback_workspace_bytes(n_lanes, max_read_len, moves_words, &need) != DIBELLA_OK)
    return DIBELLA_EINVAL;
  if (n_pairs > 0 && (!packed_words || !read_word_offsets || !read_lengths || !pairs || !results || !ops ||
                      !n_ops))
    return DIBELLA_EINVAL;
  if (!workspace || ((uintptr_t)workspace & 255)) return DIBELLA_EINVAL;
  if (workspace_bytes < need) return DIBELLA_ENOMEM;
  if (n_pairs == 0) return DIBELLA_OK;
  TbArgs a;
  a.words = packed_words;
  a.word_offsets = read_word_offsets;
  a.lengths = read_lengths;
  a.n_reads = n_reads;
  a.pairs = pairs;
  a.n_pairs = n_pairs;
  a.k = k;
  a.M = scoring.match;
  a.S = scoring.mismatch;
  a.G = scoring.gap;
  a.X = scoring.xdrop;
  a.max_len = max_read_len;
  a.results = results;
  a.ops = ops;
  a.ops_per_seed = ops_per_seed;
  a.n_ops = n_ops;
  a.n_lanes = n_lanes < n_pairs ? n_lanes : n_pairs;
  a.moves_words = moves_words;
  a.workspace = (char*)workspace;
  a.lane_bytes = tb_lane_bytes(max_read_len, moves_words);
  // The bit-sliced form by the planes that X needs, as the batch does.
  const bool unit = a.M == 1 && a.S == -1 && a.G == -1 && a.X >= 1 && a.X <= 59;
  if (unit) {  // four blocks (16 warps) are resident on an SM: more slots would only run after them
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && sms > 0 &&
        a.n_lanes > 16ll * sms)
      a.n_lanes = 16ll * sms;
  }
  const long long blocks = (a.n_lanes * 32 + kTbThreads - 1) / kTbThreads;
  const auto kernel = !unit ? traceback_kernel<0>
                            : (a.X <= 11 ? traceback_kernel<4> : (a.X <= 27 ? traceback_kernel<5> : traceback_kernel<6>));
  kernel<<<(unsigned)blocks, kTbThreads, 0, (cudaStream_t)stream>>>(a);
  return cudaGetLastError() == cudaSuccess ? DIBELLA_OK : DIBELLA_ECUDA;
}

}  // extern "C"
