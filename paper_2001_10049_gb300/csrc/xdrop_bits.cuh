// Bit-sliced X-drop extension for unit scores (match +1, mismatch -1, gap -1).
//
// Included by dibella_xdrop.cu inside its anonymous namespace (it uses that
// file's Item and kFull).  The code is per lane; a CPU test compiles it against
// an emulation of the warp intrinsics.
//
// What a cell holds.  With best = the best score of all earlier antidiagonals,
// a live cell's drop best - H lies in [0, X], and on the antidiagonal that
// improves the best it is -1.  A cell is stored as s = drop + 1, in NB bits,
// relative to the best as it was before its own antidiagonal; a dead cell is
// kD = 2^NB - 2.  As both a mismatch and a gap cost 1,
//     s(d, i) = 1 + r1 + min(s(d-1, i-1), s(d-1, i), s(d-2, i-1) + r2 - 2 eq)
// where r1 (r2) is 1 if antidiagonal d-1 (d-2) improved the best: scores rise
// by at most 1 per diagonal step, so an antidiagonal improves the best by 0 or
// 1.  The cell is live iff the minimum is at most X - r1; the subtraction
// borrows exactly on the cells that reach best + 1 (when r1 = 0), whose lowest
// i is the argmax.  A dead cell's value stays above X through all of it while
// X <= 2^NB - 5.  Nothing here is approximate: the results are those of the
// int16 and int32 forms, cell counts included.
//
// How cells are laid out.  Bit t of plane k of a lane's word w is bit k of one
// cell, so one 3-input logic instruction works on 32 cells of a lane: about
// 10 NB + 8 instructions for 32 cells and lane, where the packed int16 form
// takes 9 for one cell and lane.  A group of G lanes with W words each holds a
// window of 32 G W consecutive cells of one extension.  The window moves up by
// one cell on every second antidiagonal (even steps "E" move it, odd steps "O"
// do not), so that the diagonal predecessor never needs a shift and the two
// gap predecessors need one shift of one row between them; of the two
// sequences only the one that enters on that side moves (a at E, b at O).
// Words shift into each other; across lanes the bit comes by one shuffle per
// plane.
//
// Band.  The cells evaluated on antidiagonal d run from the first live cell of
// d-1 to one past its last, clipped to the matrix: the live mask widened by a
// cell, filled between its ends (x | -x for the lower end, a leading-zero count
// for the upper one, one ballot for the lanes above and below), and masked
// with the validity planes that shift along with the sequences.  Its
// population count is the evaluated-cell count.  A finished extension has an
// empty band and changes nothing, so the ends are looked at only every T
// antidiagonals (a checkpoint), where the window is also moved back under the
// band if it has come near an end, the next bases are loaded, and an extension
// whose band no longer fits is handed on.

// What bounds it: the integer pipe.  An antidiagonal of a warp (5 planes, one word
// a lane) is 107 instructions, 89 of them on that pipe at one per two cycles a
// scheduler; a warp alone takes 234 cycles for it, and two warps a scheduler keep
// the pipe about 95% busy.  Memory traffic is one word of bases per lane and 32
// antidiagonals.  Batches in ms, this form / the int16 forms: E. coli-sized reads
// at X = 7 (400,000 seeds) 28.2 / 147 and at X = 25 (150,000) 53.5 / 365, the
// repeat-rich reads at X = 15 (150,000) 44 / 310, reads of 500 b to 100 kb at
// X = 50 (12,000) 73 / 380, one seed of 4 kb reads 0.16 / 1.2.

template <int LUT>
__device__ __forceinline__ uint32_t lop3(uint32_t a, uint32_t b, uint32_t c) {
#ifdef XDROP_BITS_EMULATE
  uint32_t r = 0;
  for (int i = 0; i < 8; ++i)
    if ((LUT >> i) & 1) r |= ((i & 4) ? a : ~a) & ((i & 2) ? b : ~b) & ((i & 1) ? c : ~c);
  return r;
#else
  uint32_t r;
  asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(r) : "r"(a), "r"(b), "r"(c), "n"(LUT));
  return r;
#endif
}
constexpr int kLA = 0xF0, kLB = 0xCC, kLC = 0xAA;  // truth tables of the three operands
__host__ __device__ constexpr int lnot(int x) { return ~x & 0xFF; }

// x >> n and x << n with n clamped at 32 (PTX shift semantics).
__device__ __forceinline__ uint32_t shr_clamp(uint32_t x, uint32_t n) { return __funnelshift_rc(x, 0u, n); }
__device__ __forceinline__ uint32_t shl_clamp(uint32_t x, uint32_t n) { return __funnelshift_lc(0u, x, n); }

// 16 bases (base q at bits 2q) to their low bits (bits 0-15) and high bits (16-31).
__device__ __forceinline__ uint32_t split_planes(uint32_t x) {
  uint32_t t;
  t = (x ^ (x >> 1)) & 0x22222222u; x ^= t ^ (t << 1);
  t = (x ^ (x >> 2)) & 0x0C0C0C0Cu; x ^= t ^ (t << 2);
  t = (x ^ (x >> 4)) & 0x00F000F0u; x ^= t ^ (t << 4);
  t = (x ^ (x >> 8)) & 0x0000FF00u; x ^= t ^ (t << 8);
  return x;
}

// The lanes of this lane's group, those of them below and above it, and all
// ones in the group's lowest / highest lane.
struct GroupMasks {
  uint32_t grp, low, high, end_lo, end_hi;
};

// Lanes first .. first + len - 1 form a group.
__device__ __forceinline__ GroupMasks group_masks(int lane, int first, int len) {
  GroupMasks g;
  g.grp = shr_clamp(0xFFFFFFFFu, (uint32_t)(32 - len)) << first;
  g.low = g.grp & ((1u << lane) - 1u);
  g.high = g.grp & ~((2u << lane) - 1u);
  g.end_lo = lane == first ? 0xFFFFFFFFu : 0u;
  g.end_hi = lane == first + len - 1 ? 0xFFFFFFFFu : 0u;
  return g;
}

// x / -x over a group: the place (bit of the group's window) of its lowest /
// highest set bit; -1 if there is none.  Every lane of the warp calls it.
template <int W>
__device__ __forceinline__ void group_ends(const uint32_t (&x)[W], int lane, int first, uint32_t grp, int& lo, int& hi) {
  uint32_t any = 0;
  int l = 0, h = 0;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    if (x[w]) {
      if (!any) l = 32 * (W * (lane - first) + w) + __ffs((int)x[w]) - 1;
      h = 32 * (W * (lane - first) + w) + 31 - __clz((int)x[w]);
    }
    any |= x[w];
  }
  const uint32_t bal = __ballot_sync(kFull, any != 0) & grp;
  l = __shfl_sync(kFull, l, bal ? __ffs((int)bal) - 1 : lane);
  h = __shfl_sync(kFull, h, bal ? 31 - __clz((int)bal) : lane);
  lo = bal ? l : -1;
  hi = bal ? h : -1;
}

template <int NB, int W>
struct BitLane {
  // r[row][word][plane]: r[0] is the newest antidiagonal at a checkpoint, r[1] the one before it.
  uint32_t r[2][W][NB];
  uint32_t dead[W];                  // dead cells of the newest antidiagonal
  uint32_t a0[W], a1[W], va[W];      // a[i-1] (two planes) and i <= m of the window's cells
  uint32_t b0[W], b1[W], vb[W];      // b[j-1] and j <= n
  uint32_t fa0, fa1, fva;            // what enters above the lane's window: next at bit 0
  uint32_t fb0, fb1, fvb;            // what enters below it: next at bit 31
  uint32_t r1, r2;                   // all ones if d-1 (d-2) improved the best
  uint32_t imp[W];                   // improving cells of the last improving step since the layout last changed
  int imp_d;                         // its antidiagonal, or -1
  int d;                             // the newest antidiagonal
  int best;
  uint32_t cells;                    // evaluated in this lane since the layout last changed
};

template <int NB, int W>
struct BitForm {
  static constexpr int kMaxX = (1 << NB) - 5;
  __host__ __device__ static constexpr uint32_t dead_plane(int k) { return k == 0 ? 0u : 0xFFFFFFFFu; }
  using Lane = BitLane<NB, W>;

  // One antidiagonal: row P (d-1) and row Q (d-2, overwritten with d).
  // kx[k] / ky[k]: bit k of X / X - 1 as a mask.
  template <bool E>
  __device__ static __forceinline__ void step(Lane& L, uint32_t (&P)[W][NB], uint32_t (&Q)[W][NB],
                                              const uint32_t (&kx)[NB], const uint32_t (&ky)[NB],
                                              const GroupMasks& gm) {
    // Neighbour lane's word for the one-cell shift (E: from above, O: from
    // below).  At a group's ends the plane bits that come in are whatever the
    // neighbour group holds: those places are outside every band.
    uint32_t nb[NB], nd;
#pragma unroll
    for (int k = 0; k < NB; ++k)
      nb[k] = E ? __shfl_down_sync(kFull, P[0][k], 1) : __shfl_up_sync(kFull, P[W - 1][k], 1);
    nd = E ? (__shfl_down_sync(kFull, L.dead[0], 1) | gm.end_hi) : (__shfl_up_sync(kFull, L.dead[W - 1], 1) | gm.end_lo);
    ++L.d;
    // Sequences.
    if (E) {
#pragma unroll
      for (int w = 0; w < W; ++w) {
        L.a0[w] = __funnelshift_r(L.a0[w], w + 1 < W ? L.a0[w + 1 < W ? w + 1 : w] : L.fa0, 1);
        L.a1[w] = __funnelshift_r(L.a1[w], w + 1 < W ? L.a1[w + 1 < W ? w + 1 : w] : L.fa1, 1);
        L.va[w] = __funnelshift_r(L.va[w], w + 1 < W ? L.va[w + 1 < W ? w + 1 : w] : L.fva, 1);
      }
      L.fa0 >>= 1;
      L.fa1 >>= 1;
      L.fva >>= 1;
    } else {
#pragma unroll
      for (int w = W - 1; w >= 0; --w) {
        L.b0[w] = __funnelshift_l(w > 0 ? L.b0[w > 0 ? w - 1 : 0] : L.fb0, L.b0[w], 1);
        L.b1[w] = __funnelshift_l(w > 0 ? L.b1[w > 0 ? w - 1 : 0] : L.fb1, L.b1[w], 1);
        L.vb[w] = __funnelshift_l(w > 0 ? L.vb[w > 0 ? w - 1 : 0] : L.fvb, L.vb[w], 1);
      }
      L.fb0 <<= 1;
      L.fb1 <<= 1;
      L.fvb <<= 1;
    }
    // Band: the live mask widened by a cell, filled between its ends.
    uint32_t band[W];
    {
      uint32_t x[W], any = 0;
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const uint32_t s = E ? __funnelshift_r(L.dead[w], w + 1 < W ? L.dead[w + 1 < W ? w + 1 : w] : nd, 1)
                             : __funnelshift_l(w > 0 ? L.dead[w > 0 ? w - 1 : 0] : nd, L.dead[w], 1);
        x[w] = ~(L.dead[w] & s);
        any |= x[w];
      }
      // all ones if a lower / higher lane of the group has a cell
      const uint32_t bal = __ballot_sync(kFull, any != 0);
      const uint32_t below = (bal & gm.low) ? 0xFFFFFFFFu : 0u, above = (bal & gm.high) ? 0xFFFFFFFFu : 0u;
      // lower end: x | -x over the lane's words; upper end: all ones below the highest set bit
      uint32_t up = below, dn[W];
      uint32_t acc = above;
#pragma unroll
      for (int w = W - 1; w >= 0; --w) {
        dn[w] = acc | shr_clamp(0xFFFFFFFFu, (uint32_t)__clz((int)x[w]));
        if (w > 0) acc |= x[w] ? 0xFFFFFFFFu : 0u;
      }
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const uint32_t u = up | x[w] | (0u - x[w]);
        if (w + 1 < W) up |= x[w] ? 0xFFFFFFFFu : 0u;
        band[w] = u & dn[w] & L.va[w] & L.vb[w];
        L.cells += __popc(band[w]);
      }
    }
    uint32_t kc[NB];  // bits of X - r1
#pragma unroll
    for (int k = 0; k < NB; ++k) kc[k] = lop3<(kLA & kLB) | (lnot(kLA) & kLC)>(L.r1, ky[k], kx[k]);
    uint32_t imp[W], any_imp = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const uint32_t t0 = L.a0[w] ^ L.b0[w];
      const uint32_t eq = lop3<(kLA ^ kLB) & kLC>(L.a1[w], L.b1[w], t0);
      // q = s(d-2) + r2 - 2 eq: the carry (eq = 0) or borrow (eq = 1) runs up the planes
      uint32_t q[NB];
      uint32_t c = lop3<kLA ^ (kLB & kLC)>(eq, Q[w][0], L.r2);
      q[0] = Q[w][0] ^ L.r2;
#pragma unroll
      for (int k = 1; k < NB; ++k) {
        q[k] = Q[w][k] ^ c;
        c = lop3<kLA & (kLB ^ kLC)>(c, Q[w][k], eq);
      }
      const uint32_t bor = c;  // s(d-2) + r2 - 2 eq = -1
      // g = min of the two gap predecessors
      uint32_t s[NB], g[NB], lt = 0;
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        s[k] = E ? __funnelshift_r(P[w][k], w + 1 < W ? P[w + 1 < W ? w + 1 : w][k] : nb[k], 1)
                 : __funnelshift_l(w > 0 ? P[w > 0 ? w - 1 : 0][k] : nb[k], P[w][k], 1);
        // borrow of P - s
        lt = k == 0 ? (~P[w][0] & s[0])
                    : lop3<(lnot(kLA) & kLB) | (lnot(kLA ^ kLB) & kLC)>(P[w][k], s[k], lt);
      }
#pragma unroll
      for (int k = 0; k < NB; ++k) g[k] = lop3<(kLA & kLB) | (lnot(kLA) & kLC)>(lt, P[w][k], s[k]);
      // m = min(q, g), a borrowed q below everything
      uint32_t lq = 0;
#pragma unroll
      for (int k = 0; k < NB; ++k)
        lq = k == 0 ? (~q[0] & g[0]) : lop3<(lnot(kLA) & kLB) | (lnot(kLA ^ kLB) & kLC)>(q[k], g[k], lq);
      lq |= bor;
      uint32_t m[NB], gt = 0;
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        m[k] = lop3<(kLA & kLB) | (lnot(kLA) & kLC)>(lq, q[k], g[k]);
        gt = k == 0 ? (m[0] & ~kc[0]) : lop3<(kLA & lnot(kLB)) | (lnot(kLA ^ kLB) & kLC)>(m[k], kc[k], gt);
      }
      const uint32_t dd = lop3<(kLA & lnot(kLB)) | lnot(kLC)>(gt, bor, band[w]);
      imp[w] = lop3<kLA & kLB & lnot(kLC)>(bor, band[w], L.r1);
      any_imp |= imp[w];
      // s(d) = m + 1 + r1, dead cells to kD
      Q[w][0] = lop3<lnot(kLA ^ kLB) & lnot(kLC)>(m[0], L.r1, dd);
      uint32_t cy = m[0] | L.r1;
#pragma unroll
      for (int k = 1; k < NB; ++k) {
        Q[w][k] = lop3<(kLA ^ kLB) | kLC>(m[k], cy, dd);
        cy &= m[k];
      }
      L.dead[w] = dd;
    }
    const uint32_t rn = (__ballot_sync(kFull, any_imp != 0) & gm.grp) ? 0xFFFFFFFFu : 0u;
    L.r2 = L.r1;
    L.r1 = rn;
#pragma unroll
    for (int w = 0; w < W; ++w) L.imp[w] = lop3<(kLA & kLB) | (lnot(kLA) & kLC)>(rn, imp[w], L.imp[w]);
    L.imp_d = rn ? L.d : L.imp_d;
    L.best -= (int)rn;
  }

  // The planes of 32 store bases from index idx on.
  __device__ static __forceinline__ void load32(const uint32_t* __restrict__ words, long long idx, uint32_t& p0,
                                                uint32_t& p1) {
    const long long w = idx >> 4;
    const unsigned sh = (unsigned)(idx & 15) * 2u;
    const uint32_t w0 = ldg_word(words, w), w1 = ldg_word(words, w + 1), w2 = ldg_word(words, w + 2);
    const uint32_t lo = split_planes(__funnelshift_r(w0, w1, sh)), hi = split_planes(__funnelshift_r(w1, w2, sh));
    p0 = __byte_perm(lo, hi, 0x5410);
    p1 = __byte_perm(lo, hi, 0x7632);
  }

  // Sequence and validity planes of the lane's window, whose lowest place is
  // cell i = fl of antidiagonal d.  Only words that hold a base of the
  // extension are read (at most 31 bases to either side of it).
  __device__ static __forceinline__ void load_window(Lane& L, const uint32_t* __restrict__ words, long long a0,
                                                     long long b0, int m, int n, int fl, int d) {
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const int i0 = fl + 32 * w;         // i of bit 0
      const int x0 = i0 - 1;              // a index of bit 0 (ascending)
      const int y0 = d - i0 - 1;          // b index of bit 0 (descending)
      L.a0[w] = L.a1[w] = L.b0[w] = L.b1[w] = 0;
      if (x0 + 31 >= 0 && x0 < m) load32(words, a0 + x0, L.a0[w], L.a1[w]);
      if (y0 >= 0 && y0 - 31 < n) load32(words, b0 - y0, L.b0[w], L.b1[w]);
      L.va[w] = shr_clamp(0xFFFFFFFFu, (uint32_t)max(31 - (m - i0), 0));
      L.vb[w] = shl_clamp(0xFFFFFFFFu, (uint32_t)max(d - i0 - n, 0));
    }
  }

  // What enters the lane's window over the next 32 steps (16 bases on each side).
  __device__ static __forceinline__ void load_feed(Lane& L, const uint32_t* __restrict__ words, long long a0,
                                                   long long b0, int m, int n, int fl, int d) {
    const int x = fl + 32 * W - 1;  // a index of the first base above
    const int y = d - fl;           // b index of the first base below
    L.fa0 = L.fa1 = L.fb0 = L.fb1 = 0;
    if (x + 15 >= 0 && x < m) {
      const long long idx = a0 + x;
      const uint32_t v = split_planes(__funnelshift_r(ldg_word(words, idx >> 4), ldg_word(words, (idx >> 4) + 1),
                                                      (unsigned)(idx & 15) * 2u));
      L.fa0 = v & 0xFFFFu;
      L.fa1 = v >> 16;
    }
    if (y + 15 >= 0 && y < n) {  // bases y+15 .. y, ascending in the store
      const long long idx = b0 - y - 15;
      const uint32_t v = split_planes(__funnelshift_r(ldg_word(words, idx >> 4), ldg_word(words, (idx >> 4) + 1),
                                                      (unsigned)(idx & 15) * 2u));
      L.fb0 = v << 16;
      L.fb1 = v & 0xFFFF0000u;
    }
    // a cell entering above has i = x + 1 + q <= m; one entering below has j = y + 1 + q <= n
    L.fva = shr_clamp(0xFFFFFFFFu, (uint32_t)min(max(32 - (m - x), 0), 32));
    L.fvb = shl_clamp(0xFFFFFFFFu, (uint32_t)min(max(32 - (n - y), 0), 32));
  }

  // Row d = 0 (cell (0,0), drop 0) at the window place that is bit `bit` of
  // this lane (in [0, 32 W), or outside it); nothing before it.  The lane's
  // sequences are not touched.
  __device__ static __forceinline__ void init(Lane& L, int bit) {
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const int t = bit - 32 * w;
      const uint32_t m = t >= 0 && t < 32 ? 1u << t : 0u;
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        L.r[0][w][k] = k == 0 ? m : ~m;
        L.r[1][w][k] = dead_plane(k);
      }
      L.dead[w] = ~m;
      L.imp[w] = 0;
    }
    L.r1 = L.r2 = 0;
    L.imp_d = -1;
    L.d = 0;
    L.best = 0;
    L.cells = 0;
  }
  // A lane without work: everything dead, now and in the steps to come.
  __device__ static __forceinline__ void clear(Lane& L) {
    init(L, -1);
#pragma unroll
    for (int w = 0; w < W; ++w) {
#pragma unroll
      for (int k = 0; k < NB; ++k) L.r[0][w][k] = dead_plane(k);
      L.a0[w] = L.a1[w] = L.b0[w] = L.b1[w] = L.va[w] = L.vb[w] = 0;
    }
    L.fa0 = L.fa1 = L.fb0 = L.fb1 = L.fva = L.fvb = 0;
  }
};

// What a group of lanes works on (the same in all its lanes).
struct BitTask {
  int item, m, n;
  int f0;        // the window's lowest place on antidiagonal d is i = f0 + (d + 1) / 2
  int bi, bj;    // cell of the best score
  long long a0, b0, cells;
  bool active;
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
// another window, so it says which: words `shift` .. shift + want - 1 counted
// from the first one held.  A queue entry is the pool offset (a multiple of 32)
// plus want - 1 (of at most 32 words), or -2 - item for an extension that starts
// over because the pool was full; -1 is a slot that is not written yet.
constexpr int kDumpHead = 16;
template <int NB>
__device__ __forceinline__ unsigned dump_words(int len) {
  return (unsigned)(kDumpHead + (2 * NB + 1) * len + 31) & ~31u;
}

// Writes the extension of lanes first .. first + len - 1 (W words each) to the
// pool and its entry to `queue` (null: none).  Every lane of the warp calls it;
// `mine` says whose group it is.  Returns the entry.
template <int NB, int W>
__device__ __forceinline__ int bits_suspend(const ExtendParams& p, const BitLane<NB, W>& L, const BitTask& t, bool mine,
                                             int lane, int first, int len, int shift, int want, int* queue,
                                             int q_id) {
  const bool leader = mine && lane == first;
  const unsigned size = dump_words<NB>(W * len);
  int off = -1;
  if (leader && *((volatile unsigned*)&p.cnt->pool) < p.pool_words) {
    const unsigned at = atomicAdd(&p.cnt->pool, size);
    if (at + size <= p.pool_words) off = (int)at;
  }
  off = __shfl_sync(kFull, off, first);
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
    if (off < 0) atomicAdd(&p.cnt->cells[7], (unsigned long long)t.cells);
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

// The rows of a suspended extension: this lane's word 0 is its word x (words
// outside it are dead).
template <int NB, int W>
__device__ __forceinline__ void bits_load(const ExtendParams& p, BitLane<NB, W>& L, int v, int x) {
  const uint32_t* o = p.pool + (v & ~31);
  BitForm<NB, W>::init(L, -1);
  L.d = (int)__ldcg(o + 1);
  L.best = (int)__ldcg(o + 3);
  L.r1 = __ldcg(o + 6);
  L.r2 = __ldcg(o + 7);
  const int len = (int)__ldcg(o + 8);
  o += kDumpHead;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const bool in = x + w >= 0 && x + w < len;
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      L.r[0][w][k] = in ? __ldcg(o + (2 * k) * len + x + w) : BitForm<NB, W>::dead_plane(k);
      L.r[1][w][k] = in ? __ldcg(o + (2 * k + 1) * len + x + w) : BitForm<NB, W>::dead_plane(k);
    }
    L.dead[w] = in ? __ldcg(o + 2 * NB * len + x + w) : 0xFFFFFFFFu;
  }
}

// Brings the group's cell count and best cell up to date (before its layout changes or it ends).
template <int NB, int W>
__device__ __forceinline__ void bits_settle(BitLane<NB, W>& L, BitTask& t, int lane, int first, int len,
                                            const GroupMasks& gm) {
  uint32_t s = L.cells;  // inclusive scan within the group
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_up_sync(kFull, s, o);
    if (lane - o >= first) s += v;
  }
  t.cells += __shfl_sync(kFull, s, first + len - 1);
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

template <int NB>
__device__ __forceinline__ void bits_threshold(int X, uint32_t (&kx)[NB], uint32_t (&ky)[NB]) {
#pragma unroll
  for (int k = 0; k < NB; ++k) {
    kx[k] = (X >> k) & 1 ? 0xFFFFFFFFu : 0u;
    ky[k] = ((X - 1) >> k) & 1 ? 0xFFFFFFFFu : 0u;
  }
}

constexpr int kCheck = 16;
constexpr int kMarginTrig = kCheck / 2 + 1;  // places of the window that a band may cross until the next look
constexpr int kMarginNew = 16;               // kept free at both ends of a window that is laid out anew
constexpr int kMarginKeep = 24;              // ... and of one that gives lanes back
constexpr int kInitLanes = 2;
#ifndef XDROP_BITS_SHARED_MAX  // (the CPU test lowers it, to reach the whole-warp form with short sequences)
#define XDROP_BITS_SHARED_MAX 32
#endif
constexpr int kSharedMax = XDROP_BITS_SHARED_MAX;  // lanes that one extension may take
constexpr int kNarrowAgain = 24 * kSharedMax;      // live cells below which the whole-warp form gives one back

// Whole-warp form: the extension of queue entry v by all 32 lanes, W words
// each, for a band that outgrows one word a lane.  With BACK it is suspended to
// the shared-lane form again once its band has become narrow; a band that
// outgrows this form too goes to esc_q (from W = 4 on: to the forms that hold
// scores, from the start).
template <int NB, int W, bool BACK>
__device__ __forceinline__ void bits_warp_one(const ExtendParams& p, int v, const uint32_t (&kx)[NB],
                                              const uint32_t (&ky)[NB]) {
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
    bits_load<NB, W>(p, L, v, W * lane - off);
    t.f0 -= 32 * off;
  } else {
    if (!t.active) return;
    F::init(L, kWin / 2 - 32 * W * lane);
  }
  F::load_window(L, words, t.a0, t.b0, t.m, t.n, t.window(L.d) + 32 * W * lane, L.d);
  for (;;) {
    F::load_feed(L, words, t.a0, t.b0, t.m, t.n, t.window(L.d) + 32 * W * lane, L.d);
#pragma unroll 1
    for (int k = 0; k < 32; k += 2) {
      F::template step<true>(L, L.r[0], L.r[1], kx, ky, gm);
      F::template step<false>(L, L.r[1], L.r[0], kx, ky, gm);
    }
    uint32_t live[W];
#pragma unroll
    for (int w = 0; w < W; ++w) live[w] = ~L.dead[w];
    int lo, hi;
    group_ends<W>(live, lane, 0, kFull, lo, hi);
    const bool narrow = BACK && lo >= 0 && hi - lo < kNarrowAgain;
    if (lo >= kMargin && hi <= kWin - 1 - kMargin && !narrow) continue;
    bits_settle<NB, W>(L, t, lane, 0, 32, gm);
    if (lo < 0) {  // ended
      if (lane == 0) bits_finish(p, t, L.best);
      break;
    }
    if (narrow) {
      const int b = (lo - kMarginNew) >> 5, e = (hi + kMarginNew) >> 5;
      bits_suspend<NB, W>(p, L, t, true, lane, 0, 32, b, e - b + 1, p.res_q, p.res_q_id);
      break;
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
  uint32_t kx[NB], ky[NB];
  bits_threshold<NB>(p.sc.X, kx, ky);
  const unsigned tail = *((volatile unsigned*)&p.cnt->tail[p.wide_q_id]);
  for (;;) {
    const unsigned q = pop_warp(p.cnt, p.wide_q_id);
    if (q >= tail) break;
    bits_warp_one<NB, W, false>(p, p.wide_q[q], kx, ky);
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
  uint32_t kx[NB], ky[NB];
  bits_threshold<NB>(p.sc.X, kx, ky);
  const unsigned tail = *((volatile unsigned*)&p.cnt->tail[p.wide_q_id]);
  const uint32_t* __restrict__ words = p.words;
  typename F::Lane L;
  F::clear(L);
  BitTask t;
  t.item = t.m = t.n = t.f0 = t.bi = t.bj = 0;
  t.a0 = t.b0 = t.cells = 0;
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
    // lanes wanted: words b .. b + want - 1 of the present window
    const bool trig = lo < kMarginTrig || hi > 32 * len - 1 - kMarginTrig;
    int b = (lo - (trig ? kMarginNew : kMarginKeep)) >> 5, e = (hi + (trig ? kMarginNew : kMarginKeep)) >> 5;
    if (!trig) {
      b = max(b, 0);
      e = min(e, len - 1);
    }
    int want = t.active && lane == first ? e - b + 1 : 0;
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
      bits_warp_one<NB, 2, true>(p, alone, kx, ky);
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
    while (groups < p.max_groups) {
      int v = -1;
      if (lane == 0) {
        for (;;) {
          const unsigned h = *((volatile unsigned*)&p.cnt->head[p.res_q_id]);
          if ((long long)h >= p.res_cap || h >= *((volatile unsigned*)&p.cnt->tail[p.res_q_id])) break;
          const int c = *((volatile int*)&p.res_q[h]);
          if (c == -1 || (c >= 0 ? (c & 31) + 1 : max(kInitLanes, p.reserve)) > room) break;
          if (atomicCAS(&p.cnt->head[p.res_q_id], h, h + 1) == h) {
            v = c;
            break;
          }
        }
      }
      v = __shfl_sync(kFull, v, 0);
      if (v == -1) break;
      __threadfence();  // its words were written before its queue entry
      const int l = v >= 0 ? (v & 31) + 1 : kInitLanes;
      if (lane >= used && lane < used + l) {
        entry = v;
        efirst = used;
        elen = l;
      }
      used += l;
      room -= v >= 0 ? l : max(kInitLanes, p.reserve);
      ++groups;
    }
    int n_new = exhausted ? 0 : min(room / p.reserve, p.max_groups - groups);
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
    const int src = from + shift + (lane - nfirst);
    const bool held = lane < total && src >= from && src < from + old_len;
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      const uint32_t x = __shfl_sync(kFull, L.r[0][0][k], src & 31), y = __shfl_sync(kFull, L.r[1][0][k], src & 31);
      L.r[0][0][k] = held ? x : F::dead_plane(k);
      L.r[1][0][k] = held ? y : F::dead_plane(k);
    }
    const uint32_t dd = __shfl_sync(kFull, L.dead[0], src & 31);
    L.dead[0] = held ? dd : 0xFFFFFFFFu;
    L.r1 = __shfl_sync(kFull, L.r1, from);
    L.r2 = __shfl_sync(kFull, L.r2, from);
    L.d = __shfl_sync(kFull, L.d, from);
    L.best = __shfl_sync(kFull, L.best, from);
    t.item = __shfl_sync(kFull, t.item, from);
    t.m = __shfl_sync(kFull, t.m, from);
    t.n = __shfl_sync(kFull, t.n, from);
    t.f0 = __shfl_sync(kFull, t.f0, from) + 32 * shift;
    t.bi = __shfl_sync(kFull, t.bi, from);
    t.bj = __shfl_sync(kFull, t.bj, from);
    t.a0 = __shfl_sync(kFull, t.a0, from);
    t.b0 = __shfl_sync(kFull, t.b0, from);
    t.cells = __shfl_sync(kFull, t.cells, from);
    t.active = lane < total;
    first = nfirst;
    len = old_want;
    if (elen > 0) {
      first = efirst;
      len = elen;
      if (bits_task(p, t, entry, -16 * kInitLanes)) {
        const int from_word = (int)__ldcg(p.pool + (entry & ~31) + 11);
        t.f0 += 32 * from_word;
        bits_load<NB, 1>(p, L, entry, lane - first + from_word);
      } else {
        F::init(L, 16 * kInitLanes - 32 * (lane - first));
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
      bool look = false;
#pragma unroll 1
      for (int h = 0; h < 32 && !look; h += kCheck) {
#pragma unroll 1
        for (int k = 0; k < kCheck; k += 2) {
          F::template step<true>(L, L.r[0], L.r[1], kx, ky, gm);
          F::template step<false>(L, L.r[1], L.r[0], kx, ky, gm);
        }
        const uint32_t any = __ballot_sync(kFull, L.dead[0] != 0xFFFFFFFFu);
        look = __any_sync(kFull, t.active && ((any & gm.grp) == 0 || (~L.dead[0] & near_end) != 0));
      }
      if (look) break;
    }
  }
}

