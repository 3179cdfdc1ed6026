// Bit-sliced X-drop extension for unit scores (match +1, mismatch -1, gap -1).
//
// Included inside an anonymous namespace that has kFull (the full lane mask) and
// ldg_word (a word of the packed store): the cells and one antidiagonal.  The
// batch's persistent kernels are built on it in xdrop_bits_run.cuh, the traceback
// in dibella_traceback.cu.  The code is per lane; a CPU test compiles it against
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
// 10 NB + 8 logic operations for 32 cells and lane, where the packed int16 form
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
// a lane) is about 97 instructions, 79 of them on that pipe at one per two cycles a
// scheduler; two warps a scheduler keep the pipe 85 to 92% busy (counters at X = 7,
// 25 and 50).  Memory traffic is at most four words of bases per lane and 32
// antidiagonals.
// Carrying r1 into the comparison with X instead of selecting X - r1, leaving the
// validity planes out of loops that stay inside the matrix, and one shift for the
// mask below the highest bit took it there from 107 and 89 (E. coli-sized batches
// 6 to 8% faster).  Batches in ms, this form / the int16 forms: E. coli-sized reads
// at X = 7 (400,000 seeds) 22.6 / 147 and at X = 25 (150,000) 46.6 / 369, the
// repeat-rich reads at X = 15 (150,000, on the device) 35.7 / 310, reads of 500 b
// to 100 kb at X = 50 (12,000) 55 to 71 / 380, one seed of 4 kb reads 0.16 / 1.2.

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

// All ones up to the highest set bit of x, 0 for x = 0.
__device__ __forceinline__ uint32_t ones_to_highest(uint32_t x) {
#ifdef XDROP_BITS_EMULATE
  return x ? 0xFFFFFFFFu >> __clz((int)x) : 0u;
#else
  uint32_t r;  // the shift is the leading zeros, or 2^32 - 1 for x = 0 (shr clamps at 32)
  asm("{ .reg .u32 t;\n bfind.shiftamt.u32 t, %1;\n shr.u32 %0, 0xFFFFFFFF, t; }" : "=r"(r) : "r"(x));
  return r;
#endif
}

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

template <int W>
struct BitMoves {
  uint32_t band[W], hi[W], lo[W];
};

template <int NB, int W>
struct BitForm {
  static constexpr int kMaxX = (1 << NB) - 5;
  __host__ __device__ static constexpr uint32_t dead_plane(int k) { return k == 0 ? 0u : 0xFFFFFFFFu; }
  using Lane = BitLane<NB, W>;

  // One antidiagonal: row P (d-1) and row Q (d-2, overwritten with d).
  // kx[k]: bit k of X as a mask.  CLIP: the window or what enters it reaches
  // beyond the matrix (else the validity planes are all ones and stay so).  With `moves` the cells' band
  // and the move that gave each its value (equal values: the diagonal first, then
  // the step in A, then the step in B') as two planes: 00 diagonal, 01 diagonal
  // on equal bases, 10 A, 11 B'.
  template <bool E, bool CLIP>
  __device__ static __forceinline__ void step(Lane& L, uint32_t (&P)[W][NB], uint32_t (&Q)[W][NB],
                                              const uint32_t (&kx)[NB], const GroupMasks& gm,
                                              BitMoves<W>* moves = nullptr) {
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
        if (CLIP) L.va[w] = __funnelshift_r(L.va[w], w + 1 < W ? L.va[w + 1 < W ? w + 1 : w] : L.fva, 1);
      }
      L.fa0 >>= 1;
      L.fa1 >>= 1;
      if (CLIP) L.fva >>= 1;
    } else {
#pragma unroll
      for (int w = W - 1; w >= 0; --w) {
        L.b0[w] = __funnelshift_l(w > 0 ? L.b0[w > 0 ? w - 1 : 0] : L.fb0, L.b0[w], 1);
        L.b1[w] = __funnelshift_l(w > 0 ? L.b1[w > 0 ? w - 1 : 0] : L.fb1, L.b1[w], 1);
        if (CLIP) L.vb[w] = __funnelshift_l(w > 0 ? L.vb[w > 0 ? w - 1 : 0] : L.fvb, L.vb[w], 1);
      }
      L.fb0 <<= 1;
      L.fb1 <<= 1;
      if (CLIP) L.fvb <<= 1;
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
        dn[w] = acc | ones_to_highest(x[w]);
        if (w > 0) acc |= x[w] ? 0xFFFFFFFFu : 0u;
      }
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const uint32_t u = up | x[w] | (0u - x[w]);
        if (w + 1 < W) up |= x[w] ? 0xFFFFFFFFu : 0u;
        band[w] = CLIP ? u & dn[w] & L.va[w] & L.vb[w] : u & dn[w];
        L.cells += __popc(band[w]);
      }
    }
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
      // g = min of the two gap predecessors: at E, P is the one above (the step in
      // A) and its shift the one to the left (the step in B'); at O the reverse.
      // from_b: the step in B' is strictly better.
      uint32_t s[NB], g[NB], from_b = 0;
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        s[k] = E ? __funnelshift_r(P[w][k], w + 1 < W ? P[w + 1 < W ? w + 1 : w][k] : nb[k], 1)
                 : __funnelshift_l(w > 0 ? P[w > 0 ? w - 1 : 0][k] : nb[k], P[w][k], 1);
        const uint32_t up = E ? P[w][k] : s[k], left = E ? s[k] : P[w][k];
        // borrow of left - up
        from_b = k == 0 ? (~left & up) : lop3<(lnot(kLA) & kLB) | (lnot(kLA ^ kLB) & kLC)>(left, up, from_b);
      }
#pragma unroll
      for (int k = 0; k < NB; ++k)
        g[k] = lop3<(kLA & kLB) | (lnot(kLA) & kLC)>(from_b, E ? s[k] : P[w][k], E ? P[w][k] : s[k]);
      // m = min(q, g), a borrowed q below everything; gap: g is strictly better
      uint32_t gap = 0;
#pragma unroll
      for (int k = 0; k < NB; ++k)
        gap = k == 0 ? (~g[0] & q[0]) : lop3<(lnot(kLA) & kLB) | (lnot(kLA ^ kLB) & kLC)>(g[k], q[k], gap);
      gap &= ~bor;
      if (moves != nullptr) {
        moves->band[w] = band[w];
        moves->hi[w] = gap;
        moves->lo[w] = lop3<(kLA & kLB) | (lnot(kLA) & kLC)>(gap, from_b, eq);
      }
      // gt: m > X - r1, i.e. m > X, or m = X and r1 (r1 carried in)
      uint32_t m[NB], gt = L.r1;
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        m[k] = lop3<(kLA & kLB) | (lnot(kLA) & kLC)>(gap, g[k], q[k]);
        gt = lop3<(kLA & lnot(kLB)) | (lnot(kLA ^ kLB) & kLC)>(m[k], kx[k], gt);
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

  // Whether the window or what enters it over the next 32 steps reaches beyond
  // the matrix in this lane (after load_window and load_feed).
  __device__ static __forceinline__ bool clipped(const Lane& L) {
    uint32_t all = (L.fva | 0xFFFF0000u) & (L.fvb | 0x0000FFFFu);
#pragma unroll
    for (int w = 0; w < W; ++w) all &= L.va[w] & L.vb[w];
    return all != 0xFFFFFFFFu;
  }

  // N antidiagonals, an even number, from a row at an even d.
  template <int N, bool CLIP>
  __device__ static __forceinline__ void steps(Lane& L, const uint32_t (&kx)[NB], const GroupMasks& gm) {
#pragma unroll 1
    for (int k = 0; k < N; k += 2) {
      step<true, CLIP>(L, L.r[0], L.r[1], kx, gm);
      step<false, CLIP>(L, L.r[1], L.r[0], kx, gm);
    }
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

template <int NB>
__device__ __forceinline__ void bits_threshold(int X, uint32_t (&kx)[NB]) {
#pragma unroll
  for (int k = 0; k < NB; ++k) kx[k] = (X >> k) & 1 ? 0xFFFFFFFFu : 0u;
}
