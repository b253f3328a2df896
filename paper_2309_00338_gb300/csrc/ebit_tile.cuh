// Tiled sweep kernel: one split sweep (Sec. 2.1-2.4) for a tile of the grid,
// marker-centric and bit-parallel in shared memory.
//
// Tile (sweep coordinates): vertices i in [i0, i0+64), j in [j0, j0+32) with
// their aligned edge (i,j), unaligned edge (i,j) and cell (i,j).  The region
// held in shared memory is the tile plus a halo, vertices
// [i0-4, i0+67] x [j0-2, j0+34] (72 x 37): candidate chords for line k come
// from cells k-2..k, their end markers' neighbours lie one cell further, the
// neighbours' next markers (points 1 and 4 when a neighbour is too close) one
// more, and the centre rule looks at landings on edges k-1..k+1.
//
// Colours are kept as bit rows (3 words per region row).  Marker sets,
// interface cells and new four-marker cells are word-level XORs of them, and
// all per-marker work runs from compacted lists, so a tile costs in
// proportion to the interface it holds:
//   P0 colour bits of the region (funnel shifts of the stored rows; for the y
//      sweep a warp-ballot transpose)
//   P1 marker bit sets; a tile with no marker in its region only copies its
//      colour words (P7)
//   P2 moved point of every marker (the only global reads of fractions and
//      velocities), kept by the marker's rank in its bit set; corner flips
//      (Fig. 5) by XOR into the new colour bits; landing edges claimed
//   P3 landings (Sec. 2.4), new aligned markers; list of the interface cells
//      whose chords can cross the tile's grid lines
//   P4 each chord of such a cell that crosses a grid line k of the tile
//      becomes a candidate of unaligned edge (k, j): references to A, B and
//      points 1-4, centre-rule verdicts; candidates are linked per edge
//   P5 circle fits (Sec. 2.2) of all candidates, two lanes each, so the FP64
//      pipe sees full warps
//   P6 one marker per edge from its linked candidates; new unaligned markers
//   P7 centre colours of the new four-marker cells (Sec. 2.3); colour words
#pragma once
#include "ebit_device.cuh"

namespace ebit {

constexpr int kTI = 64, kTJ = 32;
constexpr int kRX = kTI + 8, kRY = kTJ + 5;
constexpr int kRW = 3;                 // words per region bit row (72 columns used)
constexpr int kRB = kRY * kRW;         // words per region bit plane
constexpr int kNVE = (kTI + 1) * kTJ;  // unaligned edges k in [i0, i0+64], rows j0..j0+31
constexpr int kCandCap = 255;          // candidates per tile of the one-grid kernels (an
                                       // edge beyond it is done in place)
// A candidate list of CAP entries links them through heads of 8 bits (CAP
// <= 255) or 16 bits; the all-ones head marks an edge without a candidate.
template <int CAP> __host__ __device__ constexpr int head_bits() { return CAP <= 255 ? 8 : 16; }
template <int CAP> __host__ __device__ constexpr uint32_t head_none() {
  return (1u << head_bits<CAP>()) - 1u;
}
// A place of the region, (lx, ly), as 13 bits, taken apart without a division.
__device__ __forceinline__ int pack_xy(int lx, int ly) { return ly << 7 | lx; }
__device__ __forceinline__ int lx_of(int id) { return id & 127; }
__device__ __forceinline__ int ly_of(int id) { return (id >> 7) & 63; }
static_assert(kRX <= 128 && kRY <= 64, "places fit");
constexpr uint16_t kKindV = 0x8000;    // marker reference: place | kKindV if unaligned
constexpr int kSecond = 0x4000;        // segment reference: place of its cell | kSecond for the second
                                       // one of a four-marker cell

// Block shape: four warps per tile, seven tiles per SM in the FP32 form (72
// registers) and six in the FP64 form (80).  What a tile waits for is latency
// (barriers, the state's loads, the fits' FP64 chains), so many small blocks
// that are in different phases beat few large ones: 4096^2 cells, cellular
// flow over 20000 disks, microseconds a sweep in FP32 / FP64 form: 257 / 301
// with four warps, 265 / 310 with five at six and five tiles per SM, 267 / 308
// at six and five tiles of four warps, 262 / 300 at eight and seven (spills);
// seven warps at four and three tiles per SM, which the dense per-edge arrays
// of moved fractions allowed before markers were kept by rank: 306 / 397.
template <typename R> __host__ __device__ constexpr int tile_threads() { return 128; }
template <typename R> __host__ __device__ constexpr int tile_min_blocks();
template <> __host__ __device__ constexpr int tile_min_blocks<float>() { return 7; }
template <> __host__ __device__ constexpr int tile_min_blocks<double>() { return 6; }
// Moved fractions of a region kept in shared memory (tile_dense takes the tiles
// with more markers): as many as fit in the 196 KB that seven (six) tiles take
// anyway.  The next carve-out leaves less L1: a sweep of the case above took 251
// us against 239 in FP32, 301 against 292 in FP64.
template <typename R> __host__ __device__ constexpr int marker_cap() { return sizeof(R) == 4 ? 2048 : 1728; }
// Block shape of the batched kernels, whose code of both directions makes more
// warps share what each fetches: 256 uneven grids in one batch advance 2.12e10
// (FP32) and 1.69e10 (FP64) cells a second with six warps a tile, 2.02 and
// 1.64 with four, 2.10 and 1.70 with five, 2.03 and 1.66 with seven (four and
// three tiles per SM).
template <typename R> __host__ __device__ constexpr int batch_threads() { return 192; }
template <typename R> __host__ __device__ constexpr int batch_min_blocks() { return sizeof(R) == 4 ? 5 : 4; }
// Candidates per tile of the batched kernels: many small grids of uneven
// sizes hold more interface per tile than one large grid, and the longer
// list (16-bit heads) still leaves 5 (FP32) / 4 (FP64) tiles per SM.
template <typename R> __host__ __device__ constexpr int batch_cand_cap() {
  return sizeof(R) == 4 ? 511 : 383;
}

// Candidate of one unaligned edge: chord ends A (left of the line) and B,
// points 1 (p1) and 4 (p4); references to moved markers held in the tile.
// The marker beyond point 1 (or 4), used where that point is too close to A
// (B), and the centre-rule verdicts, used where the edge borders a new
// four-marker cell, are rare: they are formed from these references when
// needed (the chord's cell is k - 2 + ord / 2 of row j).
enum { CF_P1 = 1, CF_P4 = 4, CF_OWNED = 16 };
struct Cand {
  uint16_t a, b, p1, p4;
  uint16_t edge;  // pack_xy(k - i0, j - j0)
  uint8_t fl, ord;
};

// Shared memory of one tile (dynamic).  Arrays whose phases do not overlap
// share storage: the marker list of P1-P3 with the candidates of P4-P6 and the
// interface-cell list of P3-P4 with the verdicts of P6-P7.
template <typename R, int CAP = kCandCap>
struct TileMem {
  static_assert(CAP <= 65534, "candidate slots fit the 16-bit heads");
  static constexpr int kMkCap = marker_cap<R>();
  struct Cands {
    double y[CAP];           // P5-P6: where the candidates cross their lines
    Cand cand[CAP];          // P4-P6
    int16_t next[CAP];       // candidate links
    uint16_t le[CAP];        // P5-P6: unaligned edges with a linked candidate
  };
  static constexpr int kMkList = sizeof(Cands) / sizeof(uint16_t);
  static_assert(kMkList >= kMkCap, "as many markers as moved fractions");
  union {
    uint16_t mk[kMkList];    // P1-P3: place of every marker, by rank
    Cands c;
  } u;
  // moved markers' fraction along the sweep, by rank (an unaligned marker's one
  // across it is its own, read from the state)
  R fr[kMkCap];
  // first linked candidate of each unaligned edge, head_bits each (all ones: none)
  alignas(16) uint32_t head[kNVE * head_bits<CAP>() / 32];
  uint32_t kb[kRB];        // old corner colours
  uint32_t kn[kRB];        // new corner colours
  uint32_t zb[kRB];        // old centre colours (bit lx of row ly: cell (lx, ly))
  uint32_t hm[kRB];        // aligned markers (bit lx of row ly: edge (lx, ly))
  uint32_t vm[kRB];        // unaligned markers
  uint16_t hbase[kRB];     // rank of the first marker of each word
  uint16_t vbase[kRB];
  uint32_t claim[kRB];     // aligned edges some marker lands on
  uint32_t hc[kRB];        // unaligned edges with a linked candidate
  uint32_t ovf[kRB];       // unaligned edges done in place
  // 2-bit codes (planes 0 and 1): moved aligned / unaligned marker ix - x + 1,
  // landing kept source - i + 2 (0: none)
  uint32_t hq[2][kRB];
  uint32_t vq[2][kRB];
  uint32_t lq[2][kRB];
  union {
    uint16_t cl[kMkCap];   // P3-P4: the segments (at most one per marker: a marker ends two)
    // P5-P7: centre verdicts of an edge: bits 0-1 right + 1, bits 2-3 left + 1
    alignas(16) uint8_t vrl[kNVE];
  };
  // Rank of the marker on aligned (kind 0) or unaligned edge (lx, ly): aligned
  // ones first, each in region order.
  __device__ __forceinline__ int rank(int kind, int lx, int ly) const {
    const int w = ly * kRW + (lx >> 5);
    const uint32_t below = (1u << (lx & 31)) - 1u;
    return kind ? vbase[w] + __popc(vm[w] & below) : hbase[w] + __popc(hm[w] & below);
  }
};

template <typename R, int CAP = kCandCap>
constexpr size_t tile_smem_bytes() {
  return sizeof(TileMem<R, CAP>);
}

__device__ __forceinline__ int getb(const uint32_t* w, int lx, int ly) {
  return (w[ly * kRW + (lx >> 5)] >> (lx & 31)) & 1;
}

// Corner mask of region cell (lx, ly), counter-clockwise from its lower left
// (lx < kRX - 1, so the word after the one of lx only counts within its row).
__device__ __forceinline__ int corners4(const uint32_t* w, int lx, int ly) {
  const uint32_t* q = w + ly * kRW + (lx >> 5);
  const int lo = __funnelshift_r(q[0], q[1], lx & 31) & 3;
  const int up = __funnelshift_r(q[kRW], q[kRW + 1], lx & 31) & 3;
  return lo | ((up & 2) << 1) | ((up & 1) << 3);
}

// 2-bit code of region entry (lx, ly) held in two bit planes.
__device__ __forceinline__ int get2(const uint32_t (&q)[2][kRB], int lx, int ly) {
  const int w = ly * kRW + (lx >> 5), b = lx & 31;
  return ((q[0][w] >> b) & 1) | (((q[1][w] >> b) & 1) << 1);
}
__device__ __forceinline__ void put2(uint32_t (&q)[2][kRB], int lx, int ly, int code) {
  const int w = ly * kRW + (lx >> 5);
  const uint32_t bit = 1u << (lx & 31);
  if (code & 1) atomicOr(&q[0][w], bit);
  if (code & 2) atomicOr(&q[1][w], bit);
}

// Word wi of row ly shifted right by one column (bit b = column 32 wi + b + 1).
__device__ __forceinline__ uint32_t shr1(const uint32_t* w, int ly, int wi) {
  uint32_t v = w[ly * kRW + wi] >> 1;
  if (wi + 1 < kRW) v |= w[ly * kRW + wi + 1] << 31;
  return v;
}

__device__ __forceinline__ int verdict_r(uint8_t c) { return (int)(c & 3) - 1; }
__device__ __forceinline__ int verdict_l(uint8_t c) { return (int)((c >> 2) & 3) - 1; }
__device__ __forceinline__ uint8_t verdicts(int vr, int vl) {
  return (uint8_t)((vr + 1) | ((vl + 1) << 2));
}

constexpr unsigned kFull = 0xffffffffu;

// Exclusive offset of this lane's n in a block-shared list counter; one
// shared atomic per warp.  All 32 lanes call it.
__device__ __forceinline__ int warp_alloc(int n, int* count, int lane) {
  int incl = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += v;
  }
  const int total = __shfl_sync(kFull, incl, 31);
  int base = 0;
  if (lane == 31 && total) base = atomicAdd(count, total);
  return __shfl_sync(kFull, base, 31) + incl - n;
}

// Adds the lanes' v to the block's counter c, one shared atomic per warp (all
// 32 lanes call it).  Counts are kept per phase so that no counter stays live
// in registers across the kernel.
__device__ __forceinline__ void flush_count(int* s_cnt, int c, int v, int lane) {
  const int s = __reduce_add_sync(kFull, v);
  if (s != 0 && lane == 0) atomicAdd(&s_cnt[c], s);
}

// Appends the set bits of plane word t as region indices (with flag), for a
// whole warp (all 32 lanes call it).
__device__ __forceinline__ void push_bits_warp(uint32_t bits, int t, int flag, uint16_t* list,
                                               int* count, int lane) {
  int base = warp_alloc(__popc(bits), count, lane);
  const int row0 = pack_xy(32 * (t % kRW), t / kRW) | flag;
#pragma unroll 1
  while (bits) {
    const int b = __ffs(bits) - 1;
    bits &= bits - 1;
    list[base++] = (uint16_t)(row0 + b);  // the flag bits lie above every region index
  }
}

// 32 x 32 bit transpose across a warp: lane r holds row r (bit c = element
// (r, c)); returns column `lane` (bit r = element (r, lane)).
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane) {
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const int s = 16 >> q;
    const uint32_t m = q == 0 ? 0x0000ffffu : q == 1 ? 0x00ff00ffu : q == 2 ? 0x0f0f0f0fu
                     : q == 3 ? 0x33333333u : 0x55555555u;
    const uint32_t y = __shfl_xor_sync(kFull, x, s);
    x = (lane & s) ? ((x & ~m) | ((y & ~m) >> s)) : ((x & m) | ((y & m) << s));
  }
  return x;
}

// Bits c0 .. c0+31 of region row ly (c0 + 32 < 32 kRW).
__device__ __forceinline__ uint32_t bits32(const uint32_t* w, int ly, int c0) {
  const int q = c0 >> 5, r = c0 & 31;
  const uint32_t a = w[ly * kRW + q];
  return r ? ((a >> r) | (w[ly * kRW + q + 1] << (32 - r))) : a;
}

// Bits b of a 32-column window starting at column c0 with c0 + b <= last.
__device__ __forceinline__ uint32_t upto32(int c0, int last) {
  const int n = last - c0 + 1;
  return n <= 0 ? 0u : (n >= 32 ? kFull : ((1u << n) - 1u));
}


// n + f + kShift for a grid line number n and a fraction f (see xy_shifted);
// false unless f is +0 or in [2^-26, 1) (-0, whose sign bit counts as part of
// the exponent here, is not).
constexpr int kShift = 12;
__device__ __forceinline__ bool shifted_sum(int n, float f, double* s) {
  const unsigned u = __float_as_uint(f), e = u >> 23;
  const unsigned long long m = (unsigned long long)(u ? (u & 0x7fffffu) | 0x800000u : 0u) << ((e - 101u) & 31u);
  *s = __longlong_as_double((1026ll << 52) + ((long long)(n + kShift - 8) << 49) + (long long)m);
  return (unsigned)(n + 4) < 8u && (u == 0u || e - 101u < 26u);
}

// A marker's moved fraction once more, out of line.
template <typename R, int AX, int LD>
__device__ __noinline__ R fraction_again(const GView<R, AX, LD> G, int kind, int x, int y) {
  return G.moved(Mk{kind, x, y}).fx;
}

// Accessor of the tile for the shared sweep logic (beyond, walk,
// new_unaligned).  Indices are clamped into the region; the kernel only asks
// inside it.  MANY: there may be more markers than moved fractions kept.
template <typename R, int AX, int LD, int CAP, bool MANY>
struct TViewB {
  const TileMem<R, CAP>* m;
  GView<R, AX, LD> g;  // an unaligned marker's own fraction is read from the state
  int ri0, rj0, nx_, ny_;
  __device__ __forceinline__ int tnx() const { return nx_; }
  __device__ __forceinline__ int tny() const { return ny_; }
  __device__ __forceinline__ int cx(int i) const {
    return (int)min((unsigned)(i - ri0), (unsigned)(kRX - 1));
  }
  __device__ __forceinline__ int cy(int j) const {
    return (int)min((unsigned)(j - rj0), (unsigned)(kRY - 1));
  }
  __device__ __forceinline__ int k(int i, int j) const { return getb(m->kb, cx(i), cy(j)); }
  __device__ __forceinline__ int z(int i, int j) const { return getb(m->zb, cx(i), cy(j)); }
  __device__ __forceinline__ int knew(int i, int j) const { return getb(m->kn, cx(i), cy(j)); }
  __device__ __forceinline__ int corners(int i, int j) const { return corners4(m->kb, cx(i), cy(j)); }
  __device__ __forceinline__ uint16_t ref(Mk mk) const {
    return (uint16_t)(pack_xy(cx(mk.i), cy(mk.j)) | (mk.kind ? kKindV : 0));
  }
  // The marker of a reference.
  __device__ __forceinline__ Mk mk(uint16_t r) const {
    return Mk{(r & kKindV) ? 1 : 0, ri0 + lx_of(r), rj0 + ly_of(r)};
  }
  // The marker beyond point 1 (side 0) or point 4 (side 1) of candidate C on
  // the unaligned edge (k, j): points 1 and 4 are the markers beyond A and B
  // seen from the chord's cell, and this is the one beyond them in turn.
  template <class CandT>
  __device__ __forceinline__ Mk next_beyond(const CandT& C, int side, int k, int j) const {
    const int c = k - 2 + (C.ord >> 1);
    int ci = 0, cj = 0, oi = 0, oj = 0;
    const Mk n = beyond(*this, mk(side ? C.b : C.a), c, j, &ci, &cj);
    if (n.kind < 0) return n;
    return beyond(*this, n, ci, cj, &oi, &oj);
  }
  // Moved fraction of the marker on edge (lx, ly) of the region.
  __device__ __forceinline__ R frac(int kind, int lx, int ly) const {
    const int r = m->rank(kind, lx, ly);
    if (MANY && r >= marker_cap<R>()) return fraction_again(g, kind, ri0 + lx, rj0 + ly);
    return m->fr[r];
  }
  __device__ __forceinline__ AP<R> moved(Mk mk) const {
    const int lx = cx(mk.i), ly = cy(mk.j);
    AP<R> p;
    p.jy = mk.j;
    p.fx = frac(mk.kind, lx, ly);
    if (mk.kind == 0) {
      p.ix = mk.i + get2(m->hq, lx, ly) - 1;
      p.fy = R(0);
    } else {
      p.ix = mk.i + get2(m->vq, lx, ly) - 1;
      p.fy = g.v(mk.i, mk.j);
    }
    return p;
  }
  __device__ __forceinline__ Landing<R> landing(int i, int j) const {
    const int c = get2(m->lq, cx(i), cy(j));
    Landing<R> L;
    L.present = knew(i, j) ^ knew(i + 1, j);
    L.kept_src = c == 0 ? -1 : i + c - 2;
    L.kept_fx = R(0);
    L.cancelled = 0;
    L.invariant = 0;
    return L;
  }
  // Moved point of a referenced marker relative to vertex (k, j).
  __device__ __forceinline__ void xy(uint16_t r, int k, int j, double* X, double* Y) const {
    const int lx = lx_of(r), ly = ly_of(r);
    // the same values as (double)n + (double)f; the conversions run on the
    // integer pipe and an aligned marker's y needs no addition
    if (r & kKindV) {
      *X = i2d(ri0 + lx + get2(m->vq, lx, ly) - 1 - k) + to_d<R>(frac(1, lx, ly));
      *Y = i2d(rj0 + ly - j) + to_d<R>(g.v(ri0 + lx, rj0 + ly));
    } else {
      *X = i2d(ri0 + lx + get2(m->hq, lx, ly) - 1 - k) + to_d<R>(frac(0, lx, ly));
      *Y = i2d(rj0 + ly - j);
    }
  }
  // An unaligned marker's own fraction (its y in the sweep), read from the
  // state; 0 for an aligned marker.
  __device__ __forceinline__ R own_fraction(uint16_t r) const {
    if (!(r & kKindV)) return R(0);
    const int lx = lx_of(r), ly = ly_of(r);
    return g.v(ri0 + lx, rj0 + ly);
  }
  // The point in the FP32 form, given its own fraction fy, relative to an
  // origin kShift cells left of and below vertex (k, j): there the sums of a
  // small grid line number and a fraction of at least 2^-26 are exact doubles
  // in [8, 16), formed by one integer addition.  Differences of two such
  // points are those of the points relative to (k, j).  False where a sum is
  // not of that kind.  (Xf, Yf): float estimates relative to (k, j), within
  // 2^-22.
  __device__ __forceinline__ bool xy_shifted(uint16_t r, int k, int j, float fy, double* X, double* Y, float* Xf,
                                             float* Yf) const {
    const int lx = lx_of(r), ly = ly_of(r), kind = r >> 15;
    const int nx = ri0 + lx + get2(kind ? m->vq : m->hq, lx, ly) - 1 - k, ny = rj0 + ly - j;
    const float fx = (float)frac(kind, lx, ly);
    *Xf = (float)nx + fx;
    *Yf = (float)ny + fy;
    const bool ok = shifted_sum(nx, fx, X);
    return shifted_sum(ny, fy, Y) && ok;
  }
};

// One marker per edge from its linked candidates (the rule of
// select_candidates, Sec. 2.4), in registers: candidates ranked by (position,
// generation order).
// *kept receives the slot of the kept candidate (-1: none); its centre-rule
// verdicts are formed by the caller where they are needed.
template <typename R, int CAP>
__device__ __forceinline__ NewV<R> select_linked(const TileMem<R, CAP>& M, int s, int present,
                                                 int* kept) {
  *kept = -1;
  double cy[6];
  long long key[6];
  int ord[6], sl[6];
  int n = 0;
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    if (s >= 0) {
      cy[q] = M.u.c.y[s];
      key[q] = okey(cy[q]);
      ord[q] = M.u.c.cand[s].ord;
      sl[q] = s;
      n = q + 1;
      s = M.u.c.next[s];
    } else {
      cy[q] = 0.0;
      key[q] = 0;
      ord[q] = 0;
      sl[q] = -1;
    }
  }
  int rank[6];
#pragma unroll
  for (int t = 0; t < 6; ++t) {
    int r = 0;
#pragma unroll
    for (int u = 0; u < 6; ++u)
      if (u != t && u < n && (key[u] < key[t] || (key[u] == key[t] && ord[u] < ord[t]))) ++r;
    rank[t] = r;
  }
  NewV<R> out;
  out.present = present;
  out.vr = -1;
  out.vl = -1;
  out.s = R(0.5);
  out.cancelled = 0;
  out.invariant = 0;
  int want = -1;  // rank of the kept candidate
  if (present && (n & 1)) {
    want = n / 2;
    out.cancelled = n / 2;  // the pairs around the middle one
  } else if (!present && !(n & 1)) {
    out.cancelled = n / 2;
  } else {
    out.invariant = 1;
    if (present && n > 0) {  // the candidate nearest the edge's middle, first in rank order
      double bd = 0.0;
#pragma unroll
      for (int t = 0; t < 6; ++t)
        if (t < n) {
          const double d = fabs(cy[t] - 0.5);
          if (want < 0 || d < bd || (d == bd && rank[t] < want)) {
            bd = d;
            want = rank[t];
          }
        }
    }
  }
  if (want >= 0) {
    double ysel = 0.0;
#pragma unroll
    for (int t = 0; t < 6; ++t)
      if (t < n && rank[t] == want) {
        ysel = cy[t];
        *kept = sl[t];
      }
    out.s = to_fraction<R>(ysel);
  }
  return out;
}

// The parts of the tile that few tiles or few markers take are kept out of
// line, with their loops rolled: inlined they made the kernel 390 KB of code,
// three times the instruction cache.

// Landings on one edge other than a single one that stays.
template <typename R>
__device__ __noinline__ Landing<R> landing_rare(bool v0, bool v1, bool v2, R f0, R f1, R f2, int x, int present) {
  const bool valid[3] = {v0, v1, v2};
  const R fx[3] = {f0, f1, f2};
  return choose_landing3<R>(valid, fx, x, present);
}

// One marker of an edge with several candidates (or none to keep): see
// select_linked.
template <typename R, int CAP>
__device__ __noinline__ NewV<R> select_rare(const TileMem<R, CAP>& M, int s, int present, int* kept) {
  return select_linked<R>(M, s, present, kept);
}

// A referenced marker's moved point relative to vertex (k, j), out of line.
template <class V>
__device__ __noinline__ void xy_rare(const V TV, uint16_t r, int k, int j, double* X, double* Y) {
  TV.xy(r, k, j, X, Y);
}

// The marker beyond point 1 (side 0) or 4 (side 1) of a candidate, as a third
// point for its ends (ax, ay) and (bx, by).
struct NextPt {
  FitPt T;
  bool found;
};
template <class V>
__device__ __noinline__ NextPt next_point(const V TV, int slot, int side, int k, int j,
                                          double ax, double ay, double bx, double by) {
  NextPt p{};
  const Mk q = TV.next_beyond(TV.m->u.c.cand[slot], side, k, j);
  p.found = q.kind >= 0;
  if (p.found) {
    double X, Y;
    TV.xy(TV.ref(q), k, j, &X, &Y);
    p.T = fit_pt(X, Y, ax, ay, bx, by);
  }
  return p;
}

// Centre-rule verdicts (right + 1, left + 1 as in verdicts()) of the kept
// candidate of unaligned edge (k, j), for the sides asked for.
template <class V>
__device__ __noinline__ uint8_t verdicts_of(const V TV, int slot, int k, bool right, bool left) {
  const Cand& C = TV.m->u.c.cand[slot];
  int v[2] = {-1, -1};
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    if (!(side ? left : right)) continue;
    const Mk none{-1, 0, 0};
    const Mk far = (C.fl & (side ? CF_P1 : CF_P4)) ? TV.mk(side ? C.p1 : C.p4) : none;
    const int line = walk(TV, TV.mk(side ? C.a : C.b), far, side ? k - 1 : k);
    if (line >= 0) v[side] = !TV.knew(k, line);
  }
  return verdicts(v[0], v[1]);
}

// new_unaligned out of line.
template <typename R, class A>
__device__ __noinline__ NewV<R> new_unaligned_rare(const A S, bool line_only, int k, int j, int* cnt) {
  return new_unaligned<R>(S, line_only, k, j, cnt);
}

// A tile's lists' lengths, counters and largest displacement (static shared memory).
struct TileCtl {
  int nh, nm, nc, ncand, ne, novf;  // aligned markers, markers, segments, candidates, edges with
                                    // a linked candidate, edges done in place
  int cnt[D_NUSED];
  unsigned long long dmax;
};

// Region columns and rows inside the grid, of the tile with origin (i0, j0).
struct TileSpan {
  int vx0, vx1, ex1;  // vertices; aligned edges, cells
  int vy0, vy1, ey1;  // vertex rows; unaligned edges, cells
  __device__ __forceinline__ TileSpan(int tnx, int tny, int ri0, int rj0)
      : vx0(max(0, -ri0)), vx1(min(kRX - 1, tnx - ri0)), ex1(min(kRX - 2, tnx - 1 - ri0)),
        vy0(max(0, -rj0)), vy1(min(kRY - 1, tny - rj0)), ey1(min(kRY - 2, tny - 1 - rj0)) {}
};

// P0: colour bits of the region.
template <typename R, int AX, int LD, int CAP, int T>
__device__ __forceinline__ void tile_colours(const GView<R, AX, LD>& G, TileMem<R, CAP>& M, const int i0,
                                             const int j0) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kTileThreads = T, kWarps = T / 32;
  const int ri0 = i0 - 4, rj0 = j0 - 2;
  const TileSpan B(G.tnx(), G.tny(), ri0, rj0);
  if (AX == 0) {
#pragma unroll 1
    for (int t = tid; t < 2 * kRB; t += kTileThreads) {
      const int zpl = t >= kRB, u = zpl ? t - kRB : t;
      const int ly = u / kRW, wi = u % kRW;
      const int y = rj0 + ly, x0 = ri0 + 32 * wi;
      uint32_t v = 0u;
      if (!zpl && ly >= B.vy0 && ly <= B.vy1)
        v = row_bits<LD>(G.K + (long long)y * G.d.kw, G.d.kw, x0) & span_mask(wi, B.vx0, B.vx1);
      if (zpl && ly >= B.vy0 && ly <= B.ey1)
        v = row_bits<LD>(G.Z + (long long)y * G.d.zw, G.d.zw, x0) & span_mask(wi, B.vx0, B.ex1);
      (zpl ? M.zb : M.kb)[u] = v;
    }
  } else {
    // region column lx is stored row ri0 + lx and region row ly stored column
    // rj0 + ly: a warp reads three words of 32 stored rows and transposes them
    const int c0 = rj0 >> 5;  // stored word holding region rows 0 and 1
    for (int g = warp; g < 2 * kRW; g += kWarps) {
      const int zpl = g >= kRW, gw = zpl ? g - kRW : g;
      const int lx = 32 * gw + lane, yr = ri0 + lx;
      const uint32_t* base = zpl ? G.Z : G.K;
      const int nw = zpl ? G.d.zw : G.d.kw;
      const int row1 = zpl ? B.ey1 : B.vy1;
      uint32_t w[3] = {0u, 0u, 0u};
      if (lx >= B.vx0 && lx <= (zpl ? B.ex1 : B.vx1)) {
        const uint32_t* r = base + (long long)yr * nw;
#pragma unroll
        for (int q = 0; q < 3; ++q)
          if (c0 + q >= 0 && c0 + q < nw) w[q] = ld_state<LD>(&r[c0 + q]);
      }
      uint32_t* dst = zpl ? M.zb : M.kb;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const uint32_t col = transpose32(w[q], lane);
        const int ly = 32 * (c0 + q) + lane - rj0;
        if (ly >= 0 && ly < kRY) dst[ly * kRW + gw] = (ly >= B.vy0 && ly <= row1) ? col : 0u;
      }
    }
  }
}

// The phases of a tile follow.  WIN = false: for the whole tile.  WIN = true: for
// a window of its rows, [j0 + r0, j0 + r0 + rows); markers outside of the window and
// its halo are left out, and there may be more than moved fractions are kept.

// P1 for a block of T threads; returns whether there are markers (S.nm: how many).
template <typename R, int AX, int LD, int CAP, int T, bool WIN>
__device__ __forceinline__ bool tile_markers(const GView<R, AX, LD>& G, TileMem<R, CAP>& M, TileCtl& S, const int i0,
                                             const int j0, const int r0, const int rows) {
  static_assert(T >= 128, "four warps");
  constexpr int kMkList = TileMem<R, CAP>::kMkList;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kTileThreads = T;
  const int tnx = G.tnx(), tny = G.tny();
  const int ri0 = i0 - 4, rj0 = j0 - 2;
  const TileSpan B(tnx, tny, ri0, rj0);
  // P1: marker sets
  int mine = 0;
  for (int t = tid; t < kRB; t += kTileThreads) {
    const int ly = t / kRW, wi = t % kRW;
    uint32_t h = 0u, v = 0u;
    const bool here = !WIN || (ly >= r0 && ly <= r0 + rows + 4), cell = !WIN || (ly >= r0 && ly < r0 + rows + 4);
    if (ly >= B.vy0 && ly <= B.vy1 && here) h = (M.kb[t] ^ shr1(M.kb, ly, wi)) & span_mask(wi, B.vx0, B.ex1);
    if (ly >= B.vy0 && ly <= B.ey1 && cell)
      v = (M.kb[t] ^ M.kb[t + kRW]) & span_mask(wi, B.vx0, B.vx1);
    M.hm[t] = h;
    M.vm[t] = v;
    if (here) M.kn[t] = M.kb[t];  // (a row's flips are its own markers': the same in every window)
    M.claim[t] = 0u;
    M.hc[t] = 0u;
    M.ovf[t] = 0u;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      M.hq[q][t] = 0u;
      M.vq[q][t] = 0u;
      M.lq[q][t] = 0u;
    }
    mine |= (h | v) != 0u;
  }
  const bool busy = __syncthreads_or(mine) != 0;

  if (busy) {
    // ranks: warps 0 and 1 take the halves of the aligned set's words, warps 2
    // and 3 those of the unaligned set, two words a lane; the markers before a
    // warp's first word are counted by the warp itself
    static_assert(kRB <= 128, "two words a lane, two warps a set");
    if (warp < 4) {
      const int pl = warp >> 1, hf = warp & 1, t0 = 64 * hf + 2 * lane;
      const uint32_t* pm = pl ? M.vm : M.hm;
      uint32_t w0 = t0 < kRB ? pm[t0] : 0u, w1 = t0 + 1 < kRB ? pm[t0 + 1] : 0u;
      const int n0 = __popc(w0), n = n0 + __popc(w1);
      int before = 0;
      if (hf) before = __popc(pm[lane]) + __popc(pm[lane + 32]);
      if (pl) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (lane + 32 * q < kRB) before += __popc(M.hm[lane + 32 * q]);
      }
      before = __reduce_add_sync(kFull, before);
      int incl = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += v;
      }
      int at = before + incl - n;
      uint16_t* base = pl ? M.vbase : M.hbase;
      if (t0 < kRB) base[t0] = (uint16_t)at;
      if (t0 + 1 < kRB) base[t0 + 1] = (uint16_t)(at + n0);
      if (hf && lane == 31) (pl ? S.nm : S.nh) = at + n;
      const int p0 = pack_xy(32 * (t0 % kRW), t0 / kRW), p1 = pack_xy(32 * ((t0 + 1) % kRW), (t0 + 1) / kRW);
#pragma unroll 1
      for (; w0 && at < kMkList; w0 &= w0 - 1) M.u.mk[at++] = (uint16_t)(p0 + __ffs(w0) - 1);
#pragma unroll 1
      for (; w1 && at < kMkList; w1 &= w1 - 1) M.u.mk[at++] = (uint16_t)(p1 + __ffs(w1) - 1);
    }
    static_assert(sizeof(M.head) % 16 == 0, "vector initialisation");
    for (int e = tid; e < (int)(sizeof(M.head) / 16); e += kTileThreads)
      reinterpret_cast<uint4*>(M.head)[e] = make_uint4(~0u, ~0u, ~0u, ~0u);
    __syncthreads();
  }
  return busy;
}

// The interface cells (corner colours not all equal) of word u whose chords can
// cross a grid line k in [i0, i0+64], cells k-2..k, to the list of segments; here:
// of a row wanted.  All 32 lanes call it.
template <typename R, int CAP>
__device__ __forceinline__ void list_segments(TileMem<R, CAP>& M, TileCtl& S, const TileSpan& B, int u, bool here) {
  const int lane = threadIdx.x & 31, ly = u / kRW, wi = u % kRW;
  uint32_t ic = 0u, four = 0u;
  if (ly <= min(kTJ + 1, B.ey1) && here) {
    const uint32_t a = M.kb[u], b = M.kb[u + kRW], a1 = shr1(M.kb, ly, wi), b1 = shr1(M.kb, ly + 1, wi);
    const uint32_t cm = span_mask(wi, max(2, B.vx0), min(kTI + 4, B.ex1));
    ic = ((a ^ a1) | (b ^ b1) | (a ^ b)) & cm;
    four = (a ^ a1) & (b ^ b1) & (a ^ b) & cm;
  }
  push_bits_warp(ic, u, 0, M.cl, &S.nc, lane);
  if (__any_sync(kFull, four != 0u)) push_bits_warp(four, u, kSecond, M.cl, &S.nc, lane);
}

// P2 and P3 (the segments are listed here unless WIN).
template <typename R, int AX, int LD, int CAP, int T, bool WIN>
__device__ __forceinline__ void tile_moves(const GView<R, AX, LD>& G, const Buf<R>& out, TileMem<R, CAP>& M, TileCtl& S,
                                           const int i0, const int j0, const int r0, const int rows) {
  constexpr int kMkCap = marker_cap<R>();
  const int tid = threadIdx.x, lane = tid & 31;
  constexpr int kTileThreads = T;
  const int tnx = G.tnx(), tny = G.tny();
  const int ri0 = i0 - 4, rj0 = j0 - 2;
  const TileSpan B(tnx, tny, ri0, rj0);
  const long long P = G.d.P;
  const int ya = j0 + r0, yb = ya + rows;
  auto owned = [&](int x, int y) { return x >= i0 && x < i0 + kTI && y >= ya && y < yb; };
  auto in_rows = [&](int ly) { return !WIN || (ly >= r0 + 2 && ly < r0 + 2 + rows); };
  const TViewB<R, AX, LD, CAP, WIN> TV{&M, G, ri0, rj0, tnx, tny};
  // P2: moved points (aligned and unaligned markers in one pass), corner
  // flips, landing claims
  const int nh = S.nh, nm = S.nm;
  int n_cfl = 0, n_clamp = 0;
  R dmax = R(0);
#pragma unroll 1
  for (int w = tid; w < nm; w += kTileThreads) {
    const int id = M.u.mk[w], lx = lx_of(id), ly = ly_of(id);
    const int x = ri0 + lx, y = rj0 + ly;
    const bool al = w < nh;
    Flags f;
    const AP<R> p = G.advect(Mk{al ? 0 : 1, x, y}, f);
    if (!WIN || w < kMkCap) M.fr[w] = p.fx;
    put2(al ? M.hq : M.vq, lx, ly, p.ix - x + 1);
    const bool own = owned(x, y);
    if (own) {  // no flag on a wall normal to the sweep
      n_cfl += f.cfl;
      n_clamp += f.clamp;
      dmax = fmax(dmax, dabs_of<R>(f));
    }
    if (al) {
      // a marker moving right passes vertex x+1, one moving left vertex x
      if (p.ix != x) {
        const int c = lx + (p.ix > x);
        atomicXor(&M.kn[ly * kRW + (c >> 5)], 1u << (c & 31));
      }
      const int dl = p.ix - ri0;
      if (dl >= 1 && dl <= kRX - 3) atomicOr(&M.claim[ly * kRW + (dl >> 5)], 1u << (dl & 31));
    } else if (own && (x == 0 || x == tnx)) {  // a wall marker normal to the sweep stays
      if (AX) { if (in_range((long long)x * P + y, G.d.nH())) out.sH[(long long)x * P + y] = p.fy; }
      else if (in_range((long long)y * P + x, G.d.nV())) out.sV[(long long)y * P + x] = p.fy;
    }
  }
  flush_count(S.cnt, D_CFL, n_cfl, lane);
  flush_count(S.cnt, D_WALL_CLAMP, n_clamp, lane);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dmax = fmax(dmax, __shfl_xor_sync(kFull, dmax, o));
  if (lane == 0 && dmax > R(0))
    atomicMax(&S.dmax, (unsigned long long)__double_as_longlong((double)dmax));
  __syncthreads();

  // P3: landings.  Of the markers landing on an edge the one from the lowest
  // source takes the edge.  After their landings the last three warps pass over
  // the words (owned edges without a landing, interface cells).
  int n_canc = 0, n_inv = 0;
  const int kSplit = kTileThreads - kTJ * kRW;  // 96 words on the last three warps
  static_assert(kTJ * kRW == 96, "warp split");
#pragma unroll 1
  for (int w = tid; w < nh; w += kTileThreads) {
    const int id = M.u.mk[w], lx = lx_of(id), ly = ly_of(id);
    const int dl = lx + get2(M.hq, lx, ly) - 1;
    if (dl < 1 || dl > kRX - 3) continue;
    const int x = ri0 + dl, y = rj0 + ly;
    bool valid[3];
    R fx[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int e = dl - 1 + q;
      valid[q] = getb(M.hm, e, ly) && e + get2(M.hq, e, ly) - 1 == dl;
      fx[q] = valid[q] ? TV.frac(0, e, ly) : R(0);
    }
    if (lx != dl - 1 && (valid[0] || (lx != dl && valid[1]))) continue;  // a lower source's edge
    const int present = getb(M.kn, dl, ly) ^ getb(M.kn, dl + 1, ly);
    Landing<R> L;
    if (__builtin_expect(present && (int)valid[0] + (int)valid[1] + (int)valid[2] == 1, 1)) {  // it stays
      L = Landing<R>{1, ri0 + lx, 0, 0, WIN ? TV.frac(0, lx, ly) : M.fr[w]};
    } else {
      L = landing_rare<R>(valid[0], valid[1], valid[2], fx[0], fx[1], fx[2], x, present);
    }
    if (L.kept_src >= 0) put2(M.lq, dl, ly, L.kept_src - x + 2);
    if (owned(x, y)) {
      n_canc += L.cancelled;
      n_inv += L.invariant;
      if (L.present) {
        if (AX) { if (in_range((long long)x * P + y, G.d.nV())) out.sV[(long long)x * P + y] = L.kept_fx; }
        else if (in_range((long long)y * P + x, G.d.nH())) out.sH[(long long)y * P + x] = L.kept_fx;
      }
    }
  }
  if (tid >= kSplit) {
    const int t = tid - kSplit;  // one word each
    const int ly = 2 + t / kRW, wi = t % kRW, u = ly * kRW + wi;
    // owned aligned edges that gain a marker none landed on (the colour
    // bookkeeping excludes it): counted, fraction 0.5
    if (ly <= B.vy1 && in_rows(ly)) {
      uint32_t bad = (M.kn[u] ^ shr1(M.kn, ly, wi)) & ~M.claim[u] &
                     span_mask(wi, 4, min(kTI + 3, B.ex1));
#pragma unroll 1
      while (bad) {
        const int b = __ffs(bad) - 1;
        bad &= bad - 1;
        const int x = ri0 + 32 * wi + b, y = rj0 + ly;
        n_inv += 1;
        if (AX) { if (in_range((long long)x * P + y, G.d.nV())) out.sV[(long long)x * P + y] = R(0.5); }
        else if (in_range((long long)y * P + x, G.d.nH())) out.sH[(long long)y * P + x] = R(0.5);
      }
    }
    if (!WIN) list_segments(M, S, B, u, true);
  }
  flush_count(S.cnt, D_CANCELLED, n_canc, lane);
  flush_count(S.cnt, D_INVARIANT, n_inv, lane);
  __syncthreads();
}

// P4-P6 for the listed segments (WIN: those of the rows [j0 + r0, j0 + r0 + rows)).
template <typename R, int AX, int LD, int CAP, int T, bool WIN>
__device__ __forceinline__ void tile_fits(const GView<R, AX, LD>& G, const Buf<R>& out, int line_only,
                                          TileMem<R, CAP>& M, TileCtl& S, const int i0, const int j0, const int r0,
                                          const int rows) {
  constexpr int kHB = head_bits<CAP>(), kHPW = 32 / kHB;  // head bits, heads per word
  constexpr uint32_t kHNone = head_none<CAP>();
  constexpr int kWarps = T / 32, kSplit = T - kTJ * kRW;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kTileThreads = T;
  const int tnx = G.tnx(), tny = G.tny();
  const int ri0 = i0 - 4, rj0 = j0 - 2;
  const TileSpan B(tnx, tny, ri0, rj0);
  const long long P = G.d.P;
  const int ty1 = min(kTJ + 1, B.ey1);  // last cell row of the tile
  auto in_rows = [&](int ly) { return !WIN || (ly >= r0 + 2 && ly < r0 + 2 + rows); };
  const TViewB<R, AX, LD, CAP, WIN> TV{&M, G, ri0, rj0, tnx, tny};
  // P4: candidates.  A thread takes one segment: counts the grid lines its
  // moved chord crosses, takes that many slots, then fills them.
  const int nc = S.nc;
  const int kmin = max(1, i0), kmax = min(tnx - 1, i0 + kTI);
#pragma unroll 1
  for (int w0 = warp * 32; w0 < nc; w0 += kTileThreads) {
    const int w = w0 + lane;
    int lx = 0, ly = 0, second = 0, ea = 0, eb = 0, xa = 0, klo = 0, khi = -1;
    auto at = [&](int e) { return pack_xy(lx + (e == 1), ly + (e == 2)); };  // edge e of the cell
    if (w < nc) {
      const int id = M.cl[w];
      second = id >= kSecond;
      ly = ly_of(id);
      lx = lx_of(id);
      const int q = corners4(M.kb, lx, ly), em = edge_mask(q);
      ea = __ffs(em) - 1;
      eb = 31 - __clz(em);
      if (__builtin_expect(em == 15, 0)) {  // the pairs of segments()
        const bool same = (q & 1) == getb(M.zb, lx, ly);
        ea = same ? 2 * second : 3 - 2 * second;
        eb = same ? ea + 1 : 2 * second;
      }
      auto line = [&](int e) {
        return ri0 + lx + (e == 1) + get2(e & 1 ? M.vq : M.hq, lx + (e == 1), ly + (e == 2)) - 1;
      };
      xa = line(ea);
      const int xb = line(eb);
      klo = max(min(xa, xb) + 1, kmin);
      khi = min(max(xa, xb), kmax);
    }
    int slot = warp_alloc(max(0, khi - klo + 1), &S.ncand, lane);
#pragma unroll 1
    for (int k = klo; k <= khi; ++k, ++slot) {
      const int j = rj0 + ly, e = (j - j0) * (kTI + 1) + (k - i0);
      const int ex = k - ri0, eu = ly * kRW + (ex >> 5);
      const uint32_t ebit = 1u << (ex & 31);
      if (__builtin_expect(slot >= CAP, 0)) {
        atomicOr(&M.ovf[eu], ebit);
        continue;
      }
      Cand& C = M.u.c.cand[slot];
      uint8_t fl = k < i0 + kTI ? CF_OWNED : 0;
      // sides A (left of the line) and B: the chord's end, and the marker
      // beyond it (point 1, 4) in the cell across the end's edge
#pragma unroll 1
      for (int side = 0; side < 2; ++side) {
        const int se = (xa < k) == (side == 0) ? ea : eb;
        (side ? C.b : C.a) = (uint16_t)(at(se) | (se & 1 ? kKindV : 0));
        const int ox = lx + (se == 1) - (se == 3), oy = ly + (se == 2) - (se == 0);
        if ((unsigned)(ri0 + ox) < (unsigned)tnx && (unsigned)(rj0 + oy) < (unsigned)tny) {
          const int q = corners4(M.kb, ox, oy), em = edge_mask(q), in = se ^ 2;
          int pe = __ffs(em & ~(1 << in)) - 1;  // partner()
          if (em == 15) pe = (q & 1) == getb(M.zb, ox, oy) ? in ^ 1 : 3 - in;
          (side ? C.p4 : C.p1) =
              (uint16_t)(pack_xy(ox + (pe == 1), oy + (pe == 2)) | (pe & 1 ? kKindV : 0));
          fl |= side ? CF_P4 : CF_P1;
        }
      }
      C.fl = fl;
      C.edge = (uint16_t)pack_xy(k - i0, j - j0);
      C.ord = (uint8_t)((ri0 + lx - (k - 2)) * 2 + second);
      {  // push the slot on the edge's list: a head of kHB bits in a shared word
        uint32_t* hw = &M.head[e / kHPW];
        const int sh = (e % kHPW) * kHB;
        uint32_t old = *hw, seen;
        do {  // each retry follows another thread's successful update
          seen = old;
          old = atomicCAS(hw, seen, (seen & ~(kHNone << sh)) | ((uint32_t)slot << sh));
        } while (old != seen);
        const uint32_t prev = (seen >> sh) & kHNone;
        M.u.c.next[slot] = prev == kHNone ? (int16_t)-1 : (int16_t)prev;
      }
      atomicOr(&M.hc[eu], ebit);
    }
  }
  __syncthreads();

  // P5: circle fits (Sec. 2.2).  Lanes 2m and 2m+1 fit the circles through
  // point 1 and point 4 of one candidate and the even lane combines them,
  // as fit_crossing does; the warps that take candidates rotate with the
  // block so that the FP64 work spreads over the SM's sub-partitions.  The
  // last three warps first list the edges with linked candidates.
  const int ncand = min(S.ncand, CAP);
  // the interface-cell list is dead: its storage becomes the verdicts of P6
  for (int e = tid; e < kNVE / 16; e += kTileThreads)
    reinterpret_cast<uint4*>(M.vrl)[e] = make_uint4(0u, 0u, 0u, 0u);
  if (warp >= kWarps - 3) {
    const int t = (warp - (kWarps - 3)) * 32 + lane;  // kTJ * kRW = 96 words
    const int u = (2 + t / kRW) * kRW + t % kRW;
    push_bits_warp(M.hc[u], u, 0, M.u.c.le, &S.ne, lane);
    const int no = __reduce_add_sync(kFull, __popc(M.ovf[u]));  // edges done in place
    if (no != 0 && lane == 0) atomicAdd(&S.novf, no);
  }
  const int rot = (int)((blockIdx.x + blockIdx.y) & 3u);
  int n_fit[4] = {0, 0, 0, 0};  // D_FIT_ONLINE .. D_FIT_TWO
  const int vt = (((warp + rot) % kWarps) << 5) | lane;
#pragma unroll 1
  for (int b0 = 0; b0 < 2 * ncand; b0 += kTileThreads) {
    const int item = b0 + vt, side = item & 1;
    Cand& C = M.u.c.cand[min(item >> 1, CAP - 1)];
    const int k = i0 + lx_of(C.edge), j = j0 + ly_of(C.edge);
    // an edge that is done in place takes no fit here
    const bool act = item < 2 * ncand && !getb(M.ovf, k - ri0, j - rj0);
    // the pair shares the chord: the even lane forms A and cx, the odd lane
    // B and cy, and they swap (shuffles instead of FP64 work)
    const bool third = act && (C.fl & (side ? CF_P4 : CF_P1));
    double px = 0.0, py = 0.0, X = 0.0, Y = 0.0, org = 0.0;
    float pxf = 0.0f, pyf = 0.0f, Xf = 0.0f, Yf = 0.0f;
    if constexpr (sizeof(R) == 4) {
      const uint16_t r = side ? C.b : C.a, r3 = side ? C.p4 : C.p1;
      // the state reads this lane needs, issued together
      const float fy = act ? TV.own_fraction(r) : 0.0f, fy3 = third ? TV.own_fraction(r3) : 0.0f;
      bool plain = !act || TV.xy_shifted(r, k, j, fy, &px, &py, &pxf, &pyf);
      if (third) plain = TV.xy_shifted(r3, k, j, fy3, &X, &Y, &Xf, &Yf) && plain;
      org = (double)kShift;
      const unsigned odd_sums = __ballot_sync(kFull, !plain);
      if (__builtin_expect(odd_sums != 0u, 0) && (odd_sums >> (lane & 30) & 3u)) {
        // a pair with a sum of the other kind takes its points relative to (k, j)
        org = 0.0;
        xy_rare(TV, r, k, j, &px, &py);
        if (third) xy_rare(TV, r3, k, j, &X, &Y);
      }
    } else {
      if (act) TV.xy(side ? C.b : C.a, k, j, &px, &py);
      if (third) TV.xy(side ? C.p4 : C.p1, k, j, &X, &Y);
    }
    const double ox = __shfl_xor_sync(kFull, px, 1), oy = __shfl_xor_sync(kFull, py, 1);
    const float oxf = __shfl_xor_sync(kFull, pxf, 1), oyf = __shfl_xor_sync(kFull, pyf, 1);
    const float bxf = side ? pxf : oxf, byf = side ? pyf : oyf;  // B, estimated in float
    const double ax = side ? ox : px, ay = side ? oy : py;
    const double bx = side ? px : ox, by = side ? py : oy;
    const double dd = side ? by - ay : bx - ax;
    const double od = __shfl_xor_sync(kFull, dd, 1);
    const double cx = side ? od : dd, cy = side ? dd : od;
    const double sq = dd * dd, osq = __shfl_xor_sync(kFull, sq, 1);
    const double c2 = side ? osq + sq : sq + osq;  // cx*cx + cy*cy
    // A relative to (k, j): x0 = -x, y0 = y (exact)
    double x0 = -ax, y0 = ay;
    if constexpr (sizeof(R) == 4) {
      const double v = (side ? ay : org) - (side ? org : ax), ov = __shfl_xor_sync(kFull, v, 1);
      x0 = side ? ov : v;
      y0 = side ? v : ov;
    }
    const bool online = d_eq0(bx) || (sizeof(R) == 4 && dbits(bx) == dbits(org));
    // the third point, then the circle.  The warp's lanes come together
    // between the two, so that those whose point takes longer do not run
    // the circle's FP64 chain a second time.
    double ys = 0.0;
    bool ok = false;
    const bool want = third && !online && !line_only && !d_below_sep(c2);
    const unsigned wanted = __ballot_sync(kFull, want);
    if (want) {
      double rx = X - ax, ry = Y - ay, r2 = rx * rx + ry * ry;
      bool tfar, use = true;
      // in the FP32 form the distance from B only where a float estimate
      // (error below 2e-6 per component) does not already put it clearly
      // past the minimum separation
      const float txf = Xf - bxf, tyf = Yf - byf;
      if (sizeof(R) == 4 && txf * txf + tyf * tyf >= 1.5e-4f) {
        tfar = true;
      } else {
        const double tx = X - bx, ty = Y - by;
        tfar = !d_below_sep(tx * tx + ty * ty);
      }
      if (__builtin_expect(side ? !tfar : d_below_sep(r2), 0)) {  // too close to B (A): the next marker
        const NextPt q = next_point(TV, item >> 1, side, k, j, ax - org, ay - org, bx - org, by - org);
        use = q.found;
        rx = q.T.rx;
        ry = q.T.ry;
        r2 = q.T.r2;
        tfar = !d_below_sep(q.T.t2);
      }
      __syncwarp(wanted);
      if (use) ok = circle_cross_r(y0, x0, cx, cy, c2, rx, ry, r2, tfar, &ys);
    }
    const double yo = __shfl_xor_sync(kFull, ys, 1);
    const bool oko = __shfl_xor_sync(kFull, (int)ok, 1) != 0;
    if (act && side == 0) {
      double y;
      int kind;
      if (online) {
        y = by - org;
        kind = D_FIT_ONLINE;
      } else if (ok && oko) {
        y = d_scale<-1>(ys + yo);
        kind = D_FIT_TWO;
      } else if (ok || oko) {
        y = ok ? ys : yo;
        kind = D_FIT_ONE;
      } else {  // no circle: the chord's own crossing
        y = y0 + (x0 * cy) / cx;
        kind = D_FIT_LINE;
      }
      M.u.c.y[item >> 1] = y;
      if (C.fl & CF_OWNED) {  // static indices keep the counters in registers
#pragma unroll
        for (int q = 0; q < 4; ++q) n_fit[q] += kind == D_FIT_ONLINE + q;
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) flush_count(S.cnt, D_FIT_ONLINE + q, n_fit[q], lane);
  __syncthreads();

  // P6: one marker per unaligned edge (Sec. 2.4)
  const int ne = S.ne;
  int n_canc = 0, n_inv = 0;
#pragma unroll 1
  for (int w = tid; w < ne; w += kTileThreads) {
    const int id = M.u.c.le[w], ex = lx_of(id), ey = ly_of(id);
    if (getb(M.ovf, ex, ey)) continue;
    const int k = ri0 + ex, j = rj0 + ey;
    const int e = (j - j0) * (kTI + 1) + (k - i0);
    const bool own = k < i0 + kTI;
    const int present = getb(M.kn, ex, ey) ^ getb(M.kn, ex, ey + 1);
    const uint32_t hd = (M.head[e / kHPW] >> ((e % kHPW) * kHB)) & kHNone;
    int kept = -1;
    NewV<R> nv;
    if (__builtin_expect(hd != kHNone && M.u.c.next[hd] < 0 && present, 1)) {
      // one candidate on an edge that keeps a marker: it is the marker
      kept = (int)hd;
      nv.present = 1;
      nv.cancelled = 0;
      nv.invariant = 0;
      nv.s = to_fraction<R>(M.u.c.y[hd]);
    } else {
      nv = select_rare<R, CAP>(M, hd == kHNone ? -1 : (int)hd, present, &kept);
    }
    if (own) {
      n_canc += nv.cancelled;
      n_inv += nv.invariant;
    }
    // centre-rule verdicts of the kept candidate (Sec. 2.3), for the cells
    // either side of the edge that have four markers after the sweep (the
    // only ones whose centre colour the rule sets)
    if (kept >= 0) {
      auto four = [&](int x) {  // cell (x, ey) of the region, new colours
        const int q = corners4(M.kn, x, ey);
        return q == 5 || q == 10;
      };
      const bool fr = four(ex), fl = four(ex - 1);
      if (__builtin_expect(fr || fl, 0)) M.vrl[e] = verdicts_of(TV, kept, k, fr, fl);
    }
    if (own && nv.present) {
      if (AX) { if (in_range((long long)k * P + j, G.d.nH())) out.sH[(long long)k * P + j] = nv.s; }
      else if (in_range((long long)j * P + k, G.d.nV())) out.sV[(long long)j * P + k] = nv.s;
    }
  }
  if (const int ry = 2 + (tid - kSplit) / kRW; tid >= kSplit && ry <= ty1 && in_rows(ry)) {  // rows of such edges
    const int t = tid - kSplit;
    const int ly = 2 + t / kRW, wi = t % kRW, u = ly * kRW + wi;
    // owned interior edges that gain a marker without a candidate: counted,
    // fraction 0.5
    uint32_t miss = (M.kn[u] ^ M.kn[u + kRW]) & ~M.hc[u] & ~M.ovf[u] &
                    span_mask(wi, max(4, 1 - ri0), min(kTI + 3, tnx - 1 - ri0));
#pragma unroll 1
    while (miss) {
      const int b = __ffs(miss) - 1;
      miss &= miss - 1;
      const int k = ri0 + 32 * wi + b, j = rj0 + ly;
      n_inv += 1;
      if (AX) { if (in_range((long long)k * P + j, G.d.nH())) out.sH[(long long)k * P + j] = R(0.5); }
      else if (in_range((long long)j * P + k, G.d.nV())) out.sV[(long long)j * P + k] = R(0.5);
    }
  }
  // edges whose candidates did not fit in the tile's list are done in
  // place by the generic logic, spread over all threads: overflow edge m
  // (in word order) goes to thread m mod the block size
#pragma unroll 1
  for (int m = tid; m < S.novf; m += kTileThreads) {
    int u = 2 * kRW, r = m;
#pragma unroll 1
    for (; u < kRB; ++u) {
      const int c = __popc(M.ovf[u]);
      if (r < c) break;
      r -= c;
    }
    if (u >= kRB) break;  // not reached: S.novf counts these words' bits
    uint32_t o = M.ovf[u];
#pragma unroll 1
    for (; r > 0; --r) o &= o - 1;
    const int b = __ffs(o) - 1, ly = u / kRW, wi = u % kRW;
    const int k = ri0 + 32 * wi + b, j = rj0 + ly;
    const int e = (j - j0) * (kTI + 1) + (k - i0);
    const bool own = k < i0 + kTI;
    int oc[D_NUSED];
#pragma unroll
    for (int c = 0; c < D_NUSED; ++c) oc[c] = 0;
    const NewV<R> nv = new_unaligned_rare<R>(TV, line_only != 0, k, j, own ? oc : nullptr);
    for (int c = 0; c < D_NUSED; ++c)
      if (oc[c]) atomicAdd(&S.cnt[c], oc[c]);
    M.vrl[e] = verdicts(nv.vr, nv.vl);
    if (own && nv.present) {
      if (AX) { if (in_range((long long)k * P + j, G.d.nH())) out.sH[(long long)k * P + j] = nv.s; }
      else if (in_range((long long)j * P + k, G.d.nV())) out.sV[(long long)j * P + k] = nv.s;
    }
  }
  flush_count(S.cnt, D_CANCELLED, n_canc, lane);
  flush_count(S.cnt, D_INVARIANT, n_inv, lane);
  __syncthreads();
}

// P7, first part: the new centre colours of tile row j0 + lane, cells i0 + 32 ow
// + b (one lane each).  Those of new four-marker cells (all four edges with a
// marker) come from the verdicts of edges i (right) and i+1 (left); the right one wins.
template <typename R, int CAP>
__device__ __forceinline__ uint32_t tile_centres(const TileMem<R, CAP>& M, const TileSpan& B, int tnx, int i0, int j0,
                                                 int ow, bool busy, int* n_zset, int* n_zconf) {
  const int lane = threadIdx.x & 31, ly = 2 + lane, cx0 = 4 + 32 * ow;
  uint32_t zw = bits32(M.zb, ly, cx0);
  const uint32_t cmask = ly <= B.ey1 ? upto32(cx0, B.ex1) : 0u;
  if (busy && cmask) {
    const uint32_t a0 = bits32(M.kn, ly, cx0), a1 = bits32(M.kn, ly, cx0 + 1);
    const uint32_t b0 = bits32(M.kn, ly + 1, cx0), b1 = bits32(M.kn, ly + 1, cx0 + 1);
    uint32_t fm = (a0 ^ a1) & (b0 ^ b1) & (a0 ^ b0) & cmask;
#pragma unroll 1
    while (fm) {
      const int b = __ffs(fm) - 1;
      fm &= fm - 1;
      const int i = i0 + 32 * ow + b;
      const int e = lane * (kTI + 1) + (i - i0);
      const int a = (i >= 1) ? verdict_r(M.vrl[e]) : -1;
      const int bl = (i + 1 <= tnx - 1) ? verdict_l(M.vrl[e + 1]) : -1;
      int zc = -1;
      if (a >= 0) {
        zc = a;
        *n_zset += 1;
        if (bl >= 0 && bl != a) *n_zconf += 1;
      } else if (bl >= 0) {
        zc = bl;
        *n_zset += 1;
      }
      if (zc >= 0) zw = zc ? (zw | (1u << b)) : (zw & ~(1u << b));
    }
  }
  return zw & cmask;
}

// P7, second part: the colour words of the 32 x 32 vertices / cells ow of the
// tile, lane L holding row j0 + L; the y sweep transposes them into stored rows.
template <typename R, int AX, int LD, int CAP>
__device__ __forceinline__ void tile_words(const GView<R, AX, LD>& G, const Buf<R>& out, const TileMem<R, CAP>& M,
                                           const TileSpan& B, int i0, int j0, int ow, uint32_t zw) {
  const int lane = threadIdx.x & 31, ly = 2 + lane, cx0 = 4 + 32 * ow, j = j0 + lane;
  uint32_t kw = bits32(M.kn, ly, cx0) & (ly <= B.vy1 ? upto32(cx0, B.vx1) : 0u);
  if (AX) {
    kw = transpose32(kw, lane);
    zw = transpose32(zw, lane);
    const int row = i0 + 32 * ow + lane, word = j0 >> 5;
    if (row <= G.d.ny && word < G.d.kw) out.K[(long long)row * G.d.kw + word] = kw;
    if (row < G.d.ny && word < G.d.zw) out.Z[(long long)row * G.d.zw + word] = zw;
  } else {
    const int word = (i0 >> 5) + ow;
    if (j <= G.d.ny && word < G.d.kw) out.K[(long long)j * G.d.kw + word] = kw;
    if (j < G.d.ny && word < G.d.zw) out.Z[(long long)j * G.d.zw + word] = zw;
  }
}

// The block's counters to the grid's.
__device__ __forceinline__ void tile_counters(TileCtl& S, int n_zset, int n_zconf, unsigned long long* ctr,
                                              unsigned long long* cfl_bits, int* status) {
  const int tid = threadIdx.x, lane = tid & 31;
  flush_count(S.cnt, D_ZSET, n_zset, lane);
  flush_count(S.cnt, D_ZCONFLICT, n_zconf, lane);
  __syncthreads();
  if (tid < D_NUSED && S.cnt[tid] != 0) atomicAdd(&ctr[tid], (unsigned long long)S.cnt[tid]);
  if (tid == 0) {
    if (S.dmax) atomicMax(cfl_bits, S.dmax);
    if (S.cnt[D_CFL]) atomicOr(status, ST_CFL);
    if (S.cnt[D_INVARIANT]) atomicOr(status, ST_INVARIANT);
  }
}

// The rest, from P2 on, of a tile whose region holds more markers than moved
// fractions are kept (closely packed small drops, noise).  Those beyond are formed
// once more where they are needed.  The chords are taken eight rows at a time, so
// that their candidates (180 for the closest drops of radius 1.5) fit the list;
// all at once, the first case below takes 765 us.  Where the list of markers is
// too short as well, all phases run for one half of the rows and then for the other.
// Microseconds a sweep with dense per-edge arrays of moved fractions, with every
// answer recomputed from global memory, and so: 2048^2 cells of drops of radius 1.5
// on a 4.0-cell lattice (1800 markers a region) 680, 5178, 677 in FP64 (in FP32 the
// tiles keep them: 651, 2149, 469); 1024^2 cells with half of the vertices set at
// random 733, 3323, 339 in FP32 and 879, 6923, 449 in FP64; a checkerboard 1225,
// 4045, 761 and 1394, 10812, 1025.
template <typename R, int AX, int LD, int CAP, int T>
__device__ __noinline__ void tile_dense(const GView<R, AX, LD> G, const Buf<R> out, int line_only,
                                        unsigned long long* ctr, unsigned long long* cfl_bits, int* status,
                                        TileCtl* ctl, const int i0, const int j0) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TileMem<R, CAP>& M = *reinterpret_cast<TileMem<R, CAP>*>(smem_raw);
  TileCtl& S = *ctl;
  constexpr int kRows = 8;
  static_assert(kRows * kRW <= 32 && kTJ / 2 % kRows == 0, "a lane a word, whole groups");
  static_assert((2 * kRX - 1) * (kTJ / 2 + 5) <= TileMem<R, CAP>::kMkList, "the markers of half the rows fit");
  static_assert(2 * kRX * kRows <= marker_cap<R>(), "the segments of eight rows fit");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const TileSpan B(G.tnx(), G.tny(), i0 - 4, j0 - 2);
  const bool whole = S.nm <= TileMem<R, CAP>::kMkList;
  const int rows = whole ? kTJ : kTJ / 2;
  uint32_t zw = 0u;  // of row j0 + lane, kept by warps 0 and 1
  int n_zset = 0, n_zconf = 0;
#pragma unroll 1
  for (int r0 = 0; r0 < kTJ; r0 += rows) {
    if (!whole) {  // (neither half is without markers: one alone holds no more than the list)
      __syncthreads();
      tile_markers<R, AX, LD, CAP, T, true>(G, M, S, i0, j0, r0, rows);
    }
    tile_moves<R, AX, LD, CAP, T, true>(G, out, M, S, i0, j0, r0, rows);
#pragma unroll 1
    for (int q = r0; q < r0 + rows; q += kRows) {
      if (tid == 0) S.nc = S.ncand = S.ne = S.novf = 0;
      for (int t = tid; t < kRB; t += T) M.hc[t] = M.ovf[t] = 0u;
      for (int e = tid; e < (int)(sizeof(M.head) / 16); e += T)
        reinterpret_cast<uint4*>(M.head)[e] = make_uint4(~0u, ~0u, ~0u, ~0u);
      __syncthreads();
      if (tid < 32) list_segments(M, S, B, (2 + q) * kRW + tid, tid < kRows * kRW);
      __syncthreads();
      tile_fits<R, AX, LD, CAP, T, true>(G, out, line_only, M, S, i0, j0, q, kRows);
      if (warp < 2 && lane >= q && lane < q + kRows)
        zw = tile_centres<R>(M, B, G.tnx(), i0, j0, warp, true, &n_zset, &n_zconf);
      __syncthreads();
    }
  }
  if (warp < 2) tile_words<R, AX, LD>(G, out, M, B, i0, j0, warp, zw);
  tile_counters(S, n_zset, n_zconf, ctr, cfl_bits, status);
}

// The tile with origin (i0, j0) of one grid (one block of T threads runs it).
template <typename R, int AX, int LD, int CAP = kCandCap, int T = tile_threads<R>()>
__device__ __forceinline__ void sweep_tile(const GView<R, AX, LD>& G, const Buf<R>& out, int line_only,
                                           unsigned long long* ctr, unsigned long long* cfl_bits,
                                           int* status, const int i0, const int j0) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TileMem<R, CAP>& M = *reinterpret_cast<TileMem<R, CAP>*>(smem_raw);
  __shared__ TileCtl S;
  const int tid = threadIdx.x, warp = tid >> 5;
  if (tid < D_NUSED) S.cnt[tid] = 0;
  if (tid == 0) {
    S.nc = S.ncand = S.ne = S.novf = 0;
    S.dmax = 0ull;
  }
  tile_colours<R, AX, LD, CAP, T>(G, M, i0, j0);
  __syncthreads();
  const bool busy = tile_markers<R, AX, LD, CAP, T, false>(G, M, S, i0, j0, 0, kTJ);
  if (busy) {
    if (__builtin_expect(S.nm > marker_cap<R>(), 0)) {  // the same in every thread
      tile_dense<R, AX, LD, CAP, T>(G, out, line_only, ctr, cfl_bits, status, &S, i0, j0);
      return;
    }
    tile_moves<R, AX, LD, CAP, T, false>(G, out, M, S, i0, j0, 0, kTJ);
    tile_fits<R, AX, LD, CAP, T, false>(G, out, line_only, M, S, i0, j0, 0, kTJ);
  }
  chained_next();
  int n_zset = 0, n_zconf = 0;
  if (warp < 2) {
    const TileSpan B(G.tnx(), G.tny(), i0 - 4, j0 - 2);
    const uint32_t zw = tile_centres<R>(M, B, G.tnx(), i0, j0, warp, busy, &n_zset, &n_zconf);
    tile_words<R, AX, LD>(G, out, M, B, i0, j0, warp, zw);
  }
  tile_counters(S, n_zset, n_zconf, ctr, cfl_bits, status);
}

// One grid: block (bx, by) runs the tile at (64 bx, 32 by).  zero: a set of
// counters no tile of this launch adds to, set to zero for the next ones.
template <typename R, int AX, int T>
__global__ void __launch_bounds__(T, T == tile_threads<R>() ? tile_min_blocks<R>() : 4)
k_sweep_tile(GView<R, AX> G, Buf<R> out, int line_only, unsigned long long* ctr,
             unsigned long long* cfl_bits, int* status, unsigned long long* zero) {
  chained_start();
  if (zero && blockIdx.x + blockIdx.y == 0 && threadIdx.x < kCounterWords) zero[threadIdx.x] = 0ull;
  sweep_tile<R, AX, 0, kCandCap, T>(G, out, line_only, ctr, cfl_bits, status, blockIdx.x * kTI, blockIdx.y * kTJ);
}

// Many grids in one launch: per-grid sweep descriptors and a list of work
// items (grid, tile); a grid whose descriptor is inactive for this launch
// (its split order puts the other direction first this step) is skipped.
template <typename R, int AX>
struct SweepDesc {
  GView<R, AX> G;
  Buf<R> out;
  unsigned long long* ctr;
  unsigned long long* cfl_bits;
  int* status;
  int line_only;
  int active;
};

struct WorkItem {
  int grid, tx, ty;
};

// Square grids only: a grid's tiles are the same in both sweep directions, so
// one launch can take the first (or second) sweep of every grid, each tile in
// the direction its grid's split order puts there (x first on even steps):
// the x descriptor when it is active for this launch, else the y one.
// What the tile reads of its descriptor is read once, not again after each store
// (served grids in FP64: 3.22e10 -> 3.27e10 cells a second of GPU time).
template <typename R, int CAP = kCandCap>
__global__ void __launch_bounds__(batch_threads<R>(), batch_min_blocks<R>())
k_sweep_tile_both(const SweepDesc<R, 0>* __restrict__ dx, const SweepDesc<R, 1>* __restrict__ dy,
                  const WorkItem* __restrict__ items) {
  chained_start();
  const WorkItem it = items[blockIdx.x];
  const SweepDesc<R, 0>& X = dx[it.grid];
  if (X.active) {
    const GView<R, 0> G = X.G;
    const Buf<R> out = X.out;
    sweep_tile<R, 0, 0, CAP, batch_threads<R>()>(G, out, X.line_only, X.ctr, X.cfl_bits, X.status, it.tx * kTI,
                             it.ty * kTJ);
  } else {
    const SweepDesc<R, 1>& Y = dy[it.grid];
    const GView<R, 1> G = Y.G;
    const Buf<R> out = Y.out;
    sweep_tile<R, 1, 0, CAP, batch_threads<R>()>(G, out, Y.line_only, Y.ctr, Y.cfl_bits, Y.status, it.tx * kTI,
                             it.ty * kTJ);
  }
}

}  // namespace ebit
