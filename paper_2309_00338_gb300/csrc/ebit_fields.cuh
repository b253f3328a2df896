// Fused fields kernel: volume fractions C, height-function curvature kappa,
// the area (per-tile partial sums, added up by the launch's last tile) and
// the marker counts of a state (Sec. 2.5), one
// 64x32 tile of cells per block with a 3-cell halo for the 7x3 height
// stencils.
//
// Colours are read as bit rows; full, empty and interface cells are word
// operations on them.  A full or empty cell has C equal to its corner colour
// exactly: C and a NaN kappa are stored four cells at a time from the words,
// and the interface cells, listed in region order, overwrite theirs.  FP64
// work is confined to them, and there to what has to be double: the area is
// added up as integers (in any order; a tile with next to no area in double)
// and so are the heights of the double form.  What bounds it then is instruction
// issue and the dense stores: 4096^2 cells with 1.2 M interface cells, 118 -> 91
// us in FP32 and 322 -> 142 us in FP64 (with double heights and sums the FP64 pipe
// was busy 82% of the time); 3.0 and 3.8 TB/s of the dense model, state read and
// C, kappa written.
#pragma once
#include "ebit_device.cuh"

namespace ebit {

constexpr int kFX = 64, kFY = 32, kFH = 3;
constexpr int kFRX = kFX + 2 * kFH, kFRY = kFY + 2 * kFH;  // region cells (70 x 38)
constexpr int kFVX = kFRX + 1, kFVY = kFRY + 1;            // region vertices (71 x 39)
constexpr int kFW = 3;                                     // words per region bit row
constexpr int kFP = 72;  // row pitch of the region's fractions: cell lx is entry lx + 1, so that
                         // groups of four entries are groups of four of the tile's columns
// Threads per tile and blocks per SM the kernel is compiled for: 4096^2 cells
// take 91 us in FP32 with eight blocks of 32 registers (a few spilled), 98 with
// six, 109 with five; in FP64 142 us with six and with five, 171 with seven.
template <typename R> __host__ __device__ constexpr int field_threads() { return 256; }
template <typename R> __host__ __device__ constexpr int fields_min_blocks() { return sizeof(R) == 4 ? 8 : 6; }

// Reference-phase area of interface cell (i,j) in cell units from its corner
// mask q, centre colour and marker fractions; double arithmetic.  Two markers
// on edges e1 < e2 cut a corner off (legs a and b) or leave a trapezoid (sides
// a and b), each the marker's fraction or its one-minus: one sequence for all
// of them, so that a warp whose cells differ repeats no FP64 work.
template <typename R>
__device__ __forceinline__ double fraction_of(int q, int zc, const R* sH, const R* sV,
                                              const Dims& d, int i, int j) {
  const long long q0 = (long long)j * d.P + i;
  // exact conversions on the integer pipe
  auto marker = [&](int e) {
    const long long at = e == 1 ? q0 + 1 : e == 2 ? q0 + d.P : q0;
    return in_range(at, e & 1 ? d.nV() : d.nH()) ? to_d<R>(e & 1 ? sV[at] : sH[at]) : 0.0;
  };
  const int em = edge_mask(q);
  if (em != 15) {
    const int e1 = __ffs(em) - 1, e2 = 31 - __clz(em);
    double a = marker(e1), b = marker(e2);
    const bool opposite = e2 - e1 == 2;
    const int c = e2 - e1 == 3 ? 0 : e2;  // the corner cut off
    if (opposite ? !(q & 1) : (c == 1 || c == 2)) a = 1.0 - a;
    if (opposite ? !(q & 1) : c >= 2) b = 1.0 - b;
    double f = d_scale<-1>(opposite ? a + b : a * b);
    if (!opposite && !((q >> c) & 1)) f = 1.0 - f;
    return f;
  }
  // four markers: the two corners of the other colour than the centre are cut
  // off (corners 1 and 3 when corner 0 has the centre's colour, else 0 and 2)
  const double s0 = marker(0), s1 = marker(1), s2 = marker(2), s3 = marker(3);
  const double Tsum = (q & 1) == zc ? 0.5 * ((1.0 - s0) * s1) + 0.5 * (s2 * (1.0 - s3))
                                    : 0.5 * (s3 * s0) + 0.5 * ((1.0 - s1) * (1.0 - s2));
  return zc == 0 ? Tsum : 1.0 - Tsum;
}

__device__ __forceinline__ int fgetb(const uint32_t* w, int lx, int ly) {
  return (w[ly * kFW + (lx >> 5)] >> (lx & 31)) & 1;
}
__device__ __forceinline__ uint32_t fshr1(const uint32_t* w, int ly, int wi) {
  uint32_t v = w[ly * kFW + wi] >> 1;
  if (wi + 1 < kFW) v |= w[ly * kFW + wi + 1] << 31;
  return v;
}
// Corner mask of region cell (lx, ly); kw has a word after its last row.
__device__ __forceinline__ int fcorners(const uint32_t* kw, int lx, int ly) {
  const uint32_t* q = kw + ly * kFW + (lx >> 5);
  const int lo = __funnelshift_r(q[0], q[1], lx & 31) & 3;
  const int up = __funnelshift_r(q[kFW], q[kFW + 1], lx & 31) & 3;
  return lo | ((up & 2) << 1) | ((up & 1) << 3);
}

// A fraction 0 <= f <= 1 in units of 2^-60, rounded down; a positive one is at
// least one unit, so that only 0 is 0 and only 1 is 2^60.
typedef unsigned long long fix60;
constexpr fix60 kFixOne = 1ull << 60;
__device__ __forceinline__ fix60 to_fix60(double f) {
  const unsigned long long u = (unsigned long long)dbits(f) & 0x7fffffffffffffffull;
  const int sh = 1015 - (int)(u >> 52);  // f = sig 2^(8 - sh) units
  const unsigned long long sig = significand(u);
  if (u == 0) return 0;
  if (sh <= 0) return sig << -sh;
  return sh > 52 ? 1ull : sig >> sh;
}
// (double)v 2^-U for |v| < 2^63, to 53 bits (rounded toward zero).
template <int U>
__device__ __forceinline__ double from_fix(long long v) {
  if (v == 0) return 0.0;
  const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int p = 63 - __clzll((long long)a);
  const unsigned long long sig = p > 52 ? a >> (p - 52) : a << (52 - p);
  return __longlong_as_double((long long)((v < 0 ? 1ull << 63 : 0ull) |
                                          ((unsigned long long)(1023 + p - U) << 52) | (sig & (kImplicit - 1))));
}

// The area of a tile's listed interface cells (of the region; those of its halo
// are left out) in double, by one warp in a fixed order: every lane gets the sum.
// Units of 2^-60 lose relative accuracy on areas far below a cell; few tiles
// hold nothing else.
template <typename R>
__device__ __forceinline__ double small_area(const uint16_t* lst, int n, const uint32_t* kw, const uint32_t* zw,
                                             const R* sH, const R* sV, const Dims& d, int rx0, int ry0) {
  double a = 0.0;
#pragma unroll 1
  for (int e = threadIdx.x & 31; e < n; e += 32) {
    const int t = lst[e] & 0x7fff, ly = t / kFP, lx = t - ly * kFP - 1;
    if (lx < kFH || lx >= kFH + kFX || ly < kFH || ly >= kFH + kFY) continue;
    a = a + fraction_of(fcorners(kw, lx, ly), fgetb(zw, lx, ly), sH, sV, d, rx0 + lx, ry0 + ly);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a = a + __shfl_xor_sync(0xffffffffu, a, o);
  return a;
}

// a 2^-12 + b 2^-60 for a < 2^24 and b < 2^48, rounded, on the integer pipe.
__device__ __forceinline__ double tile_area(unsigned a, unsigned long long b) {
  if (a == 0u) return from_fix<60>((long long)b);
  const int p = 31 - __clz((int)a), drop = p - 4;  // bits of b beyond the 53
  unsigned long long sig = ((unsigned long long)a << (52 - p)) + (drop >= 0 ? b >> drop : b << -drop);
  if (drop > 0) sig += (b >> (drop - 1)) & 1u;
  return __longlong_as_double((long long)(((unsigned long long)(1023 - 12 + p) << 52) + (sig - kImplicit)));
}

// What the height functions add up.  The float form adds floats in stencil
// order, as the definition spells it.  The double form adds integers in units
// of 2^-60: exact sums, finer than the double fractions they are made of
// (2^-54 for those above a half), and none of the 21 additions of a stencil
// takes a slot of the FP64 pipe.
template <typename R> struct HeightOf;
template <> struct HeightOf<float> {
  typedef float T;
  static __device__ __forceinline__ float one() { return 1.0f; }
  static __device__ __forceinline__ float of(double, float f) { return f; }
};
template <> struct HeightOf<double> {
  typedef fix60 T;
  static __device__ __forceinline__ fix60 one() { return kFixOne; }
  static __device__ __forceinline__ fix60 of(double f, double) { return to_fix60(f); }
};
__device__ __forceinline__ bool is_one(float h) { return one_bits(h); }
__device__ __forceinline__ bool is_one(fix60 h) { return h == kFixOne; }
__device__ __forceinline__ bool is_zero(float h) { return zero_bits(h); }
__device__ __forceinline__ bool is_zero(fix60 h) { return h == 0; }

// kappa from the heights of the three columns.
__device__ __forceinline__ float height_kappa(const float h[3], float dx) {
  const float hp = (h[2] - h[0]) * 0.5f;
  const float hpp = (h[2] - h[1]) - (h[1] - h[0]);
  const float qv = 1.0f + hp * hp;
  const float den = dx * (qv * sqrt(qv));
  return -hpp / den;
}
__device__ __forceinline__ double height_kappa(const fix60 h[3], double dx) {
  // With one end cell full and the other empty a height lies in [1, 6] cells:
  // first differences are below 5 cells, which a signed word of 2^-60 cells
  // holds (8), and the second difference is below 10, which takes units of 2^-59.
  const long long up = (long long)(h[2] - h[1]), down = (long long)(h[1] - h[0]);
  const double hp = from_fix<61>(up + down);  // half their sum
  const double hpp = from_fix<59>((up >> 1) - (down >> 1));
  const double qv = 1.0 + hp * hp;
  const double den = dx * (qv * d_sqrt(qv));
  return -d_div(hpp, den);
}

// Heights run along y when the segments' |dx| add up to at least their |dy|.
template <typename R>
__device__ __forceinline__ bool along_y(int ns, const int seg[2][2], const R px[4], const R py[4], R* margin) {
  R ax = R(0), ay = R(0);
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    if (s >= ns) break;
    ax = ax + fabs(px[seg[s][1]] - px[seg[s][0]]);
    ay = ay + fabs(py[seg[s][1]] - py[seg[s][0]]);
  }
  *margin = fabs(ax - ay);
  return ax >= ay;
}
__device__ __forceinline__ bool heights_along_y(int ns, const int seg[2][2], const float px[4], const float py[4]) {
  float m;
  return along_y(ns, seg, px, py, &m);
}
// The double form decides on float estimates (each coordinate within 2^-20, so
// the sums' difference within 2^-17) and takes the FP64 pipe only where they
// are too close to tell.
__device__ __forceinline__ bool heights_along_y(int ns, const int seg[2][2], const double px[4],
                                                const double py[4]) {
  float fx[4], fy[4], m;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    fx[e] = d_mid(px[e]) ? d_top(px[e]) : 0.0f;
    fy[e] = d_mid(py[e]) ? d_top(py[e]) : 0.0f;
  }
  const bool y = along_y(ns, seg, fx, fy, &m);
  if (m > 0x1p-16f) return y;
  double md;
  return along_y(ns, seg, px, py, &md);
}

// Dense stores of four consecutive values of a row (16-byte aligned).
__device__ __forceinline__ void store4(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void store4(double* p, double a, double b, double c, double d) {
  reinterpret_cast<double2*>(p)[0] = make_double2(a, b);
  reinterpret_cast<double2*>(p)[1] = make_double2(c, d);
}
__device__ __forceinline__ void store4(fix60* p, fix60 a, fix60 b, fix60 c, fix60 d) {
  reinterpret_cast<ulonglong2*>(p)[0] = make_ulonglong2(a, b);
  reinterpret_cast<ulonglong2*>(p)[1] = make_ulonglong2(c, d);
}

// Where the tiles' area partials are summed: with `done` set, the last tile
// of the launch to finish (counted on *done, which it then resets to 0) adds
// all n partials in a fixed order (thread t takes partials t, t + 256, ...,
// then a tree over the threads), so the area does not depend on which tile
// finishes last, and no separate reduction launch is needed.
struct AreaSum {
  unsigned* done = nullptr;
  long long n = 0;
  double scale = 0.0;
  double* area = nullptr;
  // the counters of the step's first sweep, which block (0, 0) adds to the
  // launch's own and sets to zero
  unsigned long long* first = nullptr;
};

// The tile (bx, by) of one grid; its area partial goes to partial[slot].
// With ghf_list, the interface cells left without a 7x3 stencil are
// appended to it (ghf_count, zeroed before the launch, counts them): one
// global atomic per tile reserves its slice.
template <typename R>
__device__ __forceinline__ void fields_tile(const uint32_t* K,
                                            const uint32_t* Z,
                                            const R* sH, const R* sV,
                                            const Dims& d, R dx, R* C, R* kappa, double* partial,
                                            long long slot, unsigned long long* ctr, int bx, int by,
                                            int* ghf_list = nullptr, unsigned* ghf_count = nullptr,
                                            AreaSum sum = AreaSum()) {
  constexpr int kFieldThreads = field_threads<R>();
  typedef HeightOf<R> H;
  typedef typename H::T HT;
  __shared__ uint32_t kw[kFVY * kFW + 1];  // vertex colours
  __shared__ uint32_t zw[kFRY * kFW];  // centre colours
  __shared__ uint32_t fw[kFRY * kFW + 1];  // full cells
  __shared__ uint32_t iw[kFRY * kFW];      // interface cells
  __shared__ __align__(16) HT cs[kFRY * kFP];  // fractions of the region
  __shared__ uint16_t lst[kFRY * kFRX];        // interface cells, in region order (entries of cs)
  __shared__ int s_cnt[D_NUSED];
  // the tile's area: full cells, and its interface cells' in units of 2^-60
  // cells, s_area + s_area_hi 2^48
  __shared__ unsigned long long s_area;
  __shared__ unsigned s_area_hi, s_full;
  __shared__ unsigned s_nghf, s_ghf_base;
  __shared__ int s_last, s_n;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int i0 = bx * kFX, j0 = by * kFY;
  const int rx0 = i0 - kFH, ry0 = j0 - kFH;
  if (tid < D_NUSED) s_cnt[tid] = 0;
  if (tid == 0) {
    s_area = 0ull;
    s_area_hi = s_full = 0u;
    s_nghf = 0u;
  }
  // region columns / rows inside the grid
  const int vx0 = max(0, -rx0), vx1 = min(kFVX - 1, d.nx - rx0);  // vertices
  const int cx1 = min(kFRX - 1, d.nx - 1 - rx0);                  // cells
  const int vy0 = max(0, -ry0), vy1 = min(kFVY - 1, d.ny - ry0);
  const int cy1 = min(kFRY - 1, d.ny - 1 - ry0);
  int n_h = 0, n_v = 0, n_invalid = 0;

  // colour bits
  for (int t = tid; t < (kFVY + kFRY) * kFW; t += kFieldThreads) {
    const bool zpl = t >= kFVY * kFW;
    const int u = zpl ? t - kFVY * kFW : t;
    const int ly = u / kFW, wi = u % kFW, y = ry0 + ly, x0 = rx0 + 32 * wi;
    uint32_t v = 0u;
    if (!zpl && ly >= vy0 && ly <= vy1)
      v = row_bits(K + (long long)y * d.kw, d.kw, x0) & span_mask(wi, vx0, vx1);
    if (zpl && ly >= vy0 && ly <= cy1)
      v = row_bits(Z + (long long)y * d.zw, d.zw, x0) & span_mask(wi, vx0, cx1);
    (zpl ? zw : kw)[u] = v;
  }
  __syncthreads();

  // full / interface cells; the tile's full cells and markers are counted
  constexpr int kWords = kFRY * kFW;  // 114
  int full = 0;
  for (int t = tid; t < kWords; t += kFieldThreads) {
    const int ly = t / kFW, wi = t % kFW;
    uint32_t f = 0u, ic = 0u;
    if (ly >= vy0 && ly <= cy1) {
      const uint32_t a = kw[t], a1 = fshr1(kw, ly, wi), b = kw[t + kFW], b1 = fshr1(kw, ly + 1, wi);
      const uint32_t cm = span_mask(wi, vx0, cx1);
      f = a & a1 & b & b1 & cm;
      ic = (a | a1 | b | b1) & ~f & cm;
    }
    fw[t] = f;
    iw[t] = ic;
    if (ly >= kFH && ly < kFH + kFY) {
      const uint32_t tile = span_mask(wi, kFH, kFH + kFX - 1);
      full += __popc(f & tile);
      // markers on the tile's vertices' right and upper edges
      if (ly <= vy1) {
        const uint32_t a = kw[t];
        n_h += __popc((a ^ fshr1(kw, ly, wi)) & tile & span_mask(wi, vx0, cx1));
        if (ly + 1 <= vy1) n_v += __popc((a ^ kw[t + kFW]) & tile & span_mask(wi, vx0, vx1));
      }
    }
  }
  {
    const int fsum = __reduce_add_sync(0xffffffffu, full);
    if (lane == 0 && fsum) atomicAdd(&s_full, (unsigned)fsum);
  }
  __syncthreads();

  // interface list in region order: two words a lane of the first two warps,
  // the cells before the second warp's words counted by itself
  if (warp < 2) {
    static_assert(kWords <= 128, "two words a lane, two warps");
    const int t = 64 * warp + 2 * lane;
    uint32_t w0 = t < kWords ? iw[t] : 0u, w1 = t + 1 < kWords ? iw[t + 1] : 0u;
    const int n = __popc(w0) + __popc(w1);
    const int before = warp ? __reduce_add_sync(0xffffffffu, __popc(iw[lane]) + __popc(iw[lane + 32])) : 0;
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    int pos = before + incl - n;
    if (warp == 1 && lane == 31) s_n = pos + n;
    const int r0 = (t / kFW) * kFP + 32 * (t % kFW) + 1;
    const int r1 = ((t + 1) / kFW) * kFP + 32 * ((t + 1) % kFW) + 1;
    for (; w0; w0 &= w0 - 1) lst[pos++] = (uint16_t)(r0 + __ffs(w0) - 1);
    for (; w1; w1 &= w1 - 1) lst[pos++] = (uint16_t)(r1 + __ffs(w1) - 1);
  }
  // Full and empty cells, four at a time: the region's for the heights, and
  // the tile's straight to C, with NaN to kappa (the interface cells' entries
  // are written after the next barriers).
  {
    const bool vec = ((reinterpret_cast<uintptr_t>(C) | reinterpret_cast<uintptr_t>(kappa)) & 15) == 0;
    const HT one = H::one();
    const R nan = R(NAN);
    constexpr int kQ = kFP / 4;
    for (int g = (tid + kFieldThreads - 64) % kFieldThreads; g < kFRY * kQ; g += kFieldThreads) {
      const int ly = g / kQ, qx = g - ly * kQ, lx = 4 * qx - 1;  // its first cell (-1 for qx = 0)
      const int w = ly * kFW + (lx >> 5);
      const uint32_t f = qx == 0 ? fw[ly * kFW] << 1 : __funnelshift_r(fw[w], fw[w + 1], lx & 31);
      store4(&cs[ly * kFP + 4 * qx], f & 1 ? one : HT(0), f & 2 ? one : HT(0), f & 4 ? one : HT(0),
             f & 8 ? one : HT(0));
      const int i = i0 + 4 * qx - 4, j = ry0 + ly;
      if (qx == 0 || qx > kFX / 4 || ly < kFH || ly >= kFH + kFY || j >= d.ny || i >= d.nx) continue;
      if (!in_range((long long)j * d.P + min(i + 3, d.nx - 1), d.nV())) continue;  // this group's last cell
      R* Cp = C + (long long)j * d.P + i;
      R* Kp = kappa + (long long)j * d.P + i;
      const R c0 = f & 1 ? R(1) : R(0), c1 = f & 2 ? R(1) : R(0), c2 = f & 4 ? R(1) : R(0), c3 = f & 8 ? R(1) : R(0);
      if (vec && i + 3 < d.nx) {
        store4(Cp, c0, c1, c2, c3);
        store4(Kp, nan, nan, nan, nan);
      } else {
        Cp[0] = c0;
        Kp[0] = nan;
        if (i + 1 < d.nx) { Cp[1] = c1; Kp[1] = nan; }
        if (i + 2 < d.nx) { Cp[2] = c2; Kp[2] = nan; }
        if (i + 3 < d.nx) { Cp[3] = c3; Kp[3] = nan; }
      }
    }
  }
  __syncthreads();

  // interface fractions (FP64 on full warps) and the tile's area, added up as
  // integers: the same in any order
  const int nlist = s_n;
  fix60 acc = 0;  // at most 11 cells a thread: below 2^64
  static_assert((kFRY * kFRX + kFieldThreads - 1) / kFieldThreads <= 15, "a thread's area fits");
  for (int e = tid; e < nlist; e += kFieldThreads) {
    const int t = lst[e], ly = t / kFP, lx = t - ly * kFP - 1;
    const int i = rx0 + lx, j = ry0 + ly;
    const double f = fraction_of(fcorners(kw, lx, ly), fgetb(zw, lx, ly), sH, sV, d, i, j);
    const R c = (R)f;
    cs[t] = H::of(f, c);
    if (lx >= kFH && lx < kFH + kFX && ly >= kFH && ly < kFH + kFY) {
      acc += to_fix60(f);
      if (in_range((long long)j * d.P + i, d.nV())) C[(long long)j * d.P + i] = c;
    }
  }
  if (__any_sync(0xffffffffu, acc != 0)) {
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)acc & 0xffffffu);
    const unsigned mid = __reduce_add_sync(0xffffffffu, (unsigned)(acc >> 24) & 0xffffffu);
    const unsigned hi = __reduce_add_sync(0xffffffffu, (unsigned)(acc >> 48));
    if (lane == 0) {
      atomicAdd(&s_area, lo + ((unsigned long long)mid << 24));
      atomicAdd(&s_area_hi, hi);
    }
  }
  __syncthreads();
  // the tile's partial, and its count towards the launch's last tile, by the
  // last warp: it rarely has curvature work, so the fence and the counter's
  // round trip overlap the other threads' curvature
  if (warp == kFieldThreads / 32 - 1) {
    const unsigned long long lo = s_area, b = lo & ((1ull << 48) - 1);
    const unsigned a = (s_full << 12) + s_area_hi + (unsigned)(lo >> 48);  // at most 2048 cells
    double p = tile_area(a, b);
    // Each cell's area is cut by less than a unit, and only below 2^-8.  Where
    // the cells hold fewer than 2^50 units on average (that many keep the
    // relative error below 2^-50) and there is no full cell, they are added in
    // double.
    if (s_full == 0u && a < 0x4000u && (a | b) != 0u && (((unsigned long long)a << 48) | b) < (unsigned long long)nlist << 50)
      p = small_area<R>(lst, nlist, kw, zw, sH, sV, d, rx0, ry0);
    if (lane == 31) {
      partial[slot] = p;
      s_last = 0;
      if (sum.done) {
        __threadfence();  // the partial is visible before the count says so
        s_last = atomicAdd(sum.done, 1u) == (unsigned)(sum.n - 1);
      }
    }
  }

  chained_next();
  // height-function curvature of the tile's interface cells
  for (int e = tid; e < nlist; e += kFieldThreads) {
    const int ci = lst[e], ly = ci / kFP, lx = ci - ly * kFP - 1;
    if (lx < kFH || lx >= kFH + kFX || ly < kFH || ly >= kFH + kFY) continue;
    const int i = rx0 + lx, j = ry0 + ly;
    const int q = fcorners(kw, lx, ly);
    R out = R(NAN);
    int seg[2][2];
    const int ns = segments(q, edge_mask(q) == 15 ? fgetb(zw, lx, ly) : 0, seg);
    const long long q0 = (long long)j * d.P + i, q2 = q0 + d.P;
    const R px[4] = {in_range(q0, d.nH()) ? sH[q0] : R(0), R(1),
                     in_range(q2, d.nH()) ? sH[q2] : R(0), R(0)};
    const R py[4] = {R(0), in_range(q0 + 1, d.nV()) ? sV[q0 + 1] : R(0), R(1),
                     in_range(q0, d.nV()) ? sV[q0] : R(0)};
    const bool ycol = heights_along_y(ns, seg, px, py);
    bool valid = ycol ? (i - 1 >= 0 && i + 1 <= d.nx - 1 && j - 3 >= 0 && j + 3 <= d.ny - 1)
                      : (j - 1 >= 0 && j + 1 <= d.ny - 1 && i - 3 >= 0 && i + 3 <= d.nx - 1);
    if (valid) {
      const int along = ycol ? kFP : 1, across = ycol ? 1 : kFP;
      HT h[3];
      int orient[3];
#pragma unroll
      for (int m = -1; m <= 1; ++m) {
        const HT* c = &cs[ci + m * across - 3 * along];
        const HT lo = c[0], hi = c[6 * along];
        HT a = HT(0) + lo;
#pragma unroll
        for (int s = 1; s < 6; ++s) a = a + c[s * along];
        h[m + 1] = a + hi;
        orient[m + 1] = (is_one(lo) && is_zero(hi)) ? 1 : (is_zero(lo) && is_one(hi)) ? -1 : 0;
      }
      valid = orient[0] != 0 && orient[0] == orient[1] && orient[1] == orient[2];
      if (valid) out = height_kappa(h, dx);
    }
    if (!valid) {
      n_invalid += 1;
      if (ghf_list) {  // flag the entry for the generalised fallbacks
        lst[e] = (uint16_t)(ci | 0x8000);
        atomicAdd(&s_nghf, 1u);
      }
    }
    if (in_range((long long)j * d.P + i, d.nV())) kappa[(long long)j * d.P + i] = out;
  }
  // the counters this kernel keeps (markers, cells without a height stencil)
  {
    const int h = __reduce_add_sync(0xffffffffu, n_h), v = __reduce_add_sync(0xffffffffu, n_v);
    const int x = __reduce_add_sync(0xffffffffu, n_invalid);
    if (lane == 0 && h) atomicAdd(&s_cnt[D_NH], h);
    if (lane == 0 && v) atomicAdd(&s_cnt[D_NV], v);
    if (lane == 0 && x) atomicAdd(&s_cnt[D_HF_INVALID], x);
  }
  __syncthreads();
  if (tid < D_NUSED && s_cnt[tid] != 0) atomicAdd(&ctr[tid], (unsigned long long)s_cnt[tid]);
  if (ghf_list) {
    const unsigned nflag = s_nghf;  // final: its atomics precede the last barrier
    if (nflag != 0u) {              // the same in every thread
      __syncthreads();              // every thread has read it
      if (tid == 0) {
        s_ghf_base = atomicAdd(ghf_count, nflag);
        s_nghf = 0u;
      }
      __syncthreads();
      for (int e = tid; e < nlist; e += kFieldThreads) {
        const int ci = lst[e];
        if (!(ci & 0x8000)) continue;
        const int t = ci & 0x7fff;
        const int i = rx0 + t % kFP - 1, j = ry0 + t / kFP;
        ghf_list[s_ghf_base + atomicAdd(&s_nghf, 1u)] = j * d.nx + i;
      }
    }
  }
  __syncthreads();
  if (s_last) {  // the same in every thread of the block: set before a barrier
    static_assert(field_threads<R>() == 256, "the fixed area order assumes 256 threads");
    __shared__ double red[256];
    __threadfence();
    double a = 0.0;
    long long b = tid;
    for (; b + 7 * 256 < sum.n; b += 8 * 256) {  // eight loads in flight, added in order
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __ldcg(&partial[b + u * 256]);
#pragma unroll
      for (int u = 0; u < 8; ++u) a = a + v[u];
    }
    for (; b < sum.n; b += 256) a = a + __ldcg(&partial[b]);
    red[tid] = a;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
      if (tid < s) red[tid] = red[tid] + red[tid + s];
      __syncthreads();
    }
    if (tid == 0) {
      *sum.area = red[0] * sum.scale;
      *sum.done = 0u;  // ready for the next launch (stream order)
    }
  }
}

template <typename R>
__global__ void __launch_bounds__(field_threads<R>(), fields_min_blocks<R>())
k_fields_tile(const uint32_t* K, const uint32_t* Z,
              const R* sH, const R* sV, Dims d, R dx, R* C, R* kappa,
              double* partial, unsigned long long* ctr, int* ghf_list, unsigned* ghf_count,
              AreaSum sum) {
  chained_start();
  if (sum.first && blockIdx.x + blockIdx.y == 0 && threadIdx.x < kCounterWords) {
    const unsigned long long v = sum.first[threadIdx.x];
    sum.first[threadIdx.x] = 0ull;
    if (v && threadIdx.x < kCounters) atomicAdd(&ctr[threadIdx.x], v);
    if (v && threadIdx.x == kCounters) atomicMax(&ctr[kCounters], v);  // bits of a positive double
  }
  fields_tile<R>(K, Z, sH, sV, d, dx, C, kappa, partial,
                 (long long)blockIdx.y * gridDim.x + blockIdx.x, ctr, blockIdx.x, blockIdx.y, ghf_list,
                 ghf_count, sum);
}

// Many grids in one launch (work items: grid, tile).
template <typename R>
struct FieldDesc {
  const uint32_t* K;
  const uint32_t* Z;
  const R* sH;
  const R* sV;
  Dims d;
  R dx;
  R* C;
  R* kappa;
  double* partial;
  unsigned long long* ctr;
  int tiles_x;
  int* ghf_list;         // EBIT_CURV_GHF grids: their list of cells without a 7x3 stencil
  unsigned* ghf_count;   // (null otherwise)
};

struct FieldItem {
  int grid, tx, ty;
};

template <typename R>
__global__ void __launch_bounds__(field_threads<R>(), fields_min_blocks<R>())
k_fields_tile_batch(const FieldDesc<R>* __restrict__ descs, const FieldItem* __restrict__ items) {
  chained_start();
  const FieldItem it = items[blockIdx.x];
  const FieldDesc<R>& D = descs[it.grid];
  fields_tile<R>(D.K, D.Z, D.sH, D.sV, D.d, D.dx, D.C, D.kappa, D.partial,
                 (long long)it.ty * D.tiles_x + it.tx, D.ctr, it.tx, it.ty, D.ghf_list, D.ghf_count);
}

}  // namespace ebit
