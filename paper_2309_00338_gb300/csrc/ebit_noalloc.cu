// ebit_fraction_noalloc: the volume-fraction kernel for callers that cannot
// allocate device memory.
//
// Some callers of this library cannot call cudaMalloc: a host solver that
// allocates all of its device memory once at start-up and forbids allocation
// inside its time loop (cudaMalloc can synchronise the device, fail under a
// fixed memory budget, and fragment a pool the host framework manages), or a
// framework that hands this library only the buffers it owns.  For them this
// entry point computes fractions, total area and marker counts of a state held
// in the caller's own device buffers, and allocates nothing: its scratch (the
// per-block area partial sums and two marker counters) lives in the file-scope
// array below, which every GPU that loads the library holds until the process
// exits.
#include <cstdarg>
#include <cstdio>
#include <mutex>

#include "ebit.h"
#include "ebit_device.cuh"

// Sets the message returned by ebit_last_error() (defined with the other
// entry points; hidden from the exported interface).
__attribute__((visibility("hidden"))) void ebit_detail_set_error(const char* msg);

namespace {

// The sizes accepted are those of at most kMaxBlocks blocks of kBX x kBY
// vertices (the launch's own blocks are larger, so it needs fewer partials).
constexpr int kBX = 32, kBY = 8;
// Scratch: kMaxBlocks area partials (as double bit patterns), 2 marker
// counters and the count of finished blocks.
constexpr long long kMaxBlocks = 1 << 17;  // 131072 blocks of 32x8 vertices (1 MiB)
static __device__ __align__(256) unsigned long long g_noalloc_scratch[kMaxBlocks + 3];

std::mutex g_mu;
void* g_addr[1024] = {};  // scratch device address per device ordinal

ebit_status fail_na(ebit_status s, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  ebit_detail_set_error(buf);
  return s;
}

// Device address of the scratch array on the current device.  The first call
// on a device looks it up (with that device current) and caches it for the
// life of the process; a cudaDeviceReset would make the cached address stale,
// which the header tells callers.
ebit_status scratch_address(unsigned long long** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail_na(EBIT_ECUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
  if (dev < 0 || dev >= 1024) return fail_na(EBIT_ECUDA, "device ordinal %d out of range", dev);
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p)
      return fail_na(EBIT_ECUDA, "cudaGetSymbolAddress(scratch): %s", cudaGetErrorString(e));
    g_addr[dev] = p;
  }
  *out = static_cast<unsigned long long*>(g_addr[dev]);
  return EBIT_OK;
}

using ebit::edge_mask;

// A warp takes 128 columns of 4 rows, a block 32 rows.  The kernel is a
// stream: what bounds it is the colour bytes read and the fractions written
// (5 bytes a cell in float), so the colours are read one byte a lane, whole
// warps at a time, and become 32-bit words by ballot: no byte is read outside
// the caller's buffers whatever their alignment and row length, all of a
// strip's loads are in flight together, and full, empty and interface cells
// and the marker counts are word operations.  Full and empty cells are stored
// from the words and counted as integers.  The narrow FP64 pipe (one warp
// instruction per 16 cycles of an SM) only sees interface cells, listed per
// warp and evaluated by the whole block; only the markers that a cell has are read.
// 4096^2 cells in float (one disk of 3-12 cells per 29^2): 568 us with a
// thread per cell, every cell's area through a double tree; 1283 x 777 in
// double 39 us.  With the words and lists 65 us and 14.6 us (the second is the
// host's call time); 8 rows a warp take 74 us (fewer warps in flight), lists
// evaluated per warp 72 us (36 entries fill a warp and an eighth).
constexpr int kNCol = 128, kNRow = 4, kNWarps = 8;

// (double)s; conversions on the integer pipe, any float
__device__ __forceinline__ double wide(double s) { return s; }
__device__ __forceinline__ double wide(float s) {
  return (__float_as_uint(s) & 0x7f800000u) == 0x7f800000u ? (double)s : ebit::f2d(s);
}

// Reference-phase area of an interface cell (i,j) with corner mask q from its
// markers and colour vertices (Sec. 2.5), byte layout of ebit_state_host,
// double arithmetic.  Two markers on edges e1 < e2 cut a corner off (legs a
// and b) or leave a trapezoid (sides a and b), each the marker's fraction or
// its one-minus; four markers cut two corners off.
template <typename R>
__device__ __forceinline__ double cell_area(int q, const uint8_t* __restrict__ Z, const R* __restrict__ sH,
                                            const R* __restrict__ sV, int nx, int i, int j) {
  const long long w = nx + 1;
  auto marker = [&](int e) {
    return wide(e & 1 ? __ldg(&sV[j * w + i + (e == 1)]) : __ldg(&sH[(long long)(j + (e == 2)) * nx + i]));
  };
  const int em = edge_mask(q);
  if (em != 15) {
    const int e1 = __ffs(em) - 1, e2 = 31 - __clz(em);
    double a = marker(e1), b = marker(e2);
    const bool opposite = e2 - e1 == 2;
    const int c = e2 - e1 == 3 ? 0 : e2;  // the corner cut off
    if (opposite ? !(q & 1) : (c == 1 || c == 2)) a = 1.0 - a;
    if (opposite ? !(q & 1) : c >= 2) b = 1.0 - b;
    if (opposite) return 0.5 * (a + b);
    const double T = 0.5 * (a * b);
    return ((q >> c) & 1) ? T : 1.0 - T;
  }
  const double s0 = marker(0), s1 = marker(1), s2 = marker(2), s3 = marker(3);
  const int zc = Z[(long long)j * nx + i] != 0;
  const double Tsum = (q & 1) == zc ? 0.5 * ((1.0 - s0) * s1) + 0.5 * (s2 * (1.0 - s3))
                                    : 0.5 * (s3 * s0) + 0.5 * ((1.0 - s1) * (1.0 - s2));
  return zc == 0 ? Tsum : 1.0 - Tsum;
}

template <typename R>
__global__ void __launch_bounds__(32 * kNWarps, 7)
k_fraction_noalloc(const uint8_t* __restrict__ K, const uint8_t* __restrict__ Z,
                   const R* __restrict__ sH, const R* __restrict__ sV, int nx, int ny,
                   R* __restrict__ C, unsigned long long* scratch, double scale,
                   double* __restrict__ area, long long* __restrict__ counts) {
  __shared__ uint16_t s_list[kNWarps][kNCol * kNRow];  // (corner mask, row, column) of interface cells
  __shared__ double s_sum[32 * kNWarps];
  __shared__ int s_n[kNWarps], s_full[kNWarps], s_nh[kNWarps], s_nv[kNWarps];
  __shared__ bool s_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int x0 = blockIdx.x * kNCol, y0 = (blockIdx.y * kNWarps + warp) * kNRow;
  const long long w = (long long)nx + 1;
  uint16_t* list = s_list[warp];

  // the strip's colours, a halo row above and a halo column to the right
  uint8_t kb[kNRow + 1][5];
#pragma unroll
  for (int r = 0; r <= kNRow; ++r) {
    const uint8_t* row = K + (long long)(y0 + r) * w;
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      const int x = x0 + 32 * c + (c < 4 ? lane : 0);
      kb[r][c] = (y0 + r <= ny && x <= nx) ? __ldg(&row[x]) : 0;
    }
  }
  int nfull = 0, nh = 0, nv = 0, n = 0;  // the same in every lane
  uint32_t a[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) a[c] = __ballot_sync(0xffffffffu, kb[0][c] != 0);
#pragma unroll
  for (int r = 0; r < kNRow; ++r) {
    const int y = y0 + r;
    uint32_t b[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) b[c] = __ballot_sync(0xffffffffu, kb[r + 1][c] != 0);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int x = x0 + 32 * c + lane, cells = min(max(nx - (x0 + 32 * c), 0), 32);
      const uint32_t cm = cells == 32 ? 0xffffffffu : (1u << cells) - 1u;  // columns of cells
      const uint32_t a1 = __funnelshift_r(a[c], a[c + 1], 1), b1 = __funnelshift_r(b[c], b[c + 1], 1);
      nh += __popc((a[c] ^ a1) & cm);  // rows above ny read as zero
      if (y < ny) {
        nv += __popc(a[c] ^ b[c]);     // columns right of nx read as zero
        const uint32_t full = a[c] & a1 & b[c] & b1 & cm;
        const uint32_t ic = (a[c] | a1 | b[c] | b1) & ~full & cm;
        nfull += __popc(full);
        if ((ic >> lane) & 1u) {
          const int q = ((a[c] >> lane) & 1) | (((a1 >> lane) & 1) << 1) | (((b1 >> lane) & 1) << 2) |
                        (((b[c] >> lane) & 1) << 3);
          list[n + __popc(ic & ((1u << lane) - 1u))] = (uint16_t)((q << 10) | (r << 7) | (32 * c + lane));
        } else if (x < nx) {
          C[(long long)y * nx + x] = (full >> lane) & 1u ? R(1) : R(0);
        }
        n += __popc(ic);
      }
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) a[c] = b[c];
  }
  if (lane == 0) {
    s_n[warp] = n;
    s_full[warp] = nfull;
    s_nh[warp] = nh;
    s_nv[warp] = nv;
  }
  __syncthreads();
  // the warps' lists one after the other, by all threads (fixed order)
  int end[kNWarps];
#pragma unroll
  for (int q = 0; q < kNWarps; ++q) end[q] = s_n[q] + (q ? end[q - 1] : 0);
  double acc = 0.0;
  for (int t = threadIdx.x; t < end[kNWarps - 1]; t += 32 * kNWarps) {
    int q = 0, at = t;
#pragma unroll
    for (int u = 0; u < kNWarps - 1; ++u)
      if (t >= end[u]) {
        q = u + 1;
        at = t - end[u];
      }
    const int e = s_list[q][at], i = x0 + (e & 127);
    const int j = (blockIdx.y * kNWarps + q) * kNRow + ((e >> 7) & 7);
    const double f = cell_area(e >> 10, Z, sH, sV, nx, i, j);
    C[(long long)j * nx + i] = (R)f;
    acc = acc + f;
  }
  // the block's area partial and marker counts, in a fixed order
  s_sum[threadIdx.x] = acc;
  __syncthreads();
  const long long nblocks = (long long)gridDim.x * gridDim.y;
  if (warp == 0) {
    double p = s_sum[lane];
    int full = s_full[0], h = s_nh[0], v = s_nv[0];
#pragma unroll
    for (int q = 1; q < kNWarps; ++q) {
      p = p + s_sum[32 * q + lane];
      full += s_full[q];
      h += s_nh[q];
      v += s_nv[q];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) p = p + __shfl_down_sync(0xffffffffu, p, o);
    if (lane == 0) {
      p = p + (double)full;
      scratch[(long long)blockIdx.y * gridDim.x + blockIdx.x] = (unsigned long long)__double_as_longlong(p);
      if (h) atomicAdd(&scratch[kMaxBlocks], (unsigned long long)h);
      if (v) atomicAdd(&scratch[kMaxBlocks + 1], (unsigned long long)v);
      __threadfence();  // both are visible before the count says so
      s_last = atomicAdd(&scratch[kMaxBlocks + 2], 1ull) == (unsigned long long)(nblocks - 1);
    }
  }
  __syncthreads();
  if (!s_last) return;
  // the last block adds the partials up, in a fixed order
  __threadfence();
  double s = 0.0;
  long long k = threadIdx.x;
  constexpr int kT = 32 * kNWarps;
  for (; k + 7 * kT < nblocks; k += 8 * kT) {  // eight loads in flight
    unsigned long long v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = __ldcg(&scratch[k + u * kT]);
#pragma unroll
    for (int u = 0; u < 8; ++u) s = s + __longlong_as_double((long long)v[u]);
  }
  for (; k < nblocks; k += kT) s = s + __longlong_as_double((long long)__ldcg(&scratch[k]));
  s_sum[threadIdx.x] = s;
  __syncthreads();
  for (int o = kT / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) s_sum[threadIdx.x] = s_sum[threadIdx.x] + s_sum[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    *area = s_sum[0] * scale;
    if (counts) {
      counts[0] = (long long)__ldcg(&scratch[kMaxBlocks]);
      counts[1] = (long long)__ldcg(&scratch[kMaxBlocks + 1]);
    }
  }
}

}  // namespace

extern "C" ebit_status ebit_fraction_noalloc(const ebit_grid* grid, const uint8_t* K,
                                             const uint8_t* Z, const void* sH, const void* sV,
                                             void* C, double* area, int64_t* marker_counts,
                                             void* stream) {
  if (!grid || grid->nx < 1 || grid->ny < 1 || !(grid->dx > 0.0) ||
      (grid->prec != EBIT_FP64 && grid->prec != EBIT_FP32))
    return fail_na(EBIT_EINVAL, "invalid grid");
  if (!K || !Z || !sH || !sV || !C || !area) return fail_na(EBIT_EINVAL, "NULL buffer");
  const long long bx = ((long long)grid->nx + kBX) / kBX, by = ((long long)grid->ny + kBY) / kBY;
  const long long nblocks = bx * by;
  if (nblocks > kMaxBlocks)
    return fail_na(EBIT_EINVAL,
                   "grid %dx%d needs %lld blocks of 32x8 vertices; the no-allocation scratch holds "
                   "at most %lld (about 5790x5790 cells)",
                   grid->nx, grid->ny, nblocks, kMaxBlocks);
  if (by > 65535) return fail_na(EBIT_ECUDA, "launch: ny = %d is too tall", grid->ny);
  unsigned long long* scratch = nullptr;
  ebit_status s = scratch_address(&scratch);
  if (s != EBIT_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  // the counters accumulate with atomics: they must start at zero (on every
  // call, so that calls that overlapped leave nothing behind); the partials
  // are all written before they are read
  cudaError_t e = cudaMemsetAsync(scratch + kMaxBlocks, 0, 3 * sizeof(unsigned long long), st);
  if (e != cudaSuccess) return fail_na(EBIT_ECUDA, "cudaMemsetAsync: %s", cudaGetErrorString(e));
  const dim3 g((unsigned)((grid->nx + kNCol) / kNCol),
               (unsigned)((grid->ny + kNWarps * kNRow) / (kNWarps * kNRow)));
  const double scale = grid->dx * grid->dx;
  long long* counts = (long long*)marker_counts;
  if (grid->prec == EBIT_FP32)
    k_fraction_noalloc<float><<<g, 32 * kNWarps, 0, st>>>(K, Z, (const float*)sH, (const float*)sV, grid->nx,
                                                          grid->ny, (float*)C, scratch, scale, area, counts);
  else
    k_fraction_noalloc<double><<<g, 32 * kNWarps, 0, st>>>(K, Z, (const double*)sH, (const double*)sV, grid->nx,
                                                           grid->ny, (double*)C, scratch, scale, area, counts);
  e = cudaGetLastError();
  if (e != cudaSuccess) return fail_na(EBIT_ECUDA, "launch: %s", cudaGetErrorString(e));
  return EBIT_OK;
}
