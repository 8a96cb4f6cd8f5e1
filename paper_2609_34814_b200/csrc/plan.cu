// Planning kernels: block mask -> per-head execution order of the query blocks.
//
// Algorithm 2 of the WaveAlign paper with the adaptive skip of Section 4.5 in front:
//   row block counts n_i and column counts c = M^T 1, guard statistics and decision,
//   Algorithm 1 (matrix-free centred subspace iteration, T sweeps, then the Rayleigh-Ritz
//   ordering), polar angle (Eq. 4), angular sort, wave-sized buckets, descending-count sort
//   inside each bucket.
//
// Layout of the work: the mask is kept as a bitmap M and its bit transpose Mt (both stay
// resident in L2; a bitmap is smaller than index lists once density exceeds 1/32).  One launch
// transposes and counts; a second plans: a thread-block cluster of 1 to 16 CTAs of 1024 threads
// (as many as the device holds at once for the given number of heads) owns one head and runs every
// step for it, with the iteration blocks X, Y, Z (fp64) in shared memory, so no step needs a
// grid-wide barrier.  The CTAs of a cluster keep identical copies of the state: the cheap steps
// (QR, rotation) are done by each of them in the same order, the two mask products of an iteration
// are split by rows and each result is written into every copy through distributed shared memory;
// the lead CTA does the sorts and writes the outputs.  The products are exact integer sums on the
// matrix units (multiply_rows), the floating-point reductions use a fixed thread -> element
// assignment and a fixed combination tree, so a plan is reproducible bit for bit and does not
// depend on the cluster size.  Shapes whose digits do not fit shared memory walk the set bits in fp64
// instead (gather_rows), also in an order that does not depend on which CTA takes a row.
#include <cfloat>
#include <climits>
#include <cmath>
#include <mutex>
#include "host_common.h"

namespace {

using u64 = unsigned long long;
constexpr int kPlanThreads = 1024;
constexpr int kPlanWarps = kPlanThreads / 32;
constexpr int kMaxSort = 16384;          // largest padded row count the in-smem sort takes
constexpr size_t kSmemMax = 232448;      // 227 KB opt-in limit per CTA on sm_100
constexpr int kMaxMerge = (kSmemMax - 2048) / 24;     // rows whose two sort buffers fit: 9,600

// ------------------------------------------------------------------ format conversion

// index lists -> bitmap and row counts; one warp per (head, row), which collects the row in shared memory, kCsrCols
// columns at a time, and writes whole words: no zeroing pass and no atomics on global memory (109 us
// for 79 M indices that way).  Bound by instructions: a lane takes kRun consecutive entries in two 16-byte loads, looks once
// whether all are in range, and sets a bit for each (lanes of an ascending list then mostly have words of their own).
// Collecting the bits of a word in a register first, with the branches that takes, and entry by entry range checks: 45 us for the
// 19.7 M entries of 49,152 rows, now 27.  A run that sticks out of the row reads the row's first or last entry again instead.
// PIECES: rows of more than kCsrCols columns, which read their list once a piece; most runs of an ascending list lie in one piece,
// in front of it or behind it, and the others keep their eight entries in registers too (2,048 rows of 16,384 columns, a tenth
// set: 8.0 us, with the entries loaded again one by one 20.7).  The form for one piece does not carry the offset.
constexpr int kCsrCols = 8192, kCsrWarps = 8;
template <bool PIECES>
__global__ void __launch_bounds__(kCsrWarps * 32) k_csr_to_bitmap(const int* __restrict__ row_ptr, const int* __restrict__ idx,
                                                                  u64* __restrict__ bits, long long n_rows, int wq, int n_kv,
                                                                  int m_b, int* __restrict__ nnz, int* __restrict__ nnz_out,
                                                                  int* dev_status) {
  __shared__ __align__(8) unsigned words[kCsrWarps][kCsrCols / 32];
  waveal::let_next_kernel_start();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long row = (long long)blockIdx.x * kCsrWarps + warp;
  if (row >= n_rows) return;
  unsigned* my = words[warp];
  const int lo = row_ptr[row], len = row_ptr[row + 1] - lo;
  const int* list = idx + lo;
  constexpr int kRun = 8;
  // (runs start at 16-byte boundaries, the row's first maybe before it)
  const int first = len > 0 ? -(int)((reinterpret_cast<uintptr_t>(list) >> 2) & 3) : 0;
  int count = 0;
  for (int c0 = 0; c0 < n_kv; c0 += kCsrCols) {
    const int cols = min(kCsrCols, n_kv - c0), n = (cols + 63) / 64;
    for (int w = lane; w < 2 * n; w += 32) my[w] = 0u;
    __syncwarp();
    for (int e = first + lane * kRun; e < len; e += 32 * kRun) {
      int j[kRun];
      if (e >= 0 && e <= len - kRun) {
        const int4 a = *reinterpret_cast<const int4*>(list + e), b = *reinterpret_cast<const int4*>(list + e + 4);
        j[0] = a.x; j[1] = a.y; j[2] = a.z; j[3] = a.w;
        j[4] = b.x; j[5] = b.y; j[6] = b.z; j[7] = b.w;
      } else {
#pragma unroll
        for (int i = 0; i < kRun; ++i) j[i] = list[min(max(e + i, 0), len - 1)];
      }
      auto set = [&](int v) { atomicOr(&my[(PIECES ? v - c0 : v) >> 5], 1u << (v & 31)); };
      auto report = [&](int v) {
        if (c0 == 0 && dev_status && atomicCAS(dev_status, 0, WAVEAL_ERR_BAD_MASK) == 0) {
          dev_status[1] = 1; dev_status[2] = (int)(row / m_b); dev_status[3] = v;
        }
      };
      unsigned top = 0, bottom = ~0u, entry = 0;     // positions in this piece, and the entries themselves
#pragma unroll
      for (int i = 0; i < kRun; ++i) {
        const unsigned k = (unsigned)j[i] - (PIECES ? (unsigned)c0 : 0u);
        top = max(top, k);
        if (PIECES) { bottom = min(bottom, k); entry = max(entry, (unsigned)j[i]); }
      }
      if (top < (unsigned)cols) {
#pragma unroll
        for (int i = 0; i < kRun; ++i) set(j[i]);
      } else if (PIECES) {
        if (bottom < (unsigned)cols || entry >= (unsigned)n_kv) {      // (else all eight belong to other pieces)
#pragma unroll
          for (int i = 0; i < kRun; ++i) {
            if ((unsigned)j[i] - (unsigned)c0 < (unsigned)cols) set(j[i]);
            else if ((unsigned)j[i] >= (unsigned)n_kv) report(j[i]);
          }
        }
      } else {                                       // an entry out of range
#pragma unroll 1
        for (int i = 0; i < kRun; ++i) {
          const int v = list[min(max(e + i, 0), len - 1)];
          if ((unsigned)v < (unsigned)n_kv) set(v);
          else report(v);
        }
      }
    }
    __syncwarp();
    for (int w = lane; w < n; w += 32) {
      const u64 v = reinterpret_cast<const u64*>(my)[w];
      bits[row * wq + (c0 >> 6) + w] = v;
      count += __popcll(v);
    }
    __syncwarp();
  }
  count = __reduce_add_sync(0xffffffffu, count);
  if (lane == 0) {
    nnz[row] = count;
    if (nnz_out) nnz_out[row] = count;
  }
}

// 32 x 32 bits transposed inside a warp (lane = row on entry, column on exit): five exchanges of half
// the bits with the lane 16, 8, 4, 2, 1 away.  Bytes move by permutes, smaller pieces by a rotate and a
// select; what depends on the lane is worked out once (Transposer).
struct Transposer {
  unsigned sel16, sel8, mask[3], rot[3];
  __device__ __forceinline__ explicit Transposer(int lane) {
    sel16 = lane & 16 ? 0x3276u : 0x5410u;
    sel8 = lane & 8 ? 0x3715u : 0x6240u;
    mask[0] = lane & 4 ? 0xF0F0F0F0u : 0x0F0F0F0Fu; rot[0] = lane & 4 ? 28 : 4;
    mask[1] = lane & 2 ? 0xCCCCCCCCu : 0x33333333u; rot[1] = lane & 2 ? 30 : 2;
    mask[2] = lane & 1 ? 0xAAAAAAAAu : 0x55555555u; rot[2] = lane & 1 ? 31 : 1;
  }
  __device__ __forceinline__ unsigned operator()(unsigned x) const {
    x = __byte_perm(x, __shfl_xor_sync(0xffffffffu, x, 16), sel16);
    x = __byte_perm(x, __shfl_xor_sync(0xffffffffu, x, 8), sel8);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const unsigned y = __shfl_xor_sync(0xffffffffu, x, 4 >> k);
      x = (x & mask[k]) | (__funnelshift_l(y, y, rot[k]) & ~mask[k]);
    }
    return x;
  }
};

// One pass over the mask: its bit transpose Mt[h][j][i>>6] bit (i&63) = M[h][i][j>>6] bit (j&63), the
// column counts c = M^T 1 and the row counts n_i = M 1.
// blockIdx.x < wq (all blocks where the rows are counted already): a strip of 64 columns and all rows; a warp transposes 32 rows at a time by
// shuffles, the strip is collected in shared memory ([64 columns][stride] words of 32 rows) so that
// the columns leave in whole lines and are counted on the way.  The other blocks count 32 rows each.
// Counting here spreads what every CTA of a head's cluster used to do for itself over the whole chip.
constexpr int kStatThreads = 256, kStatRows = 32;
constexpr int kStripMax = 64 * (2 * (kMaxSort / 64) + 1) * 4;      // bytes of the longest strip: 131,328
__global__ void __launch_bounds__(kStatThreads) k_mask_stats(const u64* __restrict__ M, u64* __restrict__ Mt, int m_b, int n_b,
                                                             int wq, int wk, int* __restrict__ nnz, int* __restrict__ cnt,
                                                             int* __restrict__ nnz_out, int* __restrict__ cnt_out,
                                                             int* __restrict__ status_out) {
  extern __shared__ unsigned strip[];
  waveal::let_next_kernel_start();
  waveal::wait_for_previous_kernel();
  if (status_out && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 4) status_out[threadIdx.x] = 0;
  const int h = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const u64* Mh = M + (size_t)h * m_b * wq;
  if ((int)blockIdx.x >= wq) {
    constexpr int kPer = kStatRows * 32 / kStatThreads;             // rows of a warp, loads of all in flight
    const int r0 = ((int)blockIdx.x - wq) * kStatRows + warp * kPer;
    int c[kPer] = {};
    for (int w = lane; w < wq; w += 32)
#pragma unroll
      for (int k = 0; k < kPer; ++k)
        if (r0 + k < m_b) c[k] += __popcll(Mh[(size_t)(r0 + k) * wq + w]);
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      c[k] = __reduce_add_sync(0xffffffffu, c[k]);
      if (lane == 0 && r0 + k < m_b) {
        nnz[(size_t)h * m_b + r0 + k] = c[k];
        if (nnz_out) nnz_out[(size_t)h * m_b + r0 + k] = c[k];
      }
    }
    return;
  }
  const int jw = blockIdx.x, stride = 2 * wk + 1;                   // odd: the columns of a warp hit all banks
  const Transposer transpose(lane);
  constexpr int kFly = 4;                                           // loads in flight
  for (int i0 = warp * 32; i0 < wk * 64; i0 += kFly * kStatThreads) {
    u64 w[kFly];
#pragma unroll
    for (int k = 0; k < kFly; ++k) {
      const int i = i0 + k * kStatThreads + lane;
      w[k] = i < m_b ? Mh[(size_t)i * wq + jw] : 0ull;
    }
#pragma unroll
    for (int k = 0; k < kFly; ++k) {
      const int i = i0 + k * kStatThreads;
      if (i >= wk * 64) break;
      strip[lane * stride + (i >> 5)] = transpose((unsigned)w[k]);
      strip[(lane + 32) * stride + (i >> 5)] = transpose((unsigned)(w[k] >> 32));
    }
  }
  __syncthreads();
  for (int c0 = warp; c0 < 64; c0 += kStatThreads / 32) {
    const int j = jw * 64 + c0;
    if (j >= n_b) break;
    const unsigned* col = strip + c0 * stride;
    int c = 0;
    for (int w = lane; w < wk; w += 32) {
      const u64 v = (u64)col[2 * w] | (u64)col[2 * w + 1] << 32;
      Mt[((size_t)h * n_b + j) * wk + w] = v;
      c += __popcll(v);
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane == 0) {
      cnt[(size_t)h * n_b + j] = c;
      if (cnt_out) cnt_out[(size_t)h * n_b + j] = c;
    }
  }
}

// bitmap -> ascending index lists.  The lists of all rows lie one behind the other, so the conversion
// is one compaction of the flat word array: the place of a word's first index is the number of bits
// set before it, and the row pointer is that place at the first word of a row.  Rows shorter than a
// warp leave no lane idle.  k_count_words adds up the share of every block, k_fill_lists starts from
// the sum of the shares before its own; up to kListDirect words (128 KB) a block counts the words before its own
// itself, which is quicker than a second launch.  A serial scan over the rows in one CTA, as before, took longer
// than both passes over the data.
constexpr int kListThreads = 256;             // threads of a block = words of one of its steps
constexpr int kListBlocks = 2048;             // most blocks (every one reads the shares before its own)
constexpr int kListDirect = 16384;

// total over the block of a value per thread; before: the sum over the warps before this one
__device__ __forceinline__ int list_sum(int v, int* part, int& before) {
  const int warp = threadIdx.x >> 5;
  v = __reduce_add_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) part[warp] = v;
  __syncthreads();
  int t = 0;
  before = 0;
#pragma unroll
  for (int i = 0; i < kListThreads / 32; ++i) { before += i < warp ? part[i] : 0; t += part[i]; }
  __syncthreads();
  return t;
}

__global__ void __launch_bounds__(kListThreads) k_count_words(const u64* __restrict__ bits, long long n_words, int steps,
                                                              int* __restrict__ share) {
  __shared__ int part[kListThreads / 32];
  waveal::let_next_kernel_start();
  const long long w0 = (long long)blockIdx.x * steps * kListThreads;
  int c = 0, ignored;
#pragma unroll 4
  for (int s = 0; s < steps; ++s) {
    const long long w = w0 + s * kListThreads + threadIdx.x;
    if (w < n_words) c += __popcll(bits[w]);
  }
  c = list_sum(c, part, ignored);
  if (threadIdx.x == 0) share[blockIdx.x] = c;
}

// a warp takes 32 words at a time: every lane writes the bit positions of its word into the warp's
// staging area ((lane, bit) in 16 bits), which then leaves in whole lines
__global__ void __launch_bounds__(kListThreads) k_fill_lists(const u64* __restrict__ bits, long long n_words, int wq,
                                                             int steps, const int* __restrict__ share,
                                                             int* __restrict__ ptr, long long n_rows,
                                                             int* __restrict__ idx, long long capacity) {
  __shared__ unsigned short stage[kListThreads / 32][32 * 64];
  __shared__ int part[kListThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long w0 = (long long)blockIdx.x * steps * kListThreads;
  int base = 0, pos;
  if (share) {
    waveal::wait_for_previous_kernel();
    for (int i = threadIdx.x; i < (int)blockIdx.x; i += kListThreads) base += share[i];
  } else {
    // (16 words a thread in flight: 8.7 -> 7.6 us for 5 heads of 256 rows, with four)
    constexpr int kFly = 16;
    for (int w = threadIdx.x; w < (int)w0; w += kFly * kListThreads) {
      u64 x[kFly];
#pragma unroll
      for (int k = 0; k < kFly; ++k) x[k] = w + k * kListThreads < (int)w0 ? bits[w + k * kListThreads] : 0ull;
#pragma unroll
      for (int k = 0; k < kFly; ++k) base += __popcll(x[k]);
    }
  }
  base = list_sum(base, part, pos);
  const long long row0 = w0 / wq;
  const unsigned rem0 = (unsigned)(w0 - row0 * wq);
  u64 next = w0 + threadIdx.x < n_words ? bits[w0 + threadIdx.x] : 0ull;
  for (int s = 0; s < steps && w0 + s * kListThreads < n_words; ++s) {
    const unsigned off = (unsigned)(s * kListThreads) + threadIdx.x;
    const long long w = w0 + off;
    const u64 x = next;
    next = s + 1 < steps && w + kListThreads < n_words ? bits[w + kListThreads] : 0ull;
    const int n = __popcll(x);
    const int total = list_sum(n, part, pos);
    pos += base;
    base += total;
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    const unsigned flat = rem0 + off, row = flat / (unsigned)wq, col = flat - row * (unsigned)wq;
    if (w < n_words && col == 0) ptr[row0 + row] = pos + incl - n;
    if (w == n_words - 1) ptr[n_rows] = pos + incl;
    if (idx) {
      unsigned short* st = stage[warp] + (incl - n);
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        unsigned y = half ? (unsigned)(x >> 32) : (unsigned)x;
        while (y) {
          *st++ = (unsigned short)(lane * 64 + half * 32 + __ffs((int)y) - 1);
          y &= y - 1;
        }
      }
      __syncwarp();
      const int here = __shfl_sync(0xffffffffu, incl, 31);
      for (int i0 = 0; i0 < here; i0 += 32) {
        const int i = i0 + lane, e = i < here ? stage[warp][i] : 0;
        const int v = (int)__shfl_sync(0xffffffffu, col, e >> 6) * 64 + (e & 63);
        if (i < here && pos + i < capacity) idx[pos + i] = v;
      }
      __syncwarp();
    }
  }
}

// ------------------------------------------------------------------ block-wide helpers

// Sum of N <= 4 doubles per thread over the CTA, same result in every thread; fixed tree.  The lanes of a warp
// first hand half of their values over (lane distance 16), then half of those (8), so that from there on
// each lane sums one value: 6 exchanges instead of 5 N, which the shuffle unit (one warp a clock) would take 1,280
// clk for with 32 warps and N = 4.  Warps without elements (`any` false) only leave zeros.
template <int N>
__device__ __forceinline__ void block_sum(double (&v)[N], double* scratch, bool any) {
  static_assert(N <= 4 && kPlanWarps == 32, "one quarter of a warp per value, one lane per four warps' partial sums");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double* part = scratch + 4;                 // [warp][4]; the results stand before them
  const int k = (lane >> 3) & 3;              // the value this lane ends up with
  double x = 0.0;
  if (any) {
    double u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) u[i] = i < N ? v[i < N ? i : 0] : 0.0;
    const bool h16 = lane & 16, h8 = lane & 8;
    const double p = (h16 ? u[2] : u[0]) + __shfl_xor_sync(0xffffffffu, h16 ? u[0] : u[2], 16);
    const double q = (h16 ? u[3] : u[1]) + __shfl_xor_sync(0xffffffffu, h16 ? u[1] : u[3], 16);
    x = (h8 ? q : p) + __shfl_xor_sync(0xffffffffu, h8 ? p : q, 8);
#pragma unroll
    for (int o = 4; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  }
  if ((lane & 7) == 0) part[warp * 4 + k] = x;
  __syncthreads();
  if (warp == 0) {
    const int val = lane & 3, grp = lane >> 2;
    double y = (part[grp * 4 + val] + part[(grp + 8) * 4 + val]) + (part[(grp + 16) * 4 + val] + part[(grp + 24) * 4 + val]);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
    if (lane < 4) scratch[lane] = y;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = scratch[i];
}

// the same for whole numbers
template <int N>
__device__ __forceinline__ void block_sum_i64(long long (&v)[N], long long* scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < N; ++k) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    if (lane == 0) scratch[warp * N + k] = v[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < N; ++k) {
    v[k] = scratch[lane * N + k];
#pragma unroll
    for (int o = 16; o; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  }
  __syncthreads();
}

// maxima of N non-negative doubles / minima of N ints over the CTA, same result in every thread
template <int N>
__device__ __forceinline__ void block_max(double (&v)[N], double* scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < N; ++k) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v[k] = fmax(v[k], __shfl_xor_sync(0xffffffffu, v[k], o));
    if (lane == 0) scratch[warp * N + k] = v[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < N; ++k) {
    v[k] = scratch[lane * N + k];
#pragma unroll
    for (int o = 16; o; o >>= 1) v[k] = fmax(v[k], __shfl_xor_sync(0xffffffffu, v[k], o));
  }
  __syncthreads();
}

template <int N>
__device__ __forceinline__ void block_min(int (&v)[N], int* scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    v[k] = __reduce_min_sync(0xffffffffu, v[k]);
    if (lane == 0) scratch[warp * N + k] = v[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < N; ++k) v[k] = __reduce_min_sync(0xffffffffu, scratch[lane * N + k]);
  __syncthreads();
}

// ---- thread-block cluster helpers: the CTAs of a cluster split the rows of the two mask sweeps
// of a head between them and write every result into each other's shared memory
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync_all() { cluster_arrive(); cluster_wait(); }
// store a double2 at the same shared-memory offset of CTA `rank` of this cluster
__device__ __forceinline__ void store_peer(const double2* local_ptr, unsigned rank, double2 v) {
  unsigned laddr = (unsigned)__cvta_generic_to_shared(local_ptr), raddr;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(raddr) : "r"(laddr), "r"(rank));
  asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(raddr), "d"(v.x), "d"(v.y) : "memory");
}

__device__ __forceinline__ void store_peer(const long long* local_ptr, unsigned rank, long long v) {
  unsigned laddr = (unsigned)__cvta_generic_to_shared(local_ptr), raddr;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(raddr) : "r"(laddr), "r"(rank));
  asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(raddr), "l"(v) : "memory");
}

// number of set bits with index in [lo, hi) of a bit row; four words in flight (a wave of 148 rows lies in at most
// four; one load after the other, a head's statistics took 18,200 clk instead of 14,400 on 32 heads of 1,536 blocks)
__device__ __forceinline__ int popcount_range(const u64* __restrict__ words, int lo, int hi) {
  if (hi <= lo) return 0;
  const int w0 = lo >> 6, w1 = (hi - 1) >> 6;
  int c = 0;
  for (int w = w0; w <= w1; w += 4) {
    u64 x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = w + k <= w1 ? words[w + k] : 0ull;
    if (w == w0) x[0] &= ~0ull << (lo & 63);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (w + k == w1 && (hi & 63)) x[k] &= (1ull << (hi & 63)) - 1ull;
      c += __popcll(x[k]);
    }
  }
  return c;
}

// dst[r] = sum_{c : bit (r, c) set} src[c] - rowscale(r) * corr ; rowscale = cnt[r] or 1.
// L lanes share one bit row (lane q of the group takes words q, q+L, ...), 32/L rows per warp
// step; the partial sums meet in a fixed shuffle tree of width L.  Fewer lanes per row than a
// whole warp keeps more rows in flight and wastes fewer of the scarce fp64 adds on the tree.
// crank / csize: this CTA's rank in its cluster and the cluster's size; the CTAs take the warp
// steps in turn, and when `peers` is set (state in shared memory) every result is also written
// into the other CTAs' copy of dst.  A row is summed by the same lanes in the same order
// whichever CTA takes it, so the result does not depend on the cluster size.
template <int L>
__device__ __forceinline__ void gather_rows_l(const u64* __restrict__ bits, int n_rows, int wpr,
                                              const double2* src, double2* dst,
                                              const int* __restrict__ cnt, double2 corr,
                                              int crank, int csize, bool peers) {
  constexpr int RPW = 32 / L;                       // rows per warp step
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int grp = lane / L, q = lane % L;
  for (int r0 = (warp + crank * kPlanWarps) * RPW; r0 < n_rows; r0 += csize * kPlanWarps * RPW) {
    const int r = r0 + grp;
    const bool live = r < n_rows;
    double ax = 0.0, ay = 0.0;
    for (int w0 = 0; w0 < wpr; w0 += 4 * L) {
      u64 word[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int w = w0 + q + k * L;
        word[k] = (live && w < wpr) ? bits[(size_t)r * wpr + w] : 0ull;
      }
      // walk the set bits of each word as two 32-bit halves (64-bit bit tricks cost twice
      // the integer instructions, and this loop is bound by them)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const double2* sp = src + (w0 + q + k * L) * 64;
#pragma unroll
        for (int hw = 0; hw < 2; ++hw) {
          unsigned x = hw ? (unsigned)(word[k] >> 32) : (unsigned)word[k];
          while (x) {
            const int b = __ffs((int)x) - 1;
            x &= x - 1;
            const double2 v = sp[hw * 32 + b];
            ax += v.x;
            ay += v.y;
          }
        }
      }
    }
#pragma unroll
    for (int o = L / 2; o; o >>= 1) {
      ax += __shfl_xor_sync(0xffffffffu, ax, o);
      ay += __shfl_xor_sync(0xffffffffu, ay, o);
    }
    if (live && q == 0) {
      const double sc = cnt ? (double)cnt[r] : 1.0;
      const double2 v = make_double2(ax - sc * corr.x, ay - sc * corr.y);
      dst[r] = v;
      if (peers)
        for (int c = 0; c < csize; ++c)
          if (c != crank) store_peer(dst + r, (unsigned)c, v);
    }
  }
}

__device__ __forceinline__ void gather_rows(const u64* __restrict__ bits, int n_rows, int wpr,
                                            const double2* src, double2* dst,
                                            const int* __restrict__ cnt, double2 corr,
                                            int crank, int csize, bool peers) {
  // about three words per lane
  if (wpr <= 3) gather_rows_l<1>(bits, n_rows, wpr, src, dst, cnt, corr, crank, csize, peers);
  else if (wpr <= 6) gather_rows_l<2>(bits, n_rows, wpr, src, dst, cnt, corr, crank, csize, peers);
  else if (wpr <= 12) gather_rows_l<4>(bits, n_rows, wpr, src, dst, cnt, corr, crank, csize, peers);
  else if (wpr <= 24) gather_rows_l<8>(bits, n_rows, wpr, src, dst, cnt, corr, crank, csize, peers);
  else if (wpr <= 48) gather_rows_l<16>(bits, n_rows, wpr, src, dst, cnt, corr, crank, csize, peers);
  else gather_rows_l<32>(bits, n_rows, wpr, src, dst, cnt, corr, crank, csize, peers);
}

// Q factor of the thin QR of an m x 2 block: Gram-Schmidt with one re-orthogonalisation
// pass; numerically dependent columns become zero.  Only the coefficients are computed here, in
// two reductions (the kernel's serial part: one pass and one reduction per coefficient, five in
// all, cost more than the products on short sequences); the entries follow from them one by one:
//   q1 = z1 / n1,  x2 = ((z2 - d q1) - e q1) / n2   with  d = q1.z2,  e = q1.(z2 - d q1),
//   n2^2 = |z2 - d q1|^2 - e^2   (e is a rounding error of the first projection, so nothing cancels)
struct Qr2 {
  double inv1, inv2, d, e;      // inv1 / inv2 = 0: that column is dropped
  double2 colsum;
  __device__ __forceinline__ double2 entry(double2 z) const {
    const double q1 = z.x * inv1;
    return make_double2(q1, ((z.y - d * q1) - e * q1) * inv2);
  }
};
__device__ __forceinline__ Qr2 thin_qr2(const double2* z_in, int m, double* scratch) {
  const double tiny_sq = 1e-60 * (double)m;      // a column of norm 1e-30 sqrt(m) or less is dropped
  const int tid = threadIdx.x;
  double a[3] = {0, 0, 0};
  for (int i = tid; i < m; i += kPlanThreads) { const double2 z = z_in[i]; a[0] += z.x * z.x; a[1] += z.x * z.y; a[2] += z.y * z.y; }
  const bool any = (tid & ~31) < m;
  block_sum<3>(a, scratch, any);
  Qr2 r;
  r.inv1 = a[0] > tiny_sq ? rsqrt(a[0]) : 0.0;
  r.d = a[1] * r.inv1;
  double s[4] = {0, 0, 0, 0};
  for (int i = tid; i < m; i += kPlanThreads) {
    const double2 z = z_in[i];
    const double q1 = z.x * r.inv1, y = z.y - r.d * q1;
    s[0] += q1 * y; s[1] += y * y; s[2] += q1; s[3] += y;
  }
  block_sum<4>(s, scratch, any);
  r.e = s[0];
  const double n2_sq = s[1] - r.e * r.e;         // dropped too: 1e-9 or less of the norm before the projection
  r.inv2 = n2_sq > tiny_sq && n2_sq > 1e-18 * a[2] ? rsqrt(n2_sq) : 0.0;
  r.colsum = make_double2(s[2], (s[3] - r.e * s[2]) * r.inv2);
  return r;
}

// ---- mask products on the integer matrix units
// A product of a 0/1 mask with two columns of fp64 numbers is a contraction, and an exact one once
// the numbers are fixed point: every entry becomes a 64-bit integer q = round(v * 2^e), q is cut
// into eight signed 8-bit digits, and mask x digits accumulates in int32 without rounding, in any
// order and with any split of the columns.  The digits of both columns are the 16 columns of the
// B operand (two n8 tiles), 32 mask bits are the k of one mma.m16n8k32.  e is chosen from a bound on the entries, not from their maximum (which
// would take one more exchange between the CTAs): the quantisation error is 2^-63 of that bound,
// less than the rounding of the fp64 sums it replaces.
// Set bits cost nothing here, a row costs the same at any density: the bit walk (gather_rows) takes
// ~10 instructions per set bit with three quarters of the lanes idle.
//
// Operand layout (256 columns = four 64-bit words of a row per chunk): lane (g, t) = (lane / 4,
// lane % 4) of a warp loads word 4*chunk + t of rows g and g + 8.  Step s of a chunk takes the bits
// with index s modulo 8 of every 32-bit half: (half << (7 - s)) & 0x80808080 is four bytes, so the
// k slots of that step are the columns 256*chunk + 64*t + 32*(low/high half) + s + 8*j, j = 0..3,
// and one mask and one multiply expand four bits.  A set bit counts 128; the sums are divided at the
// end.  The digits lie in shared memory in the order the fragments need, one 16-byte item per lane
// and step: {column 0 low half, high half, column 1 low half, high half}; items are XORed with s so that
// the stores of pack_digits meet no bank conflict.
constexpr int kChunkCols = 256;
constexpr int kUnitRows = 32;            // rows one warp multiplies at a time (two m16 tiles)

__device__ __forceinline__ unsigned prmt(unsigned a, unsigned b, unsigned sel) { return __byte_perm(a, b, sel); }

// bytes of four words transposed: out[i] = byte i of w0..w3
__device__ __forceinline__ void transpose4(unsigned w0, unsigned w1, unsigned w2, unsigned w3, unsigned (&o)[4]) {
  const unsigned a = prmt(w0, w1, 0x5140), b = prmt(w2, w3, 0x5140);   // {w0.0 w1.0 w0.1 w1.1}
  const unsigned c = prmt(w0, w1, 0x7362), d = prmt(w2, w3, 0x7362);   // {w0.2 w1.2 w0.3 w1.3}
  o[0] = prmt(a, b, 0x5410); o[1] = prmt(a, b, 0x7632);
  o[2] = prmt(c, d, 0x5410); o[3] = prmt(c, d, 0x7632);
}

// digits of entry(k), k < n, into `items`; entry returns the two columns' values, `scale` = 2^e.
// One thread packs eight entries of one column.
template <class Entry>
__device__ __forceinline__ void pack_digits(uint4* items, int n, double scale, Entry entry) {
  const int total = (n + kChunkCols - 1) / kChunkCols * 64;            // (chunk, t, s, column)
  for (int w = threadIdx.x; w < total; w += kPlanThreads) {
    const int col = w & 1, s = (w >> 1) & 7, t = (w >> 4) & 3, chunk = w >> 6;
    unsigned lo[8], hi[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = chunk * kChunkCols + t * 64 + s + 8 * j;           // j >= 4: the high half of the word
      const double v = k < n ? entry(k, col) : 0.0;
      // balanced digits: add 128 to each of the lower seven bytes, then take it off byte by byte
      const u64 q = ((u64)__double2ll_rn(v * scale) + 0x0080808080808080ull) ^ 0x0080808080808080ull;
      lo[j] = (unsigned)q; hi[j] = (unsigned)(q >> 32);
    }
    unsigned d0[4], d1[4];
    uint2* base = reinterpret_cast<uint2*>(items + (size_t)(chunk * 8 + s) * 32);
#pragma unroll
    for (int half = 0; half < 2; ++half) {                             // digits 0..3, 4..7
      const unsigned* q = half ? hi : lo;
      transpose4(q[0], q[1], q[2], q[3], d0);
      transpose4(q[4], q[5], q[6], q[7], d1);
#pragma unroll
      for (int g = 0; g < 4; ++g) base[((((half * 4 + g) * 4 + t) ^ s) << 1) + col] = make_uint2(d0[g], d1[g]);
    }
  }
}

__device__ __forceinline__ void imma(int (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1) {
  asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// value of sum_k digit_sum[k] 256^k from two integers of four digits each (both below 2^53)
__device__ __forceinline__ double join_digits(long long lo, long long hi) { return (double)hi * 4294967296.0 + (double)lo; }

// dst[r] = (sum_{c : bit (r, c) set} q[c]) / scale - rowscale(r) * corr, the q from `items`.
// A warp takes 32 rows and a share of the chunks; the CTAs of a cluster take the groups of 32 rows in
// turn.  ksplit > 1: that many warps share the rows of a group (by columns) and meet in `part`
// ([32 / ksplit groups][16 digits][32 rows] int32, zero on entry and on exit; the rows XORed with 8 times the digit's pair, so that
// neither a warp's fragments nor its rows meet a bank conflict, a product of 384 x 1,536 12,970 -> 12,270 clk): integer sums, so neither the split nor the cluster size
// shows in the result.
__device__ __forceinline__ void multiply_rows(const u64* __restrict__ bits, int n_rows, int wpr, const uint4* items,
                                              int* part, int ksplit, double inv_scale, double2* dst,
                                              const int* __restrict__ cnt, double2 corr, int crank, int csize, bool peers) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int units = (n_rows + kUnitRows - 1) / kUnitRows, chunks = (wpr + 3) >> 2;
  const int slots = kPlanWarps / ksplit, slot = warp / ksplit, kp = warp - slot * ksplit;
  auto put = [&](int r, int c_r, double x, double y) {
    const double sc = (double)c_r;
    const double2 v = make_double2(x * inv_scale - sc * corr.x, y * inv_scale - sc * corr.y);
    dst[r] = v;
    if (peers)
      for (int c = 0; c < csize; ++c)
        if (c != crank) store_peer(dst + r, (unsigned)c, v);
  };
  for (int u0 = crank; u0 < units; u0 += csize * slots) {              // (the same trips for every warp)
    const int u = u0 + slot * csize;
    if (slot < slots && u < units) {
      int acc[2][2][4];                                                // [m16 tile][column][fragment]
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[i][c][e] = 0;
      const int r0 = u * kUnitRows + g;
      const int c_mine = ksplit == 1 && cnt && r0 + t * 8 < n_rows ? cnt[r0 + t * 8] : 1;    // (loaded ahead of the products)
      for (int ch = kp * chunks / ksplit; ch < (kp + 1) * chunks / ksplit; ++ch) {
        u64 w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = r0 + i * 8, wi = ch * 4 + t;
          w[i] = (r < n_rows && wi < wpr) ? bits[(size_t)r * wpr + wi] : 0ull;
        }
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          const uint4 b = items[(size_t)(ch * 8 + s) * 32 + (lane ^ s)];
          unsigned a[4][2];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            a[i][0] = ((unsigned)w[i] * (128u >> s)) & 0x80808080u;
            a[i][1] = ((unsigned)(w[i] >> 32) * (128u >> s)) & 0x80808080u;
          }
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            imma(acc[i][0], a[2 * i][0], a[2 * i + 1][0], a[2 * i][1], a[2 * i + 1][1], b.x, b.y);
            imma(acc[i][1], a[2 * i][0], a[2 * i + 1][0], a[2 * i][1], a[2 * i + 1][1], b.z, b.w);
          }
        }
      }
      // fragment: element 2*half + e of lane (g, t) is row g + 8*half, digit 2*t + e
      if (ksplit == 1) {
        double val[2][2][2];                                           // [tile][row half][column]
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int half = 0; half < 2; ++half)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              long long v = (long long)(acc[i][c][2 * half] >> 7) + ((long long)(acc[i][c][2 * half + 1] >> 7) << 8);
              v <<= (t & 1) * 16;
              v += __shfl_xor_sync(0xffffffffu, v, 1);                 // lanes t = 0, 1: digits 0..3; t = 2, 3: digits 4..7
              const long long o = __shfl_xor_sync(0xffffffffu, v, 2);
              val[i][half][c] = t < 2 ? join_digits(v, o) : join_digits(o, v);
            }
        // lane t of a quad stores row g + 8t of the group
        const double x = t == 0 ? val[0][0][0] : t == 1 ? val[0][1][0] : t == 2 ? val[1][0][0] : val[1][1][0];
        const double y = t == 0 ? val[0][0][1] : t == 1 ? val[0][1][1] : t == 2 ? val[1][0][1] : val[1][1][1];
        const int r = r0 + t * 8;
        if (r < n_rows) put(r, c_mine, x, y);
      } else {
        int* pp = part + slot * (kUnitRows * 16);
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int e = 0; e < 4; ++e)
              atomicAdd(&pp[(c * 8 + 2 * t + (e & 1)) * kUnitRows + ((i * 16 + g + 8 * (e >> 1)) ^ (8 * t))], acc[i][c][e] >> 7);
      }
    }
    if (ksplit > 1) {
      // (slots * 32 <= 512 rows: one a thread)
      const int i = threadIdx.x, uu = u0 + (i / kUnitRows) * csize, r = uu * kUnitRows + i % kUnitRows;
      const bool mine = i < slots * kUnitRows;
      int* sums = part + (i / kUnitRows) * (kUnitRows * 16);
      auto digit_at = [&](int d) { return d * kUnitRows + ((i % kUnitRows) ^ (8 * ((d >> 1) & 3))); };
      const int c_mine = mine && cnt && uu < units && r < n_rows ? cnt[r] : 1;
      __syncthreads();
      if (mine) {
        if (uu < units && r < n_rows) {
          double v[2];
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            long long s[2];                                            // digits 0..3, 4..7
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              s[k] = 0;
#pragma unroll
              for (int d = 3; d >= 0; --d) s[k] = (s[k] << 8) + sums[digit_at(c * 8 + k * 4 + d)];
            }
            v[c] = join_digits(s[0], s[1]);
          }
          put(r, c_mine, v[0], v[1]);
        }
#pragma unroll
        for (int d = 0; d < 16; ++d) sums[digit_at(d)] = 0;
      }
      __syncthreads();
    }
  }
}

__device__ __forceinline__ u64 splitmix64(u64 x) {
  u64 z = x + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// monotone map double -> u64 (no NaN expected; -0.0 is removed by the caller)
__device__ __forceinline__ u64 sortable(double v) {
  u64 b = (u64)__double_as_longlong(v);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}

// Ascending merge sort of n (key, val) pairs, stable, between two buffers; the result is in the buffer
// returned (0 or 1).  Runs of 32 by counting (a warp's own elements, read as broadcasts), then
// every element finds its place in the neighbouring run by a binary search.  Against the bitonic
// network below: 8 barriers instead of 78 at 4096 elements, no padding to a power of two, and an
// element is moved 8 times.
__device__ __forceinline__ int merge_sort(u64* k0, int* v0, u64* k1, int* v1, int n) {
  for (int i = threadIdx.x; i < n; i += kPlanThreads) {
    const int g0 = i & ~31, g1 = min(g0 + 32, n);
    const u64 key = k0[i];
    int pos = g0;
    for (int j = g0; j < g1; ++j) {
      const u64 kj = k0[j];
      pos += (kj < key || (kj == key && j < i)) ? 1 : 0;
    }
    k1[pos] = key;
    v1[pos] = v0[i];
  }
  int at = 1;
  for (int len = 32; len < n; len <<= 1, at ^= 1) {
    __syncthreads();
    const u64* ks = at ? k1 : k0;
    const int* vs = at ? v1 : v0;
    u64* kd = at ? k0 : k1;
    int* vd = at ? v0 : v1;
    for (int i = threadIdx.x; i < n; i += kPlanThreads) {
      const u64 key = ks[i];
      const bool right = (i & len) != 0;               // of the two runs: equal keys of the left one come first
      const int sib = right ? (i & ~(len - 1)) - len : (i & ~(len - 1)) + len;
      int lo = min(sib, n), hi = min(sib + len, n);
      const int s0 = lo;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        const u64 km = ks[mid];
        const bool before = km < key || (right && km == key);
        lo = before ? mid + 1 : lo;
        hi = before ? hi : mid;
      }
      const int pos = (right ? i - len : i) + (lo - s0);
      kd[pos] = key;
      vd[pos] = vs[i];
    }
  }
  __syncthreads();
  return at;
}

// Exclusive prefix sums of n ints in shared memory, in place.  part: 32 ints.  Ends with a barrier.
__device__ __forceinline__ void exclusive_scan(int* a, int n, int* part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = (n + kPlanThreads - 1) / kPlanThreads, i0 = min((int)threadIdx.x * per, n), i1 = min(i0 + per, n);
  int mine = 0;
  for (int i = i0; i < i1; ++i) mine += a[i];
  int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) part[warp] = incl;
  __syncthreads();
  int at = __reduce_add_sync(0xffffffffu, lane < warp ? part[lane] : 0) + incl - mine;
  for (int i = i0; i < i1; ++i) { const int v = a[i]; a[i] = at; at += v; }
  __syncthreads();
}

// Ascending sort of n pairs (key, val) with distinct pairs, ties of the key by val, through bins that are themselves in
// ascending order: `bin(key)` < n_bins never falls as the key grows.  Counts per bin, prefix sums, a scatter, and every
// element counts the elements of its own bin that go before it: the work per element is the size of its bin, where the
// merge sort walks log2(n) binary searches.  43,800 -> 9,100 clk for 2,841 rows of a video mask, 10,400 -> 8,100 for 591, 24,000 ->
// 12,400 for 1,536 of which a tenth have one angle (rows that select everything).  (Bins cut at
// the quantiles of a sample of the keys: 41,700 for the 2,841 rows, their bins of 22 and more are walked for longer.)
// The sorted values go to v0.  False, with the pairs as they were, if a bin holds more than `most`.  (The order inside a
// bin before the count depends on the atomics, the result does not.)
template <class Bin>
__device__ __forceinline__ bool bin_sort(const u64* k0, int* v0, u64* k1, int* v1, int n, int* bins, int n_bins, int most, int* part, Bin bin) {
  for (int i = threadIdx.x; i < n_bins; i += kPlanThreads) bins[i] = 0;
  __syncthreads();
  bool big = false;
  for (int i = threadIdx.x; i < n; i += kPlanThreads) big |= atomicAdd(&bins[bin(k0[i])], 1) >= most;
  if (__syncthreads_or(big)) return false;
  exclusive_scan(bins, n_bins, part);
  for (int i = threadIdx.x; i < n; i += kPlanThreads) {
    const u64 key = k0[i];
    const int at = atomicAdd(&bins[bin(key)], 1);          // leaves the end of every bin
    k1[at] = key;
    v1[at] = v0[i];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += kPlanThreads) {
    const u64 key = k1[i];
    const int val = v1[i], b = bin(key), from = b ? bins[b - 1] : 0, to = bins[b];
    int at = from;
#pragma unroll 4
    for (int j = from; j < to; ++j) {                      // (both are always read, several rows under way)
      const u64 kj = k1[j];
      const int vj = v1[j];
      at += (int)(kj < key) | ((int)(kj == key) & (int)(vj < val));
    }
    v0[at] = val;
  }
  __syncthreads();
  return true;
}

// 256 keys ascending, eight neighbours a lane: a bitonic network in registers (steps inside a lane by min and max, the others by
// a shuffle).  In a descending stretch the keys are complemented instead of the comparisons turned around.
__device__ __forceinline__ void warp_sort256(unsigned (&a)[8]) {
  const unsigned lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 2; k <= 256; k <<= 1) {
    // (stretches of up to eight keys lie inside a lane, where the direction is known while compiling)
    const unsigned flip = k >= 8 && k < 256 && (lane & (k >> 3)) ? ~0u : 0u;
    if (k >= 8)
#pragma unroll
      for (int e = 0; e < 8; ++e) a[e] ^= flip;
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= 8) {
        const bool upper = lane & (j >> 3);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const unsigned b = __shfl_xor_sync(0xffffffffu, a[e], j >> 3);
          a[e] = upper ? max(a[e], b) : min(a[e], b);
        }
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if ((e & j) == 0) {
            const unsigned lo = min(a[e], a[e | j]), hi = max(a[e], a[e | j]);
            const bool up = k >= 8 || (e & k) == 0;
            a[e] = up ? lo : hi;
            a[e | j] = up ? hi : lo;
          }
      }
    }
    if (k >= 8)
#pragma unroll
      for (int e = 0; e < 8; ++e) a[e] ^= flip;
  }
}

// ascending bitonic sort of (key, val) pairs, ties by val; n is a power of two (row counts whose
// second buffer does not fit shared memory)
__device__ __forceinline__ void bitonic_sort(u64* keys, int* vals, int n) {
  for (int k = 2; k <= n; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < n; t += kPlanThreads) {
        int p = t ^ j;
        if (p > t) {
          u64 ka = keys[t], kb = keys[p];
          int va = vals[t], vb = vals[p];
          bool a_gt_b = ka > kb || (ka == kb && va > vb);
          bool asc = (t & k) == 0;
          if (a_gt_b == asc) { keys[t] = kb; keys[p] = ka; vals[t] = vb; vals[p] = va; }
        }
      }
      __syncthreads();
    }
  }
}

struct PlanParams {
  const u64* M;
  const u64* Mt;
  int m_b, n_b, wq, wk, wave, iters, mode, n_pow2, state_in_smem;
  int ring_cut;         // open the angular ring at its largest gap instead of at -pi
  int csize;            // CTAs per head (thread-block cluster size)
  int mma;              // mask products on the integer matrix units (else: walk over the set bits)
  int count_stage2;     // Stage 2 by counting inside the buckets (else: by a sort)
  int warp_stage2;      // Stage 2 by a warp per bucket
  int bins, bin_max;    // bins of the angular sort (0: by merging) and the most rows one may hold
  int alias_yz;         // Y and Z share one buffer (two barriers more per iteration)
  int ksplit_y, ksplit_z, part_ints;
  unsigned off_items, off_part;     // bytes from the start of shared memory
  u64 seed;
  long long kv_bytes, l2_bytes, min_nnz;
  int fit_num, fit_den, min_ppm, loc_num, loc_den;
  const int* ws_nnz;    // [heads][m_b], k_mask_stats
  const int* ws_cnt;    // [heads][n_b], k_mask_stats
  double2* ws_state;    // [heads][2*m_b + n_b] when the blocks do not fit shared memory
  int* row_order; unsigned char* flags; int* order1;
  double* embedding; long long* stats;
};

// (one copy of the function, in a rolled loop: sixteen in line were fetched one behind the other, 17,700 clk for 1,536
// rows against 4,500)
__device__ __noinline__ double polar_angle(double y, double x) { return atan2(y, x); }

__global__ void __launch_bounds__(kPlanThreads, 1) k_plan_head(PlanParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  double* scratch = reinterpret_cast<double*>(smem);                 // (32 + 1) * 4 doubles
  unsigned char* region = smem + 2048;
  // A head is planned by a cluster of p.csize CTAs.  Everything cheap (counts, guard, QR,
  // rotations, sorts) is done by every CTA of the cluster on its own copy of the state, in the
  // same order, so the copies stay identical bit for bit; only the two mask sweeps of an
  // iteration, where the time goes, are split, and their results exchanged.
  const int csize = p.csize, crank = csize > 1 ? (int)cluster_rank() : 0;
  const int h = blockIdx.x / csize, tid = threadIdx.x;
  const bool lead = crank == 0;         // writes the outputs
  const int m_b = p.m_b, n_b = p.n_b;
  const u64* M = p.M + (size_t)h * m_b * p.wq;
  const u64* Mt = p.Mt + (size_t)h * n_b * p.wk;
  const int* nnz = p.ws_nnz + (size_t)h * m_b;
  const int* cnt = p.ws_cnt + (size_t)h * n_b;
  int* order_out = p.row_order + (size_t)h * m_b;
  int* order1_out = p.order1 ? p.order1 + (size_t)h * m_b : nullptr;

  waveal::wait_for_previous_kernel();
  // (a CTA writes into another's shared memory only once that one runs: waited for below)
  if (csize > 1) cluster_arrive();
  // ---- guard statistics over natural-order waves (Section 4.5): selected pairs, and for the overlap
  // sum_l (w_l - 1) t_l from the row counts, sum_l,j c_lj (c_lj - 1) / 2 from the columns (split
  // over the CTAs of the cluster; whole numbers, so the split does not show)
  const int n_waves = (m_b + p.wave - 1) / p.wave;
  long long sums[3] = {0, 0, 0};
  for (int i = tid; i < m_b; i += kPlanThreads) {
    const int lo = i / p.wave * p.wave;
    const long long c = nnz[i];
    sums[0] += c;
    sums[1] += (long long)(min(p.wave, m_b - lo) - 1) * c;
  }
  {
    const int dj = kPlanThreads / n_waves, dl = kPlanThreads % n_waves;
    int col = tid / n_waves, l = tid % n_waves;           // (column of this CTA's share, wave), 1024 such pairs a step
    for (long long j = (long long)col * csize + crank; j < n_b; j = (long long)col * csize + crank) {
      const int lo = l * p.wave;
      const long long c = popcount_range(Mt + (size_t)j * p.wk, lo, min(lo + p.wave, m_b));
      sums[2] += c * (c - 1) / 2;
      col += dj; l += dl;
      if (l >= n_waves) { l -= n_waves; ++col; }
    }
  }
  block_sum_i64<3>(sums, reinterpret_cast<long long*>(scratch));
  const long long nnz_total = sums[0], pair2 = sums[1];
  long long ov = sums[2];
  if (csize > 1) {
    cluster_wait();
    long long* slots = reinterpret_cast<long long*>(smem + 1280);      // one per CTA of the cluster
    if (tid < csize) store_peer(slots + crank, (unsigned)tid, ov);
    cluster_sync_all();
    ov = 0;
    for (int c = 0; c < csize; ++c) ov += slots[c];
  }
  unsigned flags = 0;
  if (p.kv_bytes > 0 && p.l2_bytes > 0 && p.kv_bytes * p.fit_den <= p.l2_bytes * p.fit_num)
    flags |= WAVEAL_FLAG_SHORT_SEQ;
  if (nnz_total < p.min_nnz || nnz_total * 1000000ll < (long long)p.min_ppm * m_b * n_b)
    flags |= WAVEAL_FLAG_TOO_SPARSE;
  if (pair2 > 0 && 2 * ov * p.loc_den >= (long long)p.loc_num * pair2) flags |= WAVEAL_FLAG_ALREADY_LOCAL;
  const bool skip = p.mode == WAVEAL_FORCE_NATURAL || (p.mode == WAVEAL_AUTO && flags != 0);
  if (skip) flags |= WAVEAL_FLAG_SKIPPED;
  if (tid == 0 && lead) {
    if (p.flags) p.flags[h] = (unsigned char)flags;
    if (p.stats) { long long* s = p.stats + (size_t)h * 4; s[0] = nnz_total; s[1] = ov; s[2] = pair2; s[3] = 0; }
  }
  if (skip) {
    if (lead)
    for (int i = tid; i < m_b; i += kPlanThreads) {
      order_out[i] = i;
      if (order1_out) order1_out[i] = i;
      if (p.embedding) { p.embedding[((size_t)h * m_b + i) * 2] = 0.0; p.embedding[((size_t)h * m_b + i) * 2 + 1] = 0.0; }
    }
    return;
  }

  // pairs to sort: two buffers of m_b (merge sort), or one of n_pow2 (bitonic)
  u64* keys = reinterpret_cast<u64*>(region);
  const bool merging = m_b <= kMaxMerge;
  const int n_sort = merging ? m_b : p.n_pow2;
  u64* keys2 = keys + (merging ? m_b : 0);
  int* vals = reinterpret_cast<int*>(keys + (merging ? 2 * m_b : p.n_pow2));
  int* vals2 = vals + m_b;
  int* bins = vals2 + m_b;
  auto sort_pairs = [&]() {
    if (!merging) { bitonic_sort(keys, vals, p.n_pow2); return; }
    if (merge_sort(keys, vals, keys2, vals2, m_b)) {
      u64* k = keys; keys = keys2; keys2 = k;
      int* v = vals; vals = vals2; vals2 = v;
    }
  };

  if (p.mode != WAVEAL_STAGE2_ONLY) {
    double2* X = p.state_in_smem ? reinterpret_cast<double2*>(region)
                                 : p.ws_state + (size_t)h * (2 * (size_t)m_b + n_b);
    double2* Z = X + m_b;
    double2* Y = p.alias_yz ? Z : Z + m_b;
    uint4* items = reinterpret_cast<uint4*>(smem + p.off_items);
    int* part = reinterpret_cast<int*>(smem + p.off_part);
    const double x_scale = 4611686018427387904.0;     // 2^62: |x| <= 1
    double y_scale = 1.0;
    if (p.mma) {
      // |y_j| <= sqrt(c_j (m - c_j) / m), the norm of a centred 0/1 column: the largest column count gives a power of
      // two 2^e >= |y|, and y_scale = 2^(62 - e).  (sqrt(m) / 2, which holds for any mask, is far above what columns of a
      // few blocks reach and quantises coarser than fp64 rounds: 14,336 rows of one block each, one sweep, embedding
      // against 80-bit arithmetic: 3.7e-16 with it, 1.3e-16 so and with fp64 sums.)
      int c_mine = 0;
      for (int j = tid; j < n_b; j += kPlanThreads) c_mine = max(c_mine, cnt[j]);
      double c_max[1] = {(double)c_mine};
      block_max<1>(c_max, scratch);
      const long long c = min((int)c_max[0], m_b / 2);
      int e = 0;
      while (((long long)m_b << (2 * e)) < c * (m_b - c)) ++e;
      y_scale = __longlong_as_double((long long)(1023 + 62 - e) << 52);
    }
    const bool peers = csize > 1 && p.state_in_smem;
    auto sync_head = [&]() { if (csize > 1) cluster_sync_all(); else __syncthreads(); };
    if (p.mma)
      for (int i = tid; i < p.part_ints; i += kPlanThreads) part[i] = 0;
    const double inv_m = 1.0 / (double)m_b;
    // ---- start block (counter-based) and its orthonormalisation (Algorithm 1, step 3)
    const u64 hk = (u64)h * 0x9E3779B97F4A7C15ull;
    for (int i = tid; i < m_b; i += kPlanThreads) {
      double u0 = (double)(splitmix64(p.seed ^ hk ^ (u64)(2 * i)) >> 11) * (1.0 / 9007199254740992.0);
      double u1 = (double)(splitmix64(p.seed ^ hk ^ (u64)(2 * i + 1)) >> 11) * (1.0 / 9007199254740992.0);
      Z[i] = make_double2(2.0 * u0 - 1.0, 2.0 * u1 - 1.0);
    }
    __syncthreads();
    // ---- T sweeps + one more for the Rayleigh-Ritz step
    for (int it = 0; it <= p.iters; ++it) {
      const Qr2 qr = thin_qr2(Z, m_b, scratch);
      // Y = M^T X - c (1^T X)/m
      const double2 corr_y = make_double2(qr.colsum.x * inv_m, qr.colsum.y * inv_m);
      if (!p.mma || (it == p.iters && lead))                     // (the digits are taken from Z directly)
        for (int i = tid; i < m_b; i += kPlanThreads) X[i] = qr.entry(Z[i]);
      if (p.mma) {
        pack_digits(items, m_b, x_scale, [&](int k, int col) { const double2 x = qr.entry(Z[k]); return col ? x.y : x.x; });
        if (p.alias_yz) sync_head(); else __syncthreads();
        multiply_rows(Mt, n_b, p.wk, items, part, p.ksplit_y, 1.0 / x_scale, Y, cnt, corr_y, crank, csize, peers);
      } else {
        __syncthreads();
        gather_rows(Mt, n_b, p.wk, X, Y, cnt, corr_y, crank, csize, peers);
      }
      sync_head();
      double cy[2] = {0, 0};
      for (int j = tid; j < n_b; j += kPlanThreads) { double2 y = Y[j]; double c = (double)cnt[j]; cy[0] += c * y.x; cy[1] += c * y.y; }
      if (p.mma) pack_digits(items, n_b, y_scale, [&](int k, int col) { return col ? Y[k].y : Y[k].x; });
      block_sum<2>(cy, scratch, (tid & ~31) < n_b);
      // Z = M Y - 1 (c^T Y)/m
      const double2 corr_z = make_double2(cy[0] * inv_m, cy[1] * inv_m);
      if (p.mma) {
        if (p.alias_yz) sync_head();                             // (else: the barriers of the sum above)
        multiply_rows(M, m_b, p.wq, items, part, p.ksplit_z, 1.0 / y_scale, Z, nullptr, corr_z, crank, csize, peers);
      } else {
        gather_rows(M, m_b, p.wq, Y, Z, nullptr, corr_z, crank, csize, peers);
      }
      sync_head();
    }
    // the rest (ordering, angles, sorts, outputs) is cheap: the lead CTA finishes alone.  No CTA
    // touches another's shared memory after the last exchange above.
    if (!lead) return;
    // ---- B = X^T Z, rotate onto the eigenvectors of its symmetric part, larger Ritz value first
    double b[4] = {0, 0, 0, 0};
    for (int i = tid; i < m_b; i += kPlanThreads) {
      double2 x = X[i], z = Z[i];
      b[0] += x.x * z.x; b[1] += x.x * z.y; b[2] += x.y * z.x; b[3] += x.y * z.y;
    }
    block_sum<4>(b, scratch, (tid & ~31) < m_b);
    // (one warp works the angle out: 32 of them kept the fp64 units busy with it for 4,000 cycles)
    if (tid < 32) {
      const double th = 0.5 * polar_angle(2.0 * (0.5 * (b[1] + b[2])), b[0] - b[3]);
      if (tid == 0) { scratch[4] = cos(th); scratch[5] = sin(th); }
    }
    __syncthreads();
    const double cs = scratch[4], sn = scratch[5];
    __syncthreads();
    double mx[2] = {0, 0};
    for (int i = tid; i < m_b; i += kPlanThreads) {
      double2 x = X[i];
      double2 u = make_double2(x.x * cs + x.y * sn, x.y * cs - x.x * sn);
      X[i] = u;
      mx[0] = fmax(mx[0], fabs(u.x));
      mx[1] = fmax(mx[1], fabs(u.y));
    }
    block_max<2>(mx, scratch);
    // ---- sign: the first entry reaching half of the largest magnitude is made positive
    int f[2] = {INT_MAX, INT_MAX};
    for (int i = tid; i < m_b; i += kPlanThreads) {
      double2 u = X[i];
      if (mx[0] > 0.0 && fabs(u.x) >= 0.5 * mx[0]) f[0] = min(f[0], i);
      if (mx[1] > 0.0 && fabs(u.y) >= 0.5 * mx[1]) f[1] = min(f[1], i);
    }
    block_min<2>(f, reinterpret_cast<int*>(scratch));
    double s1 = (f[0] != INT_MAX && X[f[0]].x < 0.0) ? -1.0 : 1.0;
    double s2 = (f[1] != INT_MAX && X[f[1]].y < 0.0) ? -1.0 : 1.0;
    __syncthreads();
    // ---- polar angle a_i = atan2(u_2[i], u_1[i]) (Eq. 4), as a sort key in the place of u_1; the keys
    //      go through registers into the shared region, where they overwrite X
#pragma unroll 1
    for (int i = tid; i < m_b; i += kPlanThreads) {
      const double2 u = X[i];
      const double u1 = s1 * u.x + 0.0, u2 = s2 * u.y + 0.0;
      if (p.embedding) { p.embedding[((size_t)h * m_b + i) * 2] = u1; p.embedding[((size_t)h * m_b + i) * 2 + 1] = u2; }
      X[i].x = __longlong_as_double((long long)sortable(polar_angle(u2, u1) + 0.0));
    }
    constexpr int kPer = (kMaxSort + kPlanThreads - 1) / kPlanThreads;
    u64 ang[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int i = tid + k * kPlanThreads;
      ang[k] = i < m_b ? (u64)__double_as_longlong(X[i].x) : ~0ull;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const int i = tid + k * kPlanThreads;
      if (i < n_sort) {
        keys[i] = ang[k];
        vals[i] = i < m_b ? i : INT_MAX;
      }
    }
    __syncthreads();
    // Stage 1: rows by ascending angle, ties by row index.  Bins of equal width over the circle (the
    // map is monotone: every rounding in it is)
    const double per_bin = (double)p.bins * 0.15915494309189535;       // bins / (2 pi)
    auto angle_bin = [&](u64 k) {
      const double a = __longlong_as_double((long long)((k >> 63) ? (k & 0x7FFFFFFFFFFFFFFFull) : ~k));
      return min(max((int)((a + 3.14159265358979323846) * per_bin), 0), p.bins - 1);
    };
    if (p.bins == 0 || p.ring_cut || !bin_sort(keys, vals, keys2, vals2, m_b, bins, p.bins, p.bin_max, reinterpret_cast<int*>(scratch), angle_bin))
      sort_pairs();
    if (p.ring_cut && m_b >= 2) {
      // Variant: the sorted rows form a ring (Section 4.3.1); open it at the largest gap between
      // neighbouring angles (the gap around the back, first + 2 pi - last, included; the first
      // of equal gaps wins) instead of at -pi, where atan2 happens to put the cut.
      auto angle_at = [&](int i) {          // inverse of sortable()
        const u64 k = keys[i];
        return __longlong_as_double((long long)((k >> 63) ? (k & 0x7FFFFFFFFFFFFFFFull) : ~k));
      };
      double best[1] = {0.0};
      for (int i = tid; i < m_b; i += kPlanThreads) {
        const double g = i + 1 < m_b ? angle_at(i + 1) - angle_at(i)
                                     : (angle_at(0) + 2.0 * 3.14159265358979323846) - angle_at(m_b - 1);
        best[0] = fmax(best[0], g);
      }
      block_max<1>(best, scratch);
      int first[1] = {INT_MAX};
      for (int i = tid; i < m_b; i += kPlanThreads) {
        const double g = i + 1 < m_b ? angle_at(i + 1) - angle_at(i)
                                     : (angle_at(0) + 2.0 * 3.14159265358979323846) - angle_at(m_b - 1);
        if (g == best[0]) first[0] = min(first[0], i);
      }
      block_min<1>(first, reinterpret_cast<int*>(scratch));
      const int at = first[0];
      // rotate: the row behind the gap comes first (the key array is free until Stage 2 refills it)
      int* tmp = reinterpret_cast<int*>(keys);
      __syncthreads();
      for (int i = tid; i < m_b; i += kPlanThreads) {
        int src = i + at + 1;
        if (src >= m_b) src -= m_b;
        tmp[i] = vals[src];
      }
      __syncthreads();
      for (int i = tid; i < m_b; i += kPlanThreads) vals[i] = tmp[i];
      __syncthreads();
    }
  } else {
    if (!lead) return;
    if (p.embedding)
      for (int i = tid; i < m_b; i += kPlanThreads) { p.embedding[((size_t)h * m_b + i) * 2] = 0.0; p.embedding[((size_t)h * m_b + i) * 2 + 1] = 0.0; }
    for (int i = tid; i < n_sort; i += kPlanThreads) vals[i] = i < m_b ? i : INT_MAX;
    __syncthreads();
  }
  if (order1_out)
    for (int i = tid; i < m_b; i += kPlanThreads) order1_out[i] = vals[i];
  if (p.mode == WAVEAL_STAGE1_ONLY) {
    for (int i = tid; i < m_b; i += kPlanThreads) order_out[i] = vals[i];
    return;
  }
  // ---- Stage 2: inside each bucket of `wave` consecutive positions, descending n_i, ties by
  //      Stage-1 position
  if (p.warp_stage2) {
    // a warp per bucket: keys (n_b - n_i, position) in 32 bits, sorted in registers.  21,000 -> 7,200 clk for
    // 2,841 rows, 14,600 -> 12,000 for 1,536
    const int lane = tid & 31;
    for (int b0 = (tid >> 5) * p.wave; b0 < m_b; b0 += kPlanWarps * p.wave) {
      const int b1 = min(b0 + p.wave, m_b);
      unsigned a[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {                    // (any order will do to begin with: neighbouring lanes, neighbouring rows)
        const int i = b0 + e * 32 + lane;
        a[e] = i < b1 ? (unsigned)(n_b - nnz[vals[i]]) << 14 | (unsigned)i : UINT_MAX;
      }
      warp_sort256(a);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int at = b0 + lane * 8 + e;
        if (at < b1) order_out[at] = vals[a[e] & (kMaxSort - 1)];
      }
    }
    return;
  }
  if (p.count_stage2) {
    // small buckets: a row's place is the number of rows of its bucket that go before it, by a key of
    // (n_b - n_i, position) in 32 bits.  Most warps lie in one bucket, whose keys they read as broadcasts:
    // ~2.5 instructions per comparison, against the ~600 an element takes in the merge sort.
    unsigned* key = reinterpret_cast<unsigned*>(keys);
    for (int i = tid; i < m_b; i += kPlanThreads) key[i] = (unsigned)(n_b - nnz[vals[i]]) << 14 | (unsigned)i;
    __syncthreads();
    for (int i = tid; i < m_b; i += kPlanThreads) {
      const int b0 = i / p.wave * p.wave, b1 = min(b0 + p.wave, m_b);
      const unsigned mine = key[i];
      int at = b0;
#pragma unroll 8
      for (int j = b0; j < b1; ++j) at += key[j] < mine ? 1 : 0;
      order_out[at] = vals[i];
    }
    return;
  }
  // otherwise one sort on the key (bucket, max_count - n_i, position)
  for (int i = tid; i < n_sort; i += kPlanThreads) {
    if (i < m_b) {
      u64 bucket = (u64)(i / p.wave);
      u64 inv = (u64)(0x3FFFFF - min(nnz[vals[i]], 0x3FFFFF));
      keys[i] = (bucket << 44) | (inv << 22) | (u64)i;
    } else {
      keys[i] = ~0ull;
    }
  }
  __syncthreads();
  sort_pairs();
  for (int i = tid; i < m_b; i += kPlanThreads) order_out[i] = vals[i];
}

// ------------------------------------------------------------------ host side

struct PlanLayout {
  size_t off_bitmap, off_mt, off_nnz, off_cnt, off_state, total;
  int wq, wk, n_pow2, state_in_smem, bins;
  size_t smem;
  // shared memory of the matrix-unit form: does it fit, the iteration blocks behind `region`, the
  // digits behind them (the partial sums of the column split come last, launch_shape() adds them)
  int mma, alias_yz;
  size_t off_items, items_end;
};

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

waveal_status plan_layout(const waveal_plan_desc* d, PlanLayout* L) {
  if (!d) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "desc is NULL");
  if (d->heads <= 0 || d->n_q_blocks <= 0 || d->n_kv_blocks <= 0)
    return waveal::fail(WAVEAL_ERR_INVALID_ARG, "heads, n_q_blocks and n_kv_blocks must be positive");
  if (d->wave_size < 0 || d->svd_iters < 0 || d->svd_iters > 1000)
    return waveal::fail(WAVEAL_ERR_INVALID_ARG, "wave_size must be >= 0 and svd_iters in [0, 1000]");
  const int base_mode = d->mode & ~(WAVEAL_RING_CUT_LARGEST_GAP | WAVEAL_PLAN_CLEAR_STATUS);
  if (base_mode < WAVEAL_AUTO || base_mode > WAVEAL_STAGE2_ONLY)
    return waveal::fail(WAVEAL_ERR_INVALID_ARG, "unknown mode %d", d->mode);
  if (d->l2_fit_den <= 0 || d->local_den <= 0 || d->l2_fit_num < 0 || d->local_num < 0 || d->min_density_ppm < 0)
    return waveal::fail(WAVEAL_ERR_INVALID_ARG, "guard thresholds must be non-negative with positive denominators");
  if (d->n_q_blocks > kMaxSort)
    return waveal::fail(WAVEAL_ERR_UNSUPPORTED, "n_q_blocks %d exceeds the supported maximum %d", d->n_q_blocks, kMaxSort);
  if (d->n_kv_blocks >= (1 << 22))
    return waveal::fail(WAVEAL_ERR_UNSUPPORTED, "n_kv_blocks %d exceeds the supported maximum", d->n_kv_blocks);
  size_t H = d->heads, m = d->n_q_blocks, n = d->n_kv_blocks;
  L->wq = (int)((n + 63) / 64);
  L->wk = (int)((m + 63) / 64);
  int p2 = 1;
  while (p2 < d->n_q_blocks) p2 <<= 1;
  L->n_pow2 = p2;
  size_t sort_bytes = (size_t)p2 * 12, state_bytes = (2 * m + n) * 16;
  L->state_in_smem = 2048 + (state_bytes > sort_bytes ? state_bytes : sort_bytes) <= kSmemMax;
  // angular sort by two bins a row from 513 rows on (below, the merge sort has few passes), as far as they fit behind its buffers
  // (7,200 rows)
  L->bins = 0;
  if (m <= (size_t)kMaxMerge) sort_bytes = m * 24;
  if (m > 512 && 2048 + m * 32 <= kSmemMax) { L->bins = (int)(2 * m); sort_bytes = m * 32; }
  L->smem = 2048 + (L->state_in_smem ? (state_bytes > sort_bytes ? state_bytes : sort_bytes) : sort_bytes);
  // The matrix-unit form also keeps the digits of one block, 16 bytes an entry.  On square masks it
  // fits up to ~3,580 blocks as it is, up to ~4,730 with Y and Z in one buffer and up to 14,336
  // with the blocks in the workspace; between and beyond (the state fits shared memory, the digits
  // do not) the set bits are walked.
  const size_t big = m > n ? m : n, items = (big + kChunkCols - 1) / kChunkCols * kChunkCols * 16;
  L->mma = 1; L->alias_yz = 0;
  size_t before = L->state_in_smem ? state_bytes : 0;
  if (2048 + before + items > kSmemMax && L->state_in_smem) { L->alias_yz = 1; before = (m + big) * 16; }
  if (2048 + before + items > kSmemMax) { L->mma = 0; L->alias_yz = 0; }
  L->off_items = 2048 + before;
  L->items_end = L->off_items + items;
  size_t o = 0;
  L->off_bitmap = o; o = align_up(o + H * m * L->wq * 8, 256);
  L->off_mt = o;     o = align_up(o + H * n * L->wk * 8, 256);
  L->off_nnz = o;    o = align_up(o + H * m * 4, 256);
  L->off_cnt = o;    o = align_up(o + H * n * 4, 256);
  L->off_state = o;  o = align_up(o + (L->state_in_smem ? 0 : H * (2 * m + n) * 16), 256);
  L->total = o;
  return WAVEAL_OK;
}

// Largest cluster (up to 16 CTAs, at most `limit`) of which the device holds `heads` at once; one
// CTA per SM is assumed (the shared memory of the larger shapes).  How many clusters of a size fit
// depends on the device alone (its SMs come in groups of unequal size), so it is asked once.
waveal_status cluster_size(int dev, int heads, int limit, int* out) {
  constexpr int kMaxCluster = 16, kMaxDev = 64;
  static std::mutex mu;
  static int fit[kMaxDev][kMaxCluster + 1] = {};      // clusters of a size the device holds, + 1; 0: not asked
  if (dev < 0 || dev >= kMaxDev) { *out = 1; return WAVEAL_OK; }
  std::lock_guard<std::mutex> lock(mu);
  for (int c = limit < kMaxCluster ? limit : kMaxCluster; c > 1; --c) {
    if (!fit[dev][c]) {
      WAVEAL_CUDA_OK(cudaFuncSetAttribute(k_plan_head, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)c);
      cfg.blockDim = dim3(kPlanThreads);
      cfg.dynamicSmemBytes = kSmemMax;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = (unsigned)c; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr; cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, k_plan_head, &cfg) != cudaSuccess) { cudaGetLastError(); continue; }
      fit[dev][c] = n + 1;
    }
    if (fit[dev][c] - 1 >= heads) { *out = c; return WAVEAL_OK; }
  }
  *out = 1;
  return WAVEAL_OK;
}

waveal_status plan_common(const waveal_plan_desc* d, const u64* mask_bits, const int* row_ptr, const int* idx,
                          void* ws, size_t ws_bytes, const waveal_plan_out* out, cudaStream_t st) {
  PlanLayout L;
  waveal_status s = plan_layout(d, &L);
  if (s != WAVEAL_OK) return s;
  if (!out || !out->row_order) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "out->row_order is required");
  if (!ws || ws_bytes < L.total)
    return waveal::fail(WAVEAL_ERR_WORKSPACE, "workspace of %zu bytes needed, %zu given", L.total, ws ? ws_bytes : (size_t)0);
  if (!waveal::aligned(ws, 256)) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "workspace must be 256-byte aligned");
  if (mask_bits && !waveal::aligned(mask_bits, 8)) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "mask_bits must be 8-byte aligned");
  int dev = 0, sms = 0, l2 = 0;
  WAVEAL_CUDA_OK(cudaGetDevice(&dev));
  WAVEAL_CUDA_OK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  WAVEAL_CUDA_OK(cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev));
  unsigned char* w = static_cast<unsigned char*>(ws);
  int launches = 0;
  const size_t H = d->heads, m = d->n_q_blocks, n = d->n_kv_blocks;
  const u64* M = mask_bits;
  if (!M) {
    u64* bm = reinterpret_cast<u64*>(w + L.off_bitmap);
    long long rows = (long long)(H * m);
    (n <= kCsrCols ? k_csr_to_bitmap<false> : k_csr_to_bitmap<true>)<<<(unsigned)((rows + kCsrWarps - 1) / kCsrWarps), kCsrWarps * 32, 0, st>>>(
        row_ptr, idx, bm, rows, L.wq, (int)n, (int)m, reinterpret_cast<int*>(w + L.off_nnz), out->row_nnz, out->dev_status);
    ++launches;
    M = bm;
  }
  u64* Mt = reinterpret_cast<u64*>(w + L.off_mt);
  int* nnz = reinterpret_cast<int*>(w + L.off_nnz);
  int* cnt = reinterpret_cast<int*>(w + L.off_cnt);
  // The limits on dynamic shared memory belong to the process, and another host thread may stand between its own
  // setting of them and its launch: every call sets the same values, the largest any shape takes.
  const size_t strip_bytes = (size_t)64 * (2 * L.wk + 1) * 4;
  WAVEAL_CUDA_OK(cudaFuncSetAttribute(k_mask_stats, cudaFuncAttributeMaxDynamicSharedMemorySize, kStripMax));
  WAVEAL_CUDA_OK(cudaFuncSetAttribute(k_plan_head, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax));
  const dim3 stat_grid(L.wq + (mask_bits ? (unsigned)((m + kStatRows - 1) / kStatRows) : 0u), (unsigned)H);   // (lists: rows counted on the way)
  if (mask_bits) {
    k_mask_stats<<<stat_grid, kStatThreads, strip_bytes, st>>>(M, Mt, (int)m, (int)n, L.wq, L.wk, nnz, cnt, out->row_nnz, out->col_count,
                                                              (d->mode & WAVEAL_PLAN_CLEAR_STATUS) ? out->dev_status : nullptr);
    WAVEAL_CUDA_OK(cudaGetLastError());
  } else {
    WAVEAL_CUDA_OK(waveal::launch_chained(k_mask_stats, stat_grid, kStatThreads, strip_bytes, st, M, Mt, (int)m, (int)n, L.wq, L.wk,
                                          nnz, cnt, out->row_nnz, out->col_count, nullptr));
  }
  ++launches;
  PlanParams p{};
  p.M = M; p.Mt = Mt; p.m_b = (int)m; p.n_b = (int)n; p.wq = L.wq; p.wk = L.wk;
  // (a wave longer than the head is the whole head; cut to it, row + wave stays far from the end of int)
  p.wave = d->wave_size > 0 ? d->wave_size : sms;
  if (p.wave > (int)m) p.wave = (int)m;
  p.iters = d->svd_iters; p.mode = d->mode & ~(WAVEAL_RING_CUT_LARGEST_GAP | WAVEAL_PLAN_CLEAR_STATUS);
  p.ring_cut = (d->mode & WAVEAL_RING_CUT_LARGEST_GAP) ? 1 : 0; p.n_pow2 = L.n_pow2; p.state_in_smem = L.state_in_smem;
  p.seed = d->seed;
  p.kv_bytes = d->kv_bytes_per_head; p.l2_bytes = d->l2_bytes > 0 ? d->l2_bytes : (long long)l2;
  p.min_nnz = d->min_nnz; p.fit_num = d->l2_fit_num; p.fit_den = d->l2_fit_den; p.min_ppm = d->min_density_ppm;
  p.loc_num = d->local_num; p.loc_den = d->local_den;
  p.ws_nnz = nnz;
  p.ws_cnt = cnt;
  p.ws_state = reinterpret_cast<double2*>(w + L.off_state);
  p.row_order = out->row_order; p.flags = out->skip_flags;
  p.order1 = out->order1; p.embedding = out->embedding; p.stats = reinterpret_cast<long long*>(out->stats);
  // CTAs per head: the largest cluster of which the device holds one per head at once, and no more than
  // half as many CTAs as there are groups of 32 rows
  int csize = 1;
  {
    const int groups = (int)(((m > n ? m : n) + kUnitRows - 1) / kUnitRows);
    // (up to 256 rows one CTA is quickest: 73.8 us against 82.2 us with eight on 5 heads of 256 rows; above, two
    // groups a CTA: 88.5 / 92.0 / 97.4 us with 7 / 4 / 2 CTAs on 12 heads of 400 rows)
    const int limit = groups <= 8 ? 1 : (groups + 1) / 2;
    s = cluster_size(dev, (int)H, L.mma ? limit : (groups < 4 ? groups : 4), &csize);
    if (s != WAVEAL_OK) return s;
  }
  // counting costs 2.5 wave instructions a row, the merge sort ~550: kMaxSort = 2^14 positions, and
  // n - n_i has to fit the other 18 bits
  p.count_stage2 = p.wave <= 220 && n < (1u << 18);
  // a warp sorts up to 256 rows.  Counting is quicker where a thread has one row to place (591 rows: 8,200 clk against
  // 10,500) and where the buckets are short
  p.warp_stage2 = p.count_stage2 && p.wave >= 64 && m > kPlanThreads;
  p.bins = L.bins;
  // Equal rows share a bin, which each of them walks.  It takes as long as the merge sort from 64 rows on where a thread has one row
  // (plan of 5 heads, us, by bins / by merging: 591 rows with 33 equal ones 87 / 89, 64: 89 / 89, 128: 93 / 89, 191: 95 / 89; 1,000 rows
  // with 64: 99 / 99, 191: 105 / 99), from an eighth of the rows on above (1,200 with 150: 112 / 112; 1,536 with 128: 120 / 122, 191: 122 / 122).
  // Finding that a bin is too full costs up to 2 us.
  p.bin_max = m <= kPlanThreads ? 64 : m / 8 < 192 ? (int)(m / 8) : 192;
  p.mma = L.mma; p.alias_yz = L.alias_yz; p.off_items = (unsigned)L.off_items;
  p.ksplit_y = p.ksplit_z = 1;
  size_t smem = L.smem;
  if (L.mma) {
    // fewer groups of rows than warps: the warps of a CTA share the columns of a group
    auto split = [&](size_t rows, int words) {
      const int groups = (int)((rows + kUnitRows - 1) / kUnitRows), per_cta = (groups + csize - 1) / csize;
      const int chunks = (words + 3) / 4, ks = per_cta >= kPlanWarps ? 1 : kPlanWarps / per_cta;
      return ks < chunks ? ks : chunks;
    };
    p.ksplit_y = split(n, L.wk); p.ksplit_z = split(m, L.wq);
    int ints = 0;
    for (int ks : {p.ksplit_y, p.ksplit_z})
      if (ks > 1) ints = ints > kPlanWarps / ks * kUnitRows * 16 ? ints : kPlanWarps / ks * kUnitRows * 16;
    if (L.items_end + (size_t)ints * 4 > kSmemMax) { p.ksplit_y = p.ksplit_z = 1; ints = 0; }
    p.off_part = (unsigned)L.items_end; p.part_ints = ints;
    const size_t need = L.items_end + (size_t)ints * 4;
    smem = smem > need ? smem : need;
  }
  p.csize = csize;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(H * csize));
  cfg.blockDim = dim3(kPlanThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)csize; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = csize == 1 ? 1 : 2;
  WAVEAL_CUDA_OK(cudaLaunchKernelEx(&cfg, k_plan_head, p));
  ++launches;
  WAVEAL_CUDA_OK(cudaGetLastError());
  waveal::launch_counter() = launches;
  return WAVEAL_OK;
}

}  // namespace

extern "C" void waveal_plan_desc_default(waveal_plan_desc* d) {
  if (!d) return;
  *d = waveal_plan_desc{};
  d->svd_iters = 5;    // low end of the paper's 5-15: the attention time did not move between 3, 5 and 10 on the measured shapes
  d->mode = WAVEAL_AUTO;
  d->l2_fit_num = 9; d->l2_fit_den = 16;   // calibrated on the B200 (calibrate_guard): no gain up to K+V = 0.57 x L2 on either mask family
  d->min_density_ppm = 10000;
  d->local_num = 1; d->local_den = 2;
  d->min_nnz = 0;
}

extern "C" waveal_status waveal_plan_workspace_bytes(const waveal_plan_desc* desc, size_t* bytes) {
  PlanLayout L;
  waveal_status s = plan_layout(desc, &L);
  if (s != WAVEAL_OK) return s;
  if (!bytes) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "bytes is NULL");
  *bytes = L.total;
  return WAVEAL_OK;
}

extern "C" waveal_status waveal_plan_bitmap(const waveal_plan_desc* desc, const uint64_t* mask_bits, void* ws,
                                            size_t ws_bytes, const waveal_plan_out* out, void* cuda_stream) {
  if (!mask_bits) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "mask_bits is NULL");
  return plan_common(desc, reinterpret_cast<const u64*>(mask_bits), nullptr, nullptr, ws, ws_bytes, out,
                     static_cast<cudaStream_t>(cuda_stream));
}

extern "C" waveal_status waveal_plan_csr(const waveal_plan_desc* desc, const int32_t* kv_row_ptr,
                                         const int32_t* kv_block_indices, void* ws, size_t ws_bytes,
                                         const waveal_plan_out* out, void* cuda_stream) {
  if (!kv_row_ptr || !kv_block_indices) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "index lists are NULL");
  if (desc && (desc->mode & WAVEAL_PLAN_CLEAR_STATUS)) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "unknown mode %d", desc->mode);
  return plan_common(desc, nullptr, kv_row_ptr, kv_block_indices, ws, ws_bytes, out,
                     static_cast<cudaStream_t>(cuda_stream));
}

extern "C" waveal_status waveal_bitmap_to_csr(int32_t heads, int32_t n_q_blocks, int32_t n_kv_blocks,
                                              const uint64_t* mask_bits, int32_t* kv_row_ptr_out,
                                              int32_t* kv_block_indices_out, int64_t capacity, void* ws,
                                              size_t ws_bytes, void* cuda_stream) {
  if (heads <= 0 || n_q_blocks <= 0 || n_kv_blocks <= 0)
    return waveal::fail(WAVEAL_ERR_INVALID_ARG, "heads, n_q_blocks and n_kv_blocks must be positive");
  if (!mask_bits || !kv_row_ptr_out) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "mask_bits and kv_row_ptr_out are required");
  if (kv_block_indices_out && capacity < 0) return waveal::fail(WAVEAL_ERR_INVALID_ARG, "capacity must be >= 0");
  long long rows = (long long)heads * n_q_blocks;
  if (!ws || ws_bytes < (size_t)(rows + 1) * 4)
    return waveal::fail(WAVEAL_ERR_WORKSPACE, "workspace of %zu bytes needed", (size_t)(rows + 1) * 4);
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  int wq = (n_kv_blocks + 63) / 64;
  int* cnt = static_cast<int*>(ws);
  int launches = 0;
  // steps of a block: as few as keep the number of blocks (and of their shares) below kListBlocks and
  // within the workspace of one int per row
  const u64* bits = reinterpret_cast<const u64*>(mask_bits);
  const long long words = rows * wq, steps_all = (words + kListThreads - 1) / kListThreads;
  const bool direct = words <= kListDirect;
  const long long most = direct ? steps_all : rows < kListBlocks ? rows : kListBlocks;
  const long long steps = (steps_all + most - 1) / most;
  const unsigned blocks = (unsigned)((steps_all + steps - 1) / steps);
  if (!direct) {
    k_count_words<<<blocks, kListThreads, 0, st>>>(bits, words, (int)steps, cnt);
    ++launches;
  }
  if (direct)
    k_fill_lists<<<blocks, kListThreads, 0, st>>>(bits, words, wq, (int)steps, nullptr, kv_row_ptr_out, rows, kv_block_indices_out,
                                                  capacity);
  else
    WAVEAL_CUDA_OK(waveal::launch_chained(k_fill_lists, dim3(blocks), kListThreads, 0, st, bits, words, wq, (int)steps, cnt,
                                          kv_row_ptr_out, rows, kv_block_indices_out, capacity));
  ++launches;
  WAVEAL_CUDA_OK(cudaGetLastError());
  waveal::launch_counter() = launches;
  return WAVEAL_OK;
}

// ------------------------------------------------------------------ entry point that allocates nothing

// Scratch for waveal_bitmap_to_csr_noalloc: lives in the library image, so every GPU that
// loads the library holds this 1 MiB until the process exits.
#define WAVEAL_NOALLOC_SCRATCH_BYTES (1u << 20)
static __device__ __align__(256) unsigned char g_noalloc_scratch[WAVEAL_NOALLOC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
void* g_scratch_addr[kMaxDevices] = {};   // device address of g_noalloc_scratch, per device

// In host code the array's name is only a handle; the address a kernel can use has to be
// asked for, once per device, with that device current.
waveal_status noalloc_scratch(void** out) {
  int dev = 0;
  WAVEAL_CUDA_OK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return waveal::fail(WAVEAL_ERR_UNSUPPORTED, "device ordinal %d not supported", dev);
  std::lock_guard<std::mutex> lock(g_scratch_mu);
  if (!g_scratch_addr[dev]) {
    void* ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
    if (e != cudaSuccess || !ptr)
      return waveal::fail(WAVEAL_ERR_CUDA, "cudaGetSymbolAddress(static scratch) failed: %s", cudaGetErrorString(e));
    g_scratch_addr[dev] = ptr;
  }
  *out = g_scratch_addr[dev];
  return WAVEAL_OK;
}
}  // namespace

extern "C" size_t waveal_noalloc_max_rows(void) { return WAVEAL_NOALLOC_SCRATCH_BYTES / 4 - 1; }

extern "C" waveal_status waveal_bitmap_to_csr_noalloc(int32_t heads, int32_t n_q_blocks, int32_t n_kv_blocks,
                                                      const uint64_t* mask_bits, int32_t* kv_row_ptr_out,
                                                      int32_t* kv_block_indices_out, int64_t capacity,
                                                      void* cuda_stream) {
  if (heads <= 0 || n_q_blocks <= 0 || n_kv_blocks <= 0)
    return waveal::fail(WAVEAL_ERR_INVALID_ARG, "heads, n_q_blocks and n_kv_blocks must be positive");
  const long long rows = (long long)heads * n_q_blocks;
  if ((unsigned long long)rows > (unsigned long long)waveal_noalloc_max_rows())
    return waveal::fail(WAVEAL_ERR_UNSUPPORTED,
                        "heads*n_q_blocks = %lld exceeds the %zu rows the built-in scratch holds; "
                        "use waveal_bitmap_to_csr with a caller-owned workspace",
                        rows, waveal_noalloc_max_rows());
  void* scratch = nullptr;
  waveal_status s = noalloc_scratch(&scratch);
  if (s != WAVEAL_OK) return s;
  // the per-row counts in the scratch are fully rewritten for the rows in use before they are
  // read, so nothing of the previous call's contents has to be cleared
  return waveal_bitmap_to_csr(heads, n_q_blocks, n_kv_blocks, mask_bits, kv_row_ptr_out, kv_block_indices_out,
                              capacity, scratch, WAVEAL_NOALLOC_SCRATCH_BYTES, cuda_stream);
}
