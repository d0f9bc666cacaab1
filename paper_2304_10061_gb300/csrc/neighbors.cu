// Ordered neighbour pairs within r_c (Sec. "Allegro": E_i = sum_j E_ij over
// ordered pairs; Sec. "Species-dependent cutoffs").
//
// Cell list: atoms are binned by fractional coordinate into cells whose
// perpendicular widths are at least r_c (1 + 1e-6), counting-sorted by cell
// (each cell's list then ordered by atom index, so the traversal is
// deterministic), and each centre scans the (2R+1)^3 stencil of cells around
// its own.  A candidate's image shift S follows from the stencil wrap and the
// two atoms' wrap counts, and the pair is kept iff the float64 displacement
//   off[x] = (S0*a[x] + S1*b[x]) + S2*c[x];  d[x] = (pos_j[x] + off[x]) - pos_i[x]
//   r2 = (d0*d0 + d1*d1) + d2*d2  <  r_c^2,   not (i == j and S == 0)
// evaluated with explicitly rounded operations (no contraction), i.e. the
// same rule the oracle applies to every candidate.  Counting pass, exclusive
// scan, fill pass: rows come out in ascending centre index.  A CSC index
// (edges grouped by neighbour j, ascending edge id) serves the force gather.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "launch.cuh"

namespace alg {

__device__ __forceinline__ int floordiv(int a, int b) {
  int q = a / b;
  if ((a % b != 0) && ((a < 0) != (b < 0))) --q;
  return q;
}

// ---------------------------------------------------------------------------
// exclusive scan of int32 (out has n+1 entries; out[n] = total).  With `clear`
// the input is zeroed as it is read (the counters the next build adds to).
// The entries are counts, and their sums stop at INT_MAX: a list of 2^32 edges and some would otherwise
// show the host a small total, and the fill pass would write its rows at wrapped offsets.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int add_sat(int a, int b) { return (int)min((unsigned)a + (unsigned)b, 0x7fffffffu); }

constexpr int kScanBlock = 1024;   // elements per block of the large scan (256 threads x 4)

__device__ __forceinline__ int warp_inclusive(int x, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x = add_sat(x, y);
  }
  return x;
}

// THREADS x PER elements by one block, thread t the elements [t PER, (t + 1) PER) of its tile
// (PER a multiple of 4: 16-byte accesses; both arrays start 16-byte aligned at a tile's first element)
template <int THREADS, int PER>
__device__ __forceinline__ int block_scan_tile(int* __restrict__ in, int* __restrict__ out, int n, int base,
                                               bool clear) {
  constexpr int kWarps = THREADS / 32;
  __shared__ int warp_tot[kWarps];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int b = base + t * PER;
  int v[PER];
#pragma unroll
  for (int k = 0; k < PER; k += 4) {
    if (b + k + 3 < n) {
      const int4 x = *reinterpret_cast<const int4*>(in + b + k);
      v[k] = x.x; v[k + 1] = x.y; v[k + 2] = x.z; v[k + 3] = x.w;
      if (clear) *reinterpret_cast<int4*>(in + b + k) = make_int4(0, 0, 0, 0);
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        v[k + q] = (b + k + q < n) ? in[b + k + q] : 0;
        if (clear && b + k + q < n) in[b + k + q] = 0;
      }
    }
  }
  int s = 0;
#pragma unroll
  for (int k = 0; k < PER; ++k) s = add_sat(s, v[k]);
  const int x = warp_inclusive(s, lane);
  const int before = __shfl_up_sync(0xffffffffu, x, 1);
  if (lane == 31) warp_tot[w] = x;
  __syncthreads();
  if (w == 0) {
    const int wt = warp_inclusive(lane < kWarps ? warp_tot[lane] : 0, lane);
    if (lane < kWarps) warp_tot[lane] = wt;
  }
  __syncthreads();
  int excl = add_sat(lane > 0 ? before : 0, w > 0 ? warp_tot[w - 1] : 0);
#pragma unroll
  for (int k = 0; k < PER; k += 4) {
    int4 y;
    y.x = excl; y.y = add_sat(y.x, v[k]); y.z = add_sat(y.y, v[k + 1]); y.w = add_sat(y.z, v[k + 2]);
    excl = add_sat(y.w, v[k + 3]);
    if (b + k + 3 <= n) {
      *reinterpret_cast<int4*>(out + b + k) = y;
    } else {
      if (b + k <= n) out[b + k] = y.x;
      if (b + k + 1 <= n) out[b + k + 1] = y.y;
      if (b + k + 2 <= n) out[b + k + 2] = y.z;
    }
  }
  return warp_tot[kWarps - 1];
}

template <int PER>
__global__ void __launch_bounds__(1024) scan_one_kernel(int* in, int* out, int n, bool clear, int* total) {
  pdl_wait();
  const int t = block_scan_tile<1024, PER>(in, out, n, 0, clear);
  if (total && threadIdx.x == 0) *total = t;
}

__global__ void scan_block_kernel(int* in, int* out, int n, int* __restrict__ block_sums, bool clear) {
  pdl_wait();
  const int total = block_scan_tile<256, 4>(in, out, n, blockIdx.x * kScanBlock, clear);
  if (threadIdx.x == 255) block_sums[blockIdx.x] = total;
}

__global__ void scan_add_kernel(int* __restrict__ out, int n, const int* __restrict__ block_pref, int* total) {
  pdl_wait();
  const int base = blockIdx.x * kScanBlock;
  const int add = block_pref[blockIdx.x];
  for (int k = threadIdx.x; k < kScanBlock; k += blockDim.x) {
    int idx = base + k;
    if (idx <= n) {
      const int v = add_sat(out[idx], add);
      out[idx] = v;
      if (total && idx == n) *total = v;
    }
  }
}

// ints of a scan's block sums (or prefixes), rounded so that the next array stays 16-byte aligned
static int scan_pitch(int nb) { return (nb + 1 + 3) / 4 * 4; }

size_t scan_tmp_bytes(int n) {
  size_t total = 0;
  int m = n + 1;
  while (m > 1) {
    int nb = (m + kScanBlock - 1) / kScanBlock;
    total += (size_t)scan_pitch(nb) * 2 * sizeof(int) + 256;
    m = nb;
  }
  return total + 256;
}

// Scans in[0..n) into out[0..n] (out[n] = total).  Up to 32 x 1024 elements one block does it in
// one launch (about 3 us against 6 for the three launches of the block-wise scan at 16k elements:
// the launches are the time at these sizes); above, block sums, their scan, and an add.
static void scan_rec(int* in, int* out, int n, char* tmp, bool clear, int* total, cudaStream_t st) {
  if (n < 4 * 1024) {
    launch(scan_one_kernel<4>, 1, 1024, 0, st, in, out, n, clear, total);
    return;
  }
  if (n < 32 * 1024) {
    launch(scan_one_kernel<32>, 1, 1024, 0, st, in, out, n, clear, total);
    return;
  }
  const int nb = (n + 1 + kScanBlock - 1) / kScanBlock;
  int* sums = reinterpret_cast<int*>(tmp);
  int* pref = sums + scan_pitch(nb);
  char* next = reinterpret_cast<char*>(pref + scan_pitch(nb)) + 256;
  launch(scan_block_kernel, nb, 256, 0, st, in, out, n, sums, clear);
  scan_rec(sums, pref, nb, next, false, nullptr, st);
  launch(scan_add_kernel, nb, 256, 0, st, out, n, pref, total);
}

int exclusive_scan_i32(int* in, int* out, int n, void* tmp, bool clear, int* total, cudaStream_t st) {
  scan_rec(in, out, n, reinterpret_cast<char*>(tmp), clear, total, st);
  int launches = 1;
  for (int m = n; m >= 32 * 1024; m = (m + 1 + kScanBlock - 1) / kScanBlock) launches += 2;
  return launches;
}

// ---------------------------------------------------------------------------
// binning
// ---------------------------------------------------------------------------
__device__ __forceinline__ void frac_of(const double* p, const double* inv, double f[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) f[k] = p[0] * inv[0 * 3 + k] + p[1] * inv[1 * 3 + k] + p[2] * inv[2 * 3 + k];
}

// monotone map double -> unsigned long long for atomic min/max
__device__ __forceinline__ unsigned long long dkey(double x) {
  unsigned long long b = __double_as_longlong(x);
  return (b & 0x8000000000000000ull) ? ~b : (b | 0x8000000000000000ull);
}

__global__ void minmax_frac_kernel(const double* __restrict__ pos, int n, CellGrid g,
                                   unsigned long long* __restrict__ mm) {
  pdl_wait();
  double lo[3] = {1e300, 1e300, 1e300}, hi[3] = {-1e300, -1e300, -1e300};
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double f[3];
    frac_of(pos + 3 * (size_t)i, g.inv, f);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      lo[k] = fmin(lo[k], f[k]);
      hi[k] = fmax(hi[k], f[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    for (int o = 16; o > 0; o >>= 1) {
      lo[k] = fmin(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
      hi[k] = fmax(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
    }
    if ((threadIdx.x & 31) == 0) {
      atomicMin(&mm[k], dkey(lo[k]));
      atomicMax(&mm[3 + k], dkey(hi[k]));
    }
  }
}

__global__ void minmax_init_kernel(unsigned long long* mm) {
  pdl_wait();
  int k = threadIdx.x;
  if (k < 3) mm[k] = ~0ull;
  else if (k < 6) mm[k] = 0ull;
}

__global__ void minmax_decode_kernel(const unsigned long long* mm, double* out) {
  pdl_wait();
  int k = threadIdx.x;
  if (k < 6) {
    unsigned long long b = mm[k];
    b = (b & 0x8000000000000000ull) ? (b & 0x7fffffffffffffffull) : ~b;
    out[k] = __longlong_as_double((long long)b);
  }
}

void nb_minmax_frac(const double* pos, int n, const double* inv, double* d_minmax, cudaStream_t st) {
  CellGrid g{};
  for (int k = 0; k < 9; ++k) g.inv[k] = inv[k];
  unsigned long long* mm = reinterpret_cast<unsigned long long*>(d_minmax + 6);
  launch(minmax_init_kernel, 1, 32, 0, st, mm);
  int blocks = (n + 255) / 256;
  if (blocks > 1184) blocks = 1184;
  if (blocks < 1) blocks = 1;
  launch(minmax_frac_kernel, blocks, 256, 0, st, pos, n, g, mm);
  launch(minmax_decode_kernel, 1, 32, 0, st, mm, d_minmax);
}

__global__ void bin_kernel(const double* __restrict__ pos, int n, CellGrid g, int* __restrict__ cell_of,
                           int* __restrict__ wrap, int* __restrict__ cell_count, int* __restrict__ cell_rank) {
  pdl_wait();
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double f[3];
  frac_of(pos + 3 * (size_t)i, g.inv, f);
  int c[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    double x;
    int w = 0;
    if (g.pbc[k]) {
      double fl = floor(f[k]);
      w = (int)fl;
      x = f[k] - fl;
    } else {
      x = (g.span[k] > 0) ? (f[k] - g.lo[k]) / g.span[k] : 0.0;
    }
    int ck = (int)floor(x * g.n[k]);
    ck = ck < 0 ? 0 : (ck >= g.n[k] ? g.n[k] - 1 : ck);
    c[k] = ck;
    wrap[3 * (size_t)i + k] = w;
  }
  int id = (c[0] * g.n[1] + c[1]) * g.n[2] + c[2];
  cell_of[i] = id;
  cell_rank[i] = atomicAdd(&cell_count[id], 1);
}

void nb_bin(const double* pos, int n, const CellGrid& g, int* cell_of, int* wrap, int* cell_count, int* cell_rank,
            cudaStream_t st) {
  if (n <= 0) return;
  launch(bin_kernel, (n + 255) / 256, 256, 0, st, pos, n, g, cell_of, wrap, cell_count, cell_rank);
}

__global__ void place_kernel(const int* __restrict__ seg_of, const int* __restrict__ rank, int n,
                             const int* __restrict__ start, int* __restrict__ sorted) {
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) sorted[start[seg_of[i]] + rank[i]] = i;
}

void nb_place(const int* seg_of, const int* rank, int n, const int* start, int* sorted, cudaStream_t st) {
  if (n <= 0) return;
  launch(place_kernel, (n + 255) / 256, 256, 0, st, seg_of, rank, n, start, sorted);
}

// The fill passes and what follows them are queued before the host knows the edge count: they take
// the arrays' capacity and read the count (row_ptr[n]); a list that does not fit is left unwritten.
__device__ __forceinline__ bool list_fits(const int* __restrict__ row_ptr, int n, int edge_cap) {
  return (unsigned)row_ptr[n] <= (unsigned)edge_cap;
}

constexpr int kEdgeBlocks = 152 * 16;   // most blocks of the passes over a list of unknown length

__global__ void __launch_bounds__(256) place_edges_kernel(const int* __restrict__ ej, const int* __restrict__ rank,
                                                          const int* __restrict__ row_ptr, int n, int edge_cap,
                                                          const int* __restrict__ col_ptr, int* __restrict__ col_edge) {
  pdl_wait();
  if (!list_fits(row_ptr, n, edge_cap)) return;
  const int E = row_ptr[n];
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < E; e += gridDim.x * blockDim.x)
    col_edge[col_ptr[ej[e]] + rank[e]] = e;
}

void nb_place_edges(const int* ej, const int* rank, const int* row_ptr, int n, int edge_cap, const int* col_ptr,
                    int* col_edge, cudaStream_t st) {
  if (edge_cap <= 0) return;
  const int blocks = std::min((int)(((int64_t)edge_cap + 255) / 256), kEdgeBlocks);
  launch(place_edges_kernel, blocks, 256, 0, st, ej, rank, row_ptr, n, edge_cap, col_ptr, col_edge);
}

// Sort each segment [start[s], start[s+1]) of distinct values: G lanes per segment hold up to 4 G
// values in registers and each value's rank is the number of smaller ones (a broadcast per value),
// so a segment takes a few dependent loads instead of an insertion sort's chain through memory.
// Longer segments are ranked 8 G values at a time against all of theirs, read from memory, and go
// through `tmp` (as long as v).  Liquids reach all of these: at the density of water a column holds 27
// edges at a cutoff of 4 Angstrom, 90 at 6, 214 at 8.  Column passes at 262,144 atoms, us, an insertion
// sort per thread / by one lane past 4 G values / now: 4 Angstrom 244 / 130 / 130, 6 Angstrom 1,107 /
// 3,259 / 638, 8 Angstrom 3,427 / 17,382 / 2,157.
// done(place, value) is called for every element of the segment.
template <int G, int K, typename Done>
__device__ __forceinline__ void sort_in_registers(int b, int len, int* __restrict__ v, unsigned mask, Done&& done) {
  const int lane = threadIdx.x & (G - 1);
  int x[K], r[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    x[k] = (k * G + lane < len) ? v[b + k * G + lane] : 0x7fffffff;
    r[k] = 0;
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int m = min(G, len - k * G);
    for (int q = 0; q < m; ++q) {
      const int y = __shfl_sync(mask, x[k], q, G);
#pragma unroll
      for (int p = 0; p < K; ++p) r[p] += (y < x[p]) ? 1 : 0;
    }
  }
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (k * G + lane < len) {
      v[b + r[k]] = x[k];
      done(b + r[k], x[k]);
    }
}

template <int G, typename Done>
__device__ __forceinline__ void sort_segment(int b, int len, int* __restrict__ v, int* __restrict__ tmp, Done&& done) {
  const int lane = threadIdx.x & (G - 1);
  const unsigned mask = ((1u << G) - 1u) << (threadIdx.x & 31 & ~(G - 1));
  if (len <= G) {
    sort_in_registers<G, 1>(b, len, v, mask, done);
  } else if (len <= 2 * G) {
    sort_in_registers<G, 2>(b, len, v, mask, done);
  } else if (len <= 4 * G) {
    sort_in_registers<G, 4>(b, len, v, mask, done);
  } else {
    constexpr int K = 8;
    for (int p0 = 0; p0 < len; p0 += K * G) {
      int x[K], r[K];
#pragma unroll
      for (int k = 0; k < K; ++k) {
        x[k] = (p0 + k * G + lane < len) ? v[b + p0 + k * G + lane] : 0x7fffffff;
        r[k] = 0;
      }
#pragma unroll 4
      for (int q = 0; q < len; ++q) {
        const int y = v[b + q];
#pragma unroll
        for (int k = 0; k < K; ++k) r[k] += (y < x[k]) ? 1 : 0;
      }
#pragma unroll
      for (int k = 0; k < K; ++k)
        if (p0 + k * G + lane < len) tmp[b + r[k]] = x[k];
    }
    __syncwarp(mask);
    for (int p = lane; p < len; p += G) {
      const int x = tmp[b + p];
      v[b + p] = x;
      done(b + p, x);
    }
  }
}

// 16 lanes per column (about 25 edges at the density of water and a cutoff of 4 Angstrom)
__global__ void __launch_bounds__(256) sort_columns_kernel(const int* __restrict__ start, int n, int* __restrict__ v,
                                                           int* __restrict__ tmp) {
  pdl_wait();
  const int s = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 4);
  if (s >= n) return;
  const int b = start[s];
  sort_segment<16>(b, start[s + 1] - b, v, tmp, [](int, int) {});
}

// Arrival order of every edge in its column, as a pass of its own: at large sizes the atomics cost
// the fill pass more than they cost here (1,048,576 atoms: fill 2.51 -> 3.09 ms with them).
__global__ void __launch_bounds__(256) col_rank_kernel(const int* __restrict__ ej, const int* __restrict__ row_ptr,
                                                       int n, int edge_cap, int* __restrict__ col_count,
                                                       int* __restrict__ col_rank) {
  pdl_wait();
  if (!list_fits(row_ptr, n, edge_cap)) return;
  const int E = row_ptr[n];
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < E; e += gridDim.x * blockDim.x)
    col_rank[e] = atomicAdd(&col_count[ej[e]], 1);
}

void nb_col_rank(const int* ej, const int* row_ptr, int n, int edge_cap, int* col_count, int* col_rank,
                 cudaStream_t st) {
  if (edge_cap <= 0) return;
  const int blocks = std::min((int)(((int64_t)edge_cap + 255) / 256), kEdgeBlocks);
  launch(col_rank_kernel, blocks, 256, 0, st, ej, row_ptr, n, edge_cap, col_count, col_rank);
}

void nb_sort_columns(const int* col_ptr, int n, int* col_edge, int* tmp, cudaStream_t st) {
  if (n <= 0) return;
  launch(sort_columns_kernel, (unsigned)(((int64_t)n * 16 + 255) / 256), 256, 0, st, col_ptr, n, col_edge, tmp);
}

// ---------------------------------------------------------------------------
// exact pair test (float64, explicitly rounded, no contraction)
// ---------------------------------------------------------------------------
// (of the home image the offset is zero and adding it leaves pos_j as it is: float64 is the slow unit
// here, so a warp without images skips the 15 operations that form it)
__device__ __forceinline__ void pair_disp(const double* __restrict__ pi, const double* __restrict__ pj,
                                          const double* cell, int S0, int S1, int S2, double d[3]) {
  double p[3] = {pj[0], pj[1], pj[2]};
  if (S0 | S1 | S2) {
    const double s0 = (double)S0, s1 = (double)S1, s2 = (double)S2;
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      const double off = __dadd_rn(__dadd_rn(__dmul_rn(s0, cell[0 * 3 + x]), __dmul_rn(s1, cell[1 * 3 + x])),
                                   __dmul_rn(s2, cell[2 * 3 + x]));
      p[x] = __dadd_rn(p[x], off);
    }
  }
#pragma unroll
  for (int x = 0; x < 3; ++x) d[x] = __dsub_rn(p[x], pi[x]);
}

__device__ __forceinline__ bool pair_test(const double* __restrict__ pi, const double* __restrict__ pj,
                                          const double* cell, int S0, int S1, int S2, double rc2,
                                          double d[3]) {
  pair_disp(pi, pj, cell, S0, S1, S2, d);
  double r2 = __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
  return r2 < rc2;
}

// ---------------------------------------------------------------------------
// Verlet-skin reuse: the exact list of the current positions, filtered from a
// candidate list built at r_c + skin (every pair now within r_c was within
// r_c + skin at the build while no atom has moved skin/2 since).  One warp per
// centre row: each lane takes candidates of the row, applies the exact rule
// (pair_test, the pair's cutoff when a table is set), the warp counts the
// kept ones with a ballot (count pass) or writes them in candidate order at
// the row's offset (fill pass).
// ---------------------------------------------------------------------------
template <bool fill>
__global__ void skin_filter_kernel(const double* __restrict__ pos, int n, const double* __restrict__ cellp,
                                   const int* __restrict__ sk_row, const int* __restrict__ sk_j,
                                   const int* __restrict__ sk_S, double rc2, const double* __restrict__ pair_rc2,
                                   const int* __restrict__ species, int ns, int* __restrict__ count,
                                   const int* __restrict__ row_ptr, int* __restrict__ ej, int* __restrict__ ei,
                                   int* __restrict__ eS, double* __restrict__ ed, int* __restrict__ col_count,
                                   int* __restrict__ col_rank, int edge_cap) {
  pdl_wait();
  if (fill && !list_fits(row_ptr, n, edge_cap)) return;
  const int lane = threadIdx.x & 31;
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (i >= n) return;
  double cell[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) cell[q] = cellp[q];
  const double pi[3] = {pos[3 * (size_t)i], pos[3 * (size_t)i + 1], pos[3 * (size_t)i + 2]};
  const int zi = pair_rc2 ? species[i] : 0;
  const int b = sk_row[i], e1 = sk_row[i + 1];
  int out = fill ? row_ptr[i] : 0;
  for (int e0 = b; e0 < e1; e0 += 32) {
    const int e = e0 + lane;
    bool keep = false;
    int j = 0, S0 = 0, S1 = 0, S2 = 0;
    double d[3] = {0.0, 0.0, 0.0};
    if (e < e1) {
      j = sk_j[e];
      S0 = sk_S[3 * (size_t)e]; S1 = sk_S[3 * (size_t)e + 1]; S2 = sk_S[3 * (size_t)e + 2];
      const double pj[3] = {pos[3 * (size_t)j], pos[3 * (size_t)j + 1], pos[3 * (size_t)j + 2]};
      const double r2c = pair_rc2 ? pair_rc2[zi * ns + species[j]] : rc2;
      keep = pair_test(pi, pj, cell, S0, S1, S2, r2c, d) && !(j == i && S0 == 0 && S1 == 0 && S2 == 0);
    }
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    if (fill && keep) {
      const int o = out + __popc(m & ((1u << lane) - 1u));
      col_rank[o] = atomicAdd(&col_count[j], 1);
      ej[o] = j;
      ei[o] = i;
      eS[3 * (size_t)o] = S0; eS[3 * (size_t)o + 1] = S1; eS[3 * (size_t)o + 2] = S2;
      ed[3 * (size_t)o] = d[0]; ed[3 * (size_t)o + 1] = d[1]; ed[3 * (size_t)o + 2] = d[2];
    }
    out += __popc(m);
  }
  if (!fill && lane == 0) count[i] = out;
}

void nb_skin_filter(bool fill, const double* pos, int n, const double* d_cell, const int* sk_row, const int* sk_j,
                    const int* sk_S, double rc2, const double* pair_rc2, const int* species, int ns, int* count,
                    const int* row_ptr, int* ej, int* ei, int* eS, double* ed, int* col_count, int* col_rank,
                    int edge_cap, cudaStream_t st) {
  if (n <= 0) return;
  const int threads = 256, blocks = (int)(((int64_t)n * 32 + threads - 1) / threads);
  if (fill)
    launch(skin_filter_kernel<true>, blocks, threads, 0, st, pos, n, d_cell, sk_row, sk_j, sk_S, rc2, pair_rc2, species,
                                                         ns, count, row_ptr, ej, ei, eS, ed, col_count, col_rank,
                                                         edge_cap);
  else
    launch(skin_filter_kernel<false>, blocks, threads, 0, st, pos, n, d_cell, sk_row, sk_j, sk_S, rc2, pair_rc2,
                                                          species, ns, count, row_ptr, ej, ei, eS, ed, col_count, col_rank,
                                                         edge_cap);
}

// Largest squared displacement of any atom since the reference positions, as
// the bits of a non-negative double (their order is the values' order).
__global__ void max_disp2_kernel(const double* __restrict__ pos, const double* __restrict__ ref, int n,
                                 unsigned long long* __restrict__ out) {
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double v = 0.0;
  if (i < n) {
    const double dx = pos[3 * (size_t)i] - ref[3 * (size_t)i], dy = pos[3 * (size_t)i + 1] - ref[3 * (size_t)i + 1],
                 dz = pos[3 * (size_t)i + 2] - ref[3 * (size_t)i + 2];
    v = dx * dx + dy * dy + dz * dz;
    if (!(v == v)) v = 1e300;   // a NaN position forces a rebuild (which then reports it)
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(v));
}

void nb_max_disp2(const double* pos, const double* ref, int n, unsigned long long* out, cudaStream_t st) {
  cudaMemsetAsync(out, 0, sizeof(unsigned long long), st);
  if (n <= 0) return;
  launch(max_disp2_kernel, (n + 255) / 256, 256, 0, st, pos, ref, n, out);
}

// The cell lists in atom order, and with them the wrapped positions pw = pos - wrap . cell in
// cell-sorted order (pos4[s] and pw[3 s ..] belong to atom sorted[s]): float32 for the prefilter,
// float64 for the displacements of accepted edges.  Eight lanes per cell (about 6.4 atoms at the
// density of water).
__global__ void __launch_bounds__(256) sort_cells_kernel(const double* __restrict__ pos,
                                                         const int* __restrict__ species, CellGrid g, int n_cells,
                                                         const int* __restrict__ cell_start,
                                                         const int* __restrict__ wrap, int* __restrict__ sorted,
                                                         int* __restrict__ tmp, float4* __restrict__ pos4, double* __restrict__ pw,
                                                         int4* __restrict__ wraps) {
  pdl_wait();
  const int c = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3);
  if (c >= n_cells) return;
  const int b = cell_start[c];
  sort_segment<8>(b, cell_start[c + 1] - b, sorted, tmp, [&](int s, int j) {
    double p[3];
    const int wj[3] = {wrap[3 * (size_t)j], wrap[3 * (size_t)j + 1], wrap[3 * (size_t)j + 2]};
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      p[x] = pos[3 * (size_t)j + x];
#pragma unroll
      for (int k = 0; k < 3; ++k) p[x] -= (double)wj[k] * g.cell[k * 3 + x];
    }
    pos4[s] = make_float4((float)p[0], (float)p[1], (float)p[2], __int_as_float(species[j]));
    pw[3 * (size_t)s] = p[0];
    pw[3 * (size_t)s + 1] = p[1];
    pw[3 * (size_t)s + 2] = p[2];
    wraps[s] = make_int4(wj[0], wj[1], wj[2], 0);
  });
}

void nb_sort_cells(const double* pos, const int* species, const CellGrid& g, int n_cells, const int* cell_start,
                   const int* wrap, int* sorted, int* tmp, float4* pos4, double* pw, int4* wraps, cudaStream_t st) {
  if (n_cells <= 0) return;
  launch(sort_cells_kernel, (unsigned)(((int64_t)n_cells * 8 + 255) / 256), 256, 0, st, pos, species, g, n_cells, cell_start,
                                                                                    wrap, sorted, tmp, pos4, pw, wraps);
}

// Neighbour search.  A float32 prefilter on the wrapped positions decides
// every candidate whose squared distance is farther than `band` from r_c^2;
// candidates inside the band take the exact float64 test.  `band` is computed
// on the host from a bound on the float32 rounding of the wrapped coordinates
// and image offsets (with a safety factor), so the prefilter never changes a
// decision.  Accepted edges get their float64 displacement for later stages:
// from the exact test inside the band, else (pw_j + q . cell) - pw_i from the
// float64 wrapped positions (the same vector up to float64 rounding; the
// edge's image shift is S = q - w_j + w_i).
constexpr int kSearchThreads = 128;
// Up to this many atoms a warp per centre, above it a thread per centre (both list the same edges in
// the same order).  Count and fill pass, us, warp / thread: 64 atoms 11 + 12 / 37 + 77; 3,072 atoms
// 17 + 18 / 81 + 124; 23,552 atoms 44 + 53 / 81 + 143; 65,536 atoms 89 + 124 / 93 + 212; 1,048,576 atoms
// 1,553 + 3,298 / 518 + 2,426 (the warp form issues more instructions per candidate).
constexpr int kSearchWarpAtoms = 65536;

// image q (three signed 10-bit fields) and the exact-test flag of a staged edge.  Stencils that reach
// further (a periodic axis thinner than 1/511 of the cutoff) go unpacked: a thread per centre writes
// every edge itself.
__host__ __device__ inline bool q_packs(const CellGrid& g) { return g.R[0] < 512 && g.R[1] < 512 && g.R[2] < 512; }
__device__ __forceinline__ int pack_q(int q0, int q1, int q2, bool exact) {
  return (q0 & 1023) | ((q1 & 1023) << 10) | ((q2 & 1023) << 20) | (exact ? (1 << 30) : 0);
}
__device__ __forceinline__ int unpack_q(int v, int f) { return (int)((unsigned)v << (22 - 10 * f)) >> 22; }

// One warp per centre atom (cell order).  Up to 32 cells of the stencil at a
// time: lane c looks up cell c's range and image offset, a warp scan of the
// range lengths flattens their atoms into one candidate sequence (stencil
// order, then cell order), and the lanes test 32 consecutive candidates per
// round; a ballot places the accepted ones, so rows keep that order.  Accepted
// candidates are compacted into a 64-entry stage in shared memory and written
// 32 at a time with lanes on consecutive edges: the float64 displacements (a
// slow unit on this part) run on full warps and the stores cover consecutive
// addresses.
// Bound: latency of the dependent loads (cell ranges, then positions), and at
// large sizes instruction issue.  Why a warp per atom: a thread per atom walks
// its ~190 candidates one after another.
struct SearchCell {
  float ox, oy, oz;   // image offset of the cell minus the centre's position (float32)
  int q;              // packed image
};

template <bool fill>
__global__ void __launch_bounds__(kSearchThreads) search_kernel(
    const double* __restrict__ pos, int n, CellGrid g, const int* __restrict__ cell_of,
    const int4* __restrict__ wraps, const int* __restrict__ cell_start, const int* __restrict__ sorted,
    const float4* __restrict__ pos4, const double* __restrict__ pw, double rc2, float band,
    const double* __restrict__ pair_rc2, const float* __restrict__ pair_rc2f, int ns, int* __restrict__ count,
    const int* __restrict__ row_ptr, int* __restrict__ ej, int* __restrict__ ei, int* __restrict__ eS, double* __restrict__ ed,
    int* __restrict__ col_count, int* __restrict__ col_rank, int edge_cap, int* __restrict__ d_err) {
  pdl_wait();
  if (fill && !list_fits(row_ptr, n, edge_cap)) return;
  constexpr int kWarps = kSearchThreads / 32;
  __shared__ SearchCell s_cell[kWarps][32];
  __shared__ int s_pref[kWarps][32];    // candidates before the cell
  __shared__ int s_first[kWarps][32];   // cell_start - candidates before it
  __shared__ int2 s_stage[kWarps][fill ? 64 : 1];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int t = blockIdx.x * kWarps + w;
  if (t >= n) return;
  const int i = sorted[t];
  if (i >= g.n_centres) {   // ghost atoms (spatial decomposition) are neighbours only, never centres
    if (!fill && lane == 0) count[i] = 0;
    return;
  }
  const int ci = cell_of[i];
  const int4 wi = wraps[t];
  const float4 pi4 = pos4[t];
  const double pi[3] = {pos[3 * (size_t)i], pos[3 * (size_t)i + 1], pos[3 * (size_t)i + 2]};
  const int c2 = ci % g.n[2], c1 = (ci / g.n[2]) % g.n[1], c0 = ci / (g.n[2] * g.n[1]);
  const float lo2 = g.rc2f - band, hi2 = g.rc2f + band;
  // per-ordered-pair cutoffs: row of the centre's species (the band of the largest
  // cutoff bounds the float32 error of every smaller one)
  const double* prow = pair_rc2 ? pair_rc2 + (size_t)__float_as_int(pi4.w) * ns : nullptr;
  const float* prowf = pair_rc2f + (size_t)(pair_rc2 ? __float_as_int(pi4.w) : 0) * ns;
  const int base = fill ? row_ptr[i] : 0;
  const int cap = fill ? (row_ptr[i + 1] - base) : 0;
  int k = 0;         // accepted so far
  int nst = 0;       // staged, not yet written (they are edges [k - nst, k))
  // the first m (<= 32) staged edges, to base + k0 + lane
  auto write = [&](int k0, int m) {
    if (lane < m && k0 + lane < cap) {
      const int2 en = s_stage[w][lane];
      const int s = en.x;
      const int q0 = unpack_q(en.y, 0), q1 = unpack_q(en.y, 1), q2 = unpack_q(en.y, 2);
      const int j = sorted[s];
      const int4 wj = wraps[s];
      const int S0 = g.pbc[0] ? q0 - wj.x + wi.x : 0;
      const int S1 = g.pbc[1] ? q1 - wj.y + wi.y : 0;
      const int S2 = g.pbc[2] ? q2 - wj.z + wi.z : 0;
      double d[3];
      if ((en.y >> 30) & 1) {
        pair_disp(pi, pos + 3 * (size_t)j, g.cell, S0, S1, S2, d);
      } else {
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          double pj = pw[3 * (size_t)s + x];
          if (q0 | q1 | q2)
            pj += ((double)q0 * g.cell[x] + (double)q1 * g.cell[3 + x]) + (double)q2 * g.cell[6 + x];
          d[x] = pj - pw[3 * (size_t)t + x];
        }
      }
      const size_t o = (size_t)base + k0 + lane;
      col_rank[o] = atomicAdd(&col_count[j], 1);
      ej[o] = j;
      ei[o] = i;
      eS[3 * o] = S0; eS[3 * o + 1] = S1; eS[3 * o + 2] = S2;
      ed[3 * o] = d[0]; ed[3 * o + 1] = d[1]; ed[3 * o + 2] = d[2];
    }
  };
  const int n1 = 2 * g.R[1] + 1, n2 = 2 * g.R[2] + 1;
  const int ncell = (2 * g.R[0] + 1) * n1 * n2;
  for (int m0 = 0; m0 < ncell; m0 += 32) {
    const int m = m0 + lane;
    int b = 0, cnt = 0;
    SearchCell sc = {0.f, 0.f, 0.f, 0};
    if (m < ncell) {
      int cc[3] = {c0 + m / (n1 * n2) - g.R[0], c1 + (m / n2) % n1 - g.R[1], c2 + m % n2 - g.R[2]};
      int q[3] = {0, 0, 0};
      bool in = true;
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        if (g.pbc[x]) {
          q[x] = floordiv(cc[x], g.n[x]);
          cc[x] -= q[x] * g.n[x];
        } else if (cc[x] < 0 || cc[x] >= g.n[x]) {
          in = false;
        }
      }
      if (in) {
        const int cell = (cc[0] * g.n[1] + cc[1]) * g.n[2] + cc[2];
        b = cell_start[cell];
        cnt = cell_start[cell + 1] - b;
        const float q0 = (float)q[0], q1 = (float)q[1], q2 = (float)q[2];
        sc.ox = q0 * g.cellf[0] + q1 * g.cellf[3] + q2 * g.cellf[6] - pi4.x;
        sc.oy = q0 * g.cellf[1] + q1 * g.cellf[4] + q2 * g.cellf[7] - pi4.y;
        sc.oz = q0 * g.cellf[2] + q1 * g.cellf[5] + q2 * g.cellf[8] - pi4.z;
        sc.q = pack_q(q[0], q[1], q[2], false);
      }
    }
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    __syncwarp();
    s_cell[w][lane] = sc;
    s_pref[w][lane] = incl - cnt;
    s_first[w][lane] = b - (incl - cnt);
    __syncwarp();
    for (int r0 = 0; r0 < total; r0 += 32) {
      const int r = r0 + lane;
      bool keep = false;
      int2 en = make_int2(0, 0);
      if (r < total) {
        int o = 0;   // the last cell with s_pref <= r
#pragma unroll
        for (int h = 16; h > 0; h >>= 1)
          if (s_pref[w][o + h] <= r) o += h;
        const SearchCell ce = s_cell[w][o];
        const int s = s_first[w][o] + r;
        const float4 pj = pos4[s];
        const float dx = pj.x + ce.ox, dy = pj.y + ce.oy, dz = pj.z + ce.oz;
        const float r2f = dx * dx + dy * dy + dz * dz;
        float lo2p = lo2, hi2p = hi2;
        if (prow) {
          const float rc2pf = prowf[__float_as_int(pj.w)];
          lo2p = rc2pf - band;
          hi2p = fminf(hi2, rc2pf + band);
        }
        if (!(r2f > hi2p)) {
          bool exact = r2f >= lo2p;
          keep = true;
          if (s == t || exact) {
            const int4 wj = wraps[s];
            const int S0 = g.pbc[0] ? unpack_q(ce.q, 0) - wj.x + wi.x : 0;
            const int S1 = g.pbc[1] ? unpack_q(ce.q, 1) - wj.y + wi.y : 0;
            const int S2 = g.pbc[2] ? unpack_q(ce.q, 2) - wj.z + wi.z : 0;
            if (s == t && S0 == 0 && S1 == 0 && S2 == 0) keep = false;   // (s = t: j = i)
            double d[3];
            if (keep && exact)
              keep = pair_test(pi, pos + 3 * (size_t)sorted[s], g.cell, S0, S1, S2,
                               prow ? prow[__float_as_int(pj.w)] : rc2, d);
          }
          en = make_int2(s, ce.q | (exact ? (1 << 30) : 0));
        }
      }
      const unsigned mask = __ballot_sync(0xffffffffu, keep);
      const int nk = __popc(mask);
      if constexpr (fill) {
        if (keep) s_stage[w][nst + __popc(mask & ((1u << lane) - 1u))] = en;
        nst += nk;
        if (nst >= 32) {
          __syncwarp();
          write(k + nk - nst, 32);
          nst -= 32;
          const int2 rest = s_stage[w][32 + lane];
          __syncwarp();
          s_stage[w][lane] = rest;
          __syncwarp();
        }
      }
      k += nk;
    }
  }
  if constexpr (fill) {
    __syncwarp();
    write(k - nst, nst);
    if (lane == 0 && k != cap) atomicOr(d_err, kErrNeighbor);
  } else {
    if (lane == 0) count[i] = k;
  }
}

// One thread per centre atom, for systems that fill the GPU with threads: neighbouring lanes share
// their stencil cells, so a candidate costs a warp a few instructions for 32 centres.  The fill pass
// writes through shared memory: a lane records each accepted candidate of its row (cell-order index s,
// image q, whether it took the exact test) in its warp's staging area, then the warp writes the 32 rows
// one after another with its lanes on consecutive edges of a row, so each store covers consecutive
// addresses (a row per lane would scatter every store over 32 rows).  Edges past kFillStage in a row
// are written by their lane directly, and so are all of them when an image does not pack (q_packs).
constexpr int kFillStage = 32;

template <bool fill>
__global__ void __launch_bounds__(kSearchThreads) search_thread_kernel(
    const double* __restrict__ pos, int n, CellGrid g, const int* __restrict__ cell_of,
    const int4* __restrict__ wraps, const int* __restrict__ cell_start, const int* __restrict__ sorted,
    const float4* __restrict__ pos4, const double* __restrict__ pw, double rc2, float band,
    const double* __restrict__ pair_rc2, const float* __restrict__ pair_rc2f, int ns, int* __restrict__ count,
    const int* __restrict__ row_ptr, int* __restrict__ ej, int* __restrict__ ei, int* __restrict__ eS, double* __restrict__ ed,
    int edge_cap, int* __restrict__ d_err) {
  pdl_wait();
  if (fill && !list_fits(row_ptr, n, edge_cap)) return;
  __shared__ int2 stage[fill ? kSearchThreads : 1][fill ? kFillStage : 1];
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  bool act = t < n;
  const int i = act ? sorted[t] : 0;
  if (act && i >= g.n_centres) {   // ghost atoms (spatial decomposition) are neighbours only, never centres
    if (!fill) count[i] = 0;
    act = false;
  }
  if constexpr (!fill) {
    if (!act) return;
  }
  int4 wi = make_int4(0, 0, 0, 0);
  double pi[3] = {0.0, 0.0, 0.0}, pwi[3] = {0.0, 0.0, 0.0};
  int k = 0, base = 0, cap = 0;
  const int nstage = q_packs(g) ? kFillStage : 0;
  if (act) {
    const int ci = cell_of[i];
    int c[3];
    c[2] = ci % g.n[2];
    c[1] = (ci / g.n[2]) % g.n[1];
    c[0] = ci / (g.n[2] * g.n[1]);
    wi = wraps[t];   // cell-order copies of the wrap counts: coalesced with pos4
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      pi[x] = pos[3 * (size_t)i + x];
      pwi[x] = pw[3 * (size_t)t + x];
    }
    const float4 pi4 = pos4[t];
    const float lo2 = g.rc2f - band, hi2 = g.rc2f + band;
    // per-ordered-pair cutoffs: row of the centre's species (the band of the largest
    // cutoff bounds the float32 error of every smaller one)
    const double* prow = pair_rc2 ? pair_rc2 + (size_t)__float_as_int(pi4.w) * ns : nullptr;
    const float* prowf = pair_rc2f + (size_t)(pair_rc2 ? __float_as_int(pi4.w) : 0) * ns;
    const float* cf = g.cellf;
    base = fill ? row_ptr[i] : 0;
    cap = fill ? (row_ptr[i + 1] - base) : 0;
    for (int d0 = -g.R[0]; d0 <= g.R[0]; ++d0) {
      int cc0 = c[0] + d0, q0 = 0;
      if (g.pbc[0]) { q0 = floordiv(cc0, g.n[0]); cc0 -= q0 * g.n[0]; }
      else if (cc0 < 0 || cc0 >= g.n[0]) continue;
      for (int d1 = -g.R[1]; d1 <= g.R[1]; ++d1) {
        int cc1 = c[1] + d1, q1 = 0;
        if (g.pbc[1]) { q1 = floordiv(cc1, g.n[1]); cc1 -= q1 * g.n[1]; }
        else if (cc1 < 0 || cc1 >= g.n[1]) continue;
        for (int d2 = -g.R[2]; d2 <= g.R[2]; ++d2) {
          int cc2 = c[2] + d2, q2 = 0;
          if (g.pbc[2]) { q2 = floordiv(cc2, g.n[2]); cc2 -= q2 * g.n[2]; }
          else if (cc2 < 0 || cc2 >= g.n[2]) continue;
          const int cell = (cc0 * g.n[1] + cc1) * g.n[2] + cc2;
          const int b = cell_start[cell], e = cell_start[cell + 1];
          // image offset of this stencil cell (float32), relative to i
          const float ox = (float)q0 * cf[0] + (float)q1 * cf[3] + (float)q2 * cf[6] - pi4.x;
          const float oy = (float)q0 * cf[1] + (float)q1 * cf[4] + (float)q2 * cf[7] - pi4.y;
          const float oz = (float)q0 * cf[2] + (float)q1 * cf[5] + (float)q2 * cf[8] - pi4.z;
          for (int s = b; s < e; ++s) {
            const float4 pj = pos4[s];
            const float dx = pj.x + ox, dy = pj.y + oy, dz = pj.z + oz;
            const float r2f = dx * dx + dy * dy + dz * dz;
            if (r2f > hi2) continue;
            float lo2p = lo2;
            if (prow) {
              const float rc2pf = prowf[__float_as_int(pj.w)];
              if (r2f > rc2pf + band) continue;
              lo2p = rc2pf - band;
            }
            const int4 wj = wraps[s];
            const int S0 = g.pbc[0] ? q0 - wj.x + wi.x : 0;
            const int S1 = g.pbc[1] ? q1 - wj.y + wi.y : 0;
            const int S2 = g.pbc[2] ? q2 - wj.z + wi.z : 0;
            if (s == t && S0 == 0 && S1 == 0 && S2 == 0) continue;   // (s = t: j = i)
            const bool exact = r2f >= lo2p;
            double d[3];
            if (exact && !pair_test(pi, pos + 3 * (size_t)sorted[s], g.cell, S0, S1, S2,
                                    prow ? prow[__float_as_int(pj.w)] : rc2, d))
              continue;
            if constexpr (fill) {
              if (k < nstage) {
                stage[threadIdx.x][k] = make_int2(s, pack_q(q0, q1, q2, exact));
              } else if (k < cap) {
                // past the staging area: this lane writes the edge itself
                if (!exact) {
#pragma unroll
                  for (int x = 0; x < 3; ++x) {
                    const double qoff = (q0 | q1 | q2) ? ((double)q0 * g.cell[x] + (double)q1 * g.cell[3 + x]) +
                                                             (double)q2 * g.cell[6 + x]
                                                       : 0.0;
                    d[x] = (pw[3 * (size_t)s + x] + qoff) - pwi[x];
                  }
                }
                const size_t o = (size_t)base + k;
                ej[o] = sorted[s];
                ei[o] = i;
                eS[3 * o] = S0; eS[3 * o + 1] = S1; eS[3 * o + 2] = S2;
                ed[3 * o] = d[0]; ed[3 * o + 1] = d[1]; ed[3 * o + 2] = d[2];
              }
            }
            ++k;
          }
        }
      }
    }
  }
  if constexpr (!fill) {
    count[i] = k;
  } else {
    if (act && k != cap) atomicOr(d_err, kErrNeighbor);
    __syncwarp();
    // the warp's rows one after another, lanes on consecutive edges
    const int lane = threadIdx.x & 31, w0 = threadIdx.x & ~31;
    const int nst = act ? min(min(k, cap), nstage) : 0;
    for (int r = 0; r < 32; ++r) {
      const int nr = __shfl_sync(0xffffffffu, nst, r);
      if (nr == 0) continue;
      const int ir = __shfl_sync(0xffffffffu, i, r);
      const int br = __shfl_sync(0xffffffffu, base, r);
      const int wx = __shfl_sync(0xffffffffu, wi.x, r), wy = __shfl_sync(0xffffffffu, wi.y, r),
                wz = __shfl_sync(0xffffffffu, wi.z, r);
      double pir[3], pwr[3];
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        pir[x] = __shfl_sync(0xffffffffu, pi[x], r);
        pwr[x] = __shfl_sync(0xffffffffu, pwi[x], r);
      }
      for (int kk = lane; kk < nr; kk += 32) {
        const int2 en = stage[w0 + r][kk];
        const int s = en.x;
        const int q0 = unpack_q(en.y, 0), q1 = unpack_q(en.y, 1), q2 = unpack_q(en.y, 2);
        const bool exact = (en.y >> 30) & 1;
        const int j = sorted[s];
        const int4 wj = wraps[s];
        const int S0 = g.pbc[0] ? q0 - wj.x + wx : 0;
        const int S1 = g.pbc[1] ? q1 - wj.y + wy : 0;
        const int S2 = g.pbc[2] ? q2 - wj.z + wz : 0;
        double d[3];
        if (exact) {
          pair_disp(pir, pos + 3 * (size_t)j, g.cell, S0, S1, S2, d);
        } else {
#pragma unroll
          for (int x = 0; x < 3; ++x) {
            const double qoff = (q0 | q1 | q2) ? ((double)q0 * g.cell[x] + (double)q1 * g.cell[3 + x]) +
                                                     (double)q2 * g.cell[6 + x]
                                               : 0.0;
            d[x] = (pw[3 * (size_t)s + x] + qoff) - pwr[x];
          }
        }
        const size_t o = (size_t)br + kk;
        ej[o] = j;
        ei[o] = ir;
        eS[3 * o] = S0; eS[3 * o + 1] = S1; eS[3 * o + 2] = S2;
        ed[3 * o] = d[0]; ed[3 * o + 1] = d[1]; ed[3 * o + 2] = d[2];
      }
    }
  }
}

bool nb_search(bool fill, const double* pos, int n, const CellGrid& g, const int* cell_of, const int4* wraps,
               const int* cell_start, const int* sorted, const float4* pos4, const double* pw, double rc2, float band,
               const double* pair_rc2, const float* pair_rc2f, int ns, int* count, const int* row_ptr, int* ej, int* ei,
               int* eS, double* ed, int* col_count, int* col_rank, int edge_cap, int* d_err, cudaStream_t st) {
  if (n <= 0) return true;
  if (n <= kSearchWarpAtoms && q_packs(g)) {
    auto kernel = fill ? search_kernel<true> : search_kernel<false>;
    launch(kernel, (n + kSearchThreads / 32 - 1) / (kSearchThreads / 32), kSearchThreads, 0, st, pos, n, g, cell_of,
        wraps, cell_start, sorted, pos4, pw, rc2, band, pair_rc2, pair_rc2f, ns, count, row_ptr, ej, ei, eS, ed,
        col_count, col_rank, edge_cap, d_err);
    return true;
  }
  auto kernel = fill ? search_thread_kernel<true> : search_thread_kernel<false>;
  launch(kernel, (n + kSearchThreads - 1) / kSearchThreads, kSearchThreads, 0, st, pos, n, g, cell_of, wraps,
      cell_start, sorted, pos4, pw, rc2, band, pair_rc2, pair_rc2f, ns, count, row_ptr, ej, ei, eS, ed, edge_cap,
      d_err);
  return false;
}

// ---------------------------------------------------------------------------
// batched structures: all pairs of each structure over its image range
// ---------------------------------------------------------------------------
__global__ void brute_batched_kernel(bool fill, const double* __restrict__ pos,
                                     const int64_t* __restrict__ offs, const double* __restrict__ cells,
                                     const int* __restrict__ pbc, const int* __restrict__ nimg,
                                     double rc2, const int* __restrict__ species,
                                     const double* __restrict__ pair_rc2, int ns,
                                     const int* __restrict__ atom_struct, int n,
                                     int* __restrict__ count, const int* __restrict__ row_ptr,
                                     int* __restrict__ ej, int* __restrict__ ei, int* __restrict__ eS,
                                     double* __restrict__ ed, int* __restrict__ col_count,
                                     int* __restrict__ col_rank, int edge_cap, int* __restrict__ d_err) {
  pdl_wait();
  if (fill && !list_fits(row_ptr, n, edge_cap)) return;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int b = atom_struct[i];
  const int j0 = (int)offs[b], j1 = (int)offs[b + 1];
  double zero_cell[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  const double* cell = cells ? cells + 9 * (size_t)b : zero_cell;
  int nI[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) nI[k] = (cells && pbc[3 * b + k]) ? nimg[3 * b + k] : 0;
  double pi[3] = {pos[3 * (size_t)i], pos[3 * (size_t)i + 1], pos[3 * (size_t)i + 2]};
  int k = 0;
  const int base = fill ? row_ptr[i] : 0;
  const int cap = fill ? (row_ptr[i + 1] - base) : 0;
  const double* prow = pair_rc2 ? pair_rc2 + (size_t)species[i] * ns : nullptr;
  for (int j = j0; j < j1; ++j) {
    const double rc2p = prow ? prow[species[j]] : rc2;   // the ordered pair's cutoff
    for (int S0 = -nI[0]; S0 <= nI[0]; ++S0)
      for (int S1 = -nI[1]; S1 <= nI[1]; ++S1)
        for (int S2 = -nI[2]; S2 <= nI[2]; ++S2) {
          if (j == i && S0 == 0 && S1 == 0 && S2 == 0) continue;
          double d[3];
          if (!pair_test(pi, pos + 3 * (size_t)j, cell, S0, S1, S2, rc2p, d)) continue;
          if (fill && k < cap) {
            size_t o = (size_t)base + k;
            col_rank[o] = atomicAdd(&col_count[j], 1);
            ej[o] = j;
            ei[o] = i;
            eS[3 * o] = S0; eS[3 * o + 1] = S1; eS[3 * o + 2] = S2;
            ed[3 * o] = d[0]; ed[3 * o + 1] = d[1]; ed[3 * o + 2] = d[2];
          }
          ++k;
        }
  }
  if (fill) {
    if (k != cap) atomicOr(d_err, kErrNeighbor);
  } else {
    count[i] = k;
  }
}

// The same search for structures without cells (molecules): 16 lanes per centre test 16 atoms of its
// structure at a time and a ballot places the accepted ones in the same order.  Without images a
// test is 8 float64 operations instead of 26 (the offset is zero), and the rows are written with
// lanes on consecutive edges.  Bound: float64 issue.
template <bool fill>
__global__ void __launch_bounds__(128) brute_nocell_kernel(const double* __restrict__ pos,
                                                           const int64_t* __restrict__ offs, double rc2,
                                                           const int* __restrict__ species,
                                                           const double* __restrict__ pair_rc2, int ns,
                                                           const int* __restrict__ atom_struct, int n,
                                                           int* __restrict__ count, const int* __restrict__ row_ptr,
                                                           int* __restrict__ ej, int* __restrict__ ei,
                                                           int* __restrict__ eS, double* __restrict__ ed,
                                                           int* __restrict__ col_count, int* __restrict__ col_rank,
                                                           int edge_cap, int* __restrict__ d_err) {
  pdl_wait();
  if (fill && !list_fits(row_ptr, n, edge_cap)) return;
  const int i = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 4);
  if (i >= n) return;
  const int lane = threadIdx.x & 15, half = threadIdx.x & 16;
  const unsigned mask = 0xffffu << half;
  const int b = atom_struct[i];
  const int j0 = (int)offs[b], j1 = (int)offs[b + 1];
  const double pi[3] = {pos[3 * (size_t)i], pos[3 * (size_t)i + 1], pos[3 * (size_t)i + 2]};
  const double* prow = pair_rc2 ? pair_rc2 + (size_t)species[i] * ns : nullptr;
  const int base = fill ? row_ptr[i] : 0;
  const int cap = fill ? (row_ptr[i + 1] - base) : 0;
  int k = 0;
  for (int jb = j0; jb < j1; jb += 16) {
    const int j = jb + lane;
    bool keep = false;
    double d[3] = {0.0, 0.0, 0.0};
    if (j < j1 && j != i) {
#pragma unroll
      for (int x = 0; x < 3; ++x) d[x] = __dsub_rn(pos[3 * (size_t)j + x], pi[x]);
      const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2]));
      keep = r2 < (prow ? prow[species[j]] : rc2);   // the ordered pair's cutoff
    }
    const unsigned m = __ballot_sync(mask, keep) >> half;
    const int kk = k + __popc(m & ((1u << lane) - 1u));
    if (fill && keep && kk < cap) {
      const size_t o = (size_t)base + kk;
      col_rank[o] = atomicAdd(&col_count[j], 1);
      ej[o] = j;
      ei[o] = i;
      eS[3 * o] = 0; eS[3 * o + 1] = 0; eS[3 * o + 2] = 0;
      ed[3 * o] = d[0]; ed[3 * o + 1] = d[1]; ed[3 * o + 2] = d[2];
    }
    k += __popc(m);
  }
  if (lane == 0) {
    if (!fill) count[i] = k;
    else if (k != cap) atomicOr(d_err, kErrNeighbor);
  }
}

void nb_bruteforce_batched(bool fill, const double* pos, const int64_t* offs, int nstruct,
                           const double* cells, const int* pbc, const int* nimg, double rc2,
                           const int* species, const double* pair_rc2, int ns,
                           const int* atom_struct, int n, int* count, const int* row_ptr, int* ej,
                           int* ei, int* eS, double* ed, int* col_count, int* col_rank, int edge_cap, int* d_err,
                           cudaStream_t st) {
  (void)nstruct;
  if (n <= 0) return;
  if (!cells) {
    auto kernel = fill ? brute_nocell_kernel<true> : brute_nocell_kernel<false>;
    launch(kernel, (unsigned)(((int64_t)n * 16 + 127) / 128), 128, 0, st, pos, offs, rc2, species, pair_rc2, ns, atom_struct,
                                                                      n, count, row_ptr, ej, ei, eS, ed, col_count,
                                                                      col_rank, edge_cap, d_err);
    return;
  }
  launch(brute_batched_kernel, (n + 127) / 128, 128, 0, st, fill, pos, offs, cells, pbc, nimg, rc2, species, pair_rc2,
                                                        ns, atom_struct, n, count, row_ptr, ej, ei, eS, ed,
                                                        col_count, col_rank, edge_cap, d_err);
}

// Per structure: spread (max - min) of the fractional coordinates, so the
// image range covers positions that are not wrapped into the cell.
__global__ void struct_span_kernel(const double* __restrict__ pos, const int64_t* __restrict__ offs,
                                   const double* __restrict__ inv, double* __restrict__ span) {
  pdl_wait();
  const int b = blockIdx.x;
  __shared__ double lo[3][128], hi[3][128];
  double l[3] = {1e300, 1e300, 1e300}, h[3] = {-1e300, -1e300, -1e300};
  for (long long i = offs[b] + threadIdx.x; i < offs[b + 1]; i += blockDim.x) {
    double f[3];
    frac_of(pos + 3 * i, inv + 9 * (size_t)b, f);
    for (int k = 0; k < 3; ++k) { l[k] = fmin(l[k], f[k]); h[k] = fmax(h[k], f[k]); }
  }
  for (int k = 0; k < 3; ++k) { lo[k][threadIdx.x] = l[k]; hi[k][threadIdx.x] = h[k]; }
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s)
      for (int k = 0; k < 3; ++k) {
        lo[k][threadIdx.x] = fmin(lo[k][threadIdx.x], lo[k][threadIdx.x + s]);
        hi[k][threadIdx.x] = fmax(hi[k][threadIdx.x], hi[k][threadIdx.x + s]);
      }
    __syncthreads();
  }
  if (threadIdx.x < 3) {
    double sp = hi[threadIdx.x][0] - lo[threadIdx.x][0];
    span[3 * b + threadIdx.x] = (sp > 0) ? sp : 0.0;
  }
}

void nb_struct_span(const double* pos, const int64_t* offs, const double* inv, int nstruct, double* span,
                    cudaStream_t st) {
  if (nstruct <= 0) return;
  launch(struct_span_kernel, nstruct, 128, 0, st, pos, offs, inv, span);
}

}  // namespace alg
