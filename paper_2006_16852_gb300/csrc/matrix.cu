// matrix.cu -- creation of the CSR operator (Section 2.2.4: "objects A ... are
// LinOp objects that store their data as matrices in CSR") and of its
// GPU-side storage formats: row-length bins, merge-path tiles, ELL and the
// hybrid ELL + overflow split.  The caller's arrays are copied into
// library-owned storage (the "give"/copy ownership of Section 2.4).
#include <algorithm>
#include <climits>
#include <memory>
#include <vector>

#include "gk_device.cuh"
#include "gk_internal.h"

namespace gk {

namespace {

// Index arrays are padded so that 16-byte bulk copies rounded up to a
// multiple of four elements never read past the allocation.
inline int64_t padded(int64_t n) { return ((n + 3) & ~int64_t(3)) + 8; }

// Creation runs on the device: one pass over the row pointers (copy, checks,
// length counts per tile and over all), one over the entries (copy, checks),
// then the format from the counts; the host reads back one struct and makes
// a 257-entry table.  Creating the operator of a 7-point grid of 1.03 M rows
// (GK_CSR), block Jacobi (bs 8) and one apply of each: 6.28 -> 0.44 ms; it
// was bound by host loops over the row pointers (checks, counting sort,
// offsets), pageable copies of the plan, and an allocation and a free per
// array (now stream-ordered, from the device's pool).
//
// What creation learns about the caller's CSR arrays in one pass over the row
// pointers and one over the entries (zero-initialised device memory).  "First
// row" words hold INT_MAX - row, so that 0 means none.
struct CsrInfo {
  int32_t rp0, rpn;      // the first and the last row pointer
  int32_t dec;           // first row whose row pointer decreases
  int32_t bad_col;       // first row with a column out of range, unsorted or repeated
  int32_t maxlen;
  int32_t n_long;        // rows of more than kSliceMaxLen entries
  unsigned long long long_slots;    // DFMA lane slots of those rows (sliced_efficiency)
  int32_t hist[kSliceMaxLen + 1];   // the other rows by length
};

constexpr int kBins = static_cast<int>(kSliceMaxLen) + 1;
constexpr int kTileThreads = 256;
constexpr int kMaxTiles = 1024;  // one block scans a length's counts over the tiles

// Rows per tile of the row-pointer passes: at least 1024, and a multiple of
// the block size that gives at most kMaxTiles tiles.
int64_t tile_rows(int64_t n_rows) {
  const int64_t t = (n_rows + kMaxTiles - 1) / kMaxTiles;
  return std::max<int64_t>(1024, (t + kTileThreads - 1) / kTileThreads * kTileThreads);
}

// Copies the row pointers (src may be dst), checks them, and counts the row
// lengths: per tile (one block) into tile_hist, over all into info; lists the
// long rows (unordered).  Rows of equal length are the rule, so a warp counts
// equal lengths together instead of one shared-memory atomic per row.
__global__ void __launch_bounds__(kTileThreads) csr_rows_kernel(const int32_t* __restrict__ src, int32_t* dst,
                                                                int64_t n_pad, int n_rows, int nnz, int tile,
                                                                CsrInfo* info, int32_t* __restrict__ tile_hist,
                                                                int32_t* __restrict__ long_rows, int long_cap) {
  __shared__ int hist[kBins];
  __shared__ int s_max;
  const int t = threadIdx.x;
  for (int b = t; b < kBins; b += kTileThreads) hist[b] = 0;
  if (t == 0) s_max = 0;
  __syncthreads();
  const int64_t r_begin = static_cast<int64_t>(blockIdx.x) * tile;
  int longest = 0;
  for (int64_t base = r_begin; base < min(r_begin + tile, static_cast<int64_t>(n_rows)); base += kTileThreads) {
    const int64_t r = base + t;
    int bin = -1;
    if (r < n_rows) {
      const int r0 = src[r], r1 = src[r + 1];
      dst[r] = r0;
      const int64_t len = static_cast<int64_t>(r1) - r0;
      if (len < 0) {
        atomicMax(&info->dec, INT_MAX - static_cast<int>(r));
      } else if (len <= nnz) {  // (else another row's pointer decreases)
        longest = max(longest, static_cast<int>(len));
        if (len <= kSliceMaxLen) {
          bin = static_cast<int>(len);
        } else {
          const int at = atomicAdd(&info->n_long, 1);
          if (at < long_cap) long_rows[at] = static_cast<int32_t>(r);
          atomicAdd(&info->long_slots, static_cast<unsigned long long>(
                                           32 * ((len + 31) / 32) + 160 * ((len + kPieceLen - 1) / kPieceLen)));
        }
      }
    }
    const unsigned int same = __match_any_sync(0xffffffffu, bin);
    if (bin >= 0 && (t & 31) == __ffs(static_cast<int>(same)) - 1) atomicAdd(&hist[bin], __popc(same));
  }
  atomicMax(&s_max, longest);
  if (blockIdx.x == 0) {
    if (t == 0) {
      info->rp0 = src[0];
      info->rpn = src[n_rows];
      dst[n_rows] = src[n_rows];
    }
    for (int64_t i = n_rows + 1 + t; i < n_pad; i += kTileThreads) dst[i] = 0;
  }
  __syncthreads();
  for (int b = t; b < kBins; b += kTileThreads) {
    tile_hist[static_cast<int64_t>(blockIdx.x) * kBins + b] = hist[b];
    if (hist[b]) atomicAdd(&info->hist[b], hist[b]);
  }
  if (t == 0) atomicMax(&info->maxlen, s_max);
}

// Copies columns and values (src may be dst) and checks the columns.  A warp
// takes 32 consecutive rows, whose entries are one contiguous run read
// coalesced, four strides of 32 in flight; a column must exceed the one
// before it unless a row starts there (one bit-or over the lanes' row starts
// per 32 entries).  Nothing is read where the row pointers are unusable.
__global__ void __launch_bounds__(256) csr_entries_kernel(const int32_t* __restrict__ rowptr, const int32_t* src_col,
                                                          const double* src_val, int32_t* col, double* val,
                                                          int64_t n_pad, int n_rows, int n_cols, int nnz,
                                                          CsrInfo* info) {
  if (info->rp0 != 0 || info->rpn != nnz || info->dec != 0) return;
  const int lane = threadIdx.x & 31;
  const int n_groups = (n_rows + 31) / 32;
  const int n_warps = (gridDim.x * blockDim.x) >> 5;
  // (the warp's index from lane 0: a loop the compiler knows to be uniform)
  const int warp0 = warp_uniform((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  for (int g = warp0; g < n_groups; g += n_warps) {
    const int r = g * 32 + lane;
    const int s = rowptr[min(r, n_rows)], e = rowptr[min(r + 1, n_rows)];
    const int e0 = __shfl_sync(0xffffffffu, s, 0), e1 = __shfl_sync(0xffffffffu, e, 31);
    int carry = -1;
    for (int base = e0; base < e1; base += 128) {
      int c[4];
      double v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int k = base + 32 * j + lane;
        c[j] = k < e1 ? __ldcs(src_col + k) : 0;
        v[j] = k < e1 ? __ldcs(src_val + k) : 0.0;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int b0 = base + 32 * j, k = b0 + lane;
        if (b0 < e1) {
          const int d = s - b0;
          const unsigned int starts = __reduce_or_sync(0xffffffffu, (s < e && d >= 0 && d < 32) ? 1u << d : 0u);
          int prev = __shfl_up_sync(0xffffffffu, c[j], 1);
          if (lane == 0) prev = carry;
          carry = __shfl_sync(0xffffffffu, c[j], 31);
          const bool bad = k < e1 && (c[j] < 0 || c[j] >= n_cols || (!((starts >> lane) & 1u) && c[j] <= prev));
          const unsigned int any = __ballot_sync(0xffffffffu, bad);
          if (any) {
            const int kb = b0 + __ffs(static_cast<int>(any)) - 1;  // its row: the last that starts at or before it
            const unsigned int before = __ballot_sync(0xffffffffu, s < e && s <= kb);
            if (lane == 0) atomicMax(&info->bad_col, INT_MAX - (g * 32 + 31 - __clz(static_cast<int>(before))));
          }
          if (k < e1) {
            if (src_col != col) col[k] = c[j];
            if (src_val != val) val[k] = v[j];
          }
        }
      }
    }
  }
  for (int64_t k = nnz + static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; k < n_pad;
       k += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    col[k] = 0;
    val[k] = 0.0;
  }
}

// The length-sorted order's table, made on the host from the histogram: by
// decreasing length (bin b holds length kSliceMaxLen - b), the first place of
// the bin's rows, the first slice that begins in the bin and its offset.
struct SliceTable {
  int32_t pos[kBins + 1];
  int32_t slice0[kBins];
  int64_t off0[kBins];
};

// tile_hist[t][len] -> the place of the tile's first row of that length (one
// block per length).
__global__ void __launch_bounds__(kMaxTiles) csr_scan_tiles_kernel(int32_t* tile_hist, int tiles,
                                                                   const SliceTable* tab) {
  __shared__ int wsum[kMaxTiles / 32];
  const int len = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int v = t < tiles ? tile_hist[static_cast<int64_t>(t) * kBins + len] : 0;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  int before = tab->pos[kBins - 1 - len];
  for (int w = 0; w < warp; ++w) before += wsum[w];
  if (t < tiles) tile_hist[static_cast<int64_t>(t) * kBins + len] = before + incl - v;
}

// perm: the rows of at most kSliceMaxLen entries by decreasing length, ties
// by increasing row.  A tile's warps take consecutive runs of its rows: first
// their counts per length, then each row's place.
__global__ void __launch_bounds__(kTileThreads) csr_perm_kernel(const int32_t* __restrict__ rowptr, int n_rows,
                                                                int tile, const int32_t* __restrict__ tile_hist,
                                                                int32_t* __restrict__ perm) {
  constexpr int kWarps = kTileThreads / 32;
  __shared__ int at[kWarps][kBins];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int i = t; i < kWarps * kBins; i += kTileThreads) (&at[0][0])[i] = 0;
  __syncthreads();
  const int per = tile / kWarps;  // a multiple of 32
  const int64_t w0 = static_cast<int64_t>(blockIdx.x) * tile + static_cast<int64_t>(warp) * per;
  auto bin_of = [&](int64_t r) {
    if (r >= n_rows) return -1;
    const int len = rowptr[r + 1] - rowptr[r];
    return len <= kSliceMaxLen ? len : -1;
  };
  for (int i = 0; i < per; i += 32) {
    const int bin = bin_of(w0 + i + lane);
    const unsigned int same = __match_any_sync(0xffffffffu, bin);
    if (bin >= 0 && lane == __ffs(static_cast<int>(same)) - 1) at[warp][bin] += __popc(same);
    __syncwarp();
  }
  __syncthreads();
  for (int b = t; b < kBins; b += kTileThreads) {
    int run = tile_hist[static_cast<int64_t>(blockIdx.x) * kBins + b];
    for (int w = 0; w < kWarps; ++w) {
      const int c = at[w][b];
      at[w][b] = run;
      run += c;
    }
  }
  __syncthreads();
  for (int i = 0; i < per; i += 32) {
    const int64_t r = w0 + i + lane;
    const int bin = bin_of(r);
    const unsigned int same = __match_any_sync(0xffffffffu, bin);
    int place = 0;
    if (bin >= 0) place = at[warp][bin] + __popc(same & ((1u << lane) - 1u));
    __syncwarp();
    if (bin >= 0) {
      perm[place] = static_cast<int32_t>(r);
      if (lane == __ffs(static_cast<int>(same)) - 1) at[warp][bin] += __popc(same);
    }
    __syncwarp();
  }
}

// Slice offsets: slice c has the length of the row at place 32 c, so they
// grow linearly within a bin.
__global__ void csr_offsets_kernel(const SliceTable* __restrict__ tab, int64_t n_slices, int64_t total,
                                   int64_t* __restrict__ off) {
  for (int64_t c = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; c <= n_slices;
       c += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    if (c == n_slices) {
      off[c] = total;
      continue;
    }
    const int64_t p = 32 * c;
    int lo = 0, hi = kBins - 1;  // the last bin with pos <= p
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (tab->pos[mid] <= p) lo = mid;
      else hi = mid - 1;
    }
    off[c] = tab->off0[lo] + 32 * (kSliceMaxLen - lo) * (c - tab->slice0[lo]);
  }
}

// HYB: rows by length (all lengths), per block in shared memory where they
// fit, else straight to memory.
__global__ void __launch_bounds__(256) csr_length_hist_kernel(const int32_t* __restrict__ rowptr, int n_rows,
                                                              int bins, int in_smem, int32_t* __restrict__ hist) {
  extern __shared__ int h[];
  if (in_smem) {
    for (int b = threadIdx.x; b < bins; b += blockDim.x) h[b] = 0;
    __syncthreads();
  }
  int* const to = in_smem ? h : hist;
  const int stride = gridDim.x * blockDim.x;
  for (int base = blockIdx.x * blockDim.x; base < n_rows; base += stride) {
    const int r = base + threadIdx.x;
    const int bin = r < n_rows ? rowptr[r + 1] - rowptr[r] : -1;
    const unsigned int same = __match_any_sync(0xffffffffu, bin);
    if (bin >= 0 && (threadIdx.x & 31) == __ffs(static_cast<int>(same)) - 1) atomicAdd(to + bin, __popc(same));
  }
  if (!in_smem) return;
  __syncthreads();
  for (int b = threadIdx.x; b < bins; b += blockDim.x)
    if (h[b]) atomicAdd(hist + b, h[b]);
}

// HYB: the tail rows (longer than K) in row order.  Pass 0 counts a tile's
// tail rows and overflow entries into tile_sum; pass 1, given the sums of
// the tiles before, writes slot (row -> tail row or -1), the tail rows and
// their first overflow entries.
__global__ void __launch_bounds__(kTileThreads) hyb_tail_kernel(const int32_t* __restrict__ rowptr, int n_rows,
                                                                int tile, int K, int2* tile_sum, int pass,
                                                                int32_t* __restrict__ slot,
                                                                int32_t* __restrict__ rows,
                                                                int32_t* __restrict__ tail_rowptr) {
  constexpr int kWarps = kTileThreads / 32;
  __shared__ int2 wsum[kWarps];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  int2 run = pass ? tile_sum[blockIdx.x] : make_int2(0, 0);
  const int64_t r_begin = static_cast<int64_t>(blockIdx.x) * tile;
  for (int64_t base = r_begin; base < min(r_begin + tile, static_cast<int64_t>(n_rows)); base += kTileThreads) {
    const int64_t r = base + t;
    const int len = r < n_rows ? rowptr[r + 1] - rowptr[r] : 0;
    const int2 v = make_int2(len > K ? 1 : 0, max(len - K, 0));
    int2 incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int ux = __shfl_up_sync(0xffffffffu, incl.x, o), uy = __shfl_up_sync(0xffffffffu, incl.y, o);
      if (lane >= o) {
        incl.x += ux;
        incl.y += uy;
      }
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int2 at = run;
    for (int w = 0; w < kWarps; ++w) {
      if (w < warp) {
        at.x += wsum[w].x;
        at.y += wsum[w].y;
      }
      run.x += wsum[w].x;
      run.y += wsum[w].y;
    }
    __syncthreads();
    if (pass && r < n_rows) {
      const int i = at.x + incl.x - v.x;
      slot[r] = v.x ? i : -1;
      if (v.x) {
        rows[i] = static_cast<int32_t>(r);
        tail_rowptr[i + 1] = at.y + incl.y;  // where the next tail row's entries begin
      }
    }
  }
  if (!pass && t == 0) tile_sum[blockIdx.x] = run;
}

// Exclusive sums of the tiles' pairs in place.
__global__ void __launch_bounds__(kMaxTiles) hyb_scan_kernel(int2* tile_sum, int tiles) {
  __shared__ int2 wsum[kMaxTiles / 32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int2 v = t < tiles ? tile_sum[t] : make_int2(0, 0);
  int2 incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int ux = __shfl_up_sync(0xffffffffu, incl.x, o), uy = __shfl_up_sync(0xffffffffu, incl.y, o);
    if (lane >= o) {
      incl.x += ux;
      incl.y += uy;
    }
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  int2 before = make_int2(0, 0);
  for (int w = 0; w < warp; ++w) {
    before.x += wsum[w].x;
    before.y += wsum[w].y;
  }
  if (t < tiles) tile_sum[t] = make_int2(before.x + incl.x - v.x, before.y + incl.y - v.y);
}

// Merge-path coordinates (rows consumed, nonzeros consumed) of every tile
// start: the largest i with rowptr[i] + i <= d such that the i-th row end
// precedes the diagonal d.
__global__ void merge_plan_kernel(const int32_t* __restrict__ rowptr, int n_rows, int nnz, int n_tiles,
                                  int32_t* tile_i, int32_t* tile_j) {
  const int stride = gridDim.x * blockDim.x;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t <= n_tiles; t += stride) {
    const long long dl = min(static_cast<long long>(t) * kMergeTile, static_cast<long long>(n_rows) + nnz);
    const int d = static_cast<int>(dl);
    int lo = max(0, d - nnz), hi = min(d, n_rows);
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (rowptr[mid + 1] <= d - mid - 1) lo = mid + 1;
      else hi = mid;
    }
    tile_i[t] = lo;
    tile_j[t] = d - lo;
  }
}

// ELL (column-major, ld rows per slot column) and, for HYB, the overflow of
// rows longer than K as COO entries (row, column, value) in row order.
__global__ void ell_fill_kernel(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                                const double* __restrict__ val, int n_rows, int K, int64_t ld,
                                int32_t* ell_col, double* ell_val, const int32_t* __restrict__ tail_slot,
                                const int32_t* __restrict__ tail_rowptr, int32_t* tail_row, int32_t* tail_col,
                                double* tail_val) {
  const int stride = gridDim.x * blockDim.x;
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n_rows; r += stride) {
    const int k0 = rowptr[r], len = rowptr[r + 1] - k0;
    for (int j = 0; j < K; ++j) {
      const int64_t o = static_cast<int64_t>(j) * ld + r;
      if (j < len) {
        ell_col[o] = col[k0 + j];
        ell_val[o] = val[k0 + j];
      } else {
        ell_col[o] = -1;
        ell_val[o] = 0.0;
      }
    }
    if (len > K && tail_slot) {
      const int base = tail_rowptr[tail_slot[r]];
      for (int j = K; j < len; ++j) {
        tail_row[base + j - K] = r;
        tail_col[base + j - K] = col[k0 + j];
        tail_val[base + j - K] = val[k0 + j];
      }
    }
  }
}

template <class T>
int upload(T** dst, const std::vector<T>& src, int64_t* bytes, cudaStream_t s) {
  GK_TRY(dalloc_async_n(dst, std::max<size_t>(src.size(), 1), bytes, s));
  if (!src.empty())
    GK_TRY_CUDA(cudaMemcpyAsync(*dst, src.data(), sizeof(T) * src.size(), cudaMemcpyHostToDevice, s));
  return GK_OK;
}

int grid1d(int64_t n, int threads) {
  int64_t g = (n + threads - 1) / threads;
  return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(g, 65535)));
}

struct MatrixDeleter {
  void operator()(Matrix* m) const { matrix_release(m); }
};

// Fill the length-sorted slices: one thread per (slice, lane); entry k of
// the lane's row at off[c] + 32 k + lane, padding with column -1 and 0.
__global__ void slice_fill_kernel(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                                  const double* __restrict__ val, const int32_t* __restrict__ perm,
                                  const int64_t* __restrict__ off, int64_t n_slices, int64_t n_sell,
                                  int32_t* __restrict__ scol, double* __restrict__ sval) {
  const int64_t total = n_slices * 32;
  for (int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; t < total;
       t += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t c = t >> 5;
    const int lane = static_cast<int>(t & 31);
    const int64_t o0 = off[c];
    const int L = static_cast<int>((off[c + 1] - o0) >> 5);
    const int row = t < n_sell ? perm[t] : -1;
    const int k0 = row >= 0 ? rowptr[row] : 0;
    const int len = row >= 0 ? rowptr[row + 1] - k0 : 0;
    for (int k = 0; k < L; ++k) {
      const int64_t d = o0 + 32 * static_cast<int64_t>(k) + lane;
      scol[d] = k < len ? col[k0 + k] : -1;
      sval[d] = k < len ? val[k0 + k] : 0.0;
    }
  }
}

// Stored entries over the DFMA lane slots the GK_CSR kernel issues (slices:
// 32 x their longest row; a long row 32 x ceil(len / 32) plus a butterfly
// per piece).
double sliced_efficiency(const CsrInfo& info, int64_t nnz) {
  double slots = static_cast<double>(info.long_slots);
  int64_t place = 0;  // rows placed so far, longest first
  for (int64_t L = kSliceMaxLen; L >= 0; --L) {
    const int64_t first = (place + 31) / 32, end = (place + info.hist[L] + 31) / 32;
    slots += 32.0 * static_cast<double>(L) * static_cast<double>(end - first);
    place += info.hist[L];
  }
  return slots > 0 ? static_cast<double>(nnz) / slots : 1.0;
}

// Scratch of one creation, freed in stream order (the creation ends with a
// synchronization of its stream).
struct Scratch {
  cudaStream_t s;
  std::vector<void*> p;
  explicit Scratch(cudaStream_t st) : s(st) {}
  ~Scratch() {
    for (void* q : p) cudaFreeAsync(q, s);
  }
  template <class T>
  int get(T** out, size_t n) {
    GK_TRY(dalloc_async_n(out, n, nullptr, s));
    p.push_back(*out);
    return GK_OK;
  }
};

__global__ void long_bounds_kernel(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ rows, int n,
                                   int4* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int r = rows[i];
    out[i] = make_int4(r, rowptr[r], rowptr[r + 1], 0);
  }
}

int long_row_pieces(const int32_t* rowptr, const int32_t* d_rows, int n, Scratch& tmp, std::vector<int4>& pc,
                    std::vector<int32_t>& lr_row, std::vector<int32_t>& lr_off, int32_t& n_slot) {
  int4* d_b = nullptr;
  GK_TRY(tmp.get(&d_b, static_cast<size_t>(n)));
  long_bounds_kernel<<<(n + 255) / 256, 256, 0, tmp.s>>>(rowptr, d_rows, n, d_b);
  GK_TRY_CUDA(cudaGetLastError());
  std::vector<int4> rows(static_cast<size_t>(n));
  GK_TRY_CUDA(cudaMemcpyAsync(rows.data(), d_b, sizeof(int4) * n, cudaMemcpyDeviceToHost, tmp.s));
  GK_TRY_CUDA(cudaStreamSynchronize(tmp.s));
  std::sort(rows.begin(), rows.end(), [](const int4& u, const int4& v) {
    const int lu = u.z - u.y, lv = v.z - v.y;
    return lu != lv ? lu > lv : u.x < v.x;
  });
  for (const int4& r : rows) {
    const bool split = r.z - r.y > kPieceLen;
    for (int32_t k = r.y; k < r.z; k += kPieceLen)
      pc.push_back(make_int4(r.x, k, std::min<int32_t>(r.z, k + kPieceLen), split ? n_slot++ : -1));
    if (split) {
      lr_row.push_back(r.x);
      lr_off.push_back(n_slot);
    }
  }
  std::stable_sort(pc.begin(), pc.end(), [](const int4& u, const int4& v) { return u.z - u.y > v.z - v.y; });
  return GK_OK;
}

// Whether kernels of the current device can read p (aligned device or managed
// memory of it); host arrays and other devices' are copied first.
bool readable_here(const void* p, size_t align, int device) {
  cudaPointerAttributes at;
  if (!p || reinterpret_cast<uintptr_t>(p) % align != 0 || cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return (at.type == cudaMemoryTypeDevice && at.device == device) || at.type == cudaMemoryTypeManaged;
}

}  // namespace

int build_merge_plan(MergePlan& P, int64_t n_rows, int64_t nnz, const int32_t* rowptr,
                     const int32_t* col, const double* val, int64_t* bytes, cudaStream_t s) {
  P.n_rows = n_rows;
  P.nnz = nnz;
  P.rowptr = rowptr;
  P.col = col;
  P.val = val;
  P.n_tiles = (n_rows + nnz + kMergeTile - 1) / kMergeTile;
  const size_t nt = static_cast<size_t>(std::max<int64_t>(P.n_tiles, 1));
  GK_TRY(dalloc_async_n(&P.tile_i, nt + 1, bytes, s));
  GK_TRY(dalloc_async_n(&P.tile_j, nt + 1, bytes, s));
  GK_TRY(dalloc_async_n(&P.head_val, nt, bytes, s));
  GK_TRY(dalloc_async_n(&P.carry_val, nt, bytes, s));
  if (P.n_tiles > 0) {
    merge_plan_kernel<<<grid1d(P.n_tiles + 1, 256), 256, 0, s>>>(
        rowptr, static_cast<int>(n_rows), static_cast<int>(nnz), static_cast<int>(P.n_tiles), P.tile_i,
        P.tile_j);
    GK_TRY_CUDA(cudaGetLastError());
  }
  P.grid = merge_grid(P.n_tiles);
  return GK_OK;
}

void matrix_release(Matrix* A) {
  if (!A) return;
  if (A->refs.fetch_sub(1) != 1) return;
  int prev = -1;
  cudaGetDevice(&prev);
  cudaSetDevice(A->device);
  void* ptrs[] = {A->rowptr, A->col, A->val, A->sl_perm, A->sl_off, A->sl_col, A->sl_val, A->pc, A->lr_row, A->lr_off, A->pc_sum,
                  A->merge.tile_i, A->merge.tile_j, A->merge.head_val, A->merge.carry_val, A->ell_col,
                  A->ell_val,
                  A->tail_rows, A->tail_rowptr, A->tail_row, A->tail_col, A->tail_val, A->tail_slot,
                  A->tail_sum, A->coo_first, A->coo_last, A->coo_head, A->coo_tail, A->partials, A->counter,
                  A->err};
  // applies are asynchronous, and a failed creation leaves kernels behind:
  // the pool must not hand these arrays out before they have finished
  dfree_pooled(ptrs, sizeof(ptrs) / sizeof(ptrs[0]), A->use);
  dfree(A->dot_st);
  dfree(A->stage_in);
  dfree(A->stage_out);
  if (prev >= 0) cudaSetDevice(prev);
  delete A;
}

}  // namespace gk

using namespace gk;

extern "C" int gk_matrix_create_csr(int64_t n_rows, int64_t n_cols, int64_t nnz, const int32_t* rowptr,
                                    const int32_t* col, const void* val, int32_t dtype, int32_t format,
                                    void* stream, gk_matrix* out) {
  if (!out) return set_error(GK_ERR_ARG, "gk_matrix_create_csr: out is NULL");
  *out = nullptr;
  if (n_rows < 0 || n_cols < 0 || nnz < 0)
    return set_error(GK_ERR_ARG, "gk_matrix_create_csr: negative size");
  if (nnz > INT32_MAX - 64 || n_rows > INT32_MAX - 64 || n_cols > INT32_MAX ||
      n_rows + nnz > static_cast<int64_t>(INT32_MAX) - 4 * kMergeTile)
    return set_error(GK_ERR_ARG, "gk_matrix_create_csr: sizes exceed int32 indexing");
  if (!rowptr || (nnz > 0 && (!col || !val)))
    return set_error(GK_ERR_ARG, "gk_matrix_create_csr: NULL array");
  if (dtype == GK_F32)
    return set_error(GK_ERR_UNSUPPORTED, "gk_matrix_create_csr: FP32 storage is not built");
  if (dtype != GK_F64) return set_error(GK_ERR_DTYPE, "gk_matrix_create_csr: unknown dtype %d", dtype);
  if (format < GK_CSR || format > GK_AUTO)
    return set_error(GK_ERR_ARG, "gk_matrix_create_csr: unknown format %d", format);
  cudaStream_t s = static_cast<cudaStream_t>(stream);

  std::unique_ptr<Matrix, MatrixDeleter> hold(new Matrix);
  Matrix* A = hold.get();
  A->device = current_device();
  A->n_rows = n_rows;
  A->n_cols = n_cols;
  A->nnz = nnz;
  A->use.on(s);
  int64_t* bytes = &A->device_bytes;

  // ---- library-owned CSR copy, checked and analysed on the way -----------------
  GK_TRY(dalloc_async_n(&A->rowptr, padded(n_rows + 1), bytes, s));
  GK_TRY(dalloc_async_n(&A->col, padded(nnz), bytes, s));
  GK_TRY(dalloc_async_n(&A->val, padded(nnz), bytes, s));
  GK_TRY(dalloc_async_n(&A->counter, 4, bytes, s));
  GK_TRY(dalloc_async_n(&A->err, 4, bytes, s));
  GK_TRY_CUDA(cudaMemsetAsync(A->counter, 0, 4 * sizeof(unsigned int), s));
  GK_TRY_CUDA(cudaMemsetAsync(A->err, 0, 4 * sizeof(int), s));
  const int32_t* src_rp = rowptr;
  const int32_t* src_col = col;
  const double* src_val = static_cast<const double*>(val);
  if (!readable_here(rowptr, 4, A->device)) {
    GK_TRY_CUDA(cudaMemcpyAsync(A->rowptr, rowptr, sizeof(int32_t) * (n_rows + 1), cudaMemcpyDefault, s));
    src_rp = A->rowptr;
  }
  if (nnz > 0 && !readable_here(col, 4, A->device)) {
    GK_TRY_CUDA(cudaMemcpyAsync(A->col, col, sizeof(int32_t) * nnz, cudaMemcpyDefault, s));
    src_col = A->col;
  }
  if (nnz > 0 && !readable_here(val, 8, A->device)) {
    GK_TRY_CUDA(cudaMemcpyAsync(A->val, val, sizeof(double) * nnz, cudaMemcpyDefault, s));
    src_val = A->val;
  }
  Scratch tmp(s);
  const int tile = static_cast<int>(tile_rows(n_rows));
  const int tiles = static_cast<int>(std::max<int64_t>(1, (n_rows + tile - 1) / tile));
  const int64_t long_cap = std::min(n_rows, nnz / (kSliceMaxLen + 1)) + 1;
  CsrInfo* d_info = nullptr;
  int32_t *tile_hist = nullptr, *long_rows = nullptr;
  GK_TRY(tmp.get(&d_info, 1));
  GK_TRY(tmp.get(&tile_hist, static_cast<size_t>(tiles) * kBins));
  GK_TRY(tmp.get(&long_rows, static_cast<size_t>(long_cap)));
  GK_TRY_CUDA(cudaMemsetAsync(d_info, 0, sizeof(CsrInfo), s));
  csr_rows_kernel<<<tiles, kTileThreads, 0, s>>>(src_rp, A->rowptr, padded(n_rows + 1), static_cast<int>(n_rows),
                                                 static_cast<int>(nnz), tile, d_info, tile_hist, long_rows,
                                                 static_cast<int>(long_cap));
  GK_TRY_CUDA(cudaGetLastError());
  csr_entries_kernel<<<grid1d(n_rows, 256), 256, 0, s>>>(A->rowptr, src_col, src_val, A->col, A->val, padded(nnz),
                                                         static_cast<int>(n_rows), static_cast<int>(n_cols),
                                                         static_cast<int>(nnz), d_info);
  GK_TRY_CUDA(cudaGetLastError());
  CsrInfo info;
  GK_TRY_CUDA(cudaMemcpyAsync(&info, d_info, sizeof(info), cudaMemcpyDeviceToHost, s));
  GK_TRY_CUDA(cudaStreamSynchronize(s));
  if (info.rp0 != 0) return set_error(GK_ERR_CSR, "rowptr[0] = %d, expected 0", info.rp0);
  if (info.dec != 0) return set_error(GK_ERR_CSR, "rowptr decreases at row %lld", (long long)(INT_MAX - info.dec));
  if (info.rpn != nnz)
    return set_error(GK_ERR_CSR, "rowptr[n_rows] = %d, expected nnz = %lld", info.rpn, (long long)nnz);
  if (info.bad_col != 0)
    return set_error(GK_ERR_CSR, "row %d: column index out of range, unsorted or repeated", INT_MAX - info.bad_col);

  // ---- format ------------------------------------------------------------------
  int fmt = format;
  if (fmt == GK_AUTO) fmt = (sliced_efficiency(info, nnz) >= 0.75) ? GK_CSR : GK_CSR_MERGE;
  A->format = fmt;
  if (fmt == GK_CSR) {
    // rows by decreasing length (ties: increasing row index) on the device,
    // from a table made of the histogram
    SliceTable tab;
    int64_t place = 0, total = 0;
    for (int b = 0; b < kBins; ++b) {
      const int64_t len = kSliceMaxLen - b, first = (place + 31) / 32;
      tab.pos[b] = static_cast<int32_t>(place);
      tab.slice0[b] = static_cast<int32_t>(first);
      tab.off0[b] = total;
      place += info.hist[len];
      total += 32 * len * ((place + 31) / 32 - first);
    }
    tab.pos[kBins] = static_cast<int32_t>(place);
    const int64_t n_sell = place, n_slices = (n_sell + 31) / 32;
    A->n_sell = n_sell;
    A->n_slices = n_slices;
    A->sl_entries = total;
    GK_TRY(dalloc_async_n(&A->sl_perm, static_cast<size_t>(std::max<int64_t>(n_sell, 1)), bytes, s));
    GK_TRY(dalloc_async_n(&A->sl_off, static_cast<size_t>(n_slices + 1), bytes, s));
    GK_TRY(dalloc_async_n(&A->sl_col, static_cast<size_t>(std::max<int64_t>(total, 1)), bytes, s));
    GK_TRY(dalloc_async_n(&A->sl_val, static_cast<size_t>(std::max<int64_t>(total, 1)), bytes, s));
    SliceTable* d_tab = nullptr;
    GK_TRY(tmp.get(&d_tab, 1));
    GK_TRY_CUDA(cudaMemcpyAsync(d_tab, &tab, sizeof(tab), cudaMemcpyHostToDevice, s));
    csr_offsets_kernel<<<grid1d(n_slices + 1, 256), 256, 0, s>>>(d_tab, n_slices, total, A->sl_off);
    GK_TRY_CUDA(cudaGetLastError());
    if (n_slices > 0) {
      csr_scan_tiles_kernel<<<kBins, kMaxTiles, 0, s>>>(tile_hist, tiles, d_tab);
      GK_TRY_CUDA(cudaGetLastError());
      csr_perm_kernel<<<tiles, kTileThreads, 0, s>>>(A->rowptr, static_cast<int>(n_rows), tile, tile_hist,
                                                     A->sl_perm);
      GK_TRY_CUDA(cudaGetLastError());
      slice_fill_kernel<<<grid1d(n_slices * 32, 256), 256, 0, s>>>(A->rowptr, A->col, A->val, A->sl_perm,
                                                                   A->sl_off, n_slices, n_sell, A->sl_col,
                                                                   A->sl_val);
      GK_TRY_CUDA(cudaGetLastError());
    }
    // long rows in pieces of kPieceLen consecutive entries (the last one
    // shorter), longest first (ties: row, then position): few, on the host
    std::vector<int4> pc;
    std::vector<int32_t> lr_row, lr_off(1, 0);
    int32_t n_slot = 0;
    A->n_long = info.n_long;
    if (info.n_long > 0) {
      GK_TRY(long_row_pieces(A->rowptr, long_rows, info.n_long, tmp, pc, lr_row, lr_off, n_slot));
    }
    A->n_pc = static_cast<int64_t>(pc.size());
    A->n_lr = static_cast<int64_t>(lr_row.size());
    GK_TRY(upload(&A->pc, pc, bytes, s));
    GK_TRY(upload(&A->lr_row, lr_row, bytes, s));
    GK_TRY(upload(&A->lr_off, lr_off, bytes, s));
    GK_TRY(dalloc_async_n(&A->pc_sum, static_cast<size_t>(std::max<int32_t>(n_slot, 1)), bytes, s));
    A->sl_deep = sliced_deep(A->n_pc + n_slices, info.maxlen);
    A->n_split = sliced_split(info.hist, A->n_pc, n_slices, static_cast<int64_t>(info.long_slots) / 32 + total / 32);
    A->grid_sl = sliced_grid(A->n_pc + A->n_slices + 3 * A->n_split, false);
    A->grid_sl_plain = sliced_grid(A->n_pc + A->n_slices + 3 * A->n_split, true);
  } else if (fmt == GK_CSR_MERGE) {
    GK_TRY(build_merge_plan(A->merge, n_rows, nnz, A->rowptr, A->col, A->val, bytes, s));
  } else {  // GK_ELL, GK_HYB
    const int64_t maxlen = info.maxlen;
    int64_t K = maxlen, tail_m = 0, tail_entries = 0;
    if (fmt == GK_ELL) {
      if (K * n_rows > 8 * nnz + n_rows)
        return set_error(GK_ERR_FORMAT,
                         "ELL would hold %lld slots for %lld entries (longest row %lld); use GK_HYB",
                         (long long)(K * n_rows), (long long)nnz, (long long)K);
    } else {
      // smallest K minimising K*n*(8+4) + overflow*(8+2*4), from the
      // histogram of row lengths
      std::vector<int32_t> hist(static_cast<size_t>(maxlen + 2), 0);
      if (n_rows > 0) {
        const int bins = static_cast<int>(maxlen) + 1;
        const int in_smem = bins <= 12 * 1024 ? 1 : 0;  // 48 KB
        int32_t* d_hist = nullptr;
        GK_TRY(tmp.get(&d_hist, static_cast<size_t>(bins)));
        GK_TRY_CUDA(cudaMemsetAsync(d_hist, 0, sizeof(int32_t) * bins, s));
        csr_length_hist_kernel<<<std::min(grid1d(n_rows, 256), 4 * sm_count()), 256,
                                 in_smem ? sizeof(int) * bins : 0, s>>>(A->rowptr, static_cast<int>(n_rows), bins,
                                                                        in_smem, d_hist);
        GK_TRY_CUDA(cudaGetLastError());
        GK_TRY_CUDA(cudaMemcpyAsync(hist.data(), d_hist, sizeof(int32_t) * bins, cudaMemcpyDeviceToHost, s));
        GK_TRY_CUDA(cudaStreamSynchronize(s));
      }
      // gt[k] = #rows longer than k, over[k] = sum max(0, len - k)
      std::vector<int64_t> over(static_cast<size_t>(maxlen + 2), 0), gt(static_cast<size_t>(maxlen + 2), 0);
      for (int64_t k = maxlen - 1; k >= 0; --k) {
        gt[k] = gt[k + 1] + hist[k + 1];
        over[k] = over[k + 1] + gt[k];
      }
      int64_t bestK = 0, bestc = -1;
      for (int64_t k = 0; k <= maxlen; ++k) {
        int64_t c = k * n_rows * 12 + over[k] * 16;
        if (bestc < 0 || c < bestc) {
          bestc = c;
          bestK = k;
        }
      }
      K = bestK;
      tail_m = gt[K];
      tail_entries = over[K];
    }
    A->K = K;
    A->ld = ((n_rows + 31) / 32) * 32;
    GK_TRY(dalloc_async_n(&A->ell_col, static_cast<size_t>(std::max<int64_t>(K * A->ld, 1)), bytes, s));
    GK_TRY(dalloc_async_n(&A->ell_val, static_cast<size_t>(std::max<int64_t>(K * A->ld, 1)), bytes, s));
    if (fmt == GK_HYB) {
      // the tail rows and the overflow entries, from the histogram's sums
      A->m_tail = tail_m;
      A->tail_nnz = tail_entries;
      int2* tile_sum = nullptr;
      GK_TRY(tmp.get(&tile_sum, static_cast<size_t>(tiles)));
      // COO arrays in whole chunks (each lane's 16-byte loads stay inside)
      A->coo_chunks = (A->tail_nnz + kCooChunk - 1) / kCooChunk;
      const int64_t coo_n = std::max<int64_t>(A->coo_chunks * kCooChunk, padded(A->tail_nnz));
      GK_TRY(dalloc_async_n(&A->tail_slot, static_cast<size_t>(std::max<int64_t>(n_rows, 1)), bytes, s));
      GK_TRY(dalloc_async_n(&A->tail_rows, static_cast<size_t>(std::max<int64_t>(A->m_tail, 1)), bytes, s));
      GK_TRY(dalloc_async_n(&A->tail_rowptr, static_cast<size_t>(padded(A->m_tail + 1)), bytes, s));
      GK_TRY(dalloc_async_n(&A->tail_row, static_cast<size_t>(coo_n), bytes, s));
      GK_TRY(dalloc_async_n(&A->tail_col, static_cast<size_t>(coo_n), bytes, s));
      GK_TRY(dalloc_async_n(&A->tail_val, static_cast<size_t>(coo_n), bytes, s));
      GK_TRY(dalloc_async_n(&A->tail_sum, static_cast<size_t>(std::max<int64_t>(A->m_tail, 1)), bytes, s));
      GK_TRY_CUDA(cudaMemsetAsync(A->tail_rowptr, 0, sizeof(int32_t) * padded(A->m_tail + 1), s));
      // the entries themselves are written by ell_fill_kernel; zero the rest
      const int64_t rest = coo_n - A->tail_nnz;
      GK_TRY_CUDA(cudaMemsetAsync(A->tail_row + A->tail_nnz, 0, sizeof(int32_t) * rest, s));
      GK_TRY_CUDA(cudaMemsetAsync(A->tail_col + A->tail_nnz, 0, sizeof(int32_t) * rest, s));
      GK_TRY_CUDA(cudaMemsetAsync(A->tail_val + A->tail_nnz, 0, sizeof(double) * rest, s));
      if (n_rows > 0) {
        for (int pass = 0; pass < 2; ++pass) {
          hyb_tail_kernel<<<tiles, kTileThreads, 0, s>>>(A->rowptr, static_cast<int>(n_rows), tile,
                                                         static_cast<int>(K), tile_sum, pass, A->tail_slot,
                                                         A->tail_rows, A->tail_rowptr);
          GK_TRY_CUDA(cudaGetLastError());
          if (pass == 0) hyb_scan_kernel<<<1, kMaxTiles, 0, s>>>(tile_sum, tiles);
          GK_TRY_CUDA(cudaGetLastError());
        }
      }
      const size_t nc = static_cast<size_t>(std::max<int64_t>(A->coo_chunks, 1));
      GK_TRY(dalloc_async_n(&A->coo_first, nc, bytes, s));
      GK_TRY(dalloc_async_n(&A->coo_last, nc, bytes, s));
      GK_TRY(dalloc_async_n(&A->coo_head, nc, bytes, s));
      GK_TRY(dalloc_async_n(&A->coo_tail, nc, bytes, s));
      A->grid_coo = coo_grid(A->coo_chunks);
    }
    if (n_rows > 0) {
      ell_fill_kernel<<<grid1d(n_rows, 256), 256, 0, s>>>(
          A->rowptr, A->col, A->val, static_cast<int>(n_rows), static_cast<int>(K), A->ld, A->ell_col,
          A->ell_val, fmt == GK_HYB ? A->tail_slot : nullptr, A->tail_rowptr, A->tail_row, A->tail_col,
          A->tail_val);
      GK_TRY_CUDA(cudaGetLastError());
    }
    A->grid_ell = ell_grid(n_rows);
  }
  A->max_grid = std::max(spmv_max_grid(*A), 4 * sm_count());
  GK_TRY(dalloc_async_n(&A->partials, static_cast<size_t>(2 * (A->max_grid + kFixupMaxGrid)), bytes, s));
  GK_TRY_CUDA(cudaStreamSynchronize(s));
  *out = reinterpret_cast<gk_matrix>(hold.release());
  return GK_OK;
}

extern "C" int gk_matrix_get_info(gk_matrix h, gk_matrix_info* info) {
  Matrix* A = as_matrix(h);
  if (!A || !info) return set_error(GK_ERR_ARG, "gk_matrix_get_info: NULL argument");
  info->n_rows = A->n_rows;
  info->n_cols = A->n_cols;
  info->nnz = A->nnz;
  info->format = A->format;
  info->dtype = GK_F64;
  info->ell_width = (A->format == GK_ELL || A->format == GK_HYB) ? A->K : 0;
  info->tail_rows = A->m_tail;
  info->tail_nnz = A->tail_nnz;
  info->short_items = A->n_slices;
  info->long_rows = A->n_long;
  info->split_rows = A->n_lr;
  info->tiles = A->merge.n_tiles;
  info->device_bytes = A->device_bytes;
  // the stored operator once (CSR: values, indices, row pointers; ELL: the
  // entries' values and indices; HYB: ELL entries + COO entries with their
  // row index), x read once, y written once
  int64_t mat = A->nnz * 12 + (A->n_rows + 1) * 4;
  if (A->format == GK_ELL) mat = A->nnz * 12;
  if (A->format == GK_HYB) mat = (A->nnz - A->tail_nnz) * 12 + A->tail_nnz * 16;
  info->spmv_bytes = mat + A->n_cols * 8 + A->n_rows * 8;
  return GK_OK;
}

extern "C" int gk_matrix_destroy(gk_matrix h) {
  if (!h) return set_error(GK_ERR_ARG, "gk_matrix_destroy: NULL handle");
  matrix_release(as_matrix(h));
  return GK_OK;
}
