// permute_csr.cu -- build A' = P_r A P_c (Eq. 1) in CSR with ascending columns
// (Section 2), values copied bit for bit.
//
//   1. len'[i'] = len(rperm[i'])                      (gather of row lengths)
//   2. rowptr' = exclusive scan of len'               (scan.cu)
//   3. bucket the new rows by where they start (buckets of kBucket = 2048
//      entries).  One CTA per bucket gathers the entries of its rows from the
//      old matrix, relabels each column c -> cinv[c], and orders every row by
//      (new column, old position), so equal columns keep their old order.  A
//      bucket holds at most 4096 entries as long as no row in it is longer than
//      kLong = 2048.
//   4. rows longer than kLong (the paper's dense-row case, Section 1) are
//      gathered into one list keyed by (long-row id, new column) and sorted
//      with the radix sort of perm.cu, then written to their rows.
#include <algorithm>

#include "handle.cuh"

namespace maxe {
namespace {

constexpr int kBucket = 2048;
constexpr int kLong = 2048;
constexpr int kSortCap = 4096;  // entries per bucket tile
constexpr int kSortThreads = 512;
constexpr int kSortItems = kSortCap / kSortThreads;

__global__ void row_lengths_kernel(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ rperm, int32_t M,
                                   int32_t* __restrict__ len) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= M) return;
  const int32_t r = rperm ? rperm[i] : static_cast<int32_t>(i);
  len[i] = rowptr[r + 1] - rowptr[r];
}

// Shared memory of a bucket.  Rows are known by where they start in the
// bucket (empty rows do not appear): `start` marks those entries, and a row's
// old place, length and column range sit at the index of its first entry.  Once
// the entries are in registers the three arrays are used again: a for the bins,
// b and c for the entries in bin order, and last b for the ordered columns and
// c and a (adjacent) for the ordered values.
struct SortSmem {
  int32_t b[kSortCap];  // first column of the row's range -> columns by bin -> ordered columns
  int32_t c[kSortCap];  // last column of the row's range -> positions by bin -> ordered values
  int32_t a[kSortCap];  // old start minus start -> bin counts, then ends
  uint16_t len[kSortCap];
  uint32_t start[kSortCap / 32];  // bit per entry: a row starts here
  int32_t before[kSortCap / 32];  // last row start before this word
  uint32_t ws[kSortThreads / 32];
  uint32_t pairs[kSortThreads / 32];
};

// Comparisons within bins (the sum of their squared counts) up to which a bucket is
// ranked by bins.  On 25 M entries (12,200 buckets) 1000 comparisons in each take
// 4.1 us and the sort takes 1050 us.
constexpr uint32_t kMaxPairs = 250000;

// Sorts sz keys (a power of two) in ascending order; the whole block.  Not inlined: its
// registers are not the bins'.
__device__ __noinline__ void sort_bucket(uint64_t* keys, int sz) {
  for (int kk = 2; kk <= sz; kk <<= 1) {
    for (int j = kk >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < (sz >> 1); t += kSortThreads) {
        const int lo = 2 * t - (t & (j - 1)), hi = lo + j;
        const bool up = (lo & kk) == 0;
        const uint64_t a = keys[lo], b = keys[hi];
        if ((a > b) == up) {
          keys[lo] = b;
          keys[hi] = a;
        }
      }
      __syncthreads();
    }
  }
}

// Start of the row that holds entry pos of the bucket.
__device__ __forceinline__ int32_t row_of(const SortSmem& sm, int pos) {
  const uint32_t bits = sm.start[pos >> 5] & (0xffffffffu >> (31 - (pos & 31)));
  return bits ? (pos & ~31) + 31 - __clz(bits) : sm.before[pos >> 5];
}

// One CTA per bucket g: rows [first[g], first[g+1]) minus a trailing long row.
//
// A row of n entries is ordered by n bins of equal width over its columns' range
// (all columns when they were permuted, which spreads them; first to last
// when not, where a row mostly is in order already): each entry counts itself
// into its bin, a scan of all bins places the bins, and an entry's rank in its
// bin is the number of smaller (column, position) pairs in it, of which there
// are few.  Columns that crowd into few bins (a band under a column permutation that
// keeps it, or one far column in rows that are otherwise close) would ask for up
// to n^2 comparisons, so a bucket with more than kMaxPairs of them is sorted instead
// (100,000 rows of 250 neighbours under an identity permutation, the whole call: 2579 us
// ranked, 1507 us sorted; under a random one 490 us).
// A bitonic sort of 64-bit keys took 1874 us for 25.4 M entries (2^20 rows), this took 417 us with two
// CTAs an SM and takes 406 us with three (40 registers, a few spilled), with ten
// barriers a bucket that leave a CTA waiting.
template <typename VT>
__global__ void __launch_bounds__(kSortThreads, 3) bucket_sort_kernel(
    const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col, const VT* __restrict__ val,
    const int32_t* __restrict__ rperm, const int32_t* __restrict__ cinv, const int32_t* __restrict__ nrowptr,
    const int32_t* __restrict__ first, int32_t M, int32_t N, int64_t Z, int32_t* __restrict__ ncol,
    VT* __restrict__ nval) {
  extern __shared__ __align__(16) unsigned char raw[];
  SortSmem& sm = *reinterpret_cast<SortSmem*>(raw);
  const int g = blockIdx.x;
  const int32_t r0 = first[g], r1 = first[g + 1];
  if (r0 >= r1) return;
  int32_t rhi = r1;
  const int64_t base = nrowptr[r0];
  int64_t end = (r1 < M) ? static_cast<int64_t>(nrowptr[r1]) : Z;
  if (nrowptr[r1 - 1] + static_cast<int64_t>(kLong) < end) {  // trailing long row: handled elsewhere
    rhi = r1 - 1;
    end = nrowptr[r1 - 1];
  }
  const int count = static_cast<int>(end - base);
  if (count <= 0) return;
  for (int t = threadIdx.x; t < kSortCap / 32; t += kSortThreads) sm.start[t] = 0u;
  __syncthreads();
  for (int32_t r = r0 + static_cast<int32_t>(threadIdx.x); r < rhi; r += kSortThreads) {
    const int32_t s = static_cast<int32_t>(nrowptr[r] - base);
    const int32_t n = (r + 1 < rhi ? static_cast<int32_t>(nrowptr[r + 1] - base) : count) - s;
    if (n <= 0) continue;
    const int32_t o = rowptr[rperm ? rperm[r] : r];
    sm.a[s] = o - s;
    sm.len[s] = static_cast<uint16_t>(n);
    if (!cinv) {
      sm.b[s] = col[o];
      sm.c[s] = col[o + n - 1];
    }
    atomicOr(&sm.start[s >> 5], 1u << (s & 31));
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp == 0) {  // before[w]: four words per lane, then a running maximum over the lanes
    int32_t last[4], run = -1;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t bits = sm.start[4 * lane + u];
      last[u] = run;
      if (bits) run = 32 * (4 * lane + u) + 31 - __clz(bits);
    }
    int32_t up = run;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) up = max(up, __shfl_up_sync(0xffffffffu, up, d));
    up = __shfl_up_sync(0xffffffffu, up, 1);
    if (lane == 0) up = -1;
#pragma unroll
    for (int u = 0; u < 4; ++u) sm.before[4 * lane + u] = max(up, last[u]);
  }
  __syncthreads();
  int32_t nc[kSortItems], row[kSortItems];  // new column; start of the entry's row
  VT v[kSortItems];
#pragma unroll
  for (int u = 0; u < kSortItems; ++u) {
    const int pos = u * kSortThreads + static_cast<int>(threadIdx.x);
    if (pos < count) {
      row[u] = row_of(sm, pos);
      const int32_t src = sm.a[row[u]] + pos;
      nc[u] = __ldcs(col + src);
      v[u] = __ldcs(val + src);
    }
  }
  if (cinv) {
#pragma unroll
    for (int u = 0; u < kSortItems; ++u)
      if (u * kSortThreads + static_cast<int>(threadIdx.x) < count) nc[u] = cinv[nc[u]];
  }
  int32_t bin[kSortItems];
#pragma unroll
  for (int u = 0; u < kSortItems; ++u) {
    if (u * kSortThreads + static_cast<int>(threadIdx.x) < count) {
      // rounding is monotonic, so bins ascend with the columns; clamped to the row's own
      const int32_t n = sm.len[row[u]];
      const int32_t lo = cinv ? 0 : sm.b[row[u]], hi = cinv ? N - 1 : sm.c[row[u]];
      const float scale = __fdividef(static_cast<float>(n), fmaxf(static_cast<float>(hi) - static_cast<float>(lo), 1.f));
      const float f = (static_cast<float>(nc[u]) - static_cast<float>(lo)) * scale;
      bin[u] = row[u] + static_cast<int32_t>(fminf(fmaxf(f, 0.f), static_cast<float>(n - 1)));
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < kSortCap; t += kSortThreads) sm.a[t] = 0;
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kSortItems; ++u)
    if (u * kSortThreads + static_cast<int>(threadIdx.x) < count) atomicAdd(&sm.a[bin[u]], 1);
  __syncthreads();
  {  // exclusive sums of the bins, and the comparisons that they ask for
    int4* pa = reinterpret_cast<int4*>(sm.a) + threadIdx.x * (kSortItems / 4);
    int4 w[kSortItems / 4];
    int32_t run = 0;
    uint32_t pairs = 0;  // the block's total is at most kSortCap squared
#pragma unroll
    for (int u = 0; u < kSortItems / 4; ++u) {
      w[u] = pa[u];
      run += w[u].x + w[u].y + w[u].z + w[u].w;
      pairs += w[u].x * w[u].x + w[u].y * w[u].y + w[u].z * w[u].z + w[u].w * w[u].w;
    }
    pairs = __reduce_add_sync(0xffffffffu, pairs);
    if (lane == 0) sm.pairs[warp] = pairs;
    int32_t inc = run;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int32_t t = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= d) inc += t;
    }
    if (lane == 31) sm.ws[warp] = static_cast<uint32_t>(inc);
    __syncthreads();
    int32_t pre = inc - run;
    for (int k = 0; k < warp; ++k) pre += static_cast<int32_t>(sm.ws[k]);
#pragma unroll
    for (int u = 0; u < kSortItems / 4; ++u) {
      int4 o;
      o.x = pre;
      o.y = o.x + w[u].x;
      o.z = o.y + w[u].y;
      o.w = o.z + w[u].z;
      pre = o.w + w[u].w;
      pa[u] = o;
    }
  }
  __syncthreads();
  int32_t rank[kSortItems];
  if (__reduce_add_sync(0xffffffffu, sm.pairs[lane % (kSortThreads / 32)]) / 2 <= kMaxPairs) {
#pragma unroll
    for (int u = 0; u < kSortItems; ++u) {  // into bin order; a[bin] ends as the bin's end
      const int pos = u * kSortThreads + static_cast<int>(threadIdx.x);
      if (pos < count) {
        const int32_t p = atomicAdd(&sm.a[bin[u]], 1);
        sm.b[p] = nc[u];
        sm.c[p] = pos;
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kSortItems; ++u) {
      const int pos = u * kSortThreads + static_cast<int>(threadIdx.x);
      if (pos < count) {
        const int32_t s = bin[u] ? sm.a[bin[u] - 1] : 0, e = sm.a[bin[u]];
        rank[u] = s;
        if (e - s > 1)
          for (int32_t q = s; q < e; ++q) rank[u] += sm.b[q] < nc[u] || (sm.b[q] == nc[u] && sm.c[q] < pos);
      }
    }
  } else {
    // Columns that share bins: all entries by (row start | new column | position), 55 bits.
    uint64_t* keys = reinterpret_cast<uint64_t*>(sm.b);  // b and c
    int sz = 1;
    while (sz < count) sz <<= 1;
#pragma unroll
    for (int u = 0; u < kSortItems; ++u) {
      const int pos = u * kSortThreads + static_cast<int>(threadIdx.x);
      if (pos < count)
        keys[pos] = (static_cast<uint64_t>(row_of(sm, pos)) << 43) | (static_cast<uint64_t>(nc[u]) << 12) |
                    static_cast<uint64_t>(pos);
      else if (pos < sz)
        keys[pos] = ~0ull;
    }
    __syncthreads();
    sort_bucket(keys, sz);
    for (int p = threadIdx.x; p < count; p += kSortThreads) sm.a[keys[p] & 0xFFFull] = p;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kSortItems; ++u) {
      const int pos = u * kSortThreads + static_cast<int>(threadIdx.x);
      if (pos < count) rank[u] = sm.a[pos];
    }
  }
  __syncthreads();
  VT* sval = reinterpret_cast<VT*>(sm.c);
#pragma unroll
  for (int u = 0; u < kSortItems; ++u) {
    if (u * kSortThreads + static_cast<int>(threadIdx.x) < count) {
      sm.b[rank[u]] = nc[u];
      sval[rank[u]] = v[u];
    }
  }
  __syncthreads();
  for (int pos = threadIdx.x; pos < count; pos += kSortThreads) {
    ncol[base + pos] = sm.b[pos];
    nval[base + pos] = sval[pos];
  }
}

__global__ void long_flags_kernel(const int32_t* __restrict__ len, int32_t M, int32_t* __restrict__ flag,
                                  unsigned long long* __restrict__ stats) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= M) return;
  const int isl = len[i] > kLong;
  flag[i] = isl;
  if (isl) {
    atomicAdd(&stats[0], 1ull);
    atomicAdd(&stats[1], static_cast<unsigned long long>(len[i]));
  }
}

__global__ void long_compact_kernel(const int32_t* __restrict__ flag, const int32_t* __restrict__ ids, int32_t M,
                                    const int32_t* __restrict__ len, int32_t* __restrict__ rows,
                                    int32_t* __restrict__ lens) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= M || !flag[i]) return;
  rows[ids[i]] = static_cast<int32_t>(i);
  lens[ids[i]] = len[i];
}

// One CTA per long row: key = (id << colbits) | new column, value = old entry index.
__global__ void long_fill_kernel(const int32_t* __restrict__ lrows, const int32_t* __restrict__ seg,
                                 const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                                 const int32_t* __restrict__ rperm, const int32_t* __restrict__ cinv, int colbits,
                                 uint64_t* __restrict__ keys, int32_t* __restrict__ src) {
  const int id = blockIdx.x;
  const int32_t r = lrows[id];
  const int32_t o = rowptr[rperm ? rperm[r] : r];
  const int32_t n = rowptr[(rperm ? rperm[r] : r) + 1] - o;
  const int64_t s0 = seg[id];
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    const int32_t c = col[o + t];
    const uint64_t nc = static_cast<uint64_t>(cinv ? cinv[c] : c);
    keys[s0 + t] = (static_cast<uint64_t>(id) << colbits) | nc;
    src[s0 + t] = o + t;
  }
}

template <typename VT>
__global__ void long_write_kernel(const uint64_t* __restrict__ keys, const int32_t* __restrict__ src, int64_t n,
                                  int colbits, const int32_t* __restrict__ seg, const int32_t* __restrict__ lrows,
                                  const int32_t* __restrict__ nrowptr, const VT* __restrict__ val,
                                  int32_t* __restrict__ ncol, VT* __restrict__ nval) {
  const int64_t s = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const uint64_t key = keys[s];
  const int id = static_cast<int>(key >> colbits);
  const int64_t dst = static_cast<int64_t>(nrowptr[lrows[id]]) + (s - seg[id]);
  ncol[dst] = static_cast<int32_t>(key & ((1ull << colbits) - 1));
  nval[dst] = val[src[s]];
}

// Validation (MAXE_VALIDATE): any failure sets *bad.
__global__ void validate_csr_kernel(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col, int32_t M,
                                    int32_t N, int64_t Z, int* __restrict__ bad) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i == 0 && (rowptr[0] != 0 || rowptr[M] != Z)) atomicOr(bad, 1);
  if (i < M && rowptr[i + 1] < rowptr[i]) atomicOr(bad, 1);
  if (i < Z && (col[i] < 0 || col[i] >= N)) atomicOr(bad, 1);
}

__global__ void count_perm_kernel(const int32_t* __restrict__ perm, int32_t n, int32_t* __restrict__ seen,
                                  int* __restrict__ bad) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t p = perm[i];
  if (p < 0 || p >= n || atomicAdd(&seen[p], 1) != 0) atomicOr(bad, 1);
}

inline unsigned grid_for(int64_t n, int b = 256) { return static_cast<unsigned>(std::max<int64_t>(1, ceil_div(n, b))); }

template <typename VT>
maxe_status bucket_sort_launch(const maxe_csr* A, const int32_t* rperm, const int32_t* cinv, maxe_handle* h,
                               const int32_t* first, int64_t nb, cudaStream_t st) {
  auto kern = bucket_sort_kernel<VT>;
  const size_t smem = sizeof(SortSmem);
  MAXE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)));
  kern<<<static_cast<unsigned>(nb), kSortThreads, smem, st>>>(A->rowptr, A->col, static_cast<const VT*>(A->val),
                                                               rperm, cinv, h->rowptr, first, A->rows, A->cols,
                                                               A->nnz, h->col, static_cast<VT*>(h->val));
  MAXE_CUDA_TRY(cudaGetLastError());
  return MAXE_OK;
}

template <typename VT>
maxe_status long_write_launch(const uint64_t* keys, const int32_t* src, int64_t n, int colbits, const int32_t* seg,
                              const int32_t* lrows, maxe_handle* h, const void* val, cudaStream_t st) {
  long_write_kernel<VT><<<grid_for(n), 256, 0, st>>>(keys, src, n, colbits, seg, lrows, h->rowptr,
                                                     static_cast<const VT*>(val), h->col, static_cast<VT*>(h->val));
  MAXE_CUDA_TRY(cudaGetLastError());
  return MAXE_OK;
}

int bits_for(int64_t n) {  // bits to hold values 0..n-1 (at least 1)
  int b = 1;
  while ((int64_t(1) << b) < n) ++b;
  return b;
}

}  // namespace

maxe_status permute_csr_run(const maxe_csr* A, const int32_t* rperm, const int32_t* cperm, uint32_t flags,
                            maxe_handle* h, cudaStream_t st) {
  const int32_t M = A->rows, N = A->cols;
  const int64_t Z = A->nnz;
  const Allocator& al = h->al;
  ScratchSet scratch(al);

  if (flags & MAXE_VALIDATE) {
    int* bad = scratch.get<int>(1);
    int32_t* seen = scratch.get<int32_t>(static_cast<size_t>(std::max<int64_t>(std::max(M, N), 1)));
    if (!bad || !seen) return MAXE_ERR_OOM;
    MAXE_CUDA_TRY(cudaMemsetAsync(bad, 0, sizeof(int), st));
    validate_csr_kernel<<<grid_for(std::max<int64_t>(M + 1, Z)), 256, 0, st>>>(A->rowptr, A->col, M, N, Z, bad);
    if (rperm) {
      MAXE_CUDA_TRY(cudaMemsetAsync(seen, 0, sizeof(int32_t) * M, st));
      count_perm_kernel<<<grid_for(M), 256, 0, st>>>(rperm, M, seen, bad);
    }
    if (cperm) {
      MAXE_CUDA_TRY(cudaMemsetAsync(seen, 0, sizeof(int32_t) * N, st));
      count_perm_kernel<<<grid_for(N), 256, 0, st>>>(cperm, N, seen, bad);
    }
    MAXE_CUDA_TRY(cudaGetLastError());
    int hbad = 0;
    MAXE_CUDA_TRY(cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, st));
    MAXE_CUDA_TRY(cudaStreamSynchronize(st));
    if (hbad) return MAXE_ERR_INVALID;
  }

  // owned arrays
  const int vb = value_bytes(A->dtype);
  h->nnz_pad = round_up(Z + spmv_pad_elems(), kPadElems);
  h->rowptr = static_cast<int32_t*>(al.get(static_cast<size_t>(M + 1 + kRowptrPad) * sizeof(int32_t)));
  h->col = static_cast<int32_t*>(al.get(static_cast<size_t>(h->nnz_pad) * sizeof(int32_t)));
  h->val = al.get(static_cast<size_t>(h->nnz_pad) * vb);
  if (!h->rowptr || !h->col || !h->val) return MAXE_ERR_OOM;
  MAXE_CUDA_TRY(cudaMemsetAsync(h->rowptr + M, 0, (1 + kRowptrPad) * sizeof(int32_t), st));
  MAXE_CUDA_TRY(cudaMemsetAsync(h->col + Z, 0, (h->nnz_pad - Z) * sizeof(int32_t), st));
  MAXE_CUDA_TRY(cudaMemsetAsync(static_cast<char*>(h->val) + Z * vb, 0, (h->nnz_pad - Z) * vb, st));
  if (rperm) {
    h->rperm = static_cast<int32_t*>(al.get(static_cast<size_t>(std::max(M, 1)) * sizeof(int32_t)));
    if (!h->rperm) return MAXE_ERR_OOM;
    MAXE_CUDA_TRY(cudaMemcpyAsync(h->rperm, rperm, sizeof(int32_t) * M, cudaMemcpyDeviceToDevice, st));
  }
  if (cperm) {
    h->cperm = static_cast<int32_t*>(al.get(static_cast<size_t>(std::max(N, 1)) * sizeof(int32_t)));
    if (!h->cperm) return MAXE_ERR_OOM;
    MAXE_CUDA_TRY(cudaMemcpyAsync(h->cperm, cperm, sizeof(int32_t) * N, cudaMemcpyDeviceToDevice, st));
  }

  if (M > 0) {
    // 1-2. new row pointers
    int32_t* scan_tmp = scratch.get<int32_t>(scan_scratch_elems(M));
    int32_t* cinv = nullptr;
    if (cperm) {
      cinv = scratch.get<int32_t>(static_cast<size_t>(std::max(N, 1)));
      if (!cinv) return MAXE_ERR_OOM;
      MAXE_TRY(launch_invert(cperm, N, cinv, st));
    }
    if (!scan_tmp) return MAXE_ERR_OOM;
    row_lengths_kernel<<<grid_for(M), 256, 0, st>>>(A->rowptr, rperm, M, h->rowptr);
    MAXE_CUDA_TRY(cudaGetLastError());
    // keep the lengths for the long-row pass before scanning in place
    int32_t* len = scratch.get<int32_t>(static_cast<size_t>(M));
    if (!len) return MAXE_ERR_OOM;
    MAXE_CUDA_TRY(cudaMemcpyAsync(len, h->rowptr, sizeof(int32_t) * M, cudaMemcpyDeviceToDevice, st));
    MAXE_TRY(scan_exclusive_i32(h->rowptr, h->rowptr, M, h->rowptr + M, scan_tmp, st));

    if (Z > 0) {
      // 3. buckets of short rows
      const int64_t nb = ceil_div(Z, kBucket);
      int32_t* first = scratch.get<int32_t>(static_cast<size_t>(nb + 1));
      if (!first) return MAXE_ERR_OOM;
      MAXE_TRY(bucket_lower_bounds(h->rowptr, M, kBucket, 0, nb, first, st));
      switch (A->dtype) {
        case MAXE_F64: MAXE_TRY(bucket_sort_launch<uint64_t>(A, rperm, cinv, h, first, nb, st)); break;
        case MAXE_F32: MAXE_TRY(bucket_sort_launch<uint32_t>(A, rperm, cinv, h, first, nb, st)); break;
        case MAXE_BF16: MAXE_TRY(bucket_sort_launch<uint16_t>(A, rperm, cinv, h, first, nb, st)); break;
      }

      // 4. long rows
      int32_t* lflag = scratch.get<int32_t>(static_cast<size_t>(M));
      unsigned long long* stats = scratch.get<unsigned long long>(2);
      if (!lflag || !stats) return MAXE_ERR_OOM;
      MAXE_CUDA_TRY(cudaMemsetAsync(stats, 0, 2 * sizeof(unsigned long long), st));
      long_flags_kernel<<<grid_for(M), 256, 0, st>>>(len, M, lflag, stats);
      MAXE_CUDA_TRY(cudaGetLastError());
      unsigned long long hs[2] = {0, 0};
      MAXE_CUDA_TRY(cudaMemcpyAsync(hs, stats, sizeof(hs), cudaMemcpyDeviceToHost, st));
      MAXE_CUDA_TRY(cudaStreamSynchronize(st));
      const int64_t nlong = static_cast<int64_t>(hs[0]), tlong = static_cast<int64_t>(hs[1]);
      if (nlong > 0) {
        int32_t* ids = scratch.get<int32_t>(static_cast<size_t>(M));
        int32_t* lrows = scratch.get<int32_t>(static_cast<size_t>(nlong));
        int32_t* llen = scratch.get<int32_t>(static_cast<size_t>(nlong + 1));
        int32_t* scan2 = scratch.get<int32_t>(scan_scratch_elems(std::max<int64_t>(M, nlong)));
        if (!ids || !lrows || !llen || !scan2) return MAXE_ERR_OOM;
        MAXE_TRY(scan_exclusive_i32(lflag, ids, M, nullptr, scan2, st));
        long_compact_kernel<<<grid_for(M), 256, 0, st>>>(lflag, ids, M, len, lrows, llen);
        MAXE_CUDA_TRY(cudaGetLastError());
        MAXE_TRY(scan_exclusive_i32(llen, llen, nlong, llen + nlong, scan2, st));  // llen -> segment starts
        const int colbits = bits_for(N);
        const int idbits = bits_for(nlong);
        if (colbits + idbits > 64) return MAXE_ERR_UNSUPPORTED;
        // radix sort buffers (own allocations: the scratch set holds at most 16)
        uint64_t* k0 = static_cast<uint64_t*>(al.get(sizeof(uint64_t) * tlong));
        uint64_t* k1 = static_cast<uint64_t*>(al.get(sizeof(uint64_t) * tlong));
        int32_t* v0 = static_cast<int32_t*>(al.get(sizeof(int32_t) * tlong));
        int32_t* v1 = static_cast<int32_t*>(al.get(sizeof(int32_t) * tlong));
        void* rs = al.get(radix_scratch_bytes(tlong));
        maxe_status stt = (k0 && k1 && v0 && v1 && rs) ? MAXE_OK : MAXE_ERR_OOM;
        if (stt == MAXE_OK) {
          long_fill_kernel<<<static_cast<unsigned>(nlong), 256, 0, st>>>(lrows, llen, A->rowptr, A->col, rperm, cinv,
                                                                         colbits, k0, v0);
          stt = cudaGetLastError() == cudaSuccess ? MAXE_OK : MAXE_ERR_CUDA;
        }
        if (stt == MAXE_OK) stt = radix_sort_pairs(k0, v0, k1, v1, tlong, colbits + idbits, rs, st);
        if (stt == MAXE_OK) {
          switch (A->dtype) {
            case MAXE_F64: stt = long_write_launch<uint64_t>(k0, v0, tlong, colbits, llen, lrows, h, A->val, st); break;
            case MAXE_F32: stt = long_write_launch<uint32_t>(k0, v0, tlong, colbits, llen, lrows, h, A->val, st); break;
            case MAXE_BF16: stt = long_write_launch<uint16_t>(k0, v0, tlong, colbits, llen, lrows, h, A->val, st); break;
          }
        }
        al.put(rs);
        al.put(v1);
        al.put(v0);
        al.put(k1);
        al.put(k0);
        if (stt != MAXE_OK) return stt;
      }
    }
  } else {
    MAXE_CUDA_TRY(cudaMemsetAsync(h->rowptr, 0, sizeof(int32_t), st));
  }
  return spmv_build_partition(h, st);
}

}  // namespace maxe
