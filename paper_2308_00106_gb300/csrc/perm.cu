// perm.cu -- the random permutation of Section 3 and the vector permutations
// of Eq. 1.
//
//   keys:   key(seed, tag, i) = output number 2i+tag+1 of SplitMix64 seeded with
//           `seed` (Steele, Lea, Flood 2014), one thread per index.
//   order:  the indices in ascending (key, index) order are perm[new] = old.  The
//           keys are pseudo-random, so one split by their top bits into buckets
//           of about a thousand, then one in shared memory by the next bits into
//           bins of about one half, leaves almost nothing to compare: the keys are
//           computed where they are needed and never stored.
//   sort:   stable LSD radix sort of (key, index) pairs, 8 bits per pass, for the
//           keys that are not random (rows, cells).
//   invert: inv[perm[i]] = i.
//   gather / scatter: x' = P_c^{-1} x and y = P_r^{-1} y'.
#include <algorithm>

#include "handle.cuh"
#include "launch.cuh"

namespace maxe {
namespace {

constexpr uint64_t kGamma = 0x9e3779b97f4a7c15ull;

__device__ __forceinline__ uint64_t splitmix_output(uint64_t seed, uint64_t m) {
  uint64_t z = seed + m * kGamma;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

__device__ __forceinline__ uint64_t perm_key(uint64_t seed, int32_t tag, int32_t i) {
  return splitmix_output(seed, 2ull * static_cast<uint64_t>(i) + static_cast<uint64_t>(tag) + 1ull);
}

// ------------------------------------------- order by the Section 3 keys
// n = 2^20 took 370 us as eight radix passes over stored keys (40 launches);
// this takes four launches and reads and writes 4 bytes per index twice.
constexpr int kPoThreads = 1024;             // split kernels
constexpr int kPoItems = 8;
constexpr int kPoTile = kPoThreads * kPoItems;
constexpr int kPoSmemBuckets = 4096;         // more buckets are counted in global memory
constexpr int kPoSmallCap = 2048;            // indices of a bucket ordered in shared memory
constexpr int kPoLargeCap = 8192;            // ... and for n above kPoSmallCap / 2 * kPoSmemBuckets

struct PermOrder {
  uint64_t seed;
  int32_t tag, first, n;  // indices first .. first + n - 1
  int bits;               // buckets: the top `bits` bits of the key
};

__device__ __forceinline__ uint32_t po_bucket(uint64_t key, int bits) {
  return bits ? static_cast<uint32_t>(key >> (64 - bits)) : 0u;
}

// Counts per bucket, then (in the block that finishes last) their exclusive
// sums.  cnt: 2^bits counts and the block counter, zero before the launch.
__global__ void __launch_bounds__(kPoThreads) po_count(PermOrder o, uint32_t* cnt) {
  __shared__ uint32_t hist[kPoSmemBuckets];
  __shared__ uint32_t ws[kPoThreads / 32];
  __shared__ bool last_block;
  const uint32_t B = 1u << o.bits;
  const bool local = B <= kPoSmemBuckets;
  if (local)
    for (uint32_t b = threadIdx.x; b < B; b += kPoThreads) hist[b] = 0u;
  __syncthreads();
  const int64_t base = static_cast<int64_t>(blockIdx.x) * kPoTile;
#pragma unroll
  for (int u = 0; u < kPoItems; ++u) {
    const int64_t i = base + u * kPoThreads + threadIdx.x;
    if (i < o.n)
      atomicAdd((local ? hist : cnt) + po_bucket(perm_key(o.seed, o.tag, o.first + static_cast<int32_t>(i)), o.bits),
                1u);
  }
  __syncthreads();
  if (local)
    for (uint32_t b = threadIdx.x; b < B; b += kPoThreads)
      if (hist[b]) atomicAdd(cnt + b, hist[b]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last_block = atomicAdd(cnt + B, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last_block) return;
  __threadfence();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t carry = 0;
  for (uint32_t b0 = 0; b0 < B; b0 += 4 * kPoThreads) {  // four consecutive buckets per thread
    uint32_t v[4], run = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t b = b0 + 4 * threadIdx.x + u;
      v[u] = run;
      run += b < B ? __ldcg(cnt + b) : 0u;
    }
    uint32_t inc = run;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= d) inc += t;
    }
    __syncthreads();  // the previous round's reads of ws
    if (lane == 31) ws[w] = inc;
    __syncthreads();
    uint32_t pre = carry + inc - run, total = 0;
    for (int k = 0; k < kPoThreads / 32; ++k) {
      if (k < w) pre += ws[k];
      total += ws[k];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t b = b0 + 4 * threadIdx.x + u;
      if (b < B) cnt[b] = pre + v[u];
    }
    carry += total;
  }
}

// Indices into their buckets, in any order within a bucket; cursor[b] goes from
// the bucket's start to its end.  A block reserves its share of each bucket
// with one atomic.
__global__ void __launch_bounds__(kPoThreads) po_split(PermOrder o, uint32_t* cursor, int32_t* __restrict__ out) {
  __shared__ uint32_t hist[kPoSmemBuckets];
  const uint32_t B = 1u << o.bits;
  const bool local = B <= kPoSmemBuckets;
  if (local)
    for (uint32_t b = threadIdx.x; b < B; b += kPoThreads) hist[b] = 0u;
  __syncthreads();
  const int64_t base = static_cast<int64_t>(blockIdx.x) * kPoTile;
  uint32_t bk[kPoItems], at[kPoItems];
#pragma unroll
  for (int u = 0; u < kPoItems; ++u) {
    const int64_t i = base + u * kPoThreads + threadIdx.x;
    if (i < o.n) {
      bk[u] = po_bucket(perm_key(o.seed, o.tag, o.first + static_cast<int32_t>(i)), o.bits);
      at[u] = atomicAdd((local ? hist : cursor) + bk[u], 1u);
    }
  }
  __syncthreads();
  if (local)
    for (uint32_t b = threadIdx.x; b < B; b += kPoThreads)
      if (hist[b]) hist[b] = atomicAdd(cursor + b, hist[b]);
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kPoItems; ++u) {
    const int64_t i = base + u * kPoThreads + threadIdx.x;
    if (i < o.n) out[(local ? hist[bk[u]] : 0u) + at[u]] = o.first + static_cast<int32_t>(i);
  }
}

// One block per bucket: its indices in ascending (key, index) order.  in: the
// split indices (null: one bucket of all indices); ends[b]: the end of bucket b.
template <int CAP>
struct PoSmem {
  uint64_t key[CAP];
  int32_t idx[CAP];
  uint32_t bin[CAP];
};

template <int CAP, int THREADS>
__global__ void __launch_bounds__(THREADS) po_order(PermOrder o, const int32_t* __restrict__ in,
                                                    const uint32_t* __restrict__ ends, int32_t* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char po_raw[];
  PoSmem<CAP>& sm = *reinterpret_cast<PoSmem<CAP>*>(po_raw);
  __shared__ uint32_t ws[THREADS / 32];
  constexpr int kItems = CAP / THREADS;
  const uint32_t lo = in && blockIdx.x ? ends[blockIdx.x - 1] : 0u;
  const uint32_t m = (in ? ends[blockIdx.x] : static_cast<uint32_t>(o.n)) - lo;
  if (m > CAP) {
    // More than twice the expected size never happens with these keys (above
    // thirty standard deviations); ranked by counting, so that it would be right.
    for (uint32_t p = threadIdx.x; p < m; p += THREADS) {
      const int32_t ip = in ? in[lo + p] : o.first + static_cast<int32_t>(p);
      const uint64_t kp = perm_key(o.seed, o.tag, ip);
      uint32_t rank = 0;
      for (uint32_t q = 0; q < m; ++q) {
        const int32_t iq = in ? in[lo + q] : o.first + static_cast<int32_t>(q);
        const uint64_t kq = perm_key(o.seed, o.tag, iq);
        rank += kq < kp || (kq == kp && iq < ip);
      }
      out[lo + rank] = ip;
    }
    return;
  }
  constexpr int kBinBits = CAP == 2048 ? 11 : 13;
  static_assert((1 << kBinBits) == CAP, "one bin per slot");
  auto bin_of = [&](uint64_t key) { return static_cast<uint32_t>((key << o.bits) >> (64 - kBinBits)); };
  for (int b = threadIdx.x; b < CAP; b += THREADS) sm.bin[b] = 0u;
  __syncthreads();
  uint64_t key[kItems];
  int32_t idx[kItems];
#pragma unroll
  for (int u = 0; u < kItems; ++u) {
    const uint32_t p = u * THREADS + threadIdx.x;
    if (p < m) idx[u] = in ? in[lo + p] : o.first + static_cast<int32_t>(p);
  }
#pragma unroll
  for (int u = 0; u < kItems; ++u) {
    if (u * THREADS + threadIdx.x < m) {
      key[u] = perm_key(o.seed, o.tag, idx[u]);
      atomicAdd(&sm.bin[bin_of(key[u])], 1u);
    }
  }
  __syncthreads();
  {  // exclusive sums of the bin counts
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t v[kItems], run = 0;
#pragma unroll
    for (int u = 0; u < kItems; ++u) {
      v[u] = run;
      run += sm.bin[threadIdx.x * kItems + u];
    }
    uint32_t inc = run;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= d) inc += t;
    }
    if (lane == 31) ws[w] = inc;
    __syncthreads();
    uint32_t pre = inc - run;
    for (int k = 0; k < w; ++k) pre += ws[k];
#pragma unroll
    for (int u = 0; u < kItems; ++u) sm.bin[threadIdx.x * kItems + u] = pre + v[u];
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kItems; ++u) {  // into the bins; bin[b] ends as the bin's end
    if (u * THREADS + threadIdx.x < m) {
      const uint32_t p = atomicAdd(&sm.bin[bin_of(key[u])], 1u);
      sm.key[p] = key[u];
      sm.idx[p] = idx[u];
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kItems; ++u) {  // rank within the bin
    if (u * THREADS + threadIdx.x < m) {
      const uint32_t b = bin_of(key[u]);
      const uint32_t s = b ? sm.bin[b - 1] : 0u, e = sm.bin[b];
      uint32_t rank = s;
      for (uint32_t q = s; q < e; ++q) rank += sm.key[q] < key[u] || (sm.key[q] == key[u] && sm.idx[q] < idx[u]);
      out[lo + rank] = idx[u];
    }
  }
}

// Buckets of at most half a shared-memory tile on average.
int po_bits(int64_t n, int64_t mean) {
  int bits = 0;
  while ((mean << bits) < n) ++bits;
  return bits;
}

int64_t po_mean(int64_t n) {
  return n <= static_cast<int64_t>(kPoSmallCap / 2) * kPoSmemBuckets ? kPoSmallCap / 2 : kPoLargeCap / 2;
}

// ------------------------------------------------------------ radix sort
constexpr int kRsThreads = 256;
constexpr int kRsWarps = kRsThreads / 32;
constexpr int kRsItems = 16;
constexpr int kRsTile = kRsThreads * kRsItems;  // 4096 keys per tile
constexpr int kRsWarpKeys = 32 * kRsItems;      // 512 keys per warp
constexpr int kBins = 256;

// counts[d * ntiles + tile] = number of keys of the tile with digit d.
__global__ void __launch_bounds__(kRsThreads) rs_upsweep(const uint64_t* __restrict__ keys, int64_t n, int shift,
                                                         int32_t* __restrict__ counts, int64_t ntiles) {
  __shared__ uint32_t hist[kBins];
  hist[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = static_cast<int64_t>(blockIdx.x) * kRsTile;
#pragma unroll 4
  for (int i = 0; i < kRsItems; ++i) {
    int64_t e = base + threadIdx.x + i * kRsThreads;
    if (e < n) atomicAdd(&hist[(keys[e] >> shift) & 0xFF], 1u);
  }
  __syncthreads();
  counts[static_cast<int64_t>(threadIdx.x) * ntiles + blockIdx.x] = static_cast<int32_t>(hist[threadIdx.x]);
}

// Stable scatter of one tile: warp w owns keys [w*512, w*512+512) of the tile,
// visited 32 at a time in index order, so rank order equals index order.
__global__ void __launch_bounds__(kRsThreads) rs_scatter(const uint64_t* __restrict__ kin,
                                                         const int32_t* __restrict__ vin,
                                                         uint64_t* __restrict__ kout, int32_t* __restrict__ vout,
                                                         int64_t n, int shift, const int32_t* __restrict__ offs,
                                                         int64_t ntiles) {
  __shared__ uint32_t wcount[kRsWarps][kBins];
  __shared__ uint32_t tile_off[kBins];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kRsWarps * kBins; i += kRsThreads) (&wcount[0][0])[i] = 0;
  tile_off[threadIdx.x] = static_cast<uint32_t>(offs[static_cast<int64_t>(threadIdx.x) * ntiles + blockIdx.x]);
  __syncthreads();

  const int64_t base = static_cast<int64_t>(blockIdx.x) * kRsTile + w * kRsWarpKeys;
  const unsigned lt_mask = (1u << lane) - 1u;
  uint64_t k[kRsItems];
  int32_t v[kRsItems];
  uint32_t rank[kRsItems];
#pragma unroll
  for (int j = 0; j < kRsItems; ++j) {
    const int64_t e = base + j * 32 + lane;
    const bool valid = e < n;
    k[j] = valid ? kin[e] : 0ull;
    v[j] = valid ? vin[e] : 0;
    const uint32_t d = valid ? static_cast<uint32_t>((k[j] >> shift) & 0xFF) : static_cast<uint32_t>(kBins);
    const unsigned peers = __match_any_sync(0xffffffffu, d);
    const int leader = __ffs(peers) - 1;
    uint32_t old = 0;
    if (valid && lane == leader) {
      old = wcount[w][d];
      wcount[w][d] = old + __popc(peers);
    }
    old = __shfl_sync(0xffffffffu, old, leader);
    rank[j] = old + __popc(peers & lt_mask);
    __syncwarp();
  }
  __syncthreads();
  {  // exclusive prefix over warps, per digit
    const int d = threadIdx.x;
    uint32_t run = 0;
#pragma unroll
    for (int ww = 0; ww < kRsWarps; ++ww) {
      uint32_t t = wcount[ww][d];
      wcount[ww][d] = run;
      run += t;
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kRsItems; ++j) {
    const int64_t e = base + j * 32 + lane;
    if (e < n) {
      const uint32_t d = static_cast<uint32_t>((k[j] >> shift) & 0xFF);
      const int64_t pos = static_cast<int64_t>(tile_off[d]) + wcount[w][d] + rank[j];
      kout[pos] = k[j];
      vout[pos] = v[j];
    }
  }
}

__global__ void invert_kernel(const int32_t* __restrict__ perm, int32_t n, int32_t* __restrict__ inv) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n) inv[perm[i]] = static_cast<int32_t>(i);
}

constexpr int kGatherThreads = 256;
constexpr int kGatherRows = 4;  // rows per thread, their loads in flight together

// out row i = in row perm[i], row_elems elements each, in pieces of V = VE
// elements (16 bytes where the rows are aligned, else one element): a group of
// 2^shift lanes takes a row, piece after piece, and a thread has kGatherRows
// rows in flight.  Bound by the random reads of `in`: a 16-byte row still
// moves a 32-byte sector (4.19M rows of 4 FP32: 16 us of sectors and 20 us of
// the rest at 6.8 TB/s).  One element per thread with a 64-bit division to
// find its row took 87 us there.
template <typename T, typename V>
__global__ void __launch_bounds__(kGatherThreads) gather_kernel(const int32_t* __restrict__ perm, int64_t n,
                                                                int row_elems, int shift, const T* __restrict__ in,
                                                                int64_t ld_in, T* __restrict__ out, int64_t ld_out) {
  start_next();
  after_previous();
  constexpr int VE = sizeof(V) / sizeof(T);
  const int rows = kGatherThreads >> shift;  // per step of the block
  const int c0 = (threadIdx.x & ((1 << shift) - 1)) * VE;
  const int64_t i0 = static_cast<int64_t>(blockIdx.x) * rows * kGatherRows + (threadIdx.x >> shift);
  int64_t src[kGatherRows];
#pragma unroll
  for (int u = 0; u < kGatherRows; ++u) {
    const int64_t i = i0 + u * rows;
    src[u] = i < n ? static_cast<int64_t>(perm[i]) * ld_in : 0;
  }
  for (int c = c0; c < row_elems; c += VE << shift) {
    if (c + VE <= row_elems) {
      V v[kGatherRows];
#pragma unroll
      for (int u = 0; u < kGatherRows; ++u)
        if (i0 + u * rows < n) v[u] = *reinterpret_cast<const V*>(in + src[u] + c);
#pragma unroll
      for (int u = 0; u < kGatherRows; ++u)
        if (i0 + u * rows < n) *reinterpret_cast<V*>(out + (i0 + u * rows) * ld_out + c) = v[u];
    } else {  // the row's last piece, shorter: its elements alone
      for (int u = 0; u < kGatherRows; ++u)
        if (i0 + u * rows < n)
          for (int e = c; e < row_elems; ++e) out[(i0 + u * rows) * ld_out + e] = in[src[u] + e];
    }
  }
}

template <typename T, typename V>
void gather_launch(const int32_t* perm, int64_t n, int64_t row_elems, const void* in, int64_t ld_in, void* out,
                   int64_t ld_out, cudaStream_t st) {
  constexpr int VE = sizeof(V) / sizeof(T);
  int shift = 0;  // lanes per row: a power of two, at most 32
  while (shift < 5 && (static_cast<int64_t>(VE) << shift) < row_elems) ++shift;
  const int64_t rows = static_cast<int64_t>(kGatherThreads >> shift) * kGatherRows;
  launch_after(gather_kernel<T, V>, static_cast<unsigned>(ceil_div(n, rows)), kGatherThreads, 0, st, perm, n,
               static_cast<int>(row_elems), shift, static_cast<const T*>(in), ld_in, static_cast<T*>(out), ld_out);
}

// 16-byte pieces when rows of more than one element start on 16-byte boundaries on both sides.
template <typename T>
void gather_any(const int32_t* perm, int64_t n, int64_t row_elems, const void* in, int64_t ld_in, void* out,
                int64_t ld_out, cudaStream_t st) {
  constexpr int64_t VE = 16 / sizeof(T);
  const bool wide = row_elems > 1 && ld_in % VE == 0 && ld_out % VE == 0 &&
                    ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15u) == 0;
  if (wide)
    gather_launch<T, uint4>(perm, n, row_elems, in, ld_in, out, ld_out, st);
  else
    gather_launch<T, T>(perm, n, row_elems, in, ld_in, out, ld_out, st);
}

template <typename T>
__global__ void scatter_kernel(const int32_t* __restrict__ perm, int64_t n, const T* __restrict__ in,
                               T* __restrict__ out) {
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n) out[perm[i]] = in[i];
}

}  // namespace

size_t radix_scratch_bytes(int64_t n) {
  const int64_t ntiles = ceil_div(n > 0 ? n : 1, kRsTile);
  const int64_t counts = kBins * ntiles;
  return static_cast<size_t>(counts + static_cast<int64_t>(scan_scratch_elems(counts))) * sizeof(int32_t);
}

maxe_status radix_sort_pairs(uint64_t* keys, int32_t* vals, uint64_t* keys_alt, int32_t* vals_alt, int64_t n,
                             int bits, void* scratch, cudaStream_t st) {
  if (n <= 1 || bits <= 0) return MAXE_OK;
  const int64_t ntiles = ceil_div(n, kRsTile);
  int32_t* counts = static_cast<int32_t*>(scratch);
  int32_t* scan_tmp = counts + kBins * ntiles;
  const int passes = (bits + 7) / 8;
  uint64_t* kin = keys;
  int32_t* vin = vals;
  uint64_t* kout = keys_alt;
  int32_t* vout = vals_alt;
  for (int p = 0; p < passes; ++p) {
    const int shift = 8 * p;
    rs_upsweep<<<static_cast<unsigned>(ntiles), kRsThreads, 0, st>>>(kin, n, shift, counts, ntiles);
    MAXE_TRY(scan_exclusive_i32(counts, counts, kBins * ntiles, nullptr, scan_tmp, st));
    rs_scatter<<<static_cast<unsigned>(ntiles), kRsThreads, 0, st>>>(kin, vin, kout, vout, n, shift, counts,
                                                                      ntiles);
    MAXE_CUDA_TRY(cudaGetLastError());
    uint64_t* tk = kin;
    kin = kout;
    kout = tk;
    int32_t* tv = vin;
    vin = vout;
    vout = tv;
  }
  if (kin != keys) {  // odd number of passes: bring the result home
    MAXE_CUDA_TRY(cudaMemcpyAsync(keys, kin, n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, st));
    MAXE_CUDA_TRY(cudaMemcpyAsync(vals, vin, n * sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
  }
  return MAXE_OK;
}

size_t perm_order_scratch_bytes(int64_t n) {
  if (n <= kPoSmallCap) return 0;
  return (static_cast<size_t>(n) + (size_t(1) << po_bits(n, po_mean(n))) + 1) * sizeof(int32_t);
}

maxe_status perm_order(uint64_t seed, int32_t tag, int32_t first, int32_t n, int32_t* out, void* scratch,
                       cudaStream_t st) {
  if (n <= 0) return MAXE_OK;
  PermOrder o{seed, tag, first, n, 0};
  constexpr size_t small_smem = sizeof(PoSmem<kPoSmallCap>), large_smem = sizeof(PoSmem<kPoLargeCap>);
  static_assert(small_smem <= 48 * 1024, "no opt-in for the small tile");
  if (n <= kPoSmallCap) {  // one bucket: one launch
    po_order<kPoSmallCap, 256><<<1, 256, small_smem, st>>>(o, nullptr, nullptr, out);
    MAXE_CUDA_TRY(cudaGetLastError());
    return MAXE_OK;
  }
  o.bits = po_bits(n, po_mean(n));
  const unsigned B = 1u << o.bits;
  int32_t* idx = static_cast<int32_t*>(scratch);
  uint32_t* cnt = reinterpret_cast<uint32_t*>(idx + n);
  const unsigned tiles = static_cast<unsigned>(ceil_div(n, kPoTile));
  MAXE_CUDA_TRY(cudaMemsetAsync(cnt, 0, (static_cast<size_t>(B) + 1) * sizeof(uint32_t), st));
  po_count<<<tiles, kPoThreads, 0, st>>>(o, cnt);
  po_split<<<tiles, kPoThreads, 0, st>>>(o, cnt, idx);
  if (po_mean(n) == kPoSmallCap / 2) {
    po_order<kPoSmallCap, 256><<<B, 256, small_smem, st>>>(o, idx, cnt, out);
  } else {
    static PerDeviceOnce once;
    MAXE_TRY(once.run([] {
      MAXE_CUDA_TRY(cudaFuncSetAttribute(po_order<kPoLargeCap, 1024>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(large_smem)));
      return MAXE_OK;
    }));
    po_order<kPoLargeCap, 1024><<<B, 1024, large_smem, st>>>(o, idx, cnt, out);
  }
  MAXE_CUDA_TRY(cudaGetLastError());
  return MAXE_OK;
}

maxe_status launch_invert(const int32_t* perm, int32_t n, int32_t* inv, cudaStream_t st) {
  if (n <= 0) return MAXE_OK;
  invert_kernel<<<static_cast<unsigned>(ceil_div(n, 256)), 256, 0, st>>>(perm, n, inv);
  MAXE_CUDA_TRY(cudaGetLastError());
  return MAXE_OK;
}

maxe_status launch_gather(const int32_t* perm, int64_t n, int elem_bytes, int64_t row_elems, const void* in,
                          int64_t ld_in, void* out, int64_t ld_out, cudaStream_t st) {
  if (n <= 0 || row_elems <= 0) return MAXE_OK;
  switch (elem_bytes) {
    case 2: gather_any<uint16_t>(perm, n, row_elems, in, ld_in, out, ld_out, st); break;
    case 4: gather_any<uint32_t>(perm, n, row_elems, in, ld_in, out, ld_out, st); break;
    case 8: gather_any<uint64_t>(perm, n, row_elems, in, ld_in, out, ld_out, st); break;
    default: return MAXE_ERR_INVALID;
  }
  MAXE_CUDA_TRY(cudaGetLastError());
  return MAXE_OK;
}

maxe_status launch_scatter(const int32_t* perm, int64_t n, int elem_bytes, const void* in, void* out,
                           cudaStream_t st) {
  if (n <= 0) return MAXE_OK;
  const unsigned grid = static_cast<unsigned>(ceil_div(n, 256));
  switch (elem_bytes) {
    case 2:
      scatter_kernel<uint16_t><<<grid, 256, 0, st>>>(perm, n, static_cast<const uint16_t*>(in),
                                                    static_cast<uint16_t*>(out));
      break;
    case 4:
      scatter_kernel<uint32_t><<<grid, 256, 0, st>>>(perm, n, static_cast<const uint32_t*>(in),
                                                    static_cast<uint32_t*>(out));
      break;
    case 8:
      scatter_kernel<uint64_t><<<grid, 256, 0, st>>>(perm, n, static_cast<const uint64_t*>(in),
                                                    static_cast<uint64_t*>(out));
      break;
    default:
      return MAXE_ERR_INVALID;
  }
  MAXE_CUDA_TRY(cudaGetLastError());
  return MAXE_OK;
}

}  // namespace maxe
