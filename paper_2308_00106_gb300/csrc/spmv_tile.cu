// spmv_tile.cu -- SpMV for matrices with short rows: y' = A' x' (Section 2's
// CSR product) with the gathered x of a tile staged in shared memory.  Staging a
// block of whole rows entry by entry and summing the rows from there is the
// CSR-stream idea (Greathouse and Daga, SC 2014).
//
// The warp kernel of spmv.cu sums rows by a segmented scan over its entries
// and reads every row end back from it: about a quarter of a millisecond of
// instructions on a matrix of 84M entries with rows of five, whatever the
// gathers cost.  Here a CTA takes a tile of whole rows (those that START in
// [b*H, (b+1)*H)), all entries of it at once:
//   1. every thread loads column indices (16 bytes a load), gathers
//      x[column] for all of them with nothing in between, and stores the
//      gathered values in entry order; the matrix values go to shared memory
//      by 16-byte cp.async;
//   2. a group of G lanes per row sums a * x from shared memory with FMAs (two
//      running sums a lane, a fixed tree over the group), and writes y once.
// No scan, no search; several CTAs per SM, so one tile's gathers overlap
// another's sums.  A row longer than 32 G entries is summed by its whole
// warp; what reaches past the staged entries (only a tile's last row can) is
// summed by the whole CTA from global memory.  The order of every sum depends
// on the row and on G alone: deterministic.
//
// Random gathers are bound by the L1 tag stage, one line a cycle and SM (292
// G/s; 240 G/s reached while x stays in L2).  Permuted Laplacian, FP32, warp
// kernel -> tiles: 4096 x 4096 646 -> 372 us (x of 67 MB no longer fits in L2
// beside the stream), 2048 x 2048 97 -> 89 us; natural order, x in L1: 4096 x
// 4096 215 -> 150 us, FP64 464 -> 268 us.  With longer rows (Poisson, 15 to 50
// a row) the two are even, and the x-sliced form is faster where it applies, so the
// autotuner times all and takes the tiles where they are 5% faster; a handle that
// was not tuned keeps the warp kernel.
#include <algorithm>

#include "handle.cuh"
#include "launch.cuh"

namespace maxe {
namespace {

constexpr int kTileThreads = 256;
constexpr int kTileItems = 8;                            // entries per thread
constexpr int kTileCap = kTileThreads * kTileItems;      // staged entries
constexpr int kTileEntries = kTileCap - 64;              // starts of rows per tile: most tiles fit with their last row
constexpr int kTileMinEntries = 256;
constexpr int kTileWarps = kTileThreads / 32;

template <typename VT>
struct TileT;
template <>
struct TileT<double> {
  using AT = double;
  static __device__ __forceinline__ double acc(double v) { return v; }
};
template <>
struct TileT<float> {
  using AT = float;
  static __device__ __forceinline__ float acc(float v) { return v; }
};
template <>
struct TileT<uint16_t> {
  using AT = float;
  static __device__ __forceinline__ float acc(uint16_t v) { return __uint_as_float(static_cast<uint32_t>(v) << 16); }
};

struct TileParams {
  const int32_t* rowptr;
  const int32_t* col;
  const void* val;
  const int2* tile;  // [tiles + 1]: first row, its first entry
  const void* x;
  void* y;
  const int32_t* yperm;
  int shift;  // log2 of G, lanes per row
};

// Loads of a product that does not fit in L2 (BIG): the matrix, its row pointers
// and y pass through as the first to go, x is what should stay.  One that fits is
// read again by the next product and keeps plain loads (4096 x 4096 permuted
// Laplacian, FP32: 424 us plain, 380 us so; 1000 x 1000: 25 us plain, 27 us so,
// FP64 44 and 54 us).
struct TilePolicy {
  uint64_t once, keep;
};
__device__ __forceinline__ TilePolicy tile_policy() {
  TilePolicy p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p.once));
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p.keep));
  return p;
}

template <bool BIG>
__device__ __forceinline__ void tile_cp16(void* dst, const void* src, const TilePolicy& pol) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  if constexpr (BIG)
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "l"(pol.once)
                 : "memory");
  else
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
template <bool BIG>
__device__ __forceinline__ int4 tile_cols(const int32_t* p, const TilePolicy& pol) {
  if constexpr (!BIG) return __ldcs(reinterpret_cast<const int4*>(p));
  int4 v;
  asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.s32 {%0, %1, %2, %3}, [%4], %5;"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p), "l"(pol.once));
  return v;
}
template <bool BIG>
__device__ __forceinline__ int32_t tile_rowptr(const int32_t* p, const TilePolicy& pol) {
  if constexpr (!BIG) return __ldg(p);
  int32_t v;
  asm volatile("ld.global.nc.L2::cache_hint.s32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(pol.once));
  return v;
}
template <bool BIG>
__device__ __forceinline__ float tile_x(const float* p, const TilePolicy& pol) {
  if constexpr (!BIG) return *p;
  float v;
  asm volatile("ld.global.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(pol.keep));
  return v;
}
template <bool BIG>
__device__ __forceinline__ double tile_x(const double* p, const TilePolicy& pol) {
  if constexpr (!BIG) return *p;
  double v;
  asm volatile("ld.global.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(p), "l"(pol.keep));
  return v;
}

template <typename AT>
__device__ __forceinline__ void sts4(AT* p, const AT (&v)[4]) {
  if constexpr (sizeof(AT) == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
    reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
    reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
  }
}

// CTAs per SM a variant's registers are cut for.  Where x is gathered at random,
// all gathers of a thread should be in flight and no more CTAs than that takes
// (FP64 at six: 40 registers, two batches of gathers; permuted 3000 x 3000 Laplacian
// 760 us, at four 331 us).  Where x is found in L1, more CTAs hide more (natural
// 4096 x 4096, FP32: 172 us at six, 150 us at eight).  The autotuner times both.
template <typename VT, bool DENSE>
constexpr int tile_blocks() {
  return sizeof(VT) == 8 ? (DENSE ? 6 : 4) : (DENSE ? 8 : 6);
}

template <typename VT, bool BIG, bool DENSE>
__global__ void __launch_bounds__(kTileThreads, (tile_blocks<VT, DENSE>())) spmv_tile_kernel(const TileParams p) {
  using T = TileT<VT>;
  using AT = typename T::AT;
  __shared__ __align__(16) AT xs[kTileCap];
  __shared__ __align__(16) VT vs[kTileCap];
  __shared__ AT part[kTileWarps + 1];
  after_previous();
  const int t = threadIdx.x, lane = t & 31;
  const int2 lo = __ldg(p.tile + blockIdx.x), hi = __ldg(p.tile + blockIdx.x + 1);
  const uint32_t r0 = lo.x, r1 = hi.x;  // unsigned: a step past the last row cannot wrap
  const int64_t base = lo.y & ~7;  // 16-byte aligned for every value type
  const int32_t all = static_cast<int32_t>(hi.y - base);  // entries of the tile, counted from base
  const int32_t n = min(all, kTileCap);
  const AT* x = static_cast<const AT*>(p.x);

  // Whole 16-byte pieces: slots past n hold entries of later tiles or the
  // arrays' padding (columns within the matrix), and are not read back.
  const int32_t* col = p.col + base;
  const TilePolicy pol = BIG ? tile_policy() : TilePolicy{};
  int4 c[kTileItems / 4];
#pragma unroll
  for (int j = 0; j < kTileItems / 4; ++j) {
    const int s = 4 * (t + j * kTileThreads);
    if (s < n) c[j] = tile_cols<BIG>(col + s, pol);
  }
  constexpr int per = 16 / static_cast<int>(sizeof(VT));
  const VT* val = static_cast<const VT*>(p.val) + base;
#pragma unroll
  for (int j = 0; j < kTileItems / per; ++j) {
    const int s = per * (t + j * kTileThreads);
    if (s < n) tile_cp16<BIG>(vs + s, val + s, pol);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  AT xv[kTileItems / 4][4];
#pragma unroll
  for (int j = 0; j < kTileItems / 4; ++j) {
    if (4 * (t + j * kTileThreads) < n) {
      xv[j][0] = tile_x<BIG>(x + c[j].x, pol);
      xv[j][1] = tile_x<BIG>(x + c[j].y, pol);
      xv[j][2] = tile_x<BIG>(x + c[j].z, pol);
      xv[j][3] = tile_x<BIG>(x + c[j].w, pol);
    }
  }
  // the row pointers of the first rows come in under the gathers
  const int shift = p.shift, G = 1 << shift, rows = kTileThreads >> shift;
  const int sub = t & (G - 1);
  uint32_t rr = r0 + (t >> shift);
  int32_t s = 0, e = 0;
  if (rr < r1) {
    s = static_cast<int32_t>(tile_rowptr<BIG>(p.rowptr + rr, pol) - base);
    e = static_cast<int32_t>(tile_rowptr<BIG>(p.rowptr + rr + 1, pol) - base);
  }
#pragma unroll
  for (int j = 0; j < kTileItems / 4; ++j) {
    const int q = 4 * (t + j * kTileThreads);
    if (q < n) sts4(xs + q, xv[j]);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();

  AT* y = static_cast<AT*>(p.y);
  // trip count from the warp's first row: ballots and shuffles need whole warps
  for (uint32_t rb = r0 + ((t & ~31) >> shift); rb < r1; rb += rows) {
    const bool have = rr < r1;
    const int32_t em = min(e, n);  // staged entries of the row end here
    const bool wide = have && em - s > 32 * G;
    AT acc = AT(0), acc2 = AT(0);
    if (have && !wide) {
      int32_t q = s + sub;
      for (; q + G < em; q += 2 * G) {
        acc = fma(T::acc(vs[q]), xs[q], acc);
        acc2 = fma(T::acc(vs[q + G]), xs[q + G], acc2);
      }
      if (q < em) acc = fma(T::acc(vs[q]), xs[q], acc);
      acc += acc2;
    }
    for (int d = G >> 1; d > 0; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
    unsigned m = __ballot_sync(0xffffffffu, wide && sub == 0);
    while (m) {  // a long row by the whole warp
      const int src = __ffs(m) - 1;
      m &= m - 1;
      const int32_t ws = __shfl_sync(0xffffffffu, s, src), we = __shfl_sync(0xffffffffu, em, src);
      AT a = AT(0), b = AT(0);
      int32_t q = ws + lane;
      for (; q + 32 < we; q += 64) {
        a = fma(T::acc(vs[q]), xs[q], a);
        b = fma(T::acc(vs[q + 32]), xs[q + 32], b);
      }
      if (q < we) a = fma(T::acc(vs[q]), xs[q], a);
      a += b;
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) a += __shfl_xor_sync(0xffffffffu, a, d);
      if (lane == src) acc = a;
    }
    if (have && sub == 0) {
      if (e > n)
        part[kTileWarps] = acc;  // the tile's last row runs on past the staged entries
      else if (BIG && !p.yperm)  // (scattered y is put together in L2)
        __stcs(y + rr, acc);
      else
        y[p.yperm ? __ldg(p.yperm + rr) : rr] = acc;
    }
    rr += rows;
    if (rr < r1) {
      s = static_cast<int32_t>(tile_rowptr<BIG>(p.rowptr + rr, pol) - base);
      e = static_cast<int32_t>(tile_rowptr<BIG>(p.rowptr + rr + 1, pol) - base);
    }
  }
  if (all <= kTileCap) return;
  // entries [kTileCap, all) all belong to the last row: by the whole CTA
  AT a[4] = {AT(0), AT(0), AT(0), AT(0)};
  for (int64_t q = kTileCap + t; q < all; q += 4 * kTileThreads) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t w = q + u * kTileThreads;
      if (w < all) a[u] = fma(T::acc(val[w]), x[col[w]], a[u]);
    }
  }
  AT sum = (a[0] + a[1]) + (a[2] + a[3]);
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
  if (lane == 0) part[t >> 5] = sum;
  __syncthreads();
  if (t == 0) {
    sum = part[kTileWarps];
    for (int w = 0; w < kTileWarps; ++w) sum += part[w];
    const uint32_t r = r1 - 1;
    y[p.yperm ? __ldg(p.yperm + r) : r] = sum;
  }
}

// tile[b] = (first row of tile b, its first entry)
__global__ void tile_starts_kernel(const int32_t* __restrict__ first, const int32_t* __restrict__ rowptr, int32_t rows,
                                   int64_t tiles, int2* __restrict__ tile) {
  const int64_t b = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (b > tiles) return;
  const int32_t r = b < tiles ? first[b] : rows;
  tile[b] = make_int2(r, rowptr[r]);
}

template <typename VT, bool BIG>
maxe_status tile_launch(const TileParams& p, const maxe_handle* h, cudaStream_t st) {
  const unsigned grid = static_cast<unsigned>(h->tiles);
  MAXE_CUDA_TRY(h->tile_dense ? launch_after(spmv_tile_kernel<VT, BIG, true>, grid, kTileThreads, 0, st, p)
                              : launch_after(spmv_tile_kernel<VT, BIG, false>, grid, kTileThreads, 0, st, p));
  return MAXE_OK;
}

}  // namespace

maxe_status spmv_tile_build(maxe_handle* h, cudaStream_t st) {
  if (h->rows == 0 || h->nnz == 0) return MAXE_OK;
  // about eight tiles per SM on small matrices, so that all SMs have work
  const int64_t H = std::max<int64_t>(
      kTileMinEntries, std::min<int64_t>(kTileEntries, ceil_div(h->nnz, 8 * static_cast<int64_t>(std::max(h->sms, 1)))));
  const int64_t tiles = ceil_div(h->nnz, H);
  h->tile = static_cast<int2*>(h->al.get(static_cast<size_t>(tiles + 1) * sizeof(int2)));
  if (!h->tile) return MAXE_ERR_OOM;
  ScratchSet scratch(h->al);
  int32_t* first = scratch.get<int32_t>(static_cast<size_t>(tiles) + 1);
  if (!first) return MAXE_ERR_OOM;
  MAXE_TRY(bucket_lower_bounds(h->rowptr, h->rows, H, 0, tiles, first, st));
  tile_starts_kernel<<<static_cast<unsigned>(ceil_div(tiles + 1, 256)), 256, 0, st>>>(first, h->rowptr, h->rows, tiles,
                                                                                   h->tile);
  MAXE_CUDA_TRY(cudaGetLastError());
  h->tiles = tiles;
  // lanes per row: about six entries a lane
  const int64_t mean = h->nnz / h->rows;
  h->tile_shift = 0;
  while (h->tile_shift < 5 && (int64_t(8) << h->tile_shift) < mean) ++h->tile_shift;
  return MAXE_OK;
}

maxe_status spmv_tile_launch(const maxe_handle* h, const void* x, void* y, const int32_t* yperm, cudaStream_t st) {
  TileParams p{h->rowptr, h->col, h->val, h->tile, x, y, yperm, h->tile_shift};
  const bool big = beyond_l2(h, 1);
  switch (h->dtype) {
    case MAXE_F64: return big ? tile_launch<double, true>(p, h, st) : tile_launch<double, false>(p, h, st);
    case MAXE_F32: return big ? tile_launch<float, true>(p, h, st) : tile_launch<float, false>(p, h, st);
    case MAXE_BF16: return big ? tile_launch<uint16_t, true>(p, h, st) : tile_launch<uint16_t, false>(p, h, st);
  }
  return MAXE_ERR_INVALID;
}

}  // namespace maxe
