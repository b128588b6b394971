// spmm_rows.cu -- SpMM Y' = A' X' for matrices with short rows (Section 2's CSR
// product, k right-hand sides): one row per group of G lanes, single-matrix
// launch (the per-warp machinery is in spmm_rows.cuh).
//
// Each lane holds a piece of VC columns of X and Y (FP32: 16 bytes; FP64: one
// column, see RowsT), so a group of G lanes covers G * VC columns (more columns:
// more passes over the row).  A group walks its row's entries, gathers the piece of
// X row COL that is its lanes', accumulates in registers and writes its piece of
// Y once.
//
// The row's column indices come from shared memory, so that the gathers of X
// (the bytes that matter) are the only global loads a row waits for.  A warp
// works through its rows in chunks (at most kChunkR rows and kChunkE entries):
// while it multiplies chunk c, the column indices and values of chunk c + 1
// are on their way into the other half of its double buffer (16-byte cp.async
// copies, rounded out to 8-entry boundaries; the CSR arrays are padded past
// nnz) and the row pointers of chunk c + 2 into registers.  A row longer than
// kChunkE is a chunk of its own; its entries past the staged ones are read
// from global memory.
//
// Entries go four (16-byte pieces) or eight at a time, their X loads issued
// together, into four partial sums (entry j of a row: sum j % 4) added in a fixed
// order at the end: shorter dependency chains and a rounding error that grows
// with a quarter of the row's length.  The work is cut into parts of about
// kPartE entries (the handle's nnz-balanced row ranges, each split into Q
// parts of equal row counts); one resident wave of persistent warps takes them
// in turn (warp g: parts g, g + NG, ...), its chunk pipeline running on from
// part to part.  Neighbouring warps hold neighbouring parts, so the rows in
// flight at any time form one window of the matrix and the X rows that nearby
// rows share (a stencil's) are still in L2 when the second one needs them.
// Rows are never split, so each Y row is one group's sum in entry order:
// deterministic, but a long row holds its group (and its warp) -- the autotuner
// keeps this path only for matrices where it is faster.  Requires 16-byte
// aligned column and value arrays and rows of X under 2 GiB.
//
// FP32 rows of X or Y that are not whole 16-byte pieces (an odd k in contiguous
// tensors) take a variant whose lanes load 16, 8 or 4 bytes, as X's alignment
// allows, with up to 32 lanes to a row, and store Y column by column: an X row is
// still read by one load of the group.  Poisson rows of 20, 100,003 rows, FP32, k = 7
// contiguous: 59 us in seven column passes, 19 us here (k = 31: 237 -> 36 us; FP64,
// k = 7: 132 -> 58 us).
#include "launch.cuh"
#include "spmm_rows.cuh"

namespace maxe {
namespace {

using namespace rows;

constexpr int kRowsWarps = 8;
constexpr int kRowsThreads = 32 * kRowsWarps;
constexpr int64_t kPartE = 512;  // entries of a part (a warp's unit of work), about

struct RowsParams {
  RowsOperand op;
  const int32_t* wrow;
  int32_t nW, Q;
  bool once;   // the kernel's ONCE
  int32_t G;   // lanes per row, where the kernel has none of its own
  int64_t NG;  // warps of the grid: warp g takes parts g, g + NG, g + 2 NG, ...
};

// Rows [*lo, *hi) of part P: range P / Q of the warp partition, cut into Q
// parts of equal row counts.
__device__ __forceinline__ void part_rows(const RowsParams& p, int64_t P, int32_t* lo, int32_t* hi) {
  const int32_t w = static_cast<int32_t>(P / p.Q), q = static_cast<int32_t>(P % p.Q);
  const int32_t a = __ldg(p.wrow + w), bw = __ldg(p.wrow + w + 1);
  const int64_t len = bw - a;
  *lo = a + static_cast<int32_t>(len * q / p.Q);
  *hi = a + static_cast<int32_t>(len * (q + 1) / p.Q);
}

// The first chunk start at or after row r of part *P (rows up to *b): row r
// itself while r < *b, else the first row of the warp's next non-empty part.
// False when the warp has no parts left.
__device__ __forceinline__ bool next_start(const RowsParams& p, int32_t* r, int64_t* P, int32_t* b) {
  const int64_t NP = static_cast<int64_t>(p.nW) * p.Q;
  while (*r >= *b) {
    *P += p.NG;
    if (*P >= NP) return false;
    part_rows(p, *P, r, b);
  }
  return true;
}

// CTAs per SM the registers are cut for: FP64 sums take twice the registers.
template <typename AT>
constexpr int rows_blocks() {
  return sizeof(AT) == 8 ? 3 : 4;
}

// The matrix leaves L2 first (ONCE), so that X stays, where the product does not fit in
// L2.  Columns permuted, so that X rows are gathered at random: 2048 x 2048 Laplacian,
// without and with it, FP32 k = 4 151 and 136 us, k = 8 262 and 251, k = 16 392 and 386;
// BF16 k = 4 122 and 113, k = 16 406 and 402; FP64 k = 2 217 and 200, k = 4 394 and 387,
// k = 8 690 and 690, k = 12 1257 and 1263: hence X rows of up to 64 bytes.  In natural
// order, FP32: k = 4 71.2 and 73.0, k = 8 107 and 108, k = 12 177 and 172, k = 16 189.5
// and 186.8, k = 32 376 and 372: hence rows of more than 32 bytes, unless the prefetch
// was kept, which gains as much.  FP32 rows that are not 16-byte
// pieces go without: they were not timed with it.
constexpr int64_t kOnceRandomMax = 64;
constexpr int64_t kOnceOrderedMin = 32;

// GC: lanes per row (0: p.G, a power of two; a constant is worth 10% on rows of
// 40); VC, YVEC: see rows_chunk; ONCE: above.
template <typename VT, int GC, int VC, bool YVEC, bool ONCE>
__global__ void __launch_bounds__(kRowsThreads, rows_blocks<typename RowsT<VT>::AT>())
    spmm_rows_kernel(const RowsParams p) {
  extern __shared__ __align__(16) unsigned char rows_smem[];
  after_previous();
  const int G = GC ? GC : p.G;
  const int lane = threadIdx.x & 31, sub = lane % G, grp = lane / G;
  RowsStage<VT>* s = reinterpret_cast<RowsStage<VT>*>(rows_smem) + (threadIdx.x >> 5);
  // The warp's chunks, part after part, as one sequence: chunk i is multiplied
  // while the indices of chunk i + 1 load into the other buffer and the row
  // pointers of chunk i + 2 into registers.  Neighbouring warps take
  // neighbouring parts, so the rows in flight form one window of the matrix.
  int64_t P1 = (static_cast<int64_t>(blockIdx.x) * kRowsThreads + threadIdx.x) >> 5;
  if (P1 >= static_cast<int64_t>(p.nW) * p.Q) return;
  int32_t r1, b1;
  part_rows(p, P1, &r1, &b1);
  if (!next_start(p, &r1, &P1, &b1)) return;  // steps past an empty first part
  int32_t pa, pb;
  load_rp(p.op.rowptr, r1, b1, lane, &pa, &pb);
  int buf = 0;
  r1 += stage_chunk<VT, ONCE>(s, buf, p.op, r1, b1, lane, pa, pb);
  bool more = next_start(p, &r1, &P1, &b1);  // (r1, b1): the next chunk
  if (more) load_rp(p.op.rowptr, r1, b1, lane, &pa, &pb);
  while (true) {
    cp_async_wait_all();
    __syncwarp();
    int32_t r2 = r1, b2 = b1;
    int64_t P2 = P1;
    bool more2 = false;
    if (more) {  // stage the next chunk and fetch the row pointers of the one after
      r2 += stage_chunk<VT, ONCE>(s, buf ^ 1, p.op, r1, b1, lane, pa, pb);
      more2 = next_start(p, &r2, &P2, &b2);
      if (more2) load_rp(p.op.rowptr, r2, b2, lane, &pa, &pb);
    }
    rows_chunk<VT, VC, YVEC>(s, buf, p.op, G, 32 / G, grp, sub);
    __syncwarp();
    if (!more) break;
    r1 = r2;
    b1 = b2;
    P1 = P2;
    more = more2;
    buf ^= 1;
  }
}

template <typename VT, int G, int VC = RowsT<VT>::VC, bool YVEC = true, bool ONCE = false>
maxe_status launch_rows_g(RowsParams p, int sms, cudaStream_t st) {
  if constexpr (!ONCE && (YVEC || sizeof(VT) == 8))
    if (p.once) return launch_rows_g<VT, G, VC, YVEC, true>(p, sms, st);
  static PerDeviceOnce once;
  static int blocks_per_sm[64];
  constexpr size_t smem = sizeof(RowsStage<VT>) * kRowsWarps;
  int dev = 0;
  MAXE_CUDA_TRY(cudaGetDevice(&dev));
  MAXE_TRY(once.run([dev] {
    MAXE_CUDA_TRY(cudaFuncSetAttribute(spmm_rows_kernel<VT, G, VC, YVEC, ONCE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem)));
    int b = 0;
    MAXE_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, spmm_rows_kernel<VT, G, VC, YVEC, ONCE>, kRowsThreads, smem));
    blocks_per_sm[dev] = std::max(b, 1);
    return MAXE_OK;
  }));
  // one resident wave of persistent warps
  const int64_t parts = static_cast<int64_t>(p.nW) * p.Q;
  p.NG = std::max<int64_t>(1, std::min<int64_t>(parts, static_cast<int64_t>(sms) * blocks_per_sm[dev] * kRowsWarps));
  const unsigned grid = static_cast<unsigned>(ceil_div(p.NG, kRowsWarps));
  MAXE_CUDA_TRY(launch_after(spmm_rows_kernel<VT, G, VC, YVEC, ONCE>, grid, kRowsThreads, smem, st, p));
  return MAXE_OK;
}

template <typename VT>
maxe_status launch_rows(RowsParams p, int sms, cudaStream_t st) {
  using AT = typename RowsT<VT>::AT;
  constexpr int VC = RowsT<VT>::VC;
  // columns per load that FP32 rows of X allow: 16 bytes, 8 or one column
  auto whole = [](const void* q, int64_t ld, int vc) {
    return ld % vc == 0 && reinterpret_cast<uintptr_t>(q) % (vc * sizeof(AT)) == 0;
  };
  if constexpr (VC == 1) {  // FP64: see RowsT
    switch (rows_lanes(p.op.k)) {
      case 1: return launch_rows_g<VT, 1, 1, false>(p, sms, st);
      case 2: return launch_rows_g<VT, 2, 1, false>(p, sms, st);
      case 4: return launch_rows_g<VT, 4, 1, false>(p, sms, st);
      case 8: return launch_rows_g<VT, 8, 1, false>(p, sms, st);
      case 16: return launch_rows_g<VT, 16, 1, false>(p, sms, st);
      default: return launch_rows_g<VT, 32, 1, false>(p, sms, st);
    }
  } else {
    if (whole(p.op.X, p.op.ldx, VC) && whole(p.op.Y, p.op.ldy, VC)) {
      switch (rows_lanes((p.op.k + VC - 1) / VC)) {
        case 1: return launch_rows_g<VT, 1>(p, sms, st);
        case 2: return launch_rows_g<VT, 2>(p, sms, st);
        case 4: return launch_rows_g<VT, 4>(p, sms, st);
        case 8: return launch_rows_g<VT, 8>(p, sms, st);
        default: return launch_rows_g<VT, 16>(p, sms, st);
      }
    }
    const int vc = whole(p.op.X, p.op.ldx, 4) ? 4 : (whole(p.op.X, p.op.ldx, 2) ? 2 : 1);
    p.G = rows_lanes((p.op.k + vc - 1) / vc);
    if (vc == 4) return launch_rows_g<VT, 0, 4, false>(p, sms, st);
    if (vc == 2) return launch_rows_g<VT, 0, 2, false>(p, sms, st);
    return launch_rows_g<VT, 0, 1, false>(p, sms, st);
  }
}

}  // namespace

bool spmm_rows_any(const maxe_handle* h, int64_t ldx) {
  const int64_t eb = h->dtype == MAXE_F64 ? 8 : 4;
  return ldx * eb < (int64_t(1) << 31) &&
         ((reinterpret_cast<uintptr_t>(h->col) | reinterpret_cast<uintptr_t>(h->val)) & 15u) == 0;
}

bool spmm_rows_ready(const maxe_handle* h, int32_t k, const void* X, int64_t ldx, const void* Y, int64_t ldy) {
  const int vc = h->dtype == MAXE_F64 ? 2 : 4;
  auto a16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15u) == 0; };
  return k >= 1 && ldx % vc == 0 && ldy % vc == 0 && a16(X) && a16(Y) && spmm_rows_any(h, ldx);
}

maxe_status spmm_rows_launch(const maxe_handle* h, int32_t k, const void* X, int64_t ldx, void* Y, int64_t ldy,
                             const int32_t* yperm, cudaStream_t st) {
  if (h->rows == 0 || k == 0) return MAXE_OK;
  RowsParams p{};
  p.op.rowptr = h->rowptr;
  p.op.col = h->col;
  p.op.val = h->val;
  p.op.X = X;
  p.op.Y = Y;
  p.op.yperm = yperm;
  p.op.ldx = ldx;
  p.op.ldy = ldy;
  p.op.k = k;
  // The autotuner's pick acts from k = 16 on, where it was timed: narrower rows lose by
  // it (natural 2048 x 2048 Laplacian, FP32, k = 8: 114 us with, 110 without; permuted
  // 4096 x 4096, FP64, k = 4: 2750 and 1932 us).  A caller's own flag acts on any k.
  p.op.pf = h->spmm_rows_pf == 2 || (h->spmm_rows_pf == 1 && k >= 16);
  const int64_t xrow = k * vector_bytes(h->dtype);
  p.once = (h->cperm ? xrow <= kOnceRandomMax : xrow > kOnceOrderedMin && !h->spmm_rows_pf) && beyond_l2(h, k);
  p.wrow = h->wrow[0];
  p.nW = h->nW[0];
  // parts of about kPartE entries: a warp's range cut into Q parts of equal row counts
  const int64_t per_range = ceil_div(std::max<int64_t>(h->nnz, 1), std::max(p.nW, 1));
  p.Q = static_cast<int32_t>(std::max<int64_t>(1, ceil_div(per_range, kPartE)));
  const int sms = std::max(h->sms, 1);
  switch (h->dtype) {
    case MAXE_F64: return launch_rows<double>(p, sms, st);
    case MAXE_F32: return launch_rows<float>(p, sms, st);
    case MAXE_BF16: return launch_rows<uint16_t>(p, sms, st);
  }
  return MAXE_ERR_INVALID;
}

}  // namespace maxe
