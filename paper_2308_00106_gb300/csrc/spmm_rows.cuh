// spmm_rows.cuh -- the per-warp machinery of SpMM with one CSR row per group
// of lanes (Section 2's CSR product, k right-hand sides), shared by the
// single-matrix kernel (spmm_rows.cu) and the batched one (batch.cu).
//
// A warp works through a range of rows in chunks (at most kChunkR rows and
// kChunkE entries): stage_chunk copies a chunk's column indices and values
// into one half of the warp's double buffer (16-byte cp.async copies rounded
// out to 8-entry boundaries; the CSR arrays are padded past nnz) and writes its
// row pointers; rows_chunk multiplies the rows of a staged chunk, a group of G
// lanes per row, each lane a piece of VC columns of the X and Y rows (4 FP32
// columns where rows are 16-byte aligned), gathering X pieces by the staged
// column indices and accumulating in registers.  Entries go four or eight at a
// time, their X loads issued together, into four partial sums (entry j of a row:
// sum j % 4) added in a fixed order, so a Y row is one group's sum in a fixed
// order: the same bits whichever warp, launch or batch computes it.  A row longer than
// kChunkE is a chunk of its own; its entries past the staged ones are read
// from global memory.
#pragma once

#include "handle.cuh"

namespace maxe {
namespace rows {

constexpr int kRowsAhead = 8;   // entries of the next row prefetched, per lane of the group
constexpr int kRowsParts = 4;   // partial sums of a group
constexpr int kChunkE = 256;    // entries of a chunk (a longer row: the first kChunkE)
constexpr int kChunkR = 63;     // rows of a chunk: its 64 row pointers are two per lane
constexpr int kSlotE = kChunkE + 8;  // staged slots: the chunk rounded out to 8-entry boundaries

template <typename VT>
struct RowsT;
template <>
struct RowsT<float> {
  using AT = float;
  static constexpr int VC = 4;  // columns a lane takes of 16-byte aligned rows
  static __device__ __forceinline__ float acc(float v) { return v; }
};
template <>
struct RowsT<uint16_t> {
  using AT = float;
  static constexpr int VC = 4;
  static __device__ __forceinline__ float acc(uint16_t v) { return __uint_as_float(static_cast<uint32_t>(v) << 16); }
};
template <>
struct RowsT<double> {
  using AT = double;
  // One column a lane whatever the alignment: twice the lanes a row, so half the
  // rows a warp, which costs fewer bank conflicts of the staged entries and less
  // waiting for the longest row than 16-byte loads save.  300,000 rows of 40, k = 4:
  // 352 -> 184 us, k = 16: 604 -> 436 us; permuted 2048 x 2048 Laplacian 534 -> 397
  // and 1300 -> 1250 us.
  static constexpr int VC = 1;
  static __device__ __forceinline__ double acc(double v) { return v; }
};

// A lane's piece of VC columns.
template <typename AT, int VC>
struct RowsPiece;
template <>
struct RowsPiece<float, 4> {
  using V = float4;
};
template <>
struct RowsPiece<float, 2> {
  using V = float2;
};
template <>
struct RowsPiece<float, 1> {
  using V = float;
};
template <>
struct RowsPiece<double, 1> {
  using V = double;
};

__device__ __forceinline__ void fma_vec(float4& acc, float a, const float4& x) {
  acc.x = fmaf(a, x.x, acc.x);
  acc.y = fmaf(a, x.y, acc.y);
  acc.z = fmaf(a, x.z, acc.z);
  acc.w = fmaf(a, x.w, acc.w);
}
__device__ __forceinline__ void fma_vec(float2& acc, float a, const float2& x) {
  acc.x = fmaf(a, x.x, acc.x);
  acc.y = fmaf(a, x.y, acc.y);
}
__device__ __forceinline__ void fma_vec(float& acc, float a, float x) { acc = fmaf(a, x, acc); }
__device__ __forceinline__ void fma_vec(double& acc, double a, double x) { acc = fma(a, x, acc); }
__device__ __forceinline__ void add_vec(float4& a, const float4& b) {
  a.x += b.x;
  a.y += b.y;
  a.z += b.z;
  a.w += b.w;
}
__device__ __forceinline__ void add_vec(float2& a, const float2& b) {
  a.x += b.x;
  a.y += b.y;
}
__device__ __forceinline__ void add_vec(float& a, float b) { a += b; }
__device__ __forceinline__ void add_vec(double& a, double b) { a += b; }
// Y piece of a row: all VC columns, or the first `left` of them (the row's last piece)
__device__ __forceinline__ void store_piece(float4* y, const float4& v, int left) {
  if (left >= 4) {
    *y = v;
    return;
  }
  float* f = reinterpret_cast<float*>(y);
  f[0] = v.x;
  if (left > 1) f[1] = v.y;
  if (left > 2) f[2] = v.z;
}
// Y rows that are not 16-byte aligned: column by column
template <typename AT, typename V>
__device__ __forceinline__ void store_columns(AT* y, const V& v, int left) {
  const AT* f = reinterpret_cast<const AT*>(&v);
#pragma unroll
  for (int c = 0; c < static_cast<int>(sizeof(V) / sizeof(AT)); ++c)
    if (c < left) y[c] = f[c];
}
__device__ __forceinline__ void zero(float2& v) { v = make_float2(0.f, 0.f); }
__device__ __forceinline__ void zero(float& v) { v = 0.f; }
__device__ __forceinline__ void zero(double& v) { v = 0.0; }
__device__ __forceinline__ void zero(float4& v) { v = make_float4(0.f, 0.f, 0.f, 0.f); }

// ONCE: the bytes are the first to leave L2.
template <bool ONCE>
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  if constexpr (ONCE) {
    uint64_t pol;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "l"(pol)
                 : "memory");
  } else {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
  }
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// One warp's double buffer: column indices, values and row pointers (slots
// relative to e0a) and extents of two chunks.
template <typename VT>
struct alignas(16) RowsStage {
  int32_t col[2][kSlotE];
  VT val[2][kSlotE];
  int32_t rp[2][kChunkR + 1];
  int64_t e0a[2];  // the chunk's first staged entry (a multiple of 8)
  int32_t r[2];    // its first row
  int32_t n[2];    // its rows
  int32_t lim[2];  // end of its staged slots: rows reaching past it are long rows
};

// The product a warp works on: Y' = A' X' with A' in CSR.
struct RowsOperand {
  const int32_t* rowptr;
  const int32_t* col;
  const void* val;
  const void* X;
  void* Y;
  const int32_t* yperm;  // Y row of row r: yperm[r] (null: r)
  int64_t ldx, ldy;
  int32_t k;
  int32_t pf;  // 1: prefetch the X rows of a group's next row into L2 (stencil-like matrices)
};

// Row pointers rowptr[r + j], j = 0 .. min(kChunkR, b - r): j = lane in *pa,
// j = 32 + lane in *pb; INT32_MAX past the warp's rows.
__device__ __forceinline__ void load_rp(const int32_t* rowptr, int32_t r, int32_t b, int lane, int32_t* pa,
                                        int32_t* pb) {
  const int32_t lim = min(kChunkR, b - r);
  *pa = lane <= lim ? __ldg(rowptr + r + lane) : INT32_MAX;
  *pb = 32 + lane <= lim ? __ldg(rowptr + r + 32 + lane) : INT32_MAX;
}

// Cuts the chunk that starts at row r (its row pointers in pa / pb): the most
// rows, up to kChunkR, whose entries fit in kChunkE, at least one row.  Stages
// its column indices and values into buffer `buf` (cp.async, committed) and
// writes its row pointers and extent; returns its row count.  Warp-uniform; all
// 32 lanes take part.
template <typename VT, bool ONCE = false>
__device__ __forceinline__ int32_t stage_chunk(RowsStage<VT>* s, int buf, const RowsOperand& p, int32_t r, int32_t b,
                                               int lane, int32_t pa, int32_t pb) {
  const int32_t rows = min(kChunkR, b - r);
  const int32_t E0 = __shfl_sync(0xffffffffu, pa, 0);
  const bool oka = lane >= 1 && lane <= rows && pa - E0 <= kChunkE;
  const bool okb = 32 + lane <= rows && pb - E0 <= kChunkE;
  int32_t n = __popc(__ballot_sync(0xffffffffu, oka)) + __popc(__ballot_sync(0xffffffffu, okb));
  n = max(n, 1);
  const int32_t ea = __shfl_sync(0xffffffffu, pa, n & 31), eb = __shfl_sync(0xffffffffu, pb, n & 31);
  const int32_t E1 = n < 32 ? ea : eb;
  const int64_t e0a = static_cast<int64_t>(E0) & ~int64_t(7);
  const int32_t lim = static_cast<int32_t>(std::min<int64_t>(E1, static_cast<int64_t>(E0) + kChunkE) - e0a);
  const int32_t slots = (lim + 7) & ~7;  // <= kSlotE
  const int32_t* gcol = p.col + e0a;
  for (int i = lane; i < slots / 4; i += 32) cp_async16<ONCE>(&s->col[buf][4 * i], gcol + 4 * i);
  constexpr int per = 16 / static_cast<int>(sizeof(VT));
  const VT* gval = static_cast<const VT*>(p.val) + e0a;
  for (int i = lane; i < slots / per; i += 32) cp_async16<ONCE>(&s->val[buf][per * i], gval + per * i);
  cp_async_commit();
  const int32_t base = static_cast<int32_t>(static_cast<int64_t>(E0) - e0a);
  if (lane <= n) s->rp[buf][lane] = pa - E0 + base;
  if (32 + lane <= n) s->rp[buf][32 + lane] = pb - E0 + base;
  if (lane == 0) {
    s->e0a[buf] = e0a;
    s->r[buf] = r;
    s->n[buf] = n;
    s->lim[buf] = lim;
  }
  return n;
}

// U entries of a row from t on (PRED: only the first `left` of them), their X
// loads issued together: entry u goes to partial sum u % kRowsParts.  COL and VAL:
// the row's column indices and values, in shared or global memory.
template <typename VT, int VC, int U, bool PRED>
__device__ __forceinline__ void rows_step(typename RowsPiece<typename RowsT<VT>::AT, VC>::V (&part)[kRowsParts],
                                          const int32_t* col, const VT* val, int left, const char* xc,
                                          int32_t ldx_bytes) {
  using T = RowsT<VT>;
  using AT = typename T::AT;
  using V = typename RowsPiece<AT, VC>::V;
  V xv[U];
  AT av[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (PRED) {
      av[u] = AT(0);
      zero(xv[u]);
    }
    if (!PRED || u < left) {
      // X piece of row COL: xc + COL * ldx_bytes (one wide multiply-add per entry)
      xv[u] = __ldg(reinterpret_cast<const V*>(xc + static_cast<int64_t>(col[u]) * static_cast<int64_t>(ldx_bytes)));
      av[u] = T::acc(val[u]);
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) fma_vec(part[u % kRowsParts], av[u], xv[u]);
}

// Entries of a row, n of them: whole steps of U entries without predicates, then
// one of kRowsParts, then a predicated rest.  Every step starts at a multiple of
// kRowsParts, so entry j of the row is in partial sum j % kRowsParts whatever U.
template <typename VT, int VC, int U>
__device__ __forceinline__ void rows_entries(typename RowsPiece<typename RowsT<VT>::AT, VC>::V (&part)[kRowsParts],
                                             const int32_t* col, const VT* val, int32_t n, const char* xc,
                                             int32_t ldx_bytes) {
  static_assert(U % kRowsParts == 0, "steps keep the entries' partial sums");
  int32_t t = 0;
#pragma unroll 1
  for (; t + U <= n; t += U) rows_step<VT, VC, U, false>(part, col + t, val + t, U, xc, ldx_bytes);
  if (U > kRowsParts && t + kRowsParts <= n) {
    rows_step<VT, VC, kRowsParts, false>(part, col + t, val + t, kRowsParts, xc, ldx_bytes);
    t += kRowsParts;
  }
  if (t < n) rows_step<VT, VC, kRowsParts - 1, true>(part, col + t, val + t, n - t, xc, ldx_bytes);
}

// Entries per whole step: as many as keep their X pieces in registers.  Eight
// 16-byte pieces do not fit beside the rest in 64 registers: the compiler then
// loads them one after the other (BF16 values: 175 us against 105 with four, on
// 300,000 rows of 40, k = 16).
template <typename AT, int VC>
constexpr int rows_unroll() {
  return sizeof(AT) * VC >= 16 ? 4 : 8;
}

// Multiplies the rows of chunk buffer `buf` and writes their Y pieces: lane
// `sub` of group `grp` (G lanes per group, GPW = 32 / G groups per warp), each
// lane VC columns.  YVEC: Y rows are 16-byte aligned and VC is a whole 16 bytes.
// A row's sum does not depend on VC, G or YVEC.
template <typename VT, int VC = RowsT<VT>::VC, bool YVEC = true>
__device__ __forceinline__ void rows_chunk(const RowsStage<VT>* s, int buf, const RowsOperand& p, int G, int GPW,
                                           int grp, int sub) {
  using T = RowsT<VT>;
  using AT = typename T::AT;
  using V = typename RowsPiece<AT, VC>::V;
  constexpr int U = rows_unroll<AT, VC>();
  const int32_t ldx_bytes = static_cast<int32_t>(p.ldx * static_cast<int64_t>(sizeof(AT)));  // < 2^31 (checked)
  const int kv = (p.k + VC - 1) / VC;
  const int32_t* scol = s->col[buf];
  const VT* sval = s->val[buf];
  const int32_t n = s->n[buf], lim = s->lim[buf];
  for (int j = grp; j < n; j += GPW) {
    const int32_t t0 = s->rp[buf][j], t1 = s->rp[buf][j + 1];
    const int32_t ts = min(t1, lim);  // staged entries of the row end here
    // the X rows of the group's next row into L2, one line each (when a row
    // spans several lanes: with one lane per row the prefetches cost more)
    if (p.pf && G > 1 && j + GPW < n) {
      const int32_t u0 = s->rp[buf][j + GPW], u1 = min(s->rp[buf][j + GPW + 1], lim);
      for (int32_t u = u0 + sub; u < u1 && u < u0 + kRowsAhead * G; u += G)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const char*>(p.X) +
                                                       static_cast<int64_t>(scol[u]) * static_cast<int64_t>(ldx_bytes)));
    }
    for (int c = sub; c < kv; c += G) {
      const char* xc = static_cast<const char*>(p.X) + static_cast<int>(sizeof(V)) * c;
      V part[kRowsParts];
#pragma unroll
      for (int u = 0; u < kRowsParts; ++u) zero(part[u]);
      rows_entries<VT, VC, U>(part, scol + t0, sval + t0, ts - t0, xc, ldx_bytes);
      // Past the staged part of a long row; it ends kChunkE entries into the
      // row, so the partial sums go on where they were.
      if (t1 > ts) {
        const int64_t e = s->e0a[buf] + ts;
        rows_entries<VT, VC, U>(part, p.col + e, static_cast<const VT*>(p.val) + e, t1 - ts, xc, ldx_bytes);
      }
      add_vec(part[0], part[1]);
      add_vec(part[2], part[3]);
      add_vec(part[0], part[2]);
      const int32_t row = s->r[buf] + j;
      const int64_t yr = p.yperm ? static_cast<int64_t>(__ldg(p.yperm + row)) : static_cast<int64_t>(row);
      if constexpr (YVEC)
        store_piece(reinterpret_cast<V*>(static_cast<AT*>(p.Y) + yr * p.ldy) + c, part[0], p.k - c * VC);
      else
        store_columns(static_cast<AT*>(p.Y) + yr * p.ldy + c * VC, part[0], p.k - c * VC);
    }
  }
}

// Lanes of a row with `pieces` pieces: a power of two, at most 32 (more pieces: passes).
__host__ __device__ __forceinline__ int rows_lanes(int pieces) {
  int g = 1;
  while (g < 32 && g < pieces) g *= 2;
  return g;
}

// Rows [r_lo, b) of the product by one warp: chunk c is multiplied while the
// indices of chunk c + 1 load into the other buffer and the row pointers of
// chunk c + 2 into registers.  Warp-uniform; all 32 lanes take part.
template <typename VT, int VC, bool YVEC, int GC>
__device__ __forceinline__ void rows_range(RowsStage<VT>* s, const RowsOperand& p, int32_t r_lo, int32_t b, int Gr,
                                           int lane) {
  if (r_lo >= b) return;
  const int G = GC ? GC : Gr;
  const int GPW = 32 / G, sub = lane % G, grp = lane / G;
  int32_t pa, pb;
  load_rp(p.rowptr, r_lo, b, lane, &pa, &pb);
  int buf = 0;
  int32_t r1 = r_lo + stage_chunk<VT>(s, buf, p, r_lo, b, lane, pa, pb);  // start of the next chunk
  if (r1 < b) load_rp(p.rowptr, r1, b, lane, &pa, &pb);
  while (true) {
    cp_async_wait_all();
    __syncwarp();
    int32_t r2 = b;
    if (r1 < b) {
      r2 = r1 + stage_chunk<VT>(s, buf ^ 1, p, r1, b, lane, pa, pb);
      if (r2 < b) load_rp(p.rowptr, r2, b, lane, &pa, &pb);
    }
    rows_chunk<VT, VC, YVEC>(s, buf, p, G, GPW, grp, sub);
    __syncwarp();
    if (r1 >= b) break;
    r1 = r2;
    buf ^= 1;
  }
}

}  // namespace rows
}  // namespace maxe
