// The four LM-head contractions of the BGPO ELBO path on sm_103a tensor cores.
//
// Each is a persistent, warp-specialised kernel launched as 2-CTA clusters. A
// CTA pair computes 256 x 256 fp32 tiles with tcgen05.mma.cta_group::2: CTA r
// of the pair stages rows [128 r, 128 r + 128) of the A tile and columns
// [128 r, 128 r + 128) of the B tile, and holds accumulator rows
// [128 r, 128 r + 128) in its TMEM. The dX GEMM's tiles are one or two such
// tiles side by side, sharing their A tile. Roles in each CTA (224 threads):
//   warps 0, 6  TMA producers of A and of B: 128-byte-swizzled bf16 boxes into a
//               6-stage ring of 32 KB (dX at two accumulators: 4 stages of 48
//               KB); every copy of both CTAs completes on the even CTA's
//               "full" barrier, which the even CTA alone arms with both CTAs'
//               transaction bytes (a negative transaction count in between is
//               allowed)
//   warp 1      TMEM allocation (pair, 512 columns = two accumulators); in the
//               even CTA also the MMA issuer (M = 256, N = 256, K = 16; the
//               dX GEMM issues one per accumulator of its tile)
//   warps 2-5   epilogue: tcgen05.ld of this CTA's accumulator rows, fused
//               per-kind epilogue, TMA stores / reductions from shared memory
// The epilogue of tile n overlaps the main loop of tile n+1, except in the dX
// GEMM when its tiles occupy both accumulators.
//
// Kinds (Xm = gathered masked hidden states [M, H], W = LM head [V, H]):
//   GEMM_FWD  z = Xm W^T; epilogue: online max / sum-exp per (row, vocab tile)
//             and the target logit (Eq. 4: log softmax gathered at y^i); when
//             the workspace has a logit region the fp32 tile also leaves
//             through TMA stores, for the backward.
//   GEMM_DZ   z = Xm W^T recomputed (when the forward kept no logits) for one
//             vocabulary chunk of the backward; epilogue: dz = w_r (onehot -
//             e^{z - lse}) stored as bf16 (gradient of Eq. 4 weighted by
//             Eq. 13's dL/dl).
//   GEMM_DX   dXm += dZ_c W_c (K = the chunk's vocabulary; 256 x 256 or 256 x 512 tiles): split-K partials in
//             fp32, stored by the first chunk and added by the later ones, or,
//             when the launch needs no split, added straight into the dX rows.
//   GEMM_DW   dW[chunk rows] += dZ_c^T Xm (K = masked rows; Xm read as its
//             transpose, so that the B operand is K-major), fp32 TMA
//             reduce-add. With dW pairing (whole-vocabulary dZ), K also covers
//             the rows of the pending sample before.
//
// Every wait is bounded (time and polls); a wait that runs out sets the
// workspace error word to BGPO_ERR_TIMEOUT and both CTAs drain and exit.
#include <math.h>

#include <mutex>

#include "bgpo_device.cuh"
#include "bgpo_internal.h"

namespace bgpo {

namespace {

constexpr float kLog2e = 1.4426950408889634f;
constexpr int32_t kStatusInvalidArg = 1;  // BGPO_ERR_INVALID_ARG
constexpr int32_t kStatusTimeout = 8;     // BGPO_ERR_TIMEOUT
constexpr int kThreads = 224;             // 7 warps
// The B producer. One thread issuing both operands' copies was busy for 375 cycles
// a K block (counted with clock64; a K block's MMAs take 512), more with dX's and
// dW's 64-column boxes. From two warps: 256-wide dX tiles 720 -> 585 cycles a K
// block (500 rows, H 512, V 38912: 35.3 -> 29.8 us), dW 1205 -> 1163 us at 1,679
// rows of the 4096 x 126464 head, forward and dZ as before.
constexpr int kWarpB = 6;
constexpr uint32_t kTmemCols = 2 * kBN;   // two accumulators
constexpr uint32_t kMnChunkBytes = 64 * 64 * 2;   // one 64 x 64 bf16 TMA box (MN-major)
constexpr uint16_t kBothCtas = 0x3;

struct GemmParams {
  Geometry g;
  int num_pairs;
  int32_t j;
  int64_t v_begin, v_end, dz_col0, chunk;
  WsPtrs w;
  const float* coef;
  float* dW;
  float* dX;
  bool pair_consume;
};

// (32 bits hold every count: at most 2^14 row blocks, 2^16 vocabulary tiles, 64
// hidden-size tiles, 2^18 K blocks)
struct Work {
  int32_t units, tiles_m, tiles_n, kb_total;
  int32_t kb_first;  // first K block (dW: a partner already added is skipped)
  int32_t groups;    // forward and dZ: row groups (xm_row_groups)
  int32_t splits;
  int32_t wide;      // accumulators per tile (dX: one or two)
  int32_t rows;      // A rows that hold data: CTAs and warps wholly past them skip theirs
};

struct Unit {
  int32_t m_blk, n_blk, split, kb0, kb_n;
};

// `roff`: the first dZ / Xm^T row of the sample (dW pairing; 0 otherwise). The
// dW GEMM's K range [k0, roff + M) then covers a pending sample's rows too when
// k0 = 0.
template <int KIND>
__device__ __forceinline__ Work make_work(const GemmParams& p, int32_t M, int64_t roff,
                                          int64_t k0) {
  Work w;
  w.splits = 1;
  w.wide = 1;
  w.kb_first = 0;
  w.groups = 1;
  w.rows = M;
  if (KIND == GEMM_FWD || KIND == GEMM_DZ) {
    w.tiles_m = (int32_t)ceil_div(M, kPairM);
    w.tiles_n = (int32_t)(KIND == GEMM_FWD ? p.g.n_vt : ceil_div(p.v_end - p.v_begin, kBN));
    // a last K block past H reads the tensor maps' zero fill
    w.kb_total = (int32_t)ceil_div(p.g.H, kBK);
    w.units = w.tiles_m * w.tiles_n;
    w.groups = (int32_t)xm_row_groups(w.tiles_m, p.g.H);
  } else if (KIND == GEMM_DX) {
    w.tiles_m = (int32_t)ceil_div(M, kPairM);
    w.kb_total = (int32_t)ceil_div(p.v_end - p.v_begin, kBK);
    // one plan for every chunk of the sample (the partials of split s
    // accumulate over the chunks), left by the kernel that transposed Xm
    bool fits;
    w.splits = dx_splits_stored(p.g, M, p.w.err[ERR_DX_SPLITS], &fits);
    w.wide = dx_wide_stored(p.w.err[ERR_DX_WIDE]);
    if (!fits && M > 0 && blockIdx.x == 0 && threadIdx.x == 0)
      set_device_error(p.w.err, kStatusInvalidArg, KID_DX_GEMM * 16 + 6);
    w.tiles_n = (int32_t)dx_tiles_n(p.g.tiles_h, w.wide);
    w.units = w.tiles_m * w.tiles_n * w.splits;
  } else {  // GEMM_DW
    w.tiles_m = (int32_t)ceil_div(p.v_end - p.v_begin, kPairM);
    w.tiles_n = (int32_t)p.g.tiles_h;
    w.kb_total = (int32_t)ceil_div(roff + M, kBK);
    w.kb_first = (int32_t)(k0 / kBK);
    w.units = w.kb_total > w.kb_first ? w.tiles_m * w.tiles_n : 0;
  }
  return w;
}

template <int KIND>
__device__ __forceinline__ Unit unit_of(const Work& w, int32_t u) {
  Unit t;
  t.split = 0;
  if (KIND == GEMM_FWD || KIND == GEMM_DZ) {
    // consecutive units share a vocabulary tile of W: it is read from HBM once
    // per row group
    int64_t m, n;
    row_group_tile(u, w.tiles_m, w.tiles_n, w.groups, &m, &n);
    t.m_blk = (int32_t)m;
    t.n_blk = (int32_t)n;
    t.kb0 = 0;
    t.kb_n = w.kb_total;
  } else if (KIND == GEMM_DX) {
    // consecutive units share a row block of dZ (measured 2% faster than
    // sharing a column block of W, and than grouped rasters)
    const uint32_t per_split = (uint32_t)(w.tiles_m * w.tiles_n);
    const uint32_t split = (uint32_t)u / per_split, rem = (uint32_t)u % per_split;
    t.split = (int32_t)split;
    t.m_blk = (int32_t)(rem / (uint32_t)w.tiles_n);
    t.n_blk = (int32_t)(rem % (uint32_t)w.tiles_n);
    const uint32_t k0 = split * (uint32_t)w.kb_total / (uint32_t)w.splits;
    const uint32_t k1 = (split + 1) * (uint32_t)w.kb_total / (uint32_t)w.splits;
    t.kb0 = (int32_t)k0;
    t.kb_n = (int32_t)(k1 - k0);
  } else {
    // consecutive units share a vocabulary block of dZ^T
    t.m_blk = (int32_t)((uint32_t)u / (uint32_t)w.tiles_n);
    t.n_blk = (int32_t)((uint32_t)u % (uint32_t)w.tiles_n);
    t.kb0 = w.kb_first;
    t.kb_n = w.kb_total - w.kb_first;
  }
  return t;
}

// Shared-memory plan of one kind: 6 pipeline stages (dX with two accumulators
// per tile: 4 larger ones in the same bytes) and the epilogue's staging buffers
// (the forward GEMM stages its fp32 logits there when it keeps them).
template <int KIND>
struct SmemPlan {
  static constexpr uint32_t epi_bytes = kEpiBytes;
  static constexpr uint32_t bytes = kStages * kStageBytes + epi_bytes + 1024 + 1024;
  static_assert(bytes <= 232448, "shared memory per CTA");
};

// Operand majorness: forward and dZ read Xm and W K-major; dX reads dZ K-major
// and W MN-major; dW reads dZ^T MN-major and Xm^T (a transposed copy) K-major.
// Four MN-major boxes per stage (dW on Xm itself) measured 12% slower.
template <int KIND>
struct Majors {
  static constexpr bool a_mn = (KIND == GEMM_DW);
  static constexpr bool b_mn = (KIND == GEMM_DX);
};

// Rows of the K-major B operand (W for forward and dZ, Xm^T for dW).
template <int KIND>
__device__ __forceinline__ int64_t b_rows(const GemmParams& p) {
  return KIND == GEMM_DW ? p.g.H : p.g.V;
}

// First row of the K-major B operand in this launch: dZ's W rows start at the
// chunk's first vocabulary entry.
template <int KIND>
__device__ __forceinline__ int64_t b_base(const GemmParams& p) {
  return KIND == GEMM_DZ ? p.v_begin : 0;
}

// Whether this CTA loads its 128 rows of a K-major A tile: when they hold a masked
// row. A tile past them is not read by any epilogue; the MMA then multiplies what
// the stage happens to hold. With the epilogues' row checks this leaves out up to
// three quarters of dZ's traffic at few rows: 4096 x 126464 head, one response of
// 99 and 221 masked rows, step 2087 -> 2004 us; 2048 x 32000 head, 301 to 424
// rows, 1125 -> 1060 us (with the split rule in integers). From two row blocks on
// the forward and dZ GEMMs load Xm's zero rows all the same: they are bound by
// power, and zeros cost the multipliers less of it than stale numbers (1,124 and
// 983 rows, forwards 1473 -> 1456 us; 568 and 1,515 rows, step 6209 -> 6170; 1,336
// and 828 rows of a 1536 x 50001 head 1373 -> 1364).
template <int KIND>
__device__ __forceinline__ bool loads_a(const Work& w, const Unit& t, uint32_t rank) {
  return t.m_blk * kPairM + (int32_t)rank * kBM < w.rows || (KIND != GEMM_DX && w.tiles_m > 1);
}

// The copies of one CTA for the stages of one unit: everything about them that
// does not change from one K block to the next. The producer and the MMA issuer
// are one thread each, and their instructions per stage are time in which no
// copy and no MMA starts: with coordinates, box tests and descriptors worked out
// per unit instead of per K block, the forward and dZ GEMMs of 1,679 rows on the
// 4096 x 126464 head take 1012 and 1029 us instead of 1028 and 1038 (means of
// three runs in turn), of 495 rows on a 1536 x 50001 one 55.4 and 54.0 instead of
// 56.0 and 54.7. Boxes that would lie
// wholly outside the operand are not issued; their MMA outputs are discarded.
// The dX GEMM's dZ rows start at `roff`; its K blocks count from the chunk's
// first vocabulary entry, which lies at dZ column dz_col0 and W row v_begin.
struct LoadPlan {
  int32_t a_x, a_y, b_x, b_y;   // coordinates of the first boxes at K block 0
  int32_t a_boxes, b_boxes;     // K-major: 0 or 1; MN-major: 64-column boxes
};

template <int KIND>
__device__ __forceinline__ LoadPlan load_plan(const GemmParams& p, const Work& w, const Unit& t,
                                              uint32_t rank, int64_t roff) {
  LoadPlan q;
  const int32_t a0 = t.m_blk * kPairM + (int32_t)rank * kBM;
  const int64_t b0 =
      b_base<KIND>(p) + (int64_t)t.n_blk * w.wide * kBN + (int64_t)rank * kBNHalf;
  if (!Majors<KIND>::a_mn) {
    q.a_x = KIND == GEMM_DX ? (int32_t)p.dz_col0 : 0;
    q.a_y = a0 + (KIND == GEMM_DX ? (int32_t)roff : 0);
    q.a_boxes = loads_a<KIND>(w, t, rank) ? 1 : 0;
  } else {
    // dZ^T: 2 boxes of 64 vocabulary columns x 64 masked rows, inside the dZ buffer
    q.a_x = (int32_t)(p.dz_col0 + a0);
    q.a_y = 0;
    q.a_boxes = 0;
    for (int c = 0; c < kBM / 64; ++c)
      if (p.dz_col0 + a0 + c * 64 < p.w.dz_cols) q.a_boxes = c + 1;
  }
  if (!Majors<KIND>::b_mn) {
    q.b_x = 0;
    q.b_y = (int32_t)b0;
    q.b_boxes = b0 < b_rows<KIND>(p) ? 1 : 0;
  } else {
    // W (dX): 2 boxes of 64 x 64 per accumulator of the tile, inside H
    q.b_x = (int32_t)b0;
    q.b_y = (int32_t)p.v_begin;
    q.b_boxes = 0;
    for (int i = 0; i < 2 * w.wide; ++i)
      if (b0 + (i >> 1) * kBN + (i & 1) * 64 < p.g.H) q.b_boxes = i + 1;
  }
  return q;
}

// Bytes those copies deliver per stage.
template <int KIND>
__device__ __forceinline__ uint32_t stage_bytes(const LoadPlan& q) {
  return (uint32_t)q.a_boxes * (Majors<KIND>::a_mn ? kMnChunkBytes : kTileABytes) +
         (uint32_t)q.b_boxes * (Majors<KIND>::b_mn ? kMnChunkBytes : kTileBBytes);
}

// Issue the A and the B copies of the K block that starts at element k; they
// complete on `cbar`, the even CTA's full barrier (shared::cluster address).
template <int KIND>
__device__ __forceinline__ void load_a(const LoadPlan& q, const CUtensorMap* ma, uint32_t sa,
                                       uint32_t cbar, int32_t k) {
  if (!Majors<KIND>::a_mn) {
    if (q.a_boxes) tma_load_2d_pair(sa, ma, cbar, q.a_x + k, q.a_y);
  } else {
#pragma unroll
    for (int c = 0; c < kBM / 64; ++c)
      if (c < q.a_boxes) tma_load_2d_pair(sa + c * kMnChunkBytes, ma, cbar, q.a_x + c * 64, k);
  }
}

template <int KIND>
__device__ __forceinline__ void load_b(const LoadPlan& q, const CUtensorMap* mb, uint32_t sb,
                                       uint32_t cbar, int32_t k) {
  if (!Majors<KIND>::b_mn) {
    if (q.b_boxes) tma_load_2d_pair(sb, mb, cbar, k, q.b_y);
  } else {
#pragma unroll
    for (int i = 0; i < 2 * kDxWide; ++i)
      if (i < q.b_boxes)
        tma_load_2d_pair(sb + (i >> 1) * kTileBBytes + (i & 1) * kMnChunkBytes, mb, cbar,
                         q.b_x + (i >> 1) * kBN + (i & 1) * 64, q.b_y + k);
  }
}

__device__ __forceinline__ float bits_f(uint32_t v) { return __uint_as_float(v); }

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// ---- epilogues: one thread per accumulator row; row0 = first row of the warp --------

// Epilogue staging of one warp: two 32-row x 128-byte buffers in the 128-byte
// swizzled layout the TMA tensor maps use (16-byte chunk q of row r stored at
// chunk q ^ (r & 7)), so that 32 lanes writing one row each hit 8 bank groups.
struct EpiStage {
  uint32_t base;   // shared address of this warp's first buffer (1024-aligned)
  int buf;         // buffer the next sub-tile goes to

  // Returns the shared address of a buffer free for writing: the bulk group
  // that last read it (two sub-tiles ago) has finished reading.
  __device__ __forceinline__ uint32_t acquire(int lane) {
    if (lane == 0) bulk_wait_group_read<1>();
    __syncwarp();
    return base + (uint32_t)buf * kEpiBufBytes;
  }
  // Hands the written buffer to lane 0, which issues the bulk copy `issue`.
  template <class Issue>
  __device__ __forceinline__ void release(int lane, uint32_t sbuf, Issue issue) {
    fence_proxy_async_shared();
    __syncwarp();
    if (lane == 0) {
      issue(sbuf);
      bulk_commit_group();
    }
    buf ^= 1;
  }
};

// Writes 8 16-byte chunks (one 128-byte row of the sub-tile) for row `lane`.
__device__ __forceinline__ void stage_row(uint32_t sbuf, int lane, const uint4 (&chunk)[8]) {
  const uint32_t row = sbuf + (uint32_t)lane * 128u;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const uint32_t a = row + (uint32_t)((q ^ (lane & 7)) * 16);
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(chunk[q].x),
                 "r"(chunk[q].y), "r"(chunk[q].z), "r"(chunk[q].w)
                 : "memory");
  }
}

// What an epilogue lane needs to know about its accumulator row, loaded before
// the wait for the accumulator: the chain of loads (row, sequence, coefficient)
// otherwise follows it where a launch's tiles all run in one wave (lmhead_dz,
// start to start: 8.2 -> 7.7 us at 64 x 512, 13.6 -> 12.8 at 1024 x 8192).
struct RowInfo {
  int32_t y = -1;         // target token
  float w = 0.f;          // dZ: coef_b / t_b
  float lse_l2 = 0.f;     // dZ: log-sum-exp, base 2
  int32_t pos = -1;       // dX: b * R + i
};

template <int KIND>
__device__ __forceinline__ RowInfo row_info(const GemmParams& p, const Work& wk, int32_t M,
                                            int64_t r) {
  RowInfo q;
  if (r >= M) return q;
  if (KIND == GEMM_FWD) {
    q.y = p.w.tgt[r];
  } else if (KIND == GEMM_DZ) {
    const int32_t pos = p.w.rows[r];
    if (BGPO_IN_BOUNDS(p.w.err, pos >= 0 && pos < p.g.m_cap, KID_LMHEAD_DZ * 16 + 10)) {
      const int32_t b = pos / (int32_t)p.g.R;
      q.w = p.coef[b] / p.w.t[b];
      q.lse_l2 = p.w.lse[r] * kLog2e;
      q.y = p.w.tgt[r];
    }
  } else if (KIND == GEMM_DX && wk.splits == 1) {
    const int32_t pos = p.w.rows[r];
    if (BGPO_IN_BOUNDS(p.w.err, pos >= 0 && pos < p.g.m_cap, KID_DX_GEMM * 16 + 10)) q.pos = pos;
  }
  return q;
}

// GEMM_FWD: per (row, vocab tile) the pair (max z, sum e^{z - max}) and, in the
// tile holding y_r, the target logit z_{r, y_r}; with a logit region, the
// fp32 logits too (32-column sub-tiles through TMA stores into [m_pad, v_pad]).
__device__ __forceinline__ void epi_fwd(const GemmParams& p, const CUtensorMap* map_c, int32_t M,
                                        const Unit& t, const RowInfo& q, int64_t row0, int lane,
                                        uint32_t tb, EpiStage& st) {
  if (row0 >= M) return;  // none of this warp's rows is masked (warp-uniform)
  const int64_t r = row0 + lane;
  const bool valid = r < M;
  const int32_t y = q.y;
  const int32_t v0 = t.n_blk * kBN;
  const int32_t V = (int32_t)p.g.V;
  float m = -INFINITY, s = 0.f, tl = 0.f;
  bool hit = false;
#pragma unroll 1
  for (int c = 0; c < kBN / 32; ++c) {
    const int32_t col0 = v0 + c * 32;
    if (col0 >= V) break;  // warp-uniform
    uint32_t raw[32];
    tmem_ld_32x32b_x32(tb + c * 32, raw);
    tmem_ld_wait();
    const int nvalid = min(32, V - col0);
    // the row's target lies in this sub-tile for about one sub-tile in 4000:
    // test it once instead of once per column
    if ((uint32_t)(y - col0) < 32u) {
#pragma unroll
      for (int k = 0; k < 32; ++k)
        if (col0 + k == y) { tl = bits_f(raw[k]); hit = true; }
    }
    float cm = -INFINITY;
    float acc = 0.f;
    float mn;
    if (nvalid == 32) {  // warp-uniform: every column lies inside the vocabulary
#pragma unroll
      for (int k = 0; k < 32; ++k) cm = fmaxf(cm, bits_f(raw[k]));
      mn = fmaxf(m, cm);
      const float mnl = mn * kLog2e;
#pragma unroll
      for (int k = 0; k < 32; ++k) acc += ex2_ftz(fmaf(bits_f(raw[k]), kLog2e, -mnl));
    } else {
#pragma unroll
      for (int k = 0; k < 32; ++k)
        if (k < nvalid) cm = fmaxf(cm, bits_f(raw[k]));
      mn = fmaxf(m, cm);
      const float mnl = mn * kLog2e;
#pragma unroll
      for (int k = 0; k < 32; ++k)
        if (k < nvalid) acc += ex2_ftz(fmaf(bits_f(raw[k]), kLog2e, -mnl));
    }
    s = s * ex2_ftz((m - mn) * kLog2e) + acc;
    m = mn;
    if (p.w.zc != nullptr) {  // kernel-uniform; col0 < V <= v_pad, both multiples of 32
      uint4 chunk[8];
#pragma unroll
      for (int q = 0; q < 8; ++q)
        chunk[q] = make_uint4(raw[4 * q], raw[4 * q + 1], raw[4 * q + 2], raw[4 * q + 3]);
      const uint32_t sbuf = st.acquire(lane);
      stage_row(sbuf, lane, chunk);
      st.release(lane, sbuf, [&](uint32_t a) { tma_store_2d(map_c, a, col0, (int32_t)row0); });
    }
  }
  if (valid) {
    p.w.part[r * p.g.n_vt + t.n_blk] = make_float2(m, s);
    if (hit) p.w.tgt_logit[r] = tl;
  }
}

// GEMM_DZ: dz_{r,v} = w_r (1[v = y_r] - e^{z_{r,v} - lse_r}) as bf16, zero for
// rows in [M, roundup(M, 64)) and vocabulary columns >= V; 64-column sub-tiles
// leave through TMA stores into dZ [dz_rows, dz_cols], from row `roff` on;
// vocabulary entry v lands in column v - v_begin + dz_col0. The TMEM load of the
// next 32 columns is in flight while these are worked on, and rows past M take
// the short path too: where short K loops (H up to about 1,024) leave the
// epilogue bare, a wave of tiles takes 3.1 us instead of 5.1 (500 rows, H 256, V
// 38912: 24.8 -> 18.8 us; H 512: 26.5 -> 21.6; H 1024: 31.4 -> 29.0; H 4096: 87.5
// -> 85.9). The same in the forward's epilogue, with its maxima and sums in four
// chains, gained nothing (H 256: 17.4 -> 17.5 us).
struct DzRow {
  float w, lse_l2;
  int32_t y;
  bool valid;
};

// 32 columns from `col` on as 16 bf16 pairs. `plain`: they lie inside the
// vocabulary and away from the row's target, as almost all do: there dz =
// -w e^{z - lse}, the same value the general expression gives (w (0 - p) = (-w) p
// exactly); rows past M give zeros whatever their z is.
__device__ __forceinline__ void dz_half(const DzRow& d, bool plain, int32_t col, int32_t V,
                                        const uint32_t (&raw)[32], uint4* chunk) {
  uint32_t packed[16];
  if (plain) {
    const float nw = -d.w;
    const uint32_t keep = d.valid ? 0xffffffffu : 0u;
#pragma unroll
    for (int k = 0; k < 32; k += 2) {
      const float d0 = nw * ex2_ftz(fmaf(bits_f(raw[k]), kLog2e, -d.lse_l2));
      const float d1 = nw * ex2_ftz(fmaf(bits_f(raw[k + 1]), kLog2e, -d.lse_l2));
      packed[k / 2] = pack_bf16x2(d0, d1) & keep;
    }
  } else {
#pragma unroll
    for (int k = 0; k < 32; k += 2) {
      float v[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float pr = ex2_ftz(fmaf(bits_f(raw[k + e]), kLog2e, -d.lse_l2));
        const float x = d.w * ((col + k + e == d.y ? 1.f : 0.f) - pr);
        v[e] = (d.valid && col + k + e < V) ? x : 0.f;
      }
      packed[k / 2] = pack_bf16x2(v[0], v[1]);
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
    chunk[q] = make_uint4(packed[4 * q], packed[4 * q + 1], packed[4 * q + 2], packed[4 * q + 3]);
}

__device__ __forceinline__ void epi_dz(const GemmParams& p, const CUtensorMap* map_c, int32_t M,
                                       const Unit& t, const RowInfo& q, int64_t row0, int64_t roff,
                                       int lane, uint32_t tb, EpiStage& st) {
  // past the dW GEMM's K padding nothing reads dZ: its rows there only reach
  // accumulator rows of the dX GEMM that no epilogue reads (warp-uniform)
  if (row0 >= round_up(M, kBK)) return;
  const DzRow d = {q.w, q.lse_l2, q.y, row0 + lane < M};
  const int32_t v0 = (int32_t)p.v_begin + t.n_blk * kBN;
  const int32_t V = (int32_t)p.g.V;
  const int32_t shift = (int32_t)(p.dz_col0 - p.v_begin);   // vocabulary entry -> dZ column
  // 64-column sub-tiles inside the dZ buffer (its width is a multiple of 64)
  const int nsub = (int)min((int64_t)(kBN / 64), (p.w.dz_cols - v0 - shift) / 64);
  if (nsub <= 0) return;  // warp-uniform
  uint32_t ra[32], rb[32];
  tmem_ld_32x32b_x32(tb, ra);
#pragma unroll 1
  for (int c = 0; c < nsub; ++c) {
    const int32_t col0 = v0 + c * 64;
    const bool plain = col0 + 64 <= V && (uint32_t)(d.y - col0) >= 64u;
    uint4 chunk[8];
    tmem_ld_wait_regs(ra);
    tmem_ld_32x32b_x32(tb + (uint32_t)c * 64 + 32, rb);
    dz_half(d, plain, col0, V, ra, chunk);
    tmem_ld_wait_regs(rb);
    if (c + 1 < nsub) tmem_ld_32x32b_x32(tb + (uint32_t)(c + 1) * 64, ra);
    dz_half(d, plain, col0 + 32, V, rb, chunk + 4);
    const uint32_t sbuf = st.acquire(lane);
    stage_row(sbuf, lane, chunk);
    st.release(lane, sbuf,
               [&](uint32_t a) { tma_store_2d(map_c, a, col0 + shift, (int32_t)(row0 + roff)); });
  }
}

// GEMM_DX: fp32 partial of split s, rows [split * tiles_m * 256 + r] of the
// partial buffer, 32-column sub-tiles through TMA stores in the first
// vocabulary chunk and TMA reduce-adds in the later ones (every element has one
// writer per launch and the chunks run in order, so the sum is deterministic;
// rows >= M are not read). Without split-K every dX element has exactly this one
// contribution in the launch, so the warp adds its sub-tile straight into the
// rows dX[b, i] (which the compaction recorded) with 16-byte atomic adds, which
// need no round trip: each element still receives one addition, and the split
// reduction after the last chunk has nothing to do. The sub-tile is turned in the
// staging buffer first, so that one instruction adds four rows' whole 128-byte
// lines instead of 16 bytes of 32 rows: 1,000 rows of 4,096, K = 2,000: 45.6 -> 25.8
// us with 256 x 256 tiles, 1,500 of 3,000, K = 12,000: 117 -> 87.
__device__ __forceinline__ void dx_sub(const GemmParams& p, const CUtensorMap* map_c,
                                       const Work& wk, const RowInfo& q, int32_t h0, int32_t prow0,
                                       int c, const uint32_t (&raw)[32], int lane, EpiStage& st) {
  uint4 chunk[8];
#pragma unroll
  for (int e = 0; e < 8; ++e)
    chunk[e] = make_uint4(raw[4 * e], raw[4 * e + 1], raw[4 * e + 2], raw[4 * e + 3]);
  if (wk.splits == 1) {  // launch-uniform
    const uint32_t buf = st.base + (uint32_t)(c & 1) * kEpiBufBytes;
    stage_row(buf, lane, chunk);
    __syncwarp();
    // 16-byte piece of this lane inside each row (H is a multiple of 8)
    const int32_t col = h0 + c * 32 + (lane & 7) * 4;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int row = 4 * k + (lane >> 3);
      const int32_t pos = __shfl_sync(0xffffffffu, q.pos, row);
      if (pos >= 0 && col < (int32_t)p.g.H) {
        float4 v;
        const uint32_t a = buf + (uint32_t)row * 128u + (uint32_t)(((lane & 7) ^ (row & 7)) * 16);
        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                     : "r"(a)
                     : "memory");
        atomicAdd(reinterpret_cast<float4*>(p.dX + (int64_t)pos * p.g.H + col), v);
      }
    }
    return;
  }
  const uint32_t sbuf = st.acquire(lane);
  stage_row(sbuf, lane, chunk);
  if (p.chunk == 0)
    st.release(lane, sbuf, [&](uint32_t a) { tma_store_2d(map_c, a, h0 + c * 32, prow0); });
  else
    st.release(lane, sbuf, [&](uint32_t a) { tma_reduce_add_2d(map_c, a, h0 + c * 32, prow0); });
}

// `nb`: the 256-column block of dX this accumulator holds. The TMEM load of
// sub-tile c + 1 is in flight while sub-tile c is written out.
__device__ __forceinline__ void epi_dx(const GemmParams& p, const CUtensorMap* map_c, int32_t M,
                                       const Work& wk, const Unit& t, const RowInfo& q, int32_t nb,
                                       int64_t row0, int lane, uint32_t tb, EpiStage& st) {
  const int32_t h0 = nb * kBN;
  const int32_t nsub = min(kBN / 32, ((int32_t)p.g.H - h0 + 31) / 32);  // inside H
  if (nsub <= 0 || row0 >= M) return;  // a column block past H, no masked row (warp-uniform)
  const int32_t prow0 = (int32_t)(t.split * wk.tiles_m * kPairM + row0);
  uint32_t ra[32], rb[32];
  tmem_ld_32x32b_x32(tb, ra);
  tmem_ld_wait_regs(ra);
#pragma unroll 1
  for (int c = 0; c < nsub; c += 2) {
    if (c + 1 < nsub) tmem_ld_32x32b_x32(tb + (uint32_t)(c + 1) * 32, rb);
    dx_sub(p, map_c, wk, q, h0, prow0, c, ra, lane, st);
    if (c + 1 < nsub) {
      tmem_ld_wait_regs(rb);
      if (c + 2 < nsub) tmem_ld_32x32b_x32(tb + (uint32_t)(c + 2) * 32, ra);
      dx_sub(p, map_c, wk, q, h0, prow0, c + 1, rb, lane, st);
      if (c + 2 < nsub) tmem_ld_wait_regs(ra);
    }
  }
}

// The dW GEMM reads and writes 8 bytes of dW per element whatever its K is; up
// to about 2,000 rows that read-modify-write, not the tensor pipe, bounds it. A
// reduce-add that misses L2 streams dW at 5.0 TB/s, one that finds its lines
// there at up to 6.7 (plain copy: 6.4), so each warp fetches the lines of the
// pair's next tile into L2 while it adds the current one, in halves (512-byte
// row segments): whole tiles at once measured 5-12% slower, quarters and eighths
// slower than no prefetch. Without -> with, in us: V 126464, H 4096: 829 -> 618
// (31 rows), 835 -> 700 (505), 911 -> 844 (1012), 1204 -> 1045 (1521), 1425 ->
// 1310 (2154), 1643 -> 1491 (2536), 1893 -> 1817 (3042), but 1901 -> 1979 (3298)
// and 3147 -> 3278 (5073); V 152064, H 3584: 855 -> 653 (62), 967 -> 907 (1012),
// 1547 -> 1445 (2282), 1999 -> 1963 (3042); V 32000, H 2048: 106 -> 90 (62), 131 ->
// 121 (1012), 199 -> 189 (2282). A dW that L2 holds needs no fetching (V 8192, H
// 1024: 14 -> 18 at 62 rows), and a hidden size that is no multiple of 32 gained
// nothing (V 50001, H 1032: 86 -> 90 at 505 rows, 106 -> 102 at 1012). Where dW starts
// does not matter: 16 bytes off a 128-byte line the 4096 x 126464 head takes 901 -> 635
// at 30 rows, 938 -> 705 at 498, 1290 -> 1095 at 1,507, 1852 -> 1637 at 2,512 (on the
// line 799 -> 608, 827 -> 676, 1205 -> 1032, 1705 -> 1551).
constexpr int64_t kDwPrefetchKb = 48;                      // K blocks: 3,072 rows
constexpr int64_t kDwPrefetchMinBytes = int64_t(1) << 27;  // about L2's size

__device__ __forceinline__ bool dw_prefetches(const GemmParams& p, const Work& w) {
  return w.kb_total - w.kb_first <= kDwPrefetchKb && p.g.H % 32 == 0 &&
         4 * (p.v_end - p.v_begin) * p.g.H >= kDwPrefetchMinBytes;
}

// Fetches half `part` (kBN / 2 columns, one 512-byte row segment per lane) of
// this warp's 32 dW rows of tile t into L2 (columns past H and rows past V are
// not touched).
__device__ __forceinline__ void prefetch_dw(const GemmParams& p, const Unit& t, uint32_t rank,
                                            int quarter, int lane, int part) {
  const int64_t v = p.v_begin + (int64_t)t.m_blk * kPairM + (int64_t)rank * kBM + quarter * 32 + lane;
  const int32_t h0 = t.n_blk * kBN + part * (kBN / 2);
  if (v < p.g.V && h0 < p.g.H)
    bulk_prefetch_l2(p.dW + v * p.g.H + h0, (uint32_t)min(kBN / 2, (int32_t)p.g.H - h0) * 4u);
}

// GEMM_DW: dW[v, h] += acc through TMA reduce-add of 32 x 32 fp32 sub-tiles
// (the read-modify-write happens at L2; vocabulary rows >= V are clipped).
// Accumulator row r is vocabulary entry v_begin + r. `ahead`: the dW lines of
// this pair's next tile `tn` are fetched into L2 meanwhile, half a tile at a time.
__device__ __forceinline__ void epi_dw(const GemmParams& p, const CUtensorMap* map_c, const Unit& t,
                                       int64_t row0, int lane, uint32_t tb, EpiStage& st,
                                       bool ahead, const Unit& tn, uint32_t rank, int quarter) {
  const int32_t h0 = t.n_blk * kBN;
  const int64_t v = p.v_begin + row0;
  if (v >= p.g.V) return;  // this warp's rows all lie past the vocabulary (warp-uniform)
#pragma unroll 1
  for (int c = 0; c < kBN / 32; ++c) {
    if (ahead && c % 4 == 0) prefetch_dw(p, tn, rank, quarter, lane, c / 4);
    if (h0 + c * 32 >= p.g.H) break;  // warp-uniform
    uint32_t raw[32];
    tmem_ld_32x32b_x32(tb + c * 32, raw);
    tmem_ld_wait();
    uint4 chunk[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      chunk[q] = make_uint4(raw[4 * q], raw[4 * q + 1], raw[4 * q + 2], raw[4 * q + 3]);
    const uint32_t sbuf = st.acquire(lane);
    stage_row(sbuf, lane, chunk);
    st.release(lane, sbuf,
               [&](uint32_t a) { tma_reduce_add_2d(map_c, a, h0 + c * 32, (int32_t)v); });
  }
}

template <int KIND>
__device__ __forceinline__ int32_t kernel_id() {
  return KIND == GEMM_FWD ? KID_LMHEAD_FWD
       : KIND == GEMM_DZ  ? KID_LMHEAD_DZ
       : KIND == GEMM_DX  ? KID_DX_GEMM
                          : KID_DW_GEMM;
}

// Sets the abort flag of both CTAs of the pair.
__device__ __forceinline__ void raise_abort(volatile int* abort_flag, uint32_t peer) {
  *abort_flag = 1;
  const uint32_t remote = map_to_cta(smem_addr(const_cast<int*>(abort_flag)), peer);
  asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(remote), "r"(1) : "memory");
}

template <int KIND>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    k_gemm(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
           const __grid_constant__ CUtensorMap map_c, const GemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  constexpr int kSt = kStages;            // barriers; the dX GEMM may use fewer stages
  uint8_t* s_epi = smem + kStages * kStageBytes;   // 4 warps x 2 staging buffers
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_epi + SmemPlan<KIND>::epi_bytes);
  uint64_t* full = bars;                      // [kSt] TMA (both CTAs) -> MMA; even CTA's
  uint64_t* empty = bars + kSt;               // [kSt] MMA -> TMA of each CTA
  uint64_t* tfull = bars + 2 * kSt;           // [2] MMA -> epilogue of each CTA
  uint64_t* tempty = bars + 2 * kSt + 2;  // [2] epilogues (both CTAs) -> MMA; even CTA's
  uint64_t* done = bars + 2 * kSt + 4;    // MMA drain on abort
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kSt + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* never = reinterpret_cast<volatile int*>(tmem_slot + 2);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();  // 0: even CTA (issues the MMAs), 1: its peer
  const uint32_t peer = rank ^ 1u;
  const int32_t pair = (int32_t)(blockIdx.x >> 1);
  const int32_t num_pairs = (int32_t)(gridDim.x >> 1);
  int32_t* err = p.w.err;

  // the prologue touches no global memory: it runs while the kernel before this
  // one finishes
  if (threadIdx.x == 0) {
    for (int s = 0; s < kSt; ++s) {
      mbar_init(smem_addr(&full[s]), 1);    // the even CTA's arrive.expect_tx
      mbar_init(smem_addr(&empty[s]), 1);   // one multicast commit
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_addr(&tfull[a]), 1);
      mbar_init(smem_addr(&tempty[a]), 2 * 4);   // 4 epilogue warps in each CTA
    }
    mbar_init(smem_addr(done), 1);
    *abort_flag = 0;
    *never = 0;
    fence_barrier_init();
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_map(&map_a);
    tma_prefetch_map(&map_b);
    tma_prefetch_map(&map_c);
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_addr(tmem_slot), kTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync();  // barriers of both CTAs initialised, TMEM allocated
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // The forward and dW GEMMs are followed by small kernels, whose blocks wait
  // beside them from here on; dZ and dX let the next kernel (a GEMM that needs the
  // SMs' whole shared memory, a reduction of up to 2,432 blocks) start once this
  // CTA's last copies are on their way. Of the 16 choices this one's chains of a
  // sample's kernels are the fastest in the mean over 8 heads: all early 42.0, 78.2
  // and 266 us (320 x 777, 256 x 2000, 2048 x 32000), this 40.9, 77.0 and 264.
  if (KIND == GEMM_FWD || KIND == GEMM_DW) pdl_launch_dependents();
  pdl_wait();

  int32_t M = 0;
  if (err[ERR_SAMPLE] == p.j) {
    M = err[ERR_M];
  } else if (blockIdx.x == 0 && threadIdx.x == 0) {
    set_device_error(err, kStatusInvalidArg, kernel_id<KIND>() * 16 + 1);
  }
  if (!BGPO_IN_BOUNDS(err, M >= 0 && M <= p.g.m_cap, kernel_id<KIND>() * 16 + 9)) M = 0;
  // first dZ / Xm^T row of this sample: nonzero only when it pairs with a
  // pending sample (the masking set it; the forward does not use dZ)
  const int64_t roff = KIND == GEMM_FWD ? 0 : row_offset(err[ERR_ROW_OFF], p.w.dz_rows, p.g.m_pad);
  // dW: first K row, a multiple of kBK in [0, roff] (see ERR_DW_K0)
  const int64_t k0 = KIND == GEMM_DW ? row_offset(err[ERR_DW_K0], roff + p.g.m_pad, p.g.m_pad) : 0;
  const Work wk = make_work<KIND>(p, M, roff, k0);
  if (KIND == GEMM_DW && blockIdx.x == 0 && threadIdx.x == 0) {
    // a dW GEMM meant to complete a pair whose first sample is not pending
    // adds this sample alone: the other sample's contribution is missing
    if (p.pair_consume && err[ERR_PAIRED] != 1)
      set_device_error(err, kStatusInvalidArg, kernel_id<KIND>() * 16 + 5);
    err[ERR_PEND] = -1;  // nothing waits any more
  }
  // tiles of two accumulators fill TMEM (one tile at a time) and take 48 KB a stage
  const int wide = KIND == GEMM_DX ? wk.wide : 1;
  const int nst = wide == 2 ? kDxStages : kStages;
  const uint32_t b_bytes = (uint32_t)wide * kTileBBytes;
  uint8_t* s_a = smem;
  uint8_t* s_b = smem + nst * kTileABytes;

  if (warp == 0 || warp == kWarpB) {
    // ---------------- TMA producers (both CTAs): A tiles, B tiles ----------------
    if (lane == 0) {
      const bool is_a = warp == 0;
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      bool issued = false;
      const uint32_t dst0 = smem_addr(is_a ? s_a : s_b);
      const uint32_t step = is_a ? kTileABytes : b_bytes;
      const uint32_t full0 = smem_addr(full), empty0 = smem_addr(empty);
      const uint32_t cfull0 = map_to_cta(full0, 0);
      for (int32_t u = pair; u < wk.units && ok; u += num_pairs) {
        const Unit t = unit_of<KIND>(wk, u);
        const LoadPlan lp = load_plan<KIND>(p, wk, t, rank, roff);
        // the even CTA's A producer arms the transaction bytes of both CTAs'
        // copies on its full barrier; the other producers' copies only
        // complete_tx on it (a per-stage remote arrive from the odd CTA halved the
        // throughput)
        const uint32_t bytes =
            stage_bytes<KIND>(lp) + stage_bytes<KIND>(load_plan<KIND>(p, wk, t, peer, roff));
        for (int32_t k = t.kb0 * kBK, end = (t.kb0 + t.kb_n) * kBK; k < end; k += kBK) {
          if (!mbar_wait(empty0 + stage * 8, phase ^ 1u, abort_flag)) { ok = false; break; }
          const uint32_t dst = dst0 + stage * step, cbar = cfull0 + stage * 8;
          if (is_a) {
            if (rank == 0) mbar_arrive_expect_tx(full0 + stage * 8, bytes);
            load_a<KIND>(lp, &map_a, dst, cbar, k);
          } else {
            load_b<KIND>(lp, &map_b, dst, cbar, k);
          }
          issued = true;
          if (++stage == nst) { stage = 0; phase ^= 1u; }
        }
      }
      if (is_a) pdl_launch_dependents();
      if (!ok) {
        raise_abort(abort_flag, peer);
        set_device_error(err, kStatusTimeout, kernel_id<KIND>() * 16 + 2);
        // let copies already issued land before this CTA can exit
        if (issued) {
          const uint64_t t0 = globaltimer_ns();
          while (globaltimer_ns() - t0 < 2000000ull) {
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer (even CTA) ----------------
    if (rank == 0 && lane == 0) {
      constexpr uint32_t idesc =
          idesc_bf16_f32(kPairM, kBN, Majors<KIND>::a_mn, Majors<KIND>::b_mn);
      // one K step of an MMA: 16 K-major elements, or 16 rows of an MN-major box
      constexpr uint32_t kAStep = (Majors<KIND>::a_mn ? 2048 : 32) >> 4;
      constexpr uint32_t kBStep = (Majors<KIND>::b_mn ? 2048 : 32) >> 4;
      const uint64_t a_desc =
          smem_desc_sw128(smem_addr(s_a), Majors<KIND>::a_mn ? kMnChunkBytes : 16, 1024);
      const uint64_t b_desc =
          smem_desc_sw128(smem_addr(s_b), Majors<KIND>::b_mn ? kMnChunkBytes : 16, 1024);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true, issued = false;
      int it = 0;
      for (int32_t u = pair; u < wk.units && ok; u += num_pairs, ++it) {
        const Unit t = unit_of<KIND>(wk, u);
        const int acc = wide == 2 ? 0 : it & 1;
        const uint32_t acc_phase = (uint32_t)(wide == 2 ? it : it >> 1) & 1u;
        if (!mbar_wait(smem_addr(&tempty[acc]), acc_phase ^ 1u, abort_flag)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * kBN);
        for (int32_t kb = 0; kb < t.kb_n; ++kb) {
          if (!mbar_wait(smem_addr(&full[stage]), phase, abort_flag)) { ok = false; break; }
          tc_fence_after();
          // the address fields of the descriptors count 16-byte units and never
          // carry out of their 14 bits (shared memory is below 2^18 bytes)
          const uint64_t ad = a_desc + (uint64_t)((uint32_t)stage * (kTileABytes >> 4));
          const uint64_t bd = b_desc + (uint64_t)((uint32_t)stage * (b_bytes >> 4));
          if (KIND == GEMM_DX && wide == 2) {
#pragma unroll
            for (int k = 0; k < kBK / kUmmaK; ++k) {
              const uint32_t add = (kb > 0 || k > 0) ? 1u : 0u;
              umma_bf16_pair(d_tmem, ad + k * kAStep, bd + k * kBStep, idesc, add);
              umma_bf16_pair(d_tmem + kBN, ad + k * kAStep, bd + (kTileBBytes >> 4) + k * kBStep,
                             idesc, add);
            }
          } else {
#pragma unroll
            for (int k = 0; k < kBK / kUmmaK; ++k)
              umma_bf16_pair(d_tmem, ad + k * kAStep, bd + k * kBStep, idesc,
                             (kb > 0 || k > 0) ? 1u : 0u);
          }
          issued = true;
          // frees this stage in both CTAs once these MMAs have read it
          umma_commit_pair(smem_addr(&empty[stage]), kBothCtas);
          if (++stage == nst) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        umma_commit_pair(smem_addr(&tfull[acc]), kBothCtas);  // accumulators ready
      }
      if (!ok) {
        raise_abort(abort_flag, peer);
        set_device_error(err, kStatusTimeout, kernel_id<KIND>() * 16 + 3);
        if (issued) {
          umma_commit_pair(smem_addr(done), 0x1);
          mbar_wait(smem_addr(done), 0, never);
        }
      }
    }
    __syncwarp();
  } else {
    // ---------------- epilogue (warps 2..5 of both CTAs) ----------------
    const int quarter = warp & 3;  // TMEM lanes this warp may access: 32*quarter ..
    EpiStage st;
    st.base = smem_addr(s_epi + (uint32_t)(warp - 2) * 2u * kEpiBufBytes);
    st.buf = 0;
    int it = 0;
    bool ok = true;
    const bool ahead = KIND == GEMM_DW && pair < wk.units && dw_prefetches(p, wk);
    if (ahead) {
      const Unit t0 = unit_of<KIND>(wk, pair);
      prefetch_dw(p, t0, rank, quarter, lane, 0);
      prefetch_dw(p, t0, rank, quarter, lane, 1);
    }
    for (int32_t u = pair; u < wk.units; u += num_pairs, ++it) {
      const Unit t = unit_of<KIND>(wk, u);
      const int acc = wide == 2 ? 0 : it & 1;
      const uint32_t acc_phase = (uint32_t)(wide == 2 ? it : it >> 1) & 1u;
      const int64_t row0 = (int64_t)t.m_blk * kPairM + (int64_t)rank * kBM + quarter * 32;
      const RowInfo q = row_info<KIND>(p, wk, M, row0 + lane);
      const bool got = mbar_wait(smem_addr(&tfull[acc]), acc_phase, abort_flag);
      if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
      tc_fence_after();
      const uint32_t tb = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * kBN);
      if (KIND == GEMM_FWD) epi_fwd(p, &map_c, M, t, q, row0, lane, tb, st);
      else if (KIND == GEMM_DZ) epi_dz(p, &map_c, M, t, q, row0, roff, lane, tb, st);
      else if (KIND == GEMM_DX) {
#pragma unroll 1
        for (int g = 0; g < wide; ++g)
          epi_dx(p, &map_c, M, wk, t, q, t.n_blk * wide + g, row0, lane,
                 tb + (uint32_t)(g * kBN), st);
      } else {
        const bool more = ahead && u + num_pairs < wk.units;
        epi_dw(p, &map_c, t, row0, lane, tb, st, more, unit_of<KIND>(wk, more ? u + num_pairs : u),
               rank, quarter);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_addr(&tempty[acc]), 0));
    }
    // every bulk store / reduction of this warp has completed before exit
    if (lane == 0) bulk_wait_group<0>();
    __syncwarp();
    if (!ok) {
      raise_abort(abort_flag, peer);
      if (lane == 0) set_device_error(err, kStatusTimeout, kernel_id<KIND>() * 16 + 4);
    }
  }

  tc_fence_before();
  cluster_sync();  // no CTA of the pair still reads the other's shared memory
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, kTmemCols);
  }
}

template <int KIND>
cudaError_t launch_kind(const CUtensorMap& ma, const CUtensorMap& mb, const CUtensorMap& mc,
                        const GemmParams& p, cudaStream_t s) {
  constexpr uint32_t smem = SmemPlan<KIND>::bytes;
  cudaError_t e = cudaFuncSetAttribute(k_gemm<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  return launch_dependent(k_gemm<KIND>, dim3(2 * p.num_pairs), kThreads, smem, s, ma, mb, mc, p);
}

}  // namespace

int gemm_num_pairs(int num_sms) {
  static int cached = 0;
  static std::once_flag once;
  std::call_once(once, [num_sms] {
    int clusters = 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)num_sms, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = SmemPlan<GEMM_DX>::bytes;
    if (cudaFuncSetAttribute(k_gemm<GEMM_DX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)SmemPlan<GEMM_DX>::bytes) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&clusters, k_gemm<GEMM_DX>, &cfg) == cudaSuccess &&
        clusters > 0)
      cached = clusters;
    else
      cudaGetLastError();
  });
  const int half = num_sms / 2;
  return (cached > 0 && cached < half) ? cached : half;
}

cudaError_t launch_gemm(GemmKind kind, const CUtensorMap& map_a, const CUtensorMap& map_b,
                        const CUtensorMap& map_c, const GemmArgs& a, const WsPtrs& w,
                        cudaStream_t s) {
  GemmParams p;
  p.g = a.g;
  p.num_pairs = a.num_pairs;
  p.j = a.j;
  p.v_begin = a.v_begin;
  p.v_end = a.v_end;
  p.dz_col0 = a.dz_col0;
  p.chunk = a.chunk;
  p.w = w;
  p.coef = a.coef;
  p.dW = a.dW;
  p.dX = a.dX;
  p.pair_consume = a.pair_consume;
  switch (kind) {
    case GEMM_FWD: return launch_kind<GEMM_FWD>(map_a, map_b, map_c, p, s);
    case GEMM_DZ: return launch_kind<GEMM_DZ>(map_a, map_b, map_c, p, s);
    case GEMM_DX: return launch_kind<GEMM_DX>(map_a, map_b, map_c, p, s);
    case GEMM_DW: return launch_kind<GEMM_DW>(map_a, map_b, map_c, p, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace bgpo
