// Workspace layout, tile geometry and work splitting shared by the host code
// and the kernels of the BGPO LM-head ELBO path.
#pragma once

#include <stddef.h>
#include <stdint.h>

#ifdef __CUDACC__
#define BGPO_HD __host__ __device__ __forceinline__
#else
#define BGPO_HD inline
#endif

namespace bgpo {

// ---- GEMM tile geometry ---------------------------------------------------------
// A pair of CTAs (a 2-CTA cluster) computes one 256 x 256 fp32 tile with
// tcgen05.mma.cta_group::2: each CTA holds 128 rows of A, 128 of the 256 B
// columns and 128 accumulator rows in its own TMEM.
constexpr int kBM = 128;         // accumulator rows per CTA = TMEM lanes
constexpr int kPairM = 256;      // rows per pair tile
constexpr int kBN = 256;         // columns per tile = TMEM columns per accumulator
constexpr int kBNHalf = 128;     // B columns staged by each CTA of the pair
constexpr int kBK = 64;          // K per pipeline stage: one 128-byte swizzle row of bf16
constexpr int kUmmaK = 16;       // K of one tcgen05.mma kind::f16 instruction
constexpr int kStages = 6;       // TMA -> MMA pipeline depth
// The dX GEMM's tiles are one or two accumulators wide (dx_plan). Two (256 x
// 512): each K block of A feeds two MMAs, so the operand stream per flop into
// shared memory is 3/4 of a 256 x 256 tile's, and a wave of tiles covers all
// of H with half as many W column blocks re-read per row block; both of the
// pair's 256-column accumulators hold one tile (the epilogue does not overlap
// the next tile's main loop), with kDxStages stages of 48 KB per CTA. One: the
// other GEMMs' kStages stages of 32 KB in the same shared memory.
constexpr int kDxWide = 2;
constexpr int kDxStages = 4;
static_assert(kDxStages * (1 + kDxWide) == kStages * 2, "both stage rings fill the same bytes");
constexpr int kMaxSplits = 16;   // split-K limit of the dX GEMM
// Widest vocabulary chunk of the backward by default: dZ is formed, used by
// the dX GEMM and the dW GEMM one chunk of at most this many columns at a
// time, so its buffer holds M x V_c instead of M x V.
constexpr int64_t kVChunkDefault = 32768;
// By default the vocabulary is walked in one piece when dZ for the whole of it
// takes at most this many bytes: chunks then save little memory and their
// launch tails cost most (few masked rows per launch).
constexpr int64_t kDzWholeMaxBytes = int64_t(1) << 30;

constexpr uint32_t kTileABytes = kBM * kBK * 2;       // 16 KB per CTA
constexpr uint32_t kTileBBytes = kBNHalf * kBK * 2;   // 16 KB per CTA
constexpr uint32_t kStageBytes = kTileABytes + kTileBBytes;
// Epilogue staging: each of the 4 epilogue warps double-buffers one 32-row x
// 128-byte sub-tile (32 fp32 or 64 bf16 columns) for its TMA stores.
constexpr uint32_t kEpiBufBytes = 32 * 128;
constexpr uint32_t kEpiBytes = 4 * 2 * kEpiBufBytes;   // 32 KB

// ---- kernel ids (trace + device error "where") --------------------------------
enum KernelId : int32_t {
  KID_MASK_COMPACT = 0,
  KID_GATHER = 1,
  KID_LMHEAD_FWD = 2,
  KID_LSE_COMBINE = 3,
  KID_SEQ_REDUCE = 4,
  KID_BOUND_COEFFS = 5,
  KID_LMHEAD_DZ = 6,
  KID_DX_GEMM = 7,
  KID_DX_REDUCE = 8,
  KID_DW_GEMM = 9,
  KID_GROUP_ADV = 10,
  KID_SELFTEST_WAIT = 11,
  KID_VRPO_COEFFS = 12,
  KID_DZ_FROM_LOGITS = 13,
  KID_XM_TRANSPOSE = 14,
  KID_COUNT = 15
};

BGPO_HD int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }
BGPO_HD int64_t round_up(int64_t a, int64_t b) { return ceil_div(a, b) * b; }

// Column tiles of the dX GEMM for `tiles_h` hidden-size blocks of kBN columns,
// `wide` of them per tile.
BGPO_HD int64_t dx_tiles_n(int64_t tiles_h, int wide = kDxWide) { return ceil_div(tiles_h, wide); }

// Row groups of the forward and dZ GEMMs. Consecutive tiles share a vocabulary
// tile of W, so every wave of tiles reads all of Xm's row blocks; once Xm
// outgrows what L2 keeps from one wave to the next (measured at the 8B head:
// no re-reads up to 36 MB, 3.5-5 reads per launch at 56-64 MB), the row blocks
// are walked in groups of at most kXmGroupBytes of Xm, each group over the
// whole vocabulary: W is then read once per group instead of Xm once per wave.
constexpr int64_t kXmGroupMinBytes = int64_t(52) << 20;
constexpr int64_t kXmGroupBytes = int64_t(40) << 20;
BGPO_HD int64_t xm_row_groups(int64_t tiles_m, int64_t H) {
  const int64_t bytes = tiles_m * kPairM * H * 2;
  if (tiles_m <= 1 || bytes <= kXmGroupMinBytes) return 1;
  const int64_t g = ceil_div(bytes, kXmGroupBytes);
  return g < tiles_m ? g : tiles_m;
}

// Tile (row block, vocabulary tile) of unit u of the forward and dZ GEMMs with
// `groups` row groups: group g holds row blocks [g tm / G, (g + 1) tm / G),
// its units follow those of the groups before it, and consecutive units of a
// group share a vocabulary tile.
// (32-bit arithmetic: at most 2^14 row blocks times 2^16 vocabulary tiles)
BGPO_HD void row_group_tile(int64_t u, int64_t tiles_m, int64_t tiles_n, int64_t groups,
                            int64_t* m_blk, int64_t* n_blk) {
  const uint32_t tm = (uint32_t)tiles_m, tn = (uint32_t)tiles_n, ng = (uint32_t)groups;
  uint32_t r0 = 0, rows = tm, local = (uint32_t)u;
  if (ng > 1) {
    uint32_t g = 0, end = tm / ng;   // end = (g + 1) tm / ng
    while (g + 1 < ng && end * tn <= local) {
      r0 = end;
      ++g;
      end = (g + 1) * tm / ng;
    }
    rows = end - r0;
    local -= r0 * tn;
  }
  *n_blk = local / rows;
  *m_blk = r0 + local % rows;
}

// Split-K count of the dX GEMM (K = vocabulary) for `mb` pair row blocks times
// `tiles_n` column tiles on `num_pairs` CTA pairs: the smallest s whose
// wave-quantised time ceil(tiles*s/pairs)/s is within 8% of the ideal
// tiles/pairs, else the best s. s * mb never exceeds `row_block_cap`, which
// bounds the partial buffer independently of the SM count.
// Integers only: every lane of the warp that makes the plan runs this, at the start of
// the backward, and 16 rounds of 64-bit and double-precision divisions took 3 us.
BGPO_HD int dx_splits(int64_t mb, int64_t tiles_n, int num_pairs, int64_t k_blocks,
                      int64_t row_block_cap) {
  if (mb * tiles_n <= 0 || num_pairs <= 0) return 1;
  const uint32_t tiles = (uint32_t)(mb * tiles_n), pairs = (uint32_t)num_pairs;
  uint32_t smax = kMaxSplits;
  if (k_blocks < (int64_t)smax) smax = k_blocks > 0 ? (uint32_t)k_blocks : 1;
  const uint32_t room = (uint32_t)row_block_cap / (uint32_t)mb;
  if (room < smax) smax = room > 0 ? room : 1;
  const uint32_t q = tiles / pairs, r = tiles % pairs;
  uint32_t full = 0, rest = 0;       // tiles * s = full * pairs + rest
  uint32_t best = 1, best_waves = 0;
  for (uint32_t s = 1; s <= smax; ++s) {
    full += q;
    rest += r;
    if (rest >= pairs) { rest -= pairs; ++full; }
    const uint32_t waves = full + (rest ? 1u : 0u);
    // waves / s <= 1.08 tiles / pairs
    if ((uint64_t)waves * pairs * 25 <= (uint64_t)tiles * s * 27) return (int)s;
    if (best_waves == 0 || waves * best < best_waves * s) { best = s; best_waves = waves; }
  }
  return (int)best;
}

// Width of the backward's vocabulary chunks. `request` 0 asks for the
// default: one chunk when dW pairing keeps the whole vocabulary's dZ anyway or
// when that dZ (m_pad rows of roundup(V, 64) bf16 values) fits
// kDzWholeMaxBytes, else the V columns split into ceil(V / kVChunkDefault)
// chunks of equal width rounded up to a tile. A positive request is a multiple
// of kBN (the host validates it). A width of V or more is a single chunk.
BGPO_HD int64_t vocab_chunk_width(int64_t V, int64_t request, bool pair_dw, int64_t m_pad) {
  int64_t w;
  if (request > 0) {
    w = request;
  } else if (pair_dw || 2 * m_pad * round_up(V, 64) <= kDzWholeMaxBytes) {
    w = V;
  } else {
    const int64_t n = ceil_div(V, kVChunkDefault);
    w = round_up(ceil_div(V, n), kBN);
  }
  return w >= V ? round_up(V, 64) : w;
}

// Geometry derived from the problem sizes (host and device agree on it).
struct Geometry {
  int64_t B, P, R, H, V;
  int64_t m_cap;      // B * R: most masked rows a sample can have
  int64_t m_pad;      // m_cap rounded up to a pair tile of rows
  int64_t v_pad;      // V rounded up to 64 (row pitch of the kept logits)
  int64_t n_vt;       // vocabulary tiles of kBN columns
  int64_t tiles_h;    // hidden-size tiles of kBN columns
  int64_t kb_v;       // K blocks of kBK over the vocabulary
  int64_t vc;         // vocabulary chunk width of the backward (v_pad when one chunk)
  int64_t n_vc;       // vocabulary chunks: chunk c covers [c vc, min(V, (c + 1) vc))
  int64_t kb_vc_min;  // K blocks of kBK of the narrowest chunk (the dX split bound)
};

BGPO_HD Geometry make_geometry(int64_t B, int64_t P, int64_t R, int64_t H, int64_t V,
                               int64_t vchunk_request = 0, bool pair_dw = false) {
  Geometry g;
  g.B = B; g.P = P; g.R = R; g.H = H; g.V = V;
  g.m_cap = B * R;
  g.m_pad = round_up(g.m_cap, kPairM);
  g.v_pad = round_up(V, 64);
  g.n_vt = ceil_div(V, kBN);
  g.tiles_h = ceil_div(H, kBN);
  g.kb_v = ceil_div(V, kBK);
  g.vc = vocab_chunk_width(V, vchunk_request, pair_dw, g.m_pad);
  g.n_vc = ceil_div(V, g.vc);
  const int64_t last = V - (g.n_vc - 1) * g.vc;
  g.kb_vc_min = ceil_div(last < g.vc ? last : g.vc, kBK);
  return g;
}

// Vocabulary range [v0, v1) of backward chunk c.
BGPO_HD int64_t chunk_begin(const Geometry& g, int64_t c) { return c * g.vc; }
BGPO_HD int64_t chunk_end(const Geometry& g, int64_t c) {
  const int64_t e = (c + 1) * g.vc;
  return e < g.V ? e : g.V;
}

// Device workspace layout. Every region starts on a 1024-byte boundary (TMA
// tiles with 128-byte swizzle want 1024-byte aligned bases).
struct WsLayout {
  size_t err;        // int32[16]: the fields of ErrField
  size_t t;          // float[B]    t_{b,j}
  size_t tnum;       // uint32[2B]  T numerator (t = T / D), (low, high) words (several mask rounds)
  size_t seg_off;    // int32[B+1]  first compacted row of each sequence
  size_t rows;       // int32[m_cap] b*R + i of each masked position, ascending
  size_t tgt;        // int32[m_pad] target token of each compacted row
  size_t tgt_logit;  // float[m_pad] z_{r, y_r}
  size_t lse;        // float[m_pad] log-sum-exp of each row's logits
  size_t logp;       // float[m_pad] log p(y_r)
  size_t part;       // float2[m_pad * n_vt] (max, sum-exp) per (row, vocab tile)
  size_t xm;         // bf16[m_pad * H] gathered masked hidden states
  size_t fwd_bytes;  // end of the regions a forward pass uses (err .. xm); the same under
                     // every flag
  size_t xmT;        // bf16[H * dz_rows] the same, transposed (the dW GEMM's K-major operand)
  size_t dz;         // bf16[dz_rows * dz_cols] dL/dz of the current sample (and of a pending
                     // one): one vocabulary chunk at a time, or the whole vocabulary
  size_t dz_rows;    // m_pad, or 2 m_pad when the dW GEMM pairs samples
  size_t dz_cols;    // vc when the buffer holds one chunk, v_pad when it holds them all
  bool dz_chunk_local;  // chunk c is formed at column 0 (else at column c vc)
  size_t dxp;        // float[dxp_elems] split-K partials of dX
  size_t dxp_elems;
  size_t zc;         // float[m_pad * v_pad] logits kept by the forward (last region)
  size_t zc_bytes;   // 0 when the forward keeps no logits
  size_t total;
};

BGPO_HD size_t align_ws(size_t x) { return (x + 1023) & ~(size_t)1023; }

// Pair row blocks (256 rows) the split-K partial buffer holds, which bounds the
// splits s of a sample with mb row blocks to s * mb <= cap: three splits at the
// largest mb, up to kMaxSplits for small mb (measured: a second split takes
// 6-8% off a dX GEMM whose unsplit tiles leave a last wave 20% full; with
// 256 x 512 tiles, room for a third split took 1.5% off the dX GEMMs of a
// step against room for two).
BGPO_HD int64_t dxp_row_block_cap(const Geometry& g) {
  const int64_t mb_max = g.m_pad / kPairM;
  const int64_t small = 4 * mb_max < 4 * kMaxSplits ? 4 * mb_max : 4 * kMaxSplits;
  int64_t cap = 3 * mb_max > small ? 3 * mb_max : small;
  return cap > kMaxSplits ? cap : kMaxSplits;
}

// Tile width and split count of the dX GEMM of a sample with M masked rows (the
// same for every chunk of the sample): 256 x 512 tiles split by dx_splits (the usual
// plan), unless another allowed pair of the two (dx_allowed) is estimated to take at
// least 5% less (dx_cost). That is so where a split's K loop is short against its
// epilogue and its partials, and where H leaves a second accumulator empty. GEMM and
// reduction, usual plan -> now, in us: M 283, H 152, V 137580: 152 -> 83; M 4429, H
// 104, V 84350: 221 -> 176; M 309, H 1024, V 8192: 23.4 -> 17.2; M 5281, H 2712, V 975
// (3 splits -> unsplit): 119 -> 66; M 107, H 808, V 14743 in chunks of 1,024: 185 ->
// 131; M 521, H 528, V 115266 in chunks of 16,384: 352 -> 166. Over 36 shapes drawn
// from H 64 .. 4096, V 512 .. 152,064, 1 .. 16,384 response rows the geometric mean is
// 1.26 times faster and none is slower by more than 1%.
struct DxPlan {
  int32_t wide, splits;
};

// K blocks of the longest of s splits, summed over the chunks: the last chunk may be
// much narrower than the others (V 115266 in chunks of 16,384 leaves one of 578).
// Charging every chunk the narrowest one's blocks made two splits look cheap there:
// GEMM and reduction 338 -> 207 us at 521 rows of 528, V 55165 in chunks of 13,568
// 566 -> 459 at 3,321 rows of 1,472, V 108141 in chunks of 15,360 337 -> 213 at 105
// rows of 3,112.
BGPO_HD uint32_t dx_kblocks(const Geometry& g, int s) {
  const uint32_t n = (uint32_t)s, full = (uint32_t)(g.vc / kBK);
  const uint32_t last = (uint32_t)ceil_div(g.V - (g.n_vc - 1) * g.vc, kBK);
  return (uint32_t)(g.n_vc - 1) * ((full + n - 1) / n) + (last + n - 1) / n;
}

// Estimated cycles of the GEMM over all chunks and of the split reduction. The
// constants are fits to 15 shapes times 10 forced plans, measured on a GB300 at
// about 2 GHz: a K block takes 590 cycles at one accumulator and 1,030 at two, a
// launch 16,000 and 19,200 beside its K loops; at two, each further wave shows its
// epilogue; unsplit tiles, which add into dX themselves, take 12,000 and 17,400
// longer; partials stream at 3,100 bytes per cycle.
BGPO_HD float dx_cost(const Geometry& g, int64_t M, int num_pairs, int wide, int s) {
  const uint32_t units =
      (uint32_t)(ceil_div(M, kPairM) * dx_tiles_n(g.tiles_h, wide)) * (uint32_t)s;
  const float waves = (float)((units + (uint32_t)num_pairs - 1) / (uint32_t)num_pairs);
  float launch = wide == 1 ? 16000.f : 9200.f + 10000.f * waves;
  if (s == 1) launch += wide == 1 ? 12000.f : 17400.f * waves;
  const float kloops = waves * (float)dx_kblocks(g, s) * (wide == 1 ? 590.f : 1030.f);
  // passes over M x H floats: each partial once and dX twice in the reduction, and
  // each partial twice for every chunk that adds to it
  const float passes = (float)(s + 2 + 2 * s * (int)(g.n_vc - 1));
  const float reduce = s == 1 ? 2600.f : 4000.f + passes * (float)M * (float)g.H * (4.f / 3100.f);
  return kloops + launch * (float)g.n_vc + reduce;
}

// Candidate i of the 32: a tile width and a split count the split buffer has room for.
BGPO_HD DxPlan dx_candidate(int i) { return DxPlan{1 + (i & 1), 1 + (i >> 1)}; }
BGPO_HD bool dx_fits(const Geometry& g, int64_t M, const DxPlan& c) {
  return c.splits <= g.kb_vc_min && c.splits * ceil_div(M, kPairM) <= dxp_row_block_cap(g);
}

// The split count that the dX GEMM and the split reduction after it run with, from the
// word the backward's first kernel left. Both take it from here, so that the reduction
// sums exactly what the GEMM stored. A word that holds no count for this sample (a
// damaged workspace: dx_plan always fits) makes an unsplit GEMM, which adds straight
// into dX, and `*fits` false. (Any tile width the other word may hold is one of the two
// that work: dx_wide_stored. The reduction need not know it.)
BGPO_HD int dx_splits_stored(const Geometry& g, int64_t M, int32_t splits, bool* fits) {
  *fits = splits >= 1 && splits <= kMaxSplits && dx_fits(g, M, DxPlan{kDxWide, splits});
  return *fits ? splits : 1;
}
BGPO_HD int dx_wide_stored(int32_t wide) { return wide == 1 ? 1 : kDxWide; }

// The usual plan of M > 0 rows.
BGPO_HD DxPlan dx_plan_usual(const Geometry& g, int64_t M, int num_pairs) {
  return DxPlan{kDxWide, dx_splits(ceil_div(M, kPairM), dx_tiles_n(g.tiles_h), num_pairs,
                                   g.kb_vc_min, dxp_row_block_cap(g))};
}

// Most K blocks that one accumulator adds up in a plan of s splits.
BGPO_HD uint32_t dx_chain(const Geometry& g, int s) {
  const uint32_t kb = (uint32_t)ceil_div(g.vc < g.V ? g.vc : g.V, kBK);
  return (kb + (uint32_t)s - 1) / (uint32_t)s;
}

// Whether candidate c may take the usual plan's place: not with fewer splits, unless
// the chains stay within kDxShortChain K blocks. The rounding error of an fp32
// accumulator grows with its chain: dX against the 64-bit product of the same bf16
// dZ and W, H 3584, V 152064, 5 chunks: 2.8e-6 with 13 splits, 6.4e-6 with 6, 1.9e-5
// with 2, 3.6e-5 unsplit. Beside the 1-2e-3 that dZ's rounding to bf16 makes, chains
// of up to 476 blocks moved dX's whole error by -0.1 to +0.4%; over 48 shapes with
// chains of up to 16 blocks instead of 1 to 10 it moved by 6e-6 of itself in the mean
// (-1.5e-4 to 2.0e-4, larger in 24 of them).
// What fewer splits would give otherwise: H 3584, V 152064, 5 chunks: 1182 -> 897 us at
// 1,259 rows, 3826 -> 3401 at 4,893; H 4096, V 126464, 4 chunks: 703 -> 691 at 951
// rows, 2906 -> 2841 at 4,286.
constexpr uint32_t kDxShortChain = 16;
BGPO_HD bool dx_allowed(const Geometry& g, int64_t M, const DxPlan& usual, const DxPlan& c) {
  return dx_fits(g, M, c) && (c.splits >= usual.splits || dx_chain(g, c.splits) <= kDxShortChain);
}

// The plan, given the allowed candidate of least cost.
BGPO_HD DxPlan dx_plan_of(const Geometry& g, int64_t M, int num_pairs, const DxPlan& usual,
                          const DxPlan& best, float cost) {
  return cost <= 0.95f * dx_cost(g, M, num_pairs, usual.wide, usual.splits) ? best : usual;
}

// The rule one candidate after the other. The device takes dx_plan_warp, one candidate
// per lane; tests hold that against this.
BGPO_HD DxPlan dx_plan(const Geometry& g, int64_t M, int num_pairs) {
  if (M <= 0) return DxPlan{kDxWide, 1};
  const DxPlan usual = dx_plan_usual(g, M, num_pairs);
  DxPlan best = usual;   // always a candidate
  float cost = dx_cost(g, M, num_pairs, best.wide, best.splits);
  for (int i = 0; i < 2 * kMaxSplits; ++i) {
    const DxPlan c = dx_candidate(i);
    if (!dx_allowed(g, M, usual, c)) continue;
    const float t = dx_cost(g, M, num_pairs, c.wide, c.splits);
    if (t < cost) { cost = t; best = c; }
  }
  return dx_plan_of(g, M, num_pairs, usual, best, cost);
}

// `keep_logits` appends the fp32 logit region. `pair_dw` doubles the rows of
// dZ and the columns of Xm^T: the rows of an even sample wait there for the
// dW GEMM of the next sample, whose rows follow them; its dZ rows then span
// the whole vocabulary. Otherwise dZ holds one vocabulary chunk.
BGPO_HD WsLayout make_ws_layout(const Geometry& g, bool keep_logits, bool pair_dw) {
  WsLayout L;
  size_t o = 0;
  L.dz_rows = (pair_dw ? 2 : 1) * (size_t)g.m_pad;
  L.dz_chunk_local = !pair_dw && g.n_vc > 1;
  L.dz_cols = L.dz_chunk_local ? (size_t)g.vc : (size_t)g.v_pad;
  L.err = o;       o = align_ws(o + 64);
  L.t = o;         o = align_ws(o + 4 * (size_t)g.B);
  L.tnum = o;      o = align_ws(o + 8 * (size_t)g.B);
  L.seg_off = o;   o = align_ws(o + 4 * (size_t)(g.B + 1));
  L.rows = o;      o = align_ws(o + 4 * (size_t)g.m_cap);
  L.tgt = o;       o = align_ws(o + 4 * (size_t)g.m_pad);
  L.tgt_logit = o; o = align_ws(o + 4 * (size_t)g.m_pad);
  L.lse = o;       o = align_ws(o + 4 * (size_t)g.m_pad);
  L.logp = o;      o = align_ws(o + 4 * (size_t)g.m_pad);
  L.part = o;      o = align_ws(o + 8 * (size_t)g.m_pad * (size_t)g.n_vt);
  L.xm = o;        o = align_ws(o + 2 * (size_t)g.m_pad * (size_t)g.H);
  L.fwd_bytes = o;
  L.xmT = o;       o = align_ws(o + 2 * (size_t)g.H * L.dz_rows);
  L.dz = o;        o = align_ws(o + 2 * L.dz_rows * L.dz_cols);
  L.dxp_elems = (size_t)dxp_row_block_cap(g) * kPairM * (size_t)g.H;
  L.dxp = o;       o = align_ws(o + 4 * L.dxp_elems);
  L.zc_bytes = keep_logits ? 4 * (size_t)g.m_pad * (size_t)g.v_pad : 0;
  L.zc = keep_logits ? o : 0;
  o = align_ws(o + L.zc_bytes);
  L.total = o;
  return L;
}

// Indices into the int32 error word:
//   ERR_STATUS, ERR_WHERE  the device error (bgpo_get_device_error)
//   ERR_SAMPLE, ERR_M      the sample j the workspace holds and its masked rows
//   ERR_LOGITS    1 while the logit region holds the current sample's logits
//                 (set by the forward that wrote them, cleared by the masking of
//                 a new sample and by a forward that keeps none)
//   ERR_DX_SPLITS, ERR_DX_WIDE  the plan of the current sample's dX GEMM (DxPlan), set by
//                 the backward's first kernel
//   ERR_PEND      pend_tag(j) while sample j's dZ and Xm^T rows wait for the dW
//                 GEMM of sample j + 1, else -1
//   ERR_PEND_OFF  the row at which sample j + 1's dZ and Xm^T rows start: M_j
//                 rounded up to a K block
//   ERR_ROW_OFF   set by the masking: the first dZ / Xm^T row of the current
//                 sample (ERR_PEND_OFF when it pairs with the pending sample,
//                 else 0)
//   ERR_PAIRED    set by the masking: 1 when the current sample pairs
//   ERR_DW_K0     set by the backward before its dW GEMM: the first K row that
//                 GEMM adds (0 while the partner is pending, ERR_ROW_OFF once
//                 an earlier backward of this sample has added the partner)
enum ErrField : int {
  ERR_STATUS = 0, ERR_WHERE = 1, ERR_SAMPLE = 2, ERR_M = 3, ERR_LOGITS = 4, ERR_DX_SPLITS = 5,
  ERR_PEND = 6, ERR_PEND_OFF = 7, ERR_ROW_OFF = 8, ERR_PAIRED = 9, ERR_DW_K0 = 10,
  ERR_DX_WIDE = 11
};

// Tag of a pending sample (n_t < 2^16): neither -1 nor a small integer that
// memory not yet written by this library is likely to hold.
BGPO_HD int32_t pend_tag(int32_t j) { return (int32_t)(0x5EED0000u | (uint32_t)j); }

// First dZ / Xm^T row of the current sample, clamped to the room the layout
// has for a pending sample (none without pairing) and to a K block.
BGPO_HD int64_t row_offset(int32_t stored, int64_t dz_rows, int64_t m_pad) {
  const int64_t room = dz_rows - m_pad;
  int64_t off = stored < 0 ? 0 : (int64_t)stored;
  if (off > room) off = room;
  return off & ~(int64_t)(kBK - 1);
}

}  // namespace bgpo
