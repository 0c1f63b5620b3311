// fewrow.cu -- tcgen05 GEMM for launches of few rows, D^T[N, rows] =
// W[N, K] * A[rows, K]^T: the products of gemm.cu where that kernel's
// 128 x 256 output tiles would leave most SMs without one.
//
// The weight rows are the M side of the product (128 per tile) and a group of
// 16 to 256 activation rows its N side, so a launch over a handful of rows
// streams each weight tile once and multiplies no padding beyond 16 rows, and
// the K range of a tile is cut over the CTAs of a cluster (1, 2, 4 or 8)
// until the tiles cover the SMs.  The CTAs of a cluster exchange their
// partial tiles through distributed shared memory (one bulk copy per pair of
// CTAs): CTA r sums a 1/S share of the group's rows over all S partials in
// rank order and finishes them (a fixed order: a row's result depends on the
// split alone, never on the rows beside it).
//
// CTA = 10 warps, one CTA per SM, persistent over (column tile, row group):
//   warp 0      TMA producer: weight tiles 64 x 128 (SwiGLU: one of the gate and
//               one of the up rows), activation tiles 64 x nb (128-byte swizzle)
//   warp 1      TMEM owner + single-thread tcgen05.mma issuer (M = 128, N = nb)
//   warps 2..9  epilogue, two groups of four (one per TMEM lane quarter): a
//               lane is an output column, its 16 registers 16 activation rows,
//               so a warp's loads and stores run along rows.  Weight tiles of
//               rotated columns are loaded (one 5-D box) in an order that puts
//               both columns of a pair in one warp, 16 lanes apart.
// What a row needs besides its products (RMSNorm scale, position, cache row)
// is gathered into shared memory while the products run.
// A decode step's rows come as bf16 pairs hi + lo (hi = bf16(x),
// lo = bf16(x - hi)) in two halves of the group: the weights bound such a
// launch, so the second half of the N side costs nothing and the activations
// carry 16 significant bits instead of 8 (Qwen2.5-7B and Llama-3-8B, 4 layers:
// the largest logit's error against 64 bits 2e-3 with single bf16 rows).
// Where a residual product's splits take whole 256-row groups, the CTAs of two
// column tiles form a pair (cta_group::2): one M = 256 product, each CTA with
// its own weight rows and half of the activation rows, 32 KB instead of 48 KB a
// k-block into its shared memory (down projection of 512 rows 76 -> 67 us, of 256
// rows 50 -> 47 us).  A pair's CTA 0 issues the products; all else stays per CTA.
// Without a split two TMEM accumulators let the epilogue of one tile overlap
// the main loop of the next; with a split the partials take the ring's
// memory, so the next tile's loads begin when the sums are done.
//
// Programmatic dependent launch: the prologue, and with one row group the
// first ring of weight tiles, run while the previous kernel finishes.
// What bounds it: with up to ~64 rows the weights' HBM bytes, above that the
// operands' way into shared memory (about 630 cycles per 48 KB k-block) and the
// tiles' ends.  Measured against the 128 x 256-tile kernel with K splits
// chained through global memory, per launch (CUDA events): Qwen2.5-7B layer,
// a 256-row chunk: q/k/v 43 -> 28 us, O 33 -> 27 us, down 71 -> 48 us (pairs,
// four splits, partials in two rounds), gate/up 75 -> 66 us; a 512-slot cache:
// down 84 -> 67 us; the 512-slot tiny model's pass 78 -> 60 us.
// Decode steps: of one to four sequences the smaller products run as GEMVs
// (gemv.cuh; a launch here waits out its cluster's set-up and exchange: one
// Qwen2.5-7B row q/k/v 20 us against 15, O 19 against 14.5); gate/up 57 -> 50 us
// (271 MB) and the LM head 186 -> 159 us (1.09 GB, 6.8 TB/s) against such GEMVs.
// 16 Llama-3-8B rows against one 128-row tile per sequence: 4.25 -> 0.71 ms.
#include "fewrow.cuh"

#include <algorithm>
#include <atomic>
#include <cmath>

namespace cc {

namespace {

constexpr int BM = 128, BK = 64;
constexpr int kEpiWarps = 8;
constexpr int kThreads = 64 + kEpiWarps * 32;
constexpr int kMaxBatch = 1024;
constexpr int W_BYTES = BM * BK * 2;          // weight tile of a stage
constexpr int kRingBytes = 192 * 1024;
constexpr int kMaxStages = 10;
constexpr int kBlock = 16;                    // activation rows of one TMEM load
constexpr int kMaxRows = 256;                 // activation rows of a group at most
constexpr size_t kPrefixBytes = ((kMaxBatch + 1) * sizeof(int) + 15) & ~size_t(15);

// What the epilogue needs of each row of a group.
struct RowTab {
  float rs[kMaxRows];          // RMSNorm scale of an unnormalised A row, else 1
  uint32_t pos[kMaxRows];      // projections: position
  long long dst[kMaxRows];     // K/V cache row (head-major: first head's vector); -1: none
  int tok[kMaxRows];           // RESID_LOGIT: the row's token
};

constexpr int kOffTab = kRingBytes;                              // [2]
constexpr int kOffRed = kOffTab + 2 * (int)sizeof(RowTab);       // float2 [2][4][kMaxRows]
constexpr int kOffBar = kOffRed + 2 * 4 * kMaxRows * 8;
constexpr int kOffPrefix = kOffBar + 512;
constexpr int kSmemBytes = 1024 /*align slack*/ + kOffPrefix + (int)kPrefixBytes;
static_assert(kSmemBytes <= 232448, "shared memory");

// Weight tiles of a stage and accumulators of an output tile.
__host__ __device__ constexpr int w_tiles(int epi) { return epi == EPI_SWIGLU ? 2 : 1; }
// (rows: activation rows that a CTA stages)
__host__ __device__ constexpr int stage_bytes(int wt, int rows) { return wt * W_BYTES + rows * BK * 2; }
__host__ __device__ constexpr int stage_count(int wt, int rows) {
  return kRingBytes / stage_bytes(wt, rows) < kMaxStages ? kRingBytes / stage_bytes(wt, rows) : kMaxStages;
}
// A split's exchange in the ring's memory: this CTA's partial rows (of wt * 128
// floats) and the share it finishes from each of the others; in one round of
// the group's nb rows, or in two of half of them.
__host__ __device__ constexpr bool round_fits(int wt, int rows, int S) {
  return (rows + (S - 1) * ((rows + S - 1) / S)) * wt * BM * 4 <= kRingBytes;
}
__host__ __device__ constexpr int split_rounds(int wt, int nb, int S) {   // 0: does not fit
  return round_fits(wt, nb, S) ? 1 : round_fits(wt, nb / 2, S) ? 2 : 0;
}
static_assert(split_rounds(1, 256, 8) == 2 && split_rounds(2, 128, 8) == 2 &&
                  split_rounds(2, 256, 2) == 2 && split_rounds(2, 256, 4) == 0,
              "partial tiles of a split");
// Tensor-memory columns of one accumulator.
__host__ __device__ constexpr int acc_cols(int nb) { return nb < 32 ? 32 : nb; }

template <int EPI>
constexpr bool is_proj = EPI == EPI_QROPE || EPI == EPI_BF16 || EPI == EPI_QKV;
template <int EPI>
constexpr bool is_resid = EPI == EPI_RESID_BF16 || EPI == EPI_RESID_F32 || EPI == EPI_RESID_LOGIT;
// Where a projection's tile goes (EPI_QKV: column tiles of Q, then K, then V).
struct ProjTile {
  void *out;
  const __nv_bfloat16 *bias;
  int ldo, N, col0;            // row stride and columns of the destination, first column of the tile
  bool rope, kv, fp8;          // rotated; K/V cache rows; e4m3 codes
  float qscale;
};
template <int EPI>
CC_DEV ProjTile proj_tile(const GemmParams &p, int nt) {
  if constexpr (EPI == EPI_QKV) {
    const int nq = p.n_q_tiles, nk = p.n_k_tiles;
    if (nt < nq) return {p.out, p.bias, p.ldo, p.ldo, nt * BM, true, false, false, 1.f};
    if (nt < nq + nk)
      return {p.out_k, p.bias_k, p.ldo_kv, p.ldo_kv, (nt - nq) * BM, true, true, p.kv_fp8 != 0,
              p.k_qscale};
    return {p.out_v, p.bias_v, p.ldo_kv, p.ldo_kv, (nt - nq - nk) * BM, false, true, p.kv_fp8 != 0,
            p.v_qscale};
  } else {
    return {p.out, p.bias, p.ldo, p.N, nt * BM, EPI == EPI_QROPE, p.kv_dest != 0, p.kv_fp8 != 0,
            EPI == EPI_QROPE ? p.k_qscale : p.v_qscale};
  }
}
// First column (relative to the tile) of lane quarter q's 16 pairs, partner
// columns `half` further: whole heads per tile.
CC_DEV int pair_base(int q, int head_dim) {
  return head_dim == 128 ? 16 * q : 64 * (q >> 1) + 16 * (q & 1);
}

// This lane's output column (or pair of columns) of the current tile.
struct LaneCol {
  int c0, c1;                  // columns (c1: the pair's second)
  bool ok;                     // c0 exists
  float b0, b1;                // bias
  float gain;                  // norm or head gain of c0
  unsigned long long turn;     // RoPE angle of the pair
  size_t e0, e1;               // element offset of the columns in a destination row
  int row_mul;                 // elements between destination rows
};

// Fills tab rows [0, max(nv, 1)) for the group whose first workspace row is
// row0: thread t of the epilogue's 256 takes row t.
template <int EPI>
CC_DEV void fill_rows(const GemmParams &p, RowTab &tab, int t, int nv, size_t row0) {
  if (t >= nv && t > 0) return;
  const bool live = t < nv;
  const size_t row = row0 + t;
  float rs = 1.f;
  if constexpr (!is_resid<EPI>) {
    if (live && p.row_ss) {
      const float *pr = p.row_ss + row * p.n_ss;
      float ss = 0.f;
#pragma unroll 8
      for (int k = 0; k < p.n_ss; ++k) ss += pr[k];
      rs = rsqrtf(ss / (float)p.ss_d + p.eps);
    }
  }
  tab.rs[t] = rs;
  if constexpr (is_proj<EPI>) {
    const int gr = live ? (p.rowmap ? p.rowmap[row] : (int)row) : -1;
    uint32_t pos = 0;
    long long dst = -1;
    if (gr >= 0) {
      const int b = gr / p.kv_cap, i = gr - b * p.kv_cap;
      pos = (uint32_t)p.pos[gr];
      if (p.pg.head_major) {
        dst = (long long)b * p.pg.hkv * p.kv_cap + i;
      } else {
        dst = kv_row(p.pg, p.kv_cap, b, i);
        if (dst < 0 && (EPI == EPI_QKV || p.kv_dest)) set_status(p.status, CC_ERR_DEVICE_ARG);
      }
    }
    tab.pos[t] = pos;
    tab.dst[t] = dst;
  }
  if constexpr (EPI == EPI_RESID_LOGIT) {
    int tok = live ? p.tokens[row] : 0;
    if (tok < 0 || tok >= p.vocab) tok = 0;   // reported by the combine
    tab.tok[t] = tok;
  }
}

CC_DEV float bf16_at(const __nv_bfloat16 *p, int i) { return p ? __bfloat162float(p[i]) : 0.f; }

template <int EPI>
CC_DEV LaneCol lane_col(const GemmParams &p, const ProjTile &d, int nt, int q, int lane) {
  LaneCol lc{};
  const int l16 = lane & 15;
  if constexpr (is_proj<EPI>) {
    const int dh = p.head_dim;
    if (d.rope) {
      lc.c0 = d.col0 + pair_base(q, dh) + l16;
      lc.c1 = lc.c0 + (dh >> 1);
      lc.turn = p.turns[lc.c0 % dh];
    } else {
      lc.c0 = lc.c1 = d.col0 + 32 * q + lane;
    }
    lc.ok = lc.c0 < d.N;
    if (lc.ok) {
      lc.b0 = bf16_at(d.bias, lc.c0);
      lc.b1 = bf16_at(d.bias, lc.c1);
    }
    const bool hm = d.kv && p.pg.head_major;
    lc.row_mul = hm ? dh : d.ldo;
    lc.e0 = hm ? (size_t)(lc.c0 / dh) * p.kv_cap * dh + lc.c0 % dh : (size_t)lc.c0;
    lc.e1 = hm ? (size_t)(lc.c1 / dh) * p.kv_cap * dh + lc.c1 % dh : (size_t)lc.c1;
  } else {
    lc.c0 = nt * BM + 32 * q + lane;
    lc.ok = lc.c0 < p.N;
    if (lc.ok) {
      if constexpr (EPI == EPI_RESID_LOGIT) lc.gain = bf16_at(p.head_gain, lc.c0);
      else if (is_resid<EPI> && p.norm_out) lc.gain = bf16_at(p.norm_gain, lc.c0);
    }
  }
  return lc;
}

// One value as the next product's operand, bf16 or fp16, without a branch: the
// batches of rows below keep their arithmetic free of control flow, so that
// rows overlap.
CC_DEV uint16_t act_bits(float y, bool f16) {
  const uint16_t h = __half_as_ushort(__float2half_rn(y));
  const uint16_t b = __bfloat16_as_ushort(__float2bfloat16_rn(y));
  return f16 ? h : b;
}
// N values y[k] to out + at[k] where live[k]: one branch each for the fp16
// range report and (lo > 0) the remainders bf16(y - hi) at that offset.
template <bool RP, int N>
CC_DEV void store_acts(uint16_t *out, const size_t (&at)[N], const float (&y)[N],
                       const bool (&live)[N], bool f16, int lo, unsigned *status) {
  uint16_t bits[N];
#pragma unroll
  for (int k = 0; k < N; ++k) bits[k] = act_bits(y[k], f16);
#pragma unroll
  for (int k = 0; k < N; ++k)
    if (live[k]) out[at[k]] = bits[k];
  if (f16) {
    bool over = false;
#pragma unroll
    for (int k = 0; k < N; ++k) over |= live[k] && f16_overflow(y[k]);
    if (over) set_status(status, CC_ERR_RANGE);
  }
  if (lo > 0) {
#pragma unroll
    for (int k = 0; k < N; ++k)
      if (live[k]) {
        const float hi = __bfloat162float(__ushort_as_bfloat16(bits[k]));
        out[at[k] + lo] = __bfloat16_as_ushort(
            __float2bfloat16_rn(RP ? pair_rest(y[k], hi) : y[k] - hi));
      }
  }
}

// Sums of 16 rows over the warp's 32 lanes: lane l returns the sum of row
// (l >> 1) & 15 with the row bits in the order the halving leaves them
// (row16_of).
CC_DEV float rows_sum(float (&v)[16], int lane) {
#pragma unroll
  for (int w = 8, o = 16; w >= 1; w >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int j = 0; j < w; ++j) {
      const float keep = up ? v[j + w] : v[j], send = up ? v[j] : v[j + w];
      v[j] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, o);
    }
  }
  return v[0] + __shfl_xor_sync(0xFFFFFFFFu, v[0], 1);
}
CC_DEV int row16_of(int lane) { return (lane >> 1) & 15; }   // bit 4 of the lane: row bit 3, ...

// Rows J .. J + 8 of finish_block for the projections and SwiGLU: no branch
// between the rows, so that their arithmetic overlaps.
template <int EPI, bool RP, int J>
CC_DEV void finish_rows8(const GemmParams &p, const ProjTile &d, const LaneCol &lc,
                         const RowTab &tab, const float (&v)[16], const float (&u)[16], int r0,
                         int n, size_t row0, int lane, bool dry) {
  const bool f16 = p.out_f16 && !(is_proj<EPI> && d.kv);
  const int lo = is_proj<EPI> && d.kv ? 0 : RP ? p.row_pairs * p.ldo : p.out_split ? p.N : 0;
  size_t at[8];
  float y[8];
  bool live[8];
  if constexpr (EPI == EPI_SWIGLU) {   // v: gate, u: up
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float rs = tab.rs[r0 + J + j];
      y[j] = silu_as<false>(v[J + j] * rs) * (u[J + j] * rs);
      at[j] = (row0 + r0 + J + j) * p.ldo + lc.c0;
      live[j] = !dry && lc.ok && J + j < n;
    }
    store_acts<RP, 8>(reinterpret_cast<uint16_t *>(p.out), at, y, live, f16, lo, p.status);
  } else {
    const int hf = lane >> 4;
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
      // rotated: lanes 0-15 take row j, lanes 16-31 row j + 1, each both
      // columns of its pair; else every lane its column of both rows
      float x0 = v[J + j], x1 = v[J + j + 1];
      int ra = r0 + J + j, rb = ra + 1;
      bool la = !dry && lc.ok && J + j < n, lb = la && J + j + 1 < n;
      const float got = __shfl_xor_sync(0xFFFFFFFFu, hf ? x0 : x1, 16);
      const float z0 = hf ? got : x0, z1 = hf ? x1 : got;
      x0 = d.rope ? z0 : x0;
      x1 = d.rope ? z1 : x1;
      la = d.rope && hf ? lb : la;
      lb = d.rope ? la : lb;
      ra += d.rope ? hf : 0;
      rb = d.rope ? ra : rb;
      x0 = fmaf(x0, tab.rs[ra], lc.b0);
      x1 = fmaf(x1, tab.rs[rb], d.rope ? lc.b1 : lc.b0);
      float c, s;
      rope_cs(tab.pos[ra], lc.turn, c, s);
      c = d.rope ? c : 1.f;
      s = d.rope ? s : 0.f;
      y[j] = d.rope ? x0 * c - x1 * s : x0;
      y[j + 1] = d.rope ? x1 * c + x0 * s : x1;
      const long long ta = tab.dst[ra], tb = tab.dst[rb];
      const long long da = d.kv ? ta : (long long)(row0 + ra);
      const long long db = d.kv ? tb : (long long)(row0 + rb);
      at[j] = (size_t)da * lc.row_mul + lc.e0;
      at[j + 1] = (size_t)db * lc.row_mul + (d.rope ? lc.e1 : lc.e0);
      live[j] = la && (ta >= 0 || !d.kv);   // a bad page has no cache row
      live[j + 1] = lb && (tb >= 0 || !d.kv);
    }
    if (d.fp8) {
      uint8_t *o = reinterpret_cast<uint8_t *>(d.out);
#pragma unroll
      for (int j = 0; j < 8; j += 2) {
        const uint32_t e = pack_e4m3x2(y[j] * d.qscale, y[j + 1] * d.qscale);
        if (live[j]) o[at[j]] = (uint8_t)e;
        if (live[j + 1]) o[at[j + 1]] = (uint8_t)(e >> 8);
      }
    } else {
      store_acts<RP, 8>(reinterpret_cast<uint16_t *>(d.out), at, y, live, f16, lo, p.status);
    }
  }
}

// Residual and LM-head rows that may still be in HBM, towards L2 while the
// products run: the 64 bytes a warp reads of each of rows [r0, r0 + 16) below end.
template <int EPI>
CC_DEV void prefetch_block(const GemmParams &p, const RowTab &tab, int r0, int end, size_t row0,
                           int nt, int q, int lane) {
  const int r = r0 + (lane & 15), col = nt * BM + 32 * q;
  if (r >= end || col >= p.N) return;
  const void *a = nullptr;
  if (EPI == EPI_RESID_BF16 && lane < 16)
    a = reinterpret_cast<const __nv_bfloat16 *>(p.resid) + (row0 + r) * p.ld_resid + col;
  if (EPI == EPI_RESID_LOGIT && lane < 16) a = p.head_w + (size_t)tab.tok[r] * p.N + col;
  if (a) asm volatile("prefetch.global.L2 [%0];" ::"l"(a));
}

// Finishes rows r0 .. r0 + n of the group (n <= 16) in this lane's column:
// v[j] is row r0 + j (SwiGLU: the gate, u the up projection).  row0: workspace
// row of the group's first row.  red: per-quarter row sums.  dry: nothing is
// stored (the code alone runs).
template <int EPI, bool RP>
CC_DEV void finish_block(const GemmParams &p, const ProjTile &d, const LaneCol &lc,
                         const RowTab &tab, float (&v)[16], const float (&u)[16], int r0, int n,
                         size_t row0, int q, int lane, float2 *red, bool dry) {
  if constexpr (is_proj<EPI> || EPI == EPI_SWIGLU) {
    finish_rows8<EPI, RP, 0>(p, d, lc, tab, v, u, r0, n, row0, lane, dry);
    if (n > 8 || dry) finish_rows8<EPI, RP, 8>(p, d, lc, tab, v, u, r0, n, row0, lane, dry);
  } else if constexpr (EPI == EPI_ARGMAX) {   // the quarter's largest logit and its first column
#pragma unroll 1
    for (int j = 0; j < n; ++j) {
      float m = -INFINITY;
      int mi = 0x7FFFFFFF;
      float x = 0.f;
#pragma unroll
      for (int k = 0; k < 16; ++k)
        if (k == j) x = v[k];
      x *= tab.rs[r0 + j];
      if (lc.ok && x > m) {   // NaN never wins
        m = x;
        mi = lc.c0;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float om = __shfl_xor_sync(0xFFFFFFFFu, m, o);
        const int oi = __shfl_xor_sync(0xFFFFFFFFu, mi, o);
        if (om > m || (om == m && oi < mi)) {
          m = om;
          mi = oi;
        }
      }
      if (lane == 0 && !dry) red[q * kMaxRows + r0 + j] = make_float2(m, __int_as_float(mi));
    }
  } else {   // residual adds, optionally fused with the next norm or with the logit head
    // every load first, from addresses clamped into the tile (rows past n and
    // columns past N are never stored), converted only afterwards
    float h[16];
    uint16_t hb[16], w[16];
    const int cc = lc.ok ? lc.c0 : 0;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int r = r0 + min(j, n - 1);
      const size_t row = row0 + r;
      if constexpr (EPI == EPI_RESID_BF16)
        hb[j] = reinterpret_cast<const uint16_t *>(p.resid)[row * p.ld_resid + cc];
      else
        h[j] = reinterpret_cast<const float *>(p.out)[row * p.ldo + cc];
      if constexpr (EPI == EPI_RESID_LOGIT)
        w[j] = reinterpret_cast<const uint16_t *>(p.head_w)[(size_t)tab.tok[r] * p.N + cc];
    }
    float z[16];   // RESID_LOGIT: the products with the LM-head row; else the next norm's input
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const bool live = j < n && lc.ok;
      if constexpr (EPI == EPI_RESID_BF16) h[j] = bf16_lo(hb[j]);
      const float x = v[j] + h[j];
      if constexpr (EPI == EPI_RESID_LOGIT) {
        z[j] = live ? x * lc.gain * bf16_lo(w[j]) : 0.f;
      } else {
        const size_t row = row0 + r0 + j;
        if (live && !dry) reinterpret_cast<float *>(p.out)[row * p.ldo + lc.c0] = x;
        z[j] = x * lc.gain;
      }
      h[j] = live ? x * x : 0.f;
    }
    if constexpr (EPI != EPI_RESID_LOGIT) {
      if (p.norm_out) {
        const int norm_lo = RP ? p.row_pairs * p.ld_norm : p.norm_split ? p.N : 0;
        size_t at[16];
        bool live[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          at[j] = (row0 + r0 + j) * p.ld_norm + lc.c0;
          live[j] = !dry && lc.ok && j < n;
        }
        store_acts<RP, 16>(reinterpret_cast<uint16_t *>(p.norm_out), at, z, live, p.out_f16 != 0,
                       norm_lo, p.status);
      }
    }
    if (EPI == EPI_RESID_LOGIT || p.norm_out) {
      const float ss = rows_sum(h, lane);
      float zz = 0.f;
      if constexpr (EPI == EPI_RESID_LOGIT) zz = rows_sum(z, lane);
      const int j = row16_of(lane);
      if ((lane & 1) == 0 && j < n && !dry) red[q * kMaxRows + r0 + j] = make_float2(ss, zz);
    }
  }
}

// Shared memory of this CTA -> shared memory of a CTA of the cluster, counted
// on an mbarrier there (addresses in the shared::cluster window).
CC_DEV void bulk_to_peer(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(dst),
      "r"(src), "r"(bytes), "r"(bar)
      : "memory");
}
// 16 rows of an accumulator (a row pair's two products added).
template <bool RP>
CC_DEV void load_block(uint32_t taddr, int row_pairs, float (&v)[16]) {
  uint32_t r[16], lo[16];
  tmem_ld16(taddr, r);
  if constexpr (RP) tmem_ld16(taddr + row_pairs, lo);
  tmem_ld_wait();
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    v[j] = __uint_as_float(r[j]);
    if constexpr (RP) v[j] += __uint_as_float(lo[j]);
  }
}
CC_DEV uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
  return a;
}

template <int EPI, bool RP, bool SPLIT, bool PAIR>
__global__ void __launch_bounds__(kThreads, 1)
    few_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmB2, const __grid_constant__ CUtensorMap tmB3,
               const __grid_constant__ GemmParams p, int nb, int one_group) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                              ~uintptr_t(1023));
  uint8_t *ring = smem;
  RowTab *tabs = reinterpret_cast<RowTab *>(smem + kOffTab);         // [2]
  float2 *reds = reinterpret_cast<float2 *>(smem + kOffRed);         // [2][4][kMaxRows]
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + kOffBar);
  uint64_t *empty = full + kMaxStages;
  uint64_t *tfull = empty + kMaxStages;     // [2]
  uint64_t *tempty = tfull + 2;             // [2]
  uint64_t *peers_done = tempty + 2;        // split: every CTA's products of the tile are done
  uint64_t *parts_in = peers_done + 1;      // split: every CTA's partial rows have arrived
  uint64_t *ring_free = parts_in + 1;       // split: the partials are summed, here and by the peers
  uint64_t *own_in = ring_free + 1;         // split: this CTA's partial rows are in its ring
  uint64_t *epi_bar = own_in + 1;           // the epilogue warps among themselves
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(epi_bar + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  int *prefix = reinterpret_cast<int *>(smem + kOffPrefix);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the cluster: S K splits (rank: this CTA's) of a column tile, or of two
  // (tile_of: this CTA's), whose CTAs of one split are a pair
  constexpr int PT = PAIR ? 2 : 1;
  const int cta = SPLIT || PAIR ? (int)cluster_ctarank() : 0;
  const int S = SPLIT ? (int)cluster_nctarank() / PT : 1;
  const int rank = cta / PT, tile_of = cta % PT;
  const int lead = cta - tile_of;                     // the pair's CTA 0
  auto peer = [&](int r) { return (uint32_t)(r * PT + tile_of); };   // this tile's CTA of split r
  const int unit0 = (int)blockIdx.x / (S * PT), n_units = (int)gridDim.x / (S * PT);
  constexpr int WT = w_tiles(EPI);
  const int a_rows = nb / PT;   // activation rows of a group that this CTA stages
  const int sb = stage_bytes(WT, a_rows), n_stages = stage_count(WT, a_rows);
  const int acc_stride = WT * acc_cols(nb);
  const int n_rounds = SPLIT ? split_rounds(WT, nb, S) : 1;   // of a split's exchange
  const int n_acc = 2 * acc_stride <= 512 ? 2 : 1;   // (one: SwiGLU groups of 256 rows)
  uint32_t tmem_cols = 64;
  while ((int)tmem_cols < n_acc * acc_stride) tmem_cols *= 2;

  pdl_trigger();
  if (threadIdx.x == 0) {
    for (int s = 0; s < n_stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tfull[a], 1);
      mbar_init(&tempty[a], PT * kEpiWarps);
    }
    mbar_init(peers_done, S);
    mbar_init(own_in, kEpiWarps);
    mbar_init(epi_bar, kEpiWarps);
    mbar_init(parts_in, 1);
    mbar_init(ring_free, kEpiWarps + S - 1);
    *abort_flag = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
    if (EPI == EPI_SWIGLU || EPI == EPI_QKV) tma_prefetch_desc(&tmB2);
    if (EPI == EPI_QKV) tma_prefetch_desc(&tmB3);
  }
  if (warp == 1) {
    if constexpr (PAIR) tmem_alloc_pair(tmem_slot, tmem_cols);
    else tmem_alloc(tmem_slot, tmem_cols);
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (SPLIT || PAIR) cluster_sync();   // every CTA's barriers exist before any remote arrival
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  const int nk = (p.K + BK - 1) / BK;
  const int nk_total = p.a_split ? 2 * nk : nk;   // split A: the hi pass, then the lo pass
  const int kb0 = rank * nk_total / S, kb1 = (rank + 1) * nk_total / S;

  // weight rows of tile nt, k-block column kw, into ring slot `dst`; a pair's
  // loads complete on the barrier of its CTA 0
  auto load2 = [&](uint8_t *dst, const CUtensorMap *m, uint64_t *bar, int c0, int c1, uint64_t pol) {
    if constexpr (PAIR) tma_load_2d_pair_hint(dst, m, cluster_addr(bar, lead), c0, c1, pol);
    else tma_load_2d_hint(dst, m, bar, c0, c1, pol);
  };
  auto load_w = [&](uint8_t *dst, uint64_t *bar, int nt, int kw, uint64_t pol) {
    if constexpr (EPI == EPI_SWIGLU) {
      load2(dst, &tmB, bar, kw, nt * BM, pol);
      load2(dst + W_BYTES, &tmB2, bar, kw, nt * BM, pol);
    } else if constexpr (EPI == EPI_QROPE || EPI == EPI_QKV) {
      // whole heads of a rotated projection: rows in the order of pair_base
      const int heads = BM / p.head_dim;
      const int nq = p.n_q_tiles, nkt = p.n_k_tiles;
      if (EPI == EPI_QROPE || nt < nq)
        tma_load_5d_hint(dst, &tmB, bar, kw, 0, 0, 0, nt * heads, pol);
      else if (nt < nq + nkt)
        tma_load_5d_hint(dst, &tmB2, bar, kw, 0, 0, 0, (nt - nq) * heads, pol);
      else
        load2(dst, &tmB3, bar, kw, (nt - nq - nkt) * BM, pol);
    } else {
      load2(dst, &tmB, bar, kw, nt * BM, pol);
    }
  };
  auto w_col = [&](int kb) { return (kb < nk ? kb : kb - nk) * BK; };

  // weights first: they depend on no earlier kernel
  int prefetched = 0;
  const uint64_t keep = make_policy_evict_last(), stream_pol = make_policy_evict_first();
  const int n_tiles_u = (p.n_tiles + PT - 1) / PT;   // tiles of a unit: PT each, the last maybe one short
  if (one_group && warp == 0 && lane == 0 && unit0 < n_tiles_u) {
    prefetched = min(n_stages, kb1 - kb0);
    for (int i = 0; i < prefetched; ++i) {
      if (tile_of == 0) mbar_arrive_expect_tx(&full[i], PT * sb);
      load_w(ring + (size_t)i * sb, &full[i], unit0 * PT + tile_of, w_col(kb0 + i), stream_pol);
    }
  }
  pdl_wait();   // the rows, their ranges and every output belong to earlier kernels until here
  if (threadIdx.x == 64)
    build_tile_prefix(p.seq_len, p.row_lo, p.batch, p.cap, nb, prefix, p.status);
  // one_group: the only group's loads may be in flight already, so it is
  // walked even when it turns out to have no row (prefix only reports its range)
  if (!one_group) __syncthreads();
  const int num_g = one_group ? 1 : prefix[p.batch];
  const int total = num_g * n_tiles_u;

  if (warp == 0) {
    if (lane == 0) {  // ---------------- TMA producer
      const uint64_t pol_w = num_g > 1 ? keep : stream_pol;
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      int it = 0;
      for (int item = unit0; ok && item < total; item += n_units, ++it) {
        const int ntu = item / num_g, g = item - ntu * num_g, nt = ntu * PT + tile_of;
        int row0 = p.row_lo ? p.row_lo[0] : 0;
        if (!one_group) {
          const int b = find_seq(prefix, p.batch, g);
          row0 = b * p.cap + (p.row_lo ? p.row_lo[b] : 0) + (g - prefix[b]) * nb;
        }
        // the ring holds the last tile's partials until they are summed
        if (SPLIT && it > 0 && !(ok = mbar_wait(ring_free, (it - 1) & 1, abort_flag, p.status))) break;
        for (int kb = kb0; kb < kb1; ++kb) {
          uint8_t *dst = ring + (size_t)stage * sb;
          if (it == 0 && kb - kb0 < prefetched) {
            ;   // armed, its weights on their way
          } else {
            if (!(ok = mbar_wait(&empty[stage], phase ^ 1, abort_flag, p.status))) break;
            if (tile_of == 0) mbar_arrive_expect_tx(&full[stage], PT * sb);
            load_w(dst, &full[stage], nt, w_col(kb), pol_w);
          }
          // A column block kb of [hi | lo] (hi and lo halves are K apart)
          const int ka = kb < nk ? kb * BK : p.K + (kb - nk) * BK;
          load2(dst + WT * W_BYTES, &tmA, &full[stage], ka, row0 + tile_of * a_rows, keep);
          if (++stage == n_stages) { stage = 0; phase ^= 1; }
        }
      }
      if (PAIR && ok) {
        // every stage's last release (a commit of the pair's CTA 0) has landed
        // before the CTA may leave
        for (int i = 0; i < n_stages; ++i) {
          if (!mbar_wait(&empty[stage], phase ^ 1, abort_flag, p.status)) break;
          if (++stage == n_stages) { stage = 0; phase ^= 1; }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && tile_of == 0) {  // ---------------- MMA issuer (a pair's CTA 0, for both)
      const uint32_t idesc =
          p.ab_f16 ? make_idesc_f16(PT * BM, nb, 0, 0) : make_idesc_bf16(PT * BM, nb, 0, 0);
      const uint16_t both = (uint16_t)(3u << lead);
      const uint64_t w_desc0 = make_sdesc_sw128(smem_u32(ring), 16, 1024);
      int stage = 0, acc = 0;
      uint32_t phase = 0, acc_phase = 0;
      for (int item = unit0; item < total; item += n_units) {
        if (!mbar_wait<PAIR>(&tempty[acc], acc_phase ^ 1, abort_flag, p.status)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem + acc * acc_stride;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait<PAIR>(&full[stage], phase, abort_flag, p.status)) goto mma_done;
          tc_fence_after();
          const uint64_t wd = w_desc0 + (uint64_t)((stage * sb) >> 4);
          const uint64_t ad = wd + ((WT * W_BYTES) >> 4);
#pragma unroll
          for (int w = 0; w < WT; ++w)
#pragma unroll
            for (int k = 0; k < BK / 16; ++k) {
              const uint32_t dt = d_tmem + w * acc_cols(nb), accum = kb != kb0 || k != 0;
              const uint64_t wk = wd + w * (W_BYTES >> 4) + 2 * k, ak = ad + 2 * k;
              if constexpr (PAIR) umma_ss_pair(dt, wk, ak, idesc, accum);
              else umma_ss(dt, wk, ak, idesc, accum);
            }
          if constexpr (PAIR) umma_commit_pair(&empty[stage], both);
          else umma_commit(&empty[stage]);
          if (++stage == n_stages) { stage = 0; phase ^= 1; }
        }
        if constexpr (PAIR) umma_commit_pair(&tfull[acc], both);
        else umma_commit(&tfull[acc]);
        if (++acc == n_acc) { acc = 0; acc_phase ^= 1; }
      }
    mma_done:;
    }
  } else {  // ------------------------------ epilogue warps 2..9
    const int q = warp & 3;             // TMEM lane quarter this warp may access
    const int ew = warp - 2;            // 0..7; group ew / 4 takes row blocks group, group + 2, ...
    const int grp = ew >> 2;
    const int c = q * 32 + lane;        // this thread's weight row of the tile
    const uint32_t tq = tmem + (uint32_t(q * 32) << 16);
    int acc = 0;
    uint32_t acc_phase = 0, bar_phase = 0;
    bool ok = true;
    auto epi_sync = [&]() {   // all eight warps (bounded)
      __syncwarp();
      if (lane == 0) mbar_arrive(epi_bar);
      const bool r = mbar_wait(epi_bar, bar_phase, abort_flag, p.status);
      bar_phase ^= 1;
      return r;
    };
    auto acc_free = [&]() {   // to the issuer of this accumulator's products
      if (PAIR && tile_of) mbar_arrive_cluster(cluster_addr(&tempty[acc], lead));
      else mbar_arrive(&tempty[acc]);
    };
    // A split's round: rows [round * per_round, + nr) of a group of nv, CTA r
    // finishing share r of them, rows [base, base + rows)
    const int per_round = nb / n_rounds;
    auto round_rows = [&](int round, int nv, int &nr, int &base, int &rows) {
      const int first = round * per_round;
      nr = !SPLIT ? nv : max(0, min(per_round, nv - first));
      const int share = (nr + S - 1) / S;
      base = first + min(nr, rank * share);
      rows = first + min(nr, (rank + 1) * share) - base;
    };
    uint32_t it = 0;
    for (int item = unit0; ok && item < total; item += n_units, ++it) {
      const int ntu = item / num_g, g = item - ntu * num_g, nt = ntu * PT + tile_of;
      const int b = one_group ? 0 : find_seq(prefix, p.batch, g);
      const int lo = p.row_lo ? p.row_lo[b] : 0;
      const int hi = p.seq_len ? p.seq_len[b] : p.cap;
      const int i0 = lo + (g - (one_group ? 0 : prefix[b])) * nb;
      // (bad ranges were reported when the prefix was built)
      const bool bad = lo < 0 || hi > p.cap || (PAIR && nt >= p.n_tiles);
      // valid rows of the group
      const int nv = bad ? 0 : max(0, min(RP ? p.row_pairs : nb, hi - i0));
      const size_t row0 = (size_t)b * p.cap + i0;
      // two tables in turn: warps are at most one item apart
      const int par = num_g == 1 ? 0 : (int)(it & 1);
      RowTab &tab = tabs[par];
      float2 *red = reds + (it & 1) * 4 * kMaxRows;
      if (it == 0 || num_g > 1) {
        fill_rows<EPI>(p, tab, (int)threadIdx.x - 64, nv, row0);
        if (!(ok = epi_sync())) break;
      }
      ProjTile d{};
      if constexpr (is_proj<EPI>) d = proj_tile<EPI>(p, nt);
      const LaneCol lc = lane_col<EPI>(p, d, nt, q, lane);
      const uint32_t tacc = tq + acc * acc_stride;
      // A CTA's first tile is preceded by a dry pass over one block: the
      // code's instruction fetches (measured several microseconds from a
      // cold instruction cache) then overlap the products
      int fin_base0 = 0, fin_rows0 = 0, fin_base1 = 0, fin_rows1 = 0;   // rows finished (per round)
      for (int pass = it == 0 && nv > 0 ? 0 : 1; ok && pass < 2; ++pass) {
        const bool dry = pass == 0;
        if (!dry) {
          if constexpr (EPI == EPI_RESID_BF16 || EPI == EPI_RESID_LOGIT) {
            for (int round = 0; round < n_rounds; ++round) {
              int nr, base, rows;
              round_rows(round, nv, nr, base, rows);
              for (int r0 = base + grp * kBlock; r0 < base + rows; r0 += 2 * kBlock)
                prefetch_block<EPI>(p, tab, r0, base + rows, row0, nt, q, lane);
            }
          }
          if (!(ok = mbar_wait(&tfull[acc], acc_phase, abort_flag, p.status))) break;
          tc_fence_after();
        }
        constexpr int ROW = WT * BM;                  // floats of a partial row
        const int rounds = dry ? 1 : n_rounds;
#pragma unroll 1
        for (int round = 0; ok && round < rounds; ++round) {
          const int lo_r = round * per_round;
          int nr = 1, base = 0, rows = 1;
          if (!dry) round_rows(round, nv, nr, base, rows);
          const int share = (nr + S - 1) / S;
          const float *own = reinterpret_cast<const float *>(ring);   // row lo_r first
          const float *recv = own + (size_t)per_round * ROW;   // [S - 1][share][ROW], peers in rank order
          if (SPLIT && !dry) {
            const uint32_t ph = (it * n_rounds + round) & 1;
            // every CTA's products are done (round 0) or its last round is summed:
            // no ring of the cluster is read any more
            if (round > 0) {
              fence_proxy_async_smem();   // generic reads before the peers' next copies
              if (!(ok = epi_sync())) break;
            }
            if (ew == 0 && lane < S) mbar_arrive_cluster(map_rank(smem_u32(peers_done), peer(lane)));
            if (!(ok = mbar_wait<true>(peers_done, ph, abort_flag, p.status))) break;
            // this CTA's partial rows of the round into its own ring
            if (ew == 0 && lane == 0)
              mbar_arrive_expect_tx(parts_in, (uint32_t)((S - 1) * rows * ROW * 4));
            for (int r0 = grp * kBlock; r0 < nr; r0 += 2 * kBlock) {
#pragma unroll
              for (int w = 0; w < WT; ++w) {
                float x[16];
                load_block<RP>(tacc + w * acc_cols(nb) + lo_r + r0, p.row_pairs, x);
                float *o = reinterpret_cast<float *>(ring) + r0 * ROW + w * BM + c;
#pragma unroll
                for (int j = 0; j < kBlock; ++j) o[j * ROW] = x[j];
              }
            }
            tc_fence_before();
            fence_proxy_async_smem();   // the bulk copies read what was just written
            __syncwarp();
            if (lane == 0) {
              if (round == n_rounds - 1) acc_free();
              mbar_arrive(own_in);
            }
            if (!(ok = mbar_wait(own_in, ph, abort_flag, p.status))) break;
            if (ew == 0 && lane < S && lane != rank) {
              const int d0 = min(nr, lane * share), dn = min(nr, d0 + share) - d0;
              const int slot = rank < lane ? rank : rank - 1;   // this CTA's place among lane's peers
              if (dn > 0)
                bulk_to_peer(map_rank(smem_u32(recv + (size_t)slot * share * ROW), peer(lane)),
                             smem_u32(own + (size_t)d0 * ROW), (uint32_t)(dn * ROW * 4),
                             map_rank(smem_u32(parts_in), peer(lane)));
            }
            if (!(ok = mbar_wait<true>(parts_in, ph, abort_flag, p.status))) break;
          }
#pragma unroll 1
          for (int r0 = dry ? 0 : grp * kBlock; r0 < rows; r0 += 2 * kBlock) {
            const int n = min(kBlock, rows - r0);
            float v[16], u[16];   // u: the up projection (SwiGLU)
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = u[j] = 0.f;
            if (!SPLIT && !dry) {
              load_block<RP>(tacc + r0, p.row_pairs, v);
              if constexpr (WT == 2) load_block<RP>(tacc + acc_cols(nb) + r0, p.row_pairs, u);
            } else if (!dry) {
#pragma unroll 1
              for (int s = 0; s < S; ++s) {   // rank order
                const float *src = (s == rank ? own + (size_t)(base - lo_r) * ROW
                                              : recv + (size_t)(s < rank ? s : s - 1) * share * ROW) +
                                   r0 * ROW + c;
#pragma unroll
                for (int j = 0; j < 16; ++j)
                  if (j < n) {
                    v[j] += src[j * ROW];
                    if constexpr (WT == 2) u[j] += src[j * ROW + BM];
                  }
              }
            }
            finish_block<EPI, RP>(p, d, lc, tab, v, u, base + r0, n, row0, q, lane, red, dry);
          }
          if (dry) continue;
          if (round == 0) {   // the rows this CTA finished, for the sums below
            fin_base0 = base;
            fin_rows0 = rows;
          } else {
            fin_base1 = base;
            fin_rows1 = rows;
          }
        }
        if (!ok) break;
        if (dry) continue;
        if constexpr (!SPLIT) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) acc_free();
        } else {
          // generic reads of the ring before the next tile's bulk writes to it;
          // the peers' copies into this CTA are done, so their sources may go
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(ring_free);
          if (ew == 0 && lane < S && lane != rank)
            mbar_arrive_cluster(map_rank(smem_u32(ring_free), peer(lane)));
        }
        if constexpr (is_resid<EPI> || EPI == EPI_ARGMAX) {
          // the four quarters' row sums (or maxima) of the tile
          const bool wanted = EPI == EPI_RESID_LOGIT || EPI == EPI_ARGMAX || p.norm_out;
          if (wanted && !(ok = epi_sync())) break;
          const int t = (int)threadIdx.x - 64;
          if (wanted && t < fin_rows0 + fin_rows1) {
            const int r = t < fin_rows0 ? fin_base0 + t : fin_base1 + t - fin_rows0;
            const float2 x0 = red[r], x1 = red[kMaxRows + r], x2 = red[2 * kMaxRows + r],
                         x3 = red[3 * kMaxRows + r];
            const size_t row = row0 + r;
            if constexpr (EPI == EPI_ARGMAX) {   // ascending columns: a later tie does not win
              float2 m = x0;
              if (x1.x > m.x) m = x1;
              if (x2.x > m.x) m = x2;
              if (x3.x > m.x) m = x3;
              if (__float_as_int(m.y) == 0x7FFFFFFF) m.y = __int_as_float(-1);
              reinterpret_cast<float2 *>(p.out)[row * p.ldo + nt] = m;
            } else {
              const float ss = (x0.x + x1.x) + (x2.x + x3.x);
              if constexpr (EPI == EPI_RESID_LOGIT)
                p.head_part[row * p.n_tiles + nt] =
                    make_float2(ss, (x0.y + x1.y) + (x2.y + x3.y));
              else
                p.ss_part[row * p.n_tiles + nt] = ss;
            }
          }
        }
      }
      if (++acc == n_acc) { acc = 0; acc_phase ^= 1; }
    }
  }

  tc_fence_before();
  __syncthreads();
  if constexpr (SPLIT || PAIR) cluster_sync();   // no CTA of the cluster still writes to this one
  if (*abort_flag) __nanosleep(1000000);   // let copies still in flight land
  if (warp == 1) {
    tc_fence_after();
    if constexpr (PAIR) tmem_dealloc_pair(tmem, tmem_cols);
    else tmem_dealloc(tmem, tmem_cols);
  }
}

template <int EPI, bool RP, bool SPLIT, bool PAIR = false>
cudaError_t launch_t(const CUtensorMap &a, const CUtensorMap &b, const CUtensorMap &b2,
                     const CUtensorMap &b3, const GemmParams &p, const FewPlan &plan,
                     bool one_group, cudaStream_t stream) {
  auto kern = few_kernel<EPI, RP, SPLIT, PAIR>;
  static std::atomic<bool> attr_set[64];
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  const int S = plan.split * (PAIR ? 2 : 1);   // CTAs of a cluster
  const int si = S == 1 ? 0 : S == 2 ? 1 : S == 4 ? 2 : 3;
  if (S != 1 << si || S > kFewMaxSplit || plan.clusters < 1 || plan.nb < 16 || plan.nb > 256 || plan.nb % 16) return cudaErrorInvalidValue;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)S;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)S);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (!attr_set[dev].load()) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return e;
    attr_set[dev].store(true);
  }
  cfg.gridDim = dim3((unsigned)(plan.clusters * S));
  return cudaLaunchKernelEx(&cfg, kern, a, b, b2, b3, p, plan.nb, one_group ? 1 : 0);
}

}  // namespace

FewClusters few_clusters(int sms) {
  return {{sms, std::max(1, sms / 2), std::max(1, sms / 4 * 19 / 20), std::max(1, sms / 10)}};
}

static int cluster_log2(int ctas) { return ctas == 1 ? 0 : ctas == 2 ? 1 : ctas == 4 ? 2 : 3; }
// Estimated SM cycles of a plan over `groups` row groups of at most rows_per_seq rows.
static double plan_cycles(int epi, int n_tiles, int K, bool a_split, double groups,
                          long long rows_per_seq, int nb, int S, int pt, const FewClusters &fit) {
  const int wt = w_tiles(epi);
  const int nk = ((K + BK - 1) / BK) * (a_split ? 2 : 1);
  const double hbm = (double)n_tiles * wt * BM * K * 2 / 3500.0;   // weight bytes at 6.7 TB/s, 1.9 GHz
  const int rounds = S > 1 ? split_rounds(wt, nb, S) : 1;
  // k-block: the products (2 cycles per row) or their operands' way into
  // shared memory (measured on the Qwen2.5 projections: 266 cycles for 18 KB,
  // 570 for 32 KB, 630 to 670 for 48 KB)
  const double tk = std::max(2.0 * nb * wt, 180.0 + stage_bytes(wt, nb / pt) / 105.0);
  const double waves = std::ceil(groups * ((n_tiles + pt - 1) / pt) / fit.n[cluster_log2(S * pt)]);
  // a tile's end: about 3600 cycles per 16-row block of a warp (SwiGLU 2600),
  // for a split the exchange before it; without a split it overlaps the
  // next tile's products while two accumulators fit
  const double fin = 1500.0 + (wt == 2 ? 80.0 : 112.0) * std::min<double>(nb, (double)rows_per_seq) / S;
  const bool overlapped = S == 1 && 2 * wt * acc_cols(nb) <= 512;
  const double fix = S > 1 ? 2500.0 * rounds + 20.0 * wt * nb + fin : overlapped ? 300.0 : fin;
  const double main = waves * std::ceil((double)nk / S) * tk;
  // (a pair's set-up and hand-overs: about 2 us for a launch alone, less
  // behind another kernel: the O projection of 512 Qwen2.5-7B rows is 35 us
  // alone either way, and all 28 layers take 6860 us without, 6710 with)
  const double ends = waves * fix + (overlapped ? fin : 0.0) + (pt == 2 ? 1500.0 : 0.0);
  // several groups read the same weight tiles at the same time, which holds
  // the SMs' requests longer (gate/up of 256 rows, 271 MB: 128-row groups
  // 70 us at 4.9 TB/s, one of 256 rows 66 us)
  return std::max(main, hbm * (groups > 1 ? 1.5 : 1.1)) + ends + 0.05 * (main + ends);
}

FewPlan few_plan(int epi, int n_tiles, int K, bool a_split, int seqs, long long rows_per_seq,
                 int row_pairs, const FewClusters &fit) {
  const int wt = w_tiles(epi);
  FewPlan best{};
  best.n_tiles = n_tiles;
  best.cycles = 1e300;
  const int nk = ((K + BK - 1) / BK) * (a_split ? 2 : 1);
  const bool resid = epi == EPI_RESID_BF16 || epi == EPI_RESID_F32 || epi == EPI_RESID_LOGIT;
  for (int nb = 16; nb <= kMaxRows; nb *= 2) {
    if (row_pairs && nb != 2 * row_pairs) continue;
    if (!row_pairs && nb > 16 && nb / 2 >= rows_per_seq) break;   // half of it holds every row
    const double groups = (double)seqs * (double)((rows_per_seq + nb - 1) / nb);
    for (int S = 1; S <= kFewMaxSplit; S *= 2) {
      if (S > 1 && (nk < 4 * S || split_rounds(wt, nb, S) == 0)) break;
      for (int pt = 1; pt <= 2; ++pt) {   // 2: CTA pairs
        // whole groups of the residual products, split (128-row groups measured
        // 62 us against 59, the projections the same, gate/up 64 against 65)
        if (pt == 2 && (!resid || nb != kMaxRows || S == 1 || 2 * S > kFewMaxSplit || row_pairs))
          break;
        const double t = plan_cycles(epi, n_tiles, K, a_split, groups, rows_per_seq, nb, S, pt, fit);
        if (t < best.cycles * 0.98) {
          best.nb = nb;
          best.split = S;
          best.pair = pt == 2;
          best.clusters = fit.n[cluster_log2(S * pt)];
          best.cycles = t;
        }
      }
    }
  }
  return best;
}

double few_cycles(const FewPlan &plan, int epi, int K, bool a_split, int seqs, long long rows_per_seq,
                  const FewClusters &fit) {
  const double groups = (double)seqs * (double)((rows_per_seq + plan.nb - 1) / plan.nb);
  return plan_cycles(epi, plan.n_tiles, K, a_split, groups, rows_per_seq, plan.nb, plan.split,
                     plan.pair ? 2 : 1, fit);
}

cudaError_t launch_few(int epi, const CUtensorMap &a, const CUtensorMap &b, const CUtensorMap &b2,
                       const CUtensorMap &b3, const GemmParams &p, const FewPlan &plan,
                       bool one_group, cudaStream_t st) {
  // (row pairs: the products of a decode step)
#define CC_FEW_T(E, R)                                                                   \
  (plan.split > 1 ? launch_t<E, R, true>(a, b, b2, b3, p, plan, one_group, st)      \
                  : launch_t<E, R, false>(a, b, b2, b3, p, plan, one_group, st))
#define CC_FEW_RESID(E)                                                                  \
  (plan.pair ? launch_t<E, false, true, true>(a, b, b2, b3, p, plan, one_group, st) \
             : CC_FEW_T(E, false))
#define CC_FEW_DECODE(E) (p.row_pairs ? CC_FEW_T(E, true) : CC_FEW_T(E, false))
  if (p.row_pairs && (epi == EPI_RESID_BF16 || epi == EPI_RESID_LOGIT)) return cudaErrorInvalidValue;
  switch (epi) {
    case EPI_QROPE: return CC_FEW_DECODE(EPI_QROPE);
    case EPI_RESID_BF16: return CC_FEW_RESID(EPI_RESID_BF16);
    case EPI_RESID_F32:
      return p.row_pairs ? CC_FEW_T(EPI_RESID_F32, true) : CC_FEW_RESID(EPI_RESID_F32);
    case EPI_SWIGLU: return CC_FEW_DECODE(EPI_SWIGLU);
    case EPI_BF16: return CC_FEW_DECODE(EPI_BF16);
    case EPI_QKV: return CC_FEW_DECODE(EPI_QKV);
    case EPI_ARGMAX: return CC_FEW_DECODE(EPI_ARGMAX);
    case EPI_RESID_LOGIT: return CC_FEW_RESID(EPI_RESID_LOGIT);
    default: return cudaErrorInvalidValue;
  }
#undef CC_FEW_DECODE
#undef CC_FEW_RESID
#undef CC_FEW_T
}

}  // namespace cc
