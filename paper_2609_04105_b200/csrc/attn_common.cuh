// Pieces shared by the attention kernels (one query tile per CTA, and two query tiles per CTA): tile sizes, the
// tensor-memory and shared-memory maps, work-item decoding, and the per-block score -> code arithmetic of
// Algorithm "direct-p-pack".
#pragma once
#include <cuda.h>

#include "common.cuh"
#include "ptx.cuh"

namespace fp4attn {
using namespace ptx;

constexpr int BM = 128;          // query rows per work item
constexpr int BN = 64;           // keys per score tile (two N32 probability blocks)
constexpr int BS = 128;          // keys per stage
constexpr int kTeams = 4;        // score slots / softmax teams
constexpr int kFirstSoftmaxWarp = 7;     // warps 3..6 are the correction warps
constexpr int kAttnThreads = 32 * (kFirstSoftmaxWarp + 4 * kTeams);
constexpr int kLazyShift = 64;   // the row reference is raised only when a block exponent exceeds it by more
                                 // than this many octaves (rescales are exact powers of 2) ...
constexpr int kRefHeadroom = 60; // ... and is then set this far ABOVE that exponent, so that a later raise
                                 // needs a jump of 124 octaves: E8M0 bytes stay within 1..191, blocks weaker
                                 // than 2^-66 of the row maximum become zero blocks
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColS = 0, kColO = 256, kColSFQ = 400, kColSFK = 416, kColSFV = 432, kColSFP = 448,
                   kColP = 456;      // P codes: [stage parity][tile] x 8 columns (64 keys x 4 bits per row)
constexpr int kItemTable = 64;   // work items of a CTA that are decoded ahead (ItemRec)
constexpr int kOnesRows = 16;    // rows of ones appended to V^T (the MMA's N must be a multiple of 16)

template <int D, bool NV>
struct Cfg {
  static constexpr int ROW_BYTES = D / 2;                       // packed bytes of one Q/K row
  static constexpr int KBLK = D / 64;                           // K64 instructions per QK stage
  static constexpr int CTQ = NV ? (D / 16 + 3) / 4 : 1;         // scale atoms per 128 rows of Q or K
  static constexpr int Q_BYTES = BM * ROW_BYTES;
  static constexpr int QSF_BYTES = CTQ * 512;
  static constexpr int K_BYTES = BS * ROW_BYTES;                // 128 keys
  static constexpr int V_BYTES = D * (BS / 2);                  // V^T: d rows x 64 bytes
  static constexpr int ONES_BYTES = kOnesRows * (BS / 2);       // constant rows of E2M1 1.0, written once
  static constexpr int DN = D + kOnesRows;                      // N of the PV instruction
  static constexpr int KSF_BYTES = CTQ * 512;
  static constexpr int VSF_BYTES = 512;
  static constexpr int OFF_KSF = K_BYTES + V_BYTES + ONES_BYTES;   // within a stage
  static constexpr int OFF_VSF = OFF_KSF + KSF_BYTES;
  static constexpr int STAGE_BYTES = OFF_VSF + VSF_BYTES;
  static constexpr int NST = 8;                                 // ring depth (stages of 128 keys); at d = 128 the affine map takes 1-2 % longer with 7, the same with 9
  static constexpr int PSF_BYTES = 512;                         // one atom per stage: bytes {0,1} tile 0, {2,3} tile 1
  static constexpr int META_BYTES = BM * 16;                    // per stage parity and row: {E_0, E_1} of tile 0, of tile 1
  // shared-memory map (offsets from a 1024-byte aligned base)
  static constexpr int OFF_Q = 0;                               // two buffers
  static constexpr int OFF_QSF = OFF_Q + 2 * Q_BYTES;           // two buffers of 1 KB
  static constexpr int OFF_PSF = OFF_QSF + 2048;
  static constexpr int OFF_ONESF = OFF_PSF + 2 * PSF_BYTES;     // scale atom of 1.0 for the rows of ones
  static constexpr int OFF_META = OFF_ONESF + 512;
  static constexpr int OFF_STAGE = (OFF_META + 2 * META_BYTES + 1023) / 1024 * 1024;
  static constexpr int OFF_OUT = (OFF_STAGE + NST * STAGE_BYTES + 1023) / 1024 * 1024; // bf16 O tile staged for TMA stores: D/64 halves of [128 rows][128 B]
  static constexpr int OUT_BYTES = (D / 64) * BM * 128;
  static constexpr int OFF_BAR = OFF_OUT + OUT_BYTES;
  static constexpr int OFF_SEQ = OFF_BAR + 1024;                // SeqTable
  static constexpr int OFF_ITEMS = OFF_SEQ + 1536;              // item table
  static constexpr int SMEM_BYTES = OFF_ITEMS + kItemTable * 32 + 1024;   // + alignment slack
  static constexpr uint64_t SWZ_QK = (ROW_BYTES == 64) ? kSwz64 : kSwz32;
  static_assert(STAGE_BYTES % 512 == 0 && OFF_STAGE % 1024 == 0 && OFF_OUT % 1024 == 0, "stage alignment");
  static_assert(SMEM_BYTES <= 227 * 1024, "shared memory");
};

struct AttnParams {
  const uint8_t *q_sf, *k_sf, *v_sf;
  const float *q_G, *k_G;
  __nv_bfloat16* O;
  float* LSE;
  int* status;
  int N, stages;           // keys, N / 128
  int n_items;             // B * H * N / 128
  float c_base;            // fl32(log2(e) * softmax_scale)
  unsigned long long c_mx2, ca_mx2;            // MXFP4 Q, K: {c, c} with c = fl32(c_base / 36), and {A c, A c}: packed multiply-add operands
  float aff_a, aff_b;      // affine classifier u = max(0, A x + B) (only read by the affine variant)
  int thr16;               // block exponent rule: 0 = ceil(max y), 1 = floor(max y + log2 1.6)
  int causal;              // 1: query row i sees keys 0..i
  int H, Hkv;              // query heads, K/V heads (H % Hkv == 0: grouped-query attention)
  int BH;                  // B * H
  unsigned long long recip_qtiles, recip_bh;   // ceil(2^64 / (N / 128)), ceil(2^64 / BH); 0 for a divisor of 1
  int ref_fixed;           // the constant row reference of the FIXREF instances (octaves)
  const int* seq_len;      // NULL, or B token counts: batch entry b is seq_len[b] tokens padded to N (masked kernels only)
  unsigned long long recip_h;                  // ceil(2^64 / H); 0 for H = 1
  int B;
  int sorted;              // seq_len given and B <= kSeqTableMax: the work items come from a SeqTable
};

// One work item = one 128-row query tile of one (batch, query head).
struct WorkItem {
  int qt;                  // query tile within the head
  int qrow0;               // first row of the tile in the [B*H*N] row space of Q, O, LSE
  int qtile_lin;           // (b*H + h) * qtiles + qt: index of the tile's Q scale atom(s)
  int kvh;                 // b*Hkv + h / (H/Hkv): the K/V head this query head reads
  int bh;                  // b*H + h
  int T2;                  // 128-key stages to walk (causal: up to and including the diagonal; padded: those with a key)
  int len;                 // keys that exist for this unit (N unless the batch entry is a padded sequence)
};
// ---- which work items a CTA takes, and in which order (masked kernels)
// The items of a causal mask or of sequences of unlike lengths differ in cost (stages).  They are numbered from the most
// expensive down and dealt to the persistent CTAs in rounds of alternating direction: dealt in one direction only, the first
// CTA gets the dearest item of every round (causal, 64 heads, N = 4096: 269 stages against 254, with a mean of 253).
template <bool MASKED>
__device__ __forceinline__ int item_at(int i) {
  return i * (int)gridDim.x + (MASKED && (i & 1) ? (int)gridDim.x - 1 - (int)blockIdx.x : (int)blockIdx.x);
}
template <bool MASKED>
__device__ __forceinline__ int items_of_cta(int n_items) {
  const int rounds = n_items / (int)gridDim.x;
  return rounds + (item_at<MASKED>(rounds) < n_items ? 1 : 0);
}
// Padded sequences: the entries ordered by length, longest first (rank r is entry b[r] with len[r] tokens in T[r] tiles), and
// the items numbered accordingly, query tiles beyond a length left out (they are only filled with zeros, fill_skipped).
// Built by every CTA from the token counts.  Without a causal mask rank r has H * T[r] items of T[r] stages each; with it,
// tile qt costs qt + 1 stages wherever it exists, so the items go tile level by tile level, from T[0] - 1 down, and the
// levels from T[r] - 1 to T[r + 1] have (r + 1) * H items each.  first[r]: number of the first item of segment r; skipped[r]:
// of the first left-out tile of rank r.  Both end with the total at [B] and the largest int beyond.
// (B = 6, H = 12, N = 2176, 436 ... 2176 tokens, d = 64, whole step: 100 -> 77 us; in batch order one CTA had 163 stages
// and item boundaries where the mean is 111.)
constexpr int kSeqTableMax = 64;
struct SeqTable {
  int first[kSeqTableMax + 1], skipped[kSeqTableMax + 1], T[kSeqTableMax + 1], b[kSeqTableMax], len[kSeqTableMax];
};
static_assert(sizeof(SeqTable) <= 1536, "the space behind the barriers");
// all threads; ends with a barrier
__device__ __forceinline__ void build_seq_table(SeqTable* st, const AttnParams& p, int qtiles) {
  const int t = threadIdx.x;
  int len = 0, rank = 0;
  if (t < p.B) {
    len = min(max(__ldcg(p.seq_len + t), 1), p.N);
    st->first[t] = len;                                          // for the comparison below
  }
  __syncthreads();
  if (t < p.B)
    for (int k = 0; k < p.B; ++k) {
      const int T = (st->first[k] + BS - 1) / BS, Tt = (len + BS - 1) / BS;
      rank += T > Tt || (T == Tt && k < t);
    }
  __syncthreads();
  if (t < p.B) {
    st->b[rank] = t;
    st->len[rank] = len;
    st->T[rank] = (len + BS - 1) / BS;
  }
  if (t == p.B) st->T[t] = 0;
  __syncthreads();
  if (t <= kSeqTableMax) {
    int items = 0, left_out = 0;
    for (int k = 0; k < min(t, p.B); ++k) {
      items += p.causal ? (st->T[k] - st->T[k + 1]) * (k + 1) : st->T[k];
      left_out += qtiles - st->T[k];
    }
    st->first[t] = t <= p.B ? items * p.H : 0x7FFFFFFF;
    st->skipped[t] = t <= p.B ? left_out * p.H : 0x7FFFFFFF;
  }
  __syncthreads();
}
// r with start[r] <= n < start[r + 1]; the whole warp, n the same in every lane
__device__ __forceinline__ int seq_segment(const int* start, int n) {
  const int lane = threadIdx.x & 31;
  return __popc(__ballot_sync(0xffffffffu, start[1 + lane] <= n)) + __popc(__ballot_sync(0xffffffffu, start[33 + lane] <= n));
}
// Zeros for O and LSE in the query tiles that no token occupies.  All threads of all CTAs.
template <int D>
__device__ __forceinline__ void fill_skipped(const SeqTable* st, const AttnParams& p, int qtiles) {
  const int total = st->skipped[p.B];
  for (int j = blockIdx.x; j < total; j += gridDim.x) {
    const int r = seq_segment(st->skipped, j), n = qtiles - st->T[r], rem = j - st->skipped[r], h = rem / n;
    const size_t row0 = ((size_t)st->b[r] * p.H + h) * p.N + (size_t)(st->T[r] + rem - h * n) * BM;
    uint4* o = reinterpret_cast<uint4*>(p.O + row0 * D);
    for (int k = threadIdx.x; k < BM * D / 8; k += blockDim.x) o[k] = make_uint4(0u, 0u, 0u, 0u);
    if (p.LSE && threadIdx.x < BM) p.LSE[row0 + threadIdx.x] = 0.f;
  }
}

// two bf16 of O, round to nearest even, the largest finite value instead of an infinity
__device__ __forceinline__ uint32_t bf16x2_finite(float lo, float hi) {
  uint32_t w;
  asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(w) : "f"(hi), "f"(lo));
  return w;
}

// floor(n / d) for n < 2^31 through the precomputed reciprocal ceil(2^64 / d) (0 stands for d = 1): the
// roles decode a work item on their critical path, and a 32-bit division costs some fifty instructions
__device__ __forceinline__ int fast_div(int n, unsigned long long recip) {
  return recip ? (int)__umul64hi((unsigned long long)n, recip) : n;
}
// MASKED: the kernels that mask the last stage of an item - the causal mask (p.causal), padded sequences
// (p.seq_len), or both.  The unmasked kernels ignore both fields.
template <bool MASKED>
__device__ __forceinline__ WorkItem decode_item(int item, const AttnParams& p, int qtiles, const SeqTable* st) {
  constexpr bool CAUSAL = MASKED;
  WorkItem w;
  int bh;
  if (MASKED && p.sorted) {
    int r = seq_segment(st->first, item), h;
    const int rem = item - st->first[r];
    w.T2 = st->T[r];
    if (p.causal) {
      const int width = (r + 1) * p.H, level = rem / width, k = rem - level * width;
      w.qt = w.T2 - 1 - level;
      w.T2 = w.qt + 1;
      r = k / p.H;
      h = k - r * p.H;
    } else {
      h = rem / w.T2;
      w.qt = rem - h * w.T2;
    }
    const int b = st->b[r];
    w.len = st->len[r];
    w.bh = b * p.H + h;
    w.qrow0 = w.bh * p.N + w.qt * BM;
    w.qtile_lin = w.bh * qtiles + w.qt;
    w.kvh = p.H != p.Hkv ? b * p.Hkv + h / (p.H / p.Hkv) : w.bh;
    return w;
  }
  if (CAUSAL) {             // longest items first, so the persistent CTAs finish together
    const int r = fast_div(item, p.recip_bh);
    w.qt = qtiles - 1 - r;
    bh = item - r * p.BH;
  } else {                  // consecutive items share K/V in L2
    bh = fast_div(item, p.recip_qtiles);
    w.qt = item - bh * qtiles;
  }
  w.qrow0 = bh * p.N + w.qt * BM;
  w.qtile_lin = bh * qtiles + w.qt;
  w.kvh = bh;
  w.bh = bh;
  if (p.H != p.Hkv) {       // grouped-query attention
    const int b = bh / p.H, h = bh - b * p.H;
    w.kvh = b * p.Hkv + h / (p.H / p.Hkv);
  }
  w.len = p.N;
  w.T2 = p.stages;
  if (MASKED) {
    if (p.seq_len) {
      const int len = __ldcg(p.seq_len + fast_div(bh, p.recip_h));
      w.len = len < 1 ? 1 : (len > p.N ? p.N : len);
      w.T2 = w.qt * BM < w.len ? (w.len + BS - 1) / BS : 1;   // a query tile beyond the length: one stage, results unused
    }
    if (p.causal && w.qt + 1 < w.T2) w.T2 = w.qt + 1;
  }
  return w;
}

// ---- the items of a CTA, decoded once
// A masked item's decoding is some two hundred instructions (integer divisions, the ranks of a SeqTable), a unit's score
// constant two loads from L2 and a division, and each of the 23 warps did both for every item, on schedulers whose issue slots
// are what these kernels are bound by.  So the CTA's first kItemTable items are decoded when it starts, one warp an item; later
// ones by every role for itself.  Attention alone from a graph, no table | table: B=2, H=32/8, N=4096, d=128, causal, one NVFP4
// factor per unit 134.8 | 130.2 us; padded batch B=6, H=12, N=2176, d=64 59.3 | 58.4; without a mask (B=4, H=16, N=4096, d=128,
// factors per unit), where an item's decoding is short, 223.9 | 224.8.
struct __align__(16) ItemRec {
  WorkItem w;
  float c;                 // the unit's score constant (NVFP4 factors per unit)
};
static_assert(sizeof(ItemRec) == 32, "the space behind the SeqTable");
__device__ __forceinline__ float unit_score_constant(const AttnParams& p, const WorkItem& w) {
  return __fdiv_rn(p.c_base, __fmul_rn(__ldcg(p.q_G + w.bh), __ldcg(p.k_G + w.kvh)));
}
// all threads; ends with a barrier
template <bool MASKED, bool UNIT_CONSTANT>
__device__ __forceinline__ void build_item_table(ItemRec* tab, int n_my, const AttnParams& p, int qtiles, const SeqTable* st) {
  for (int i = threadIdx.x >> 5; i < min(n_my, kItemTable); i += (int)blockDim.x / 32) {
    ItemRec r;
    r.w = decode_item<MASKED>(item_at<MASKED>(i), p, qtiles, st);
    r.c = UNIT_CONSTANT ? unit_score_constant(p, r.w) : 0.f;
    if ((threadIdx.x & 31) == 0) tab[i] = r;
  }
  __syncthreads();
}
template <bool MASKED>
__device__ __forceinline__ WorkItem item_of_cta(int i, const ItemRec* tab, const AttnParams& p, int qtiles, const SeqTable* st) {
  return i < kItemTable ? tab[i].w : decode_item<MASKED>(item_at<MASKED>(i), p, qtiles, st);
}

// barrier slots (8 bytes each)
enum { BAR_QFULL0 = 0, BAR_QFREE0 = 2, BAR_OFULL = 4, BAR_OFREE = 5, BAR_SFULL0 = 6, BAR_SEMPTY0 = 8,
       BAR_PFULL0 = 10, BAR_PFREE0 = 12, BAR_SMDONE0 = 14, BAR_DRAIN0 = 16, BAR_RING = 18 };

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// maximum of 32 floats held as raw bits, as a depth-4 tree of 3-input maxima
__device__ __forceinline__ float max32(const uint32_t* r) {
  float t[12];
#pragma unroll
  for (int k = 0; k < 10; ++k)
    t[k] = max3(__uint_as_float(r[3 * k]), __uint_as_float(r[3 * k + 1]), __uint_as_float(r[3 * k + 2]));
  t[10] = __uint_as_float(r[30]);
  t[11] = __uint_as_float(r[31]);
  const float a = max3(t[0], t[1], t[2]), b = max3(t[3], t[4], t[5]), c = max3(t[6], t[7], t[8]), d = max3(t[9], t[10], t[11]);
  return fmaxf(max3(a, b, c), d);
}
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
// {x0, x1} = {s0, s1} * {c, c} + {b, b}
__device__ __forceinline__ void fma2(float s0, float s1, float c, float b, float& x0, float& x1) {
  unpack2(fma2(pack2(s0, s1), pack2(c, c), pack2(b, b)), x0, x1);
}
// ---- the code of 2^x without 2^x.
// A code is the number of boundaries log2(b), b in {1/4, 3/4, 5/4, 7/4, 5/2, 7/2, 5}, below x.  The conversion to E2M1
// counts the boundaries {1/4, 3/4, 5/4, 7/4, ...} below its own argument, so three conversions of affine functions of x
// count all seven, each exactly once:
//   u0 = x/2 + k0     crosses 1/4, 3/4, 5/4 at log2 5/4, log2 5/2, log2 5
//   u1 = a1 x + k1    crosses 1/4, 3/4      at log2 1/4, log2 7/4
//   u2 = a2 x + k2    crosses 1/4, 3/4      at log2 3/4, log2 7/2
// The next crossing of each lies above 3.32, and x never exceeds log2 7.5 = 2.91 (log2 6 under the ceiling rule) by
// construction of the block exponent, which leaves room for its rounding up to |y| = 2^21 (beyond, where the exponent is
// clamped, counts of 8 and more are possible: other codes, signs and carries; the epilogue keeps what follows finite); negative arguments are clamped to code 0 by the conversion.  The three counts never sum to more than 7, so the packed
// words of eight codes simply add.  The arguments are float32, so the codes are those of the exact exponential up to the
// rounding of x at a boundary, as with ex2.approx (2-million-score sweeps at |y| up to 2000: no mismatch further than
// 0.3 spacings of y from a boundary for either).
//
// What it is for: ex2.approx costs 8 clocks per warp instruction and scheduler, so 32 of them per block would alone take
// 256.  Half the pairs on this route leave 128, and it takes less of everything else than a polynomial does: of its
// four multiply-adds three read one register pair (x; slope and offset are literals).  Register operands are what the
// dispatch is short of (about two 32-bit operands per clock and scheduler: a packed multiply-add with three register
// pairs takes 4 clocks, with two 2, a three-input maximum 2).  Clocks per 32 x 32 block and scheduler, four warps, scores
// from tensor memory: all pairs on ex2 272, 12 of 16 and a degree-6 polynomial for the rest 220, 12 / 10 / 8 / 6 / 0 of 16
// and this route for the rest 211 / 192 / 178 / 186 / 233.
constexpr float kCodeA1 = 0.1781035935540111f;                   // 1/2 / (log2 7/4 - log2 1/4)
constexpr float kCodeA2 = 0.22498276865942612f;                  // 1/2 / (log2 7/2 - log2 3/4)
constexpr float kCodeK0 = 0.0890359525563188f;                   // 1/4 - 1/2 log2 5/4
constexpr float kCodeK1 = 0.6062071871080222f;                   // 1/4 + 2 a1
constexpr float kCodeK2 = 0.34337628568523887f;                  // 1/4 - a2 log2 3/4

// One N32 score fragment of one row: E_B = ceil(max y) and the codes.  Nothing here depends on the
// row reference.
//   ideal map  (Eq. "ideal-code-path"):  q = Q_E2M1(2^x),            x = y - E_B + log2 6
//   affine map (Eq. "affine-code-map"):  q = Q_E2M1(max(0, A x + B)), folded into one fused multiply-add
//                                        per element: u = s * fl32(A c) + fma(A, log2 6 - E_B, B)
// PMAP: 0 ideal map for every element, 1 affine map for every element, 2..4 mixed (the EX2-density control
// of Appendix "SM103 launch and EX2 controls"): element pair k of the block takes the ideal map where bit
// k of the pattern is set, the affine map elsewhere.
__host__ __device__ constexpr uint32_t exact_pairs_of(int pmap) {
  return pmap == 0 ? 0xFFFFu : pmap == 1 ? 0x0000u : pmap == 2 ? 0x1111u : pmap == 3 ? 0x5555u : 0x7777u;
}
// Words (of eight keys) whose exact pairs take the conversion count instead of ex2.approx: so many that the special-function
// unit stops being the bound (8 of 16 pairs are left to it, 9 with 12 of 16 exact; with 8 or fewer exact it never is).  The
// two middle words rather than the first two: 889 against 903 us at N = 8192 (903: words 0 and 1, 934: one word).
__host__ __device__ constexpr uint32_t counted_words_of(int pmap) { return pmap == 0 ? 0x6u : pmap == 4 ? 0x1u : 0x0u; }
// RULE: block exponent from the block maximum - 0 ceiling, 1 threshold rule, 2 the better of ceiling and ceiling - 1 by
// squared error of the 32 represented values (ideal map only; see direct_p_block_mse)
__device__ __forceinline__ void direct_p_block_mse(const uint32_t* sraw, float c32, int& E, uint32_t* words);
// Keys from `visible` on (causal mask, padding) get -inf: they never raise a block maximum, and they code to 0 as long as the
// score constant is not 0 (which NVFP4 Q and K make it that are so small that the product of their encode factors overflows).
__device__ __forceinline__ void mask_scores(uint32_t* sraw, int visible) {
#pragma unroll
  for (int i = 0; i < 32; ++i) sraw[i] = (i < visible) ? sraw[i] : 0xFF800000u;
}
// The scores of a block of a masked kernel, of whose 32 keys this row sees the first `visible`.  Whole warp.  False (and the
// scores as they were): none of the warp's rows sees any.  Most blocks of a masked stage are seen by all rows of a warp or by
// none (of a diagonal tile's sixteen, six and six), so only the others are masked: 135.4 -> 130.2 us for the causal launch named
// at ItemRec.  (The FP8 P/V kernels lose 5 % with it.)
__device__ __forceinline__ bool masked_scores(uint32_t* sraw, int visible) {
  if (__all_sync(0xffffffffu, visible >= 32)) return true;
  if (!__any_sync(0xffffffffu, visible > 0)) return false;
  mask_scores(sraw, visible);
  return true;
}
// what direct_p_block makes of 32 times -inf
__device__ __forceinline__ void empty_block(int& E, uint32_t* words) {
  E = -2097152;
  words[0] = words[1] = words[2] = words[3] = 0u;
}
// The score constant for masked keys: the smallest normal number instead of 0, which changes no score by 1e-25.
__host__ __device__ __forceinline__ float nonzero(float c) { return c == 0.f ? 1.17549435e-38f : c; }
// The FP8 P/V kernels clear the bytes of masked keys instead (half the instructions of a second masking of the scores; in the
// FP4 kernels, which mask the scores for the block maximum anyway, clearing the codes too took 2.5 % of a causal step).
__device__ __forceinline__ void mask_bytes(uint32_t* words, int visible) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int n = visible - 4 * i;
    words[i] = n >= 4 ? words[i] : n <= 0 ? 0u : words[i] & ((1u << (8 * n)) - 1u);
  }
}

// c2 = {c, c}, ca2 = {fl32(A c), fl32(A c)}: 64-bit so that they can stay in uniform registers (kernel parameters)
template <int PMAP, int RULE>
__device__ __forceinline__ void direct_p_block(const uint32_t* sraw, uint64_t c2, uint64_t ca2, float A, float B, int& E, uint32_t* words) {
  const float c32 = __uint_as_float((uint32_t)c2);
  if (RULE == 2) { direct_p_block_mse(sraw, c32, E, words); return; }
  constexpr bool THR16 = RULE == 1;
  constexpr uint32_t kExact = exact_pairs_of(PMAP), kCounted = counted_words_of(PMAP);
  const float LOG2_6 = 2.5849625007211560f;
  // y is clamped to +-2^21 (scores beyond that are outside any softmax's range; a fully masked block,
  // max = -inf, lands on the lower clamp and becomes a zero block)
  const float ymax = fminf(fmaxf(__fmul_rn(max32(sraw), c32), -2097152.0f), 2097152.0f);
  // amplitude rule (Eq. "mx-scale" allows either neighbouring power of two): ceiling, or the threshold
  // rule alpha = 2^floor(log2(1.6 a)) under which values above the amplitude saturate at code 6.
  // Integer rounding on the FMA pipe (the conversion instructions share the SFU's issue slots with
  // ex2): for |y| < 2^22, y + 1.5*2^23 rounded up (down) is ceil(y) (floor(y)) + 1.5*2^23 exactly.
  const float M = 12582912.0f;
  const float t = THR16 ? __fadd_rd(__fadd_rn(ymax, 0.6780719161033630f), M) : __fadd_ru(ymax, M);
  E = (int)(__float_as_uint(t) - 0x4B400000u);
  const float bB = __fsub_rn(LOG2_6, __fsub_rn(t, M));          // t - M = (float)E, exact
  const float bA = __fmaf_rn(A, bB, B);                          // affine pairs only
  static_assert(kCounted == 0u || kExact == 0xFFFFu || kExact == 0x7777u, "a counted word has its first three pairs exact, or all four");
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    const bool counted = (kCounted >> w) & 1u;
    float pv[8], q1[8], q2[8];
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      const float s0 = __uint_as_float(sraw[8 * w + i]), s1 = __uint_as_float(sraw[8 * w + i + 1]);
      if ((kExact >> (4 * w + i / 2)) & 1u) {
        const uint64_t x = fma2(pack2(s0, s1), c2, pack2(bB, bB));
        if (counted) {
          unpack2(fma2(x, pack2(0.5f, 0.5f), pack2(kCodeK0, kCodeK0)), pv[i], pv[i + 1]);
          unpack2(fma2(x, pack2(kCodeA1, kCodeA1), pack2(kCodeK1, kCodeK1)), q1[i], q1[i + 1]);
          unpack2(fma2(x, pack2(kCodeA2, kCodeA2), pack2(kCodeK2, kCodeK2)), q2[i], q2[i + 1]);
        } else {
          float x0, x1;
          unpack2(x, x0, x1);
          pv[i] = ex2_approx(x0);
          pv[i + 1] = ex2_approx(x1);
        }
      } else {
        unpack2(fma2(pack2(s0, s1), ca2, pack2(bA, bA)), pv[i], pv[i + 1]);
      }
    }
    // the conversion clamps negative inputs to +0 (affine and counted pairs; an exponential is positive anyway)
    words[w] = (kExact == 0xFFFFu && !counted) ? cvt_e2m1x8(pv) : cvt_e2m1x8_relu(pv);
    if (counted) words[w] += kExact == 0xFFFFu ? cvt_e2m1x8_relu(q1) + cvt_e2m1x8_relu(q2) : cvt_e2m1x6_relu(q1) + cvt_e2m1x6_relu(q2);
  }
}

// Eq. "mx-scale" names both powers of two next to a block maximum.  Here every block takes, of E_c = ceil(max y) and
// E_c - 1, the one with the smaller squared error of its 32 represented probabilities.  Under E_c the code units are
// v = 6 * 2^(y - E_c) (every v through ex2.approx: the conversion count gives codes, not values); under
// E_c - 1 they are 2v, saturating at 6, in units half as large: the floor wins iff
//   sum (2v - q(2v))^2 < 4 sum (v - q(v))^2      (strictly; a block whose maximum is an integer has one candidate).
// Error sums in fp32: eight consecutive keys left to right, the four group sums as (g0 + g1) + (g2 + g3).
__device__ __forceinline__ void direct_p_block_mse(const uint32_t* sraw, float c32, int& E, uint32_t* words) {
  const float LOG2_6 = 2.5849625007211560f;
  const float ymax = fminf(fmaxf(__fmul_rn(max32(sraw), c32), -2097152.0f), 2097152.0f);
  const float M = 12582912.0f;
  const float t = __fadd_ru(ymax, M);
  const float Ec = __fsub_rn(t, M);                              // ceil(ymax), exact
  const float bB = __fsub_rn(LOG2_6, Ec);
  float gc[4], gf[4];
  uint32_t wc[4], wf[4];
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    float v[8], v2[8];
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      float x0, x1;
      fma2(__uint_as_float(sraw[8 * w + i]), __uint_as_float(sraw[8 * w + i + 1]), c32, bB, x0, x1);
      v[i] = ex2_approx(x0);
      v[i + 1] = ex2_approx(x1);
      v2[i] = __fmul_rn(2.0f, v[i]);
      v2[i + 1] = __fmul_rn(2.0f, v[i + 1]);
    }
    wc[w] = cvt_e2m1x8(v);
    wf[w] = cvt_e2m1x8(v2);                                      // saturates at 6
    gc[w] = mx_error_x8(v, wc[w]);
    gf[w] = mx_error_x8(v2, wf[w]);
  }
  const float ec = __fadd_rn(__fadd_rn(gc[0], gc[1]), __fadd_rn(gc[2], gc[3]));
  const float ef = __fadd_rn(__fadd_rn(gf[0], gf[1]), __fadd_rn(gf[2], gf[3]));
  const bool take_f = (ymax != Ec) && (ef < __fmul_rn(4.0f, ec));
  E = (int)(__float_as_uint(t) - 0x4B400000u) - (take_f ? 1 : 0);
#pragma unroll
  for (int w = 0; w < 4; ++w) words[w] = take_f ? wf[w] : wc[w];
}

// Tensor maps of a launch (Q, K, V^T, O in that order) from the calling thread's cache; nullptr if the driver
// refuses to encode one.  Defined beside the one-query kernel.
const CUtensorMap* attention_tensor_maps(int D, const fp4attn_operands* ops, void* O, int B, int H, int Hkv, int N);
// The same with V^T held as E4M3 bytes [B, Hkv, d, N] (box: 128 keys x d rows, 128-byte swizzle).
const CUtensorMap* attention_tensor_maps_fp8v(int D, const fp4attn_operands* ops, void* O, int B, int H, int Hkv, int N);

}  // namespace fp4attn
