// FP8 P/V route of the attention forward (Section "Training stability selects FP8 P/V"): Q and K stay block-scaled
// FP4 and S = Q K^T is the same product as in attn_fwd.cu, but probabilities and V are single E4M3 bytes without
// block scales, P V is a `tcgen05.mma kind::f8f6f4` product, and the row reference is the row maximum itself.
//
//   mu_i  = ceil(max_j y_ij)                         (integer, known before any probability is formed)
//   p8_ij = Q_E4M3(2^(y_ij - mu_i + 8))              (<= 256; round to nearest even; below 2^-10 it is 0)
//   O_i   = sum_j p8_ij V8_j / (G_V sum_j p8_ij),   LSE_i = ln2 (mu_i - 8 + log2 sum_j p8_ij)
//
// Without block scales a probability cannot be re-scaled after it has been rounded, so it must be formed against the
// final reference.  An online running maximum would make the rounded values depend on the tile order (E4M3 flushes
// and loses mantissa bits at the bottom of its range) and would put a reduction over the softmax teams on every
// stage.  The tensor pipe is three quarters idle in this kernel family, so the reference is taken by a first sweep
// instead: every work item walks its keys TWICE - sweep A computes S and reduces the row maxima only, sweep B
// computes S again, forms the bytes against the now final mu and feeds PV.  Nothing is ever rescaled, there is no
// correction pass, and the result equals the plain (not online) definition above.  The second sweep of one item
// and the first sweep of the CTA's next item run interleaved stage by stage (see the schedule comment in the
// kernel), so that SFU-heavy and SFU-free visits alternate on every team.
//
//   warp 0        TMA producer: Q tile per item; a ring of {K, K scales} for all steps and one of V8^T for B-steps
//   warps 1, 23   QK issuers (both kinds of step), one per team pair
//   warp 2        PV issuer (B-steps): four K32 products per 128-key stage, A operand from tensor memory
//   warps 3-6     epilogue: O = O_hw / (L_hw G_V), LSE
//   warps 7-22    softmax teams as in attn_fwd.cu (team 2p + h: h-th 64 keys of the steps with parity p)
//
// The row sum is column d of the accumulator: sixteen rows of E4M3 1.0 follow V8^T in every stage.
// Tensor memory: S slots 0..255 | O 256..399 | Q scales 400..415 | K scales 416..431 | P bytes 432..495 (per step
// parity 32 columns: 128 keys x 8 bits per row) | Q scales of the second QK issuer 496..511.
#include "attn_common.cuh"

namespace fp4attn {
using namespace ptx;

constexpr uint32_t k8ColP = 432, k8ColSFQ1 = 496;
constexpr float kP8Shift = 8.0f;
// The row references go from the teams to the epilogue through one slot an item and no barrier of their own.  A slot is written
// when the item's first sweep ends and read after its last product.  Writers: a team of EITHER pair, with the same values, for
// the products of an item of one stage come from one pair alone, and only that pair's visits are ordered before the epilogue.
// Slots: item k + 4 is written after the second sweeps of items k + 1, k + 2 and k + 3, two of which share a pair; that pair's
// later visit awaited a product of item k + 1 or later, and that product awaited that the epilogue had read item k.
constexpr int kMuSlots = 4;

template <int D, bool NV>
struct Cfg8 {
  using C1 = Cfg<D, NV>;
  static constexpr int V_BYTES = D * BS;                              // V8^T: d rows x 128 bytes
  static constexpr int ONES_BYTES = kOnesRows * BS;                   // rows of E4M3 1.0
  // Two rings: a slot of K is handed back by the score product, one of V8^T by the PV product some two steps later, and only
  // every other step needs V.  Attention alone, us, d=128 N=8192 | d=128 N=1024 | causal N=8192 | d=64 N=8192: one ring of 5 slots
  // (d=64: 8) 748 | 110 | 402 | 718, K and V slots 8 and 3 722 | 104 | 397 | 703.  With the issuers and visits as they are now: V
  // slots 3 680 | 104 | 381 | 646, 4 682 | 97 | 381 | 679; K slots 4, 6, 8 686, 684, 680; a third Q buffer 690 | 95 | 379 | 646.
  // (Short sequences at d = 64 were not timed with more than three.)
  static constexpr int KST_BYTES = (C1::K_BYTES + C1::KSF_BYTES + 1023) / 1024 * 1024;   // K, K scales
  static constexpr int VST_BYTES = V_BYTES + ONES_BYTES;
  static constexpr int KST = 8, VST = (D == 128) ? 4 : 3;
  static constexpr int OFF_Q = 0;                                     // two buffers
  static constexpr int OFF_QSF = OFF_Q + 2 * C1::Q_BYTES;             // two buffers of 1 KB
  static constexpr int OFF_RMAX = OFF_QSF + 2048;                     // [item parity][first-sweep team][row] float
  static constexpr int OFF_MU = OFF_RMAX + 2 * 4 * BM * 4;            // [item % kMuSlots][row] int
  static constexpr int OFF_K = (OFF_MU + kMuSlots * BM * 4 + 1023) / 1024 * 1024;
  static constexpr int OFF_V = OFF_K + KST * KST_BYTES;
  static constexpr int OFF_OUT = OFF_V + VST * VST_BYTES;
  static constexpr int OFF_BAR = OFF_OUT + C1::OUT_BYTES;
  static constexpr int OFF_SEQ = OFF_BAR + 1024;                      // SeqTable
  static constexpr int OFF_ITEMS = OFF_SEQ + 1536;                    // item table
  static constexpr int SMEM_BYTES = OFF_ITEMS + kItemTable * 32 + 1024;
  static_assert(OFF_K % 1024 == 0 && OFF_V % 1024 == 0 && OFF_OUT % 1024 == 0 && SMEM_BYTES <= 227 * 1024, "shared memory");
};

enum { B8_QFULL0 = 0, B8_QFREE0 = 2, B8_OFULL = 4, B8_OFREE = 5, B8_SFULL0 = 6, B8_SEMPTY0 = 8, B8_PFREE0 = 10,
       B8_SMDONE0 = 12, B8_DRAIN0 = 14, B8_MURDY0 = 16, B8_DRAIN2 = 18, B8_RING = 19 };

struct Fp8Params {
  AttnParams a;
  const float* v_G;        // one decode divisor per K/V unit: V^ = V8 / v_G[unit]
};

// D[tmem] (+)= A[tmem] * B[smem], E4M3 x E4M3, K = 32, fp32 accumulate
__device__ __forceinline__ void tc_mma_f8_ta(uint32_t d, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// Instruction descriptor of kind::f8f6f4: 4-5 accumulator format (1 = F32) | 7-9 A format, 10-12 B format (0 = E4M3) |
// 15/16 A/B major (0 = K-major) | 17-22 N >> 3 | 24-28 M >> 4
__host__ __device__ constexpr uint32_t make_idesc_f8(int M, int N) {
  return 1u << 4 | (uint32_t)(N >> 3) << 17 | (uint32_t)(M >> 4) << 24;
}
__device__ __forceinline__ uint32_t cvt_e4m3x4_pos(float a, float b, float c, float d) {   // a in bits 0-7 ... d in bits 24-31
  uint32_t w;
  asm("{\n\t.reg .b16 lo, hi;\n\t"
      "cvt.rn.satfinite.e4m3x2.f32 lo, %2, %1;\n\t"
      "cvt.rn.satfinite.e4m3x2.f32 hi, %4, %3;\n\t"
      "mov.b32 %0, {lo, hi};\n\t}"
      : "=r"(w) : "f"(a), "f"(b), "f"(c), "f"(d));
  return w;
}

// 32 scores of one row -> 32 E4M3 bytes (8 words) against the row's final reference: x = fma(s, c, 8 - mu), c2 = {c, c}
__device__ __forceinline__ void fp8_p_block(const uint32_t* sraw, uint64_t c2, float b, uint32_t* words) {
  const uint64_t bb = pack2(b, b);
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    float pv[4];
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
      float x0, x1;
      unpack2(fma2(pack2(__uint_as_float(sraw[4 * w + i]), __uint_as_float(sraw[4 * w + i + 1])), c2, bb), x0, x1);
      pv[i] = ex2_approx(x0);
      pv[i + 1] = ex2_approx(x1);
    }
    words[w] = cvt_e4m3x4_pos(pv[0], pv[1], pv[2], pv[3]);
  }
}

constexpr int kFp8Threads = kAttnThreads + 32;                 // and the second QK issuer
template <int D, int NV, bool CAUSAL>
__global__ void __launch_bounds__(kFp8Threads, 1)
attn_fwd_fp8pv_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                      const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmO,
                      const Fp8Params pp) {
  const AttnParams& p = pp.a;
  using C = Cfg<D, (NV != 0)>;
  using C8 = Cfg8<D, (NV != 0)>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* sgen = smem_raw + (sbase - smem_u32(smem_raw));
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sgen + C8::OFF_BAR + 768);
  const uint32_t abort_at = sbase + C8::OFF_BAR + 776;
  volatile int* abortf = reinterpret_cast<volatile int*>(sgen + C8::OFF_BAR + 776);
  auto bar = [&](int i) { return sbase + C8::OFF_BAR + 8u * i; };
  auto k_full = [&](int s) { return bar(B8_RING + s); };
  auto k_empty = [&](int s) { return bar(B8_RING + C8::KST + s); };
  auto v_full = [&](int s) { return bar(B8_RING + 2 * C8::KST + s); };
  auto v_empty = [&](int s) { return bar(B8_RING + 2 * C8::KST + C8::VST + s); };
  constexpr uint64_t kDescSF = (uint64_t)(16 >> 4) << 16 | (uint64_t)(128 >> 4) << 32 | 1ull << 46;
  constexpr uint64_t kDescQK = (uint64_t)(16 >> 4) << 16 | (uint64_t)((8 * C::ROW_BYTES) >> 4) << 32 | 1ull << 46 | C::SWZ_QK << 61;
  constexpr uint64_t kDescV = (uint64_t)(16 >> 4) << 16 | (uint64_t)(1024 >> 4) << 32 | 1ull << 46 | kSwz128 << 61;   // 128-byte rows
  auto at = [](uint64_t tmpl, uint32_t addr) { return tmpl | (uint64_t)((addr & 0x3FFFFu) >> 4); };

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int qtiles = p.N / BM;
  if (threadIdx.x == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar(B8_QFULL0 + b), 1);
      mbar_init(bar(B8_QFREE0 + b), 2);        // both QK issuers
      mbar_init(bar(B8_SFULL0 + b), 1);
      mbar_init(bar(B8_SEMPTY0 + b), 8);       // the two teams of the pair, four warps each
      mbar_init(bar(B8_SMDONE0 + b), 8);
      mbar_init(bar(B8_PFREE0 + b), 1);
      mbar_init(bar(B8_MURDY0 + b), 4 * kTeams);   // every softmax warp, once per item (slot by item parity)
      mbar_init(bar(B8_DRAIN0 + b), 1);
    }
    mbar_init(bar(B8_DRAIN2), 1);
    mbar_init(bar(B8_OFULL), 1);
    mbar_init(bar(B8_OFREE), 4);
    for (int s = 0; s < C8::KST; ++s) { mbar_init(k_full(s), 1); mbar_init(k_empty(s), 1); }
    for (int s = 0; s < C8::VST; ++s) { mbar_init(v_full(s), 1); mbar_init(v_empty(s), 1); }
    *abortf = 0;
    fence_barrier_init();
    prefetch_tensormap(&tmQ);
    prefetch_tensormap(&tmK);
    prefetch_tensormap(&tmV);
    prefetch_tensormap(&tmO);
  }
  if (warp == 1) { tmem_alloc(sbase + C8::OFF_BAR + 768, kTmemCols); tmem_relinquish(); }
  // constant operand rows: E4M3 1.0 (0x38) in every byte
  for (int i = threadIdx.x; i < C8::VST * (C8::ONES_BYTES / 4); i += kFp8Threads)
    reinterpret_cast<uint32_t*>(sgen + C8::OFF_V + (i / (C8::ONES_BYTES / 4)) * C8::VST_BYTES + C8::V_BYTES)[i % (C8::ONES_BYTES / 4)] = 0x38383838u;
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  wait_prior_grids();                                           // everything above is this block's own set-up
  const uint32_t tmem = *tslot;
  SeqTable* const seq = reinterpret_cast<SeqTable*>(sgen + C8::OFF_SEQ);
  if (CAUSAL && p.sorted) {
    build_seq_table(seq, p, qtiles);
    fill_skipped<D>(seq, p, qtiles);
  }
  const int n_my = items_of_cta<CAUSAL>(CAUSAL && p.sorted ? seq->first[p.B] : p.n_items);   // this CTA's items: item_at(0 .. n_my - 1)
  ItemRec* const tab = reinterpret_cast<ItemRec*>(sgen + C8::OFF_ITEMS);
  if (CAUSAL) build_item_table<true, false>(tab, n_my, p, qtiles, seq);
  auto work = [&](int i) { return CAUSAL ? item_of_cta<true>(i, tab, p, qtiles, seq) : decode_item<false>(item_at<false>(i), p, qtiles, seq); };

  // Every role walks the same schedule.  Phase ph (0 .. n_my) carries the first sweep ("A": scores -> row maxima) of
  // item ph and the second sweep ("B": scores -> bytes -> PV) of item ph - 1, stage by stage, in the order
  // A B | B A | A B | ... ; the first phase has no B part, the last no A part.  Steps are numbered g = 0, 1, 2 ... in
  // that order; step g uses score slot g & 1 and is served by the team pair g & 1 (teams 2p, 2p + 1), so each pair
  // alternates between the SFU-heavy second sweep of one item and the SFU-free first sweep of the next, and the four
  // warps of a scheduler are never all in the same kind of work.
  if (warp == 0) {
    // ===================================================================== TMA producer
    int s = 0, ph = 0, sv = 0, phv = 0;
    bool ok = true;
    for (int phs = 0; ok && phs <= n_my; ++phs) {
      WorkItem wa = {}, wb = {};
      int TA = 0, TB = 0;
      if (phs < n_my) { wa = work(phs); TA = wa.T2; }
      if (phs >= 1) { wb = work(phs - 1); TB = wb.T2; }
      if (phs < n_my) {
        const int qb = phs & 1;
        if (phs >= 2) ok = mbar_wait<false>(bar(B8_QFREE0 + qb), ((phs >> 1) - 1) & 1, abort_at);
        if (!ok) break;
        if (elect_one()) {
          mbar_arrive_expect_tx(bar(B8_QFULL0 + qb), C::Q_BYTES + C::QSF_BYTES);
          tma_load_2d(sbase + C8::OFF_Q + qb * C::Q_BYTES, &tmQ, 0, wa.qrow0, bar(B8_QFULL0 + qb));
          bulk_load_1d(sbase + C8::OFF_QSF + qb * 1024, p.q_sf + (size_t)wa.qtile_lin * C::QSF_BYTES, C::QSF_BYTES, bar(B8_QFULL0 + qb));
        }
      }
      const int TM = TA > TB ? TA : TB;
      for (int s2 = 0; ok && s2 < TM; ++s2) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int kind = j ^ (s2 & 1);                            // 0: A-step of item phs, 1: B-step of item phs - 1
          if (s2 >= (kind ? TB : TA)) continue;
          const WorkItem& wi = kind ? wb : wa;
          ok = mbar_wait<false>(k_empty(s), ph ^ 1, abort_at);      // (a fresh barrier passes)
          if (ok && kind) ok = mbar_wait<false>(v_empty(sv), phv ^ 1, abort_at);
          if (!ok) break;
          const uint32_t fb = k_full(s), st = sbase + C8::OFF_K + s * C8::KST_BYTES;
          if (elect_one()) {
            mbar_arrive_expect_tx(fb, C::K_BYTES + C::KSF_BYTES);
            tma_load_2d(st, &tmK, 0, wi.kvh * p.N + s2 * BS, fb);
            bulk_load_1d(st + C::K_BYTES, p.k_sf + ((size_t)wi.kvh * qtiles + s2) * C::KSF_BYTES, C::KSF_BYTES, fb);
            if (kind) {
              mbar_arrive_expect_tx(v_full(sv), C8::V_BYTES);
              tma_load_2d(sbase + C8::OFF_V + sv * C8::VST_BYTES, &tmV, s2 * BS, wi.kvh * D, v_full(sv));
            }
          }
          if (++s == C8::KST) { s = 0; ph ^= 1; }
          if (kind && ++sv == C8::VST) { sv = 0; phv ^= 1; }
        }
      }
    }
    if (*abortf && lane == 0) {
      for (int r = 0; r < C8::KST; ++r)
        for (int spin = 0; spin < (1 << 12) && !mbar_try_wait(k_full(r), 0) && !mbar_try_wait(k_full(r), 1); ++spin) {}
      for (int r = 0; r < C8::VST; ++r)
        for (int spin = 0; spin < (1 << 12) && !mbar_try_wait(v_full(r), 0) && !mbar_try_wait(v_full(r), 1); ++spin) {}
    }
    __syncwarp();
  } else if (warp == 1 || warp == kFirstSoftmaxWarp + 4 * kTeams) {
    // ===================================================================== QK issuers (both sweeps), one for the steps of either team pair
    // A pair waits for a score product after each of its A-visits, which are short, so what counts here is the time from the
    // last read of a slot to the next product into it.  One warp for both pairs takes some 550 clocks from issue to issue and
    // serves them in step order; two each wait for their own pair (the second on the scheduler that had no issuing warp).
    // With the visits as they are below: 745 -> 680 us at d=128, N=8192, 706 -> 646 at d=64.
    constexpr uint32_t kIdQK0 = NV ? make_idesc_fp4(BM, BS, false, 0, 0) : make_idesc_fp4(BM, BS, true, 0, 0);
    constexpr uint32_t kIdQK1 = NV ? make_idesc_fp4(BM, BS, false, 0, 0) : make_idesc_fp4(BM, BS, true, 2, 2);
    const int pr = warp == 1 ? 0 : 1;
    static_assert(C8::KST % 2 == 0, "a ring slot's steps belong to one pair");
    const uint32_t tSFK = tmem + kColSFK + 8 * pr, tS = tmem + kColS + BS * pr, tSFQ0 = tmem + (pr ? k8ColSFQ1 : kColSFQ);
    int sq = pr, phq = 0;
    uint32_t stq = sbase + C8::OFF_K + pr * C8::KST_BYTES;
    uint32_t g = 0, m = 0;                                      // steps so far (both kinds, all items); of this warp's: issued so far
    bool ok = true;
    for (int phs = 0; ok && phs <= n_my; ++phs) {
      int TA = 0, TB = 0;
      if (phs < n_my) TA = work(phs).T2;
      if (phs >= 1) TB = work(phs - 1).T2;
      if (phs < n_my) {
        const int qb = phs & 1;
        ok = mbar_wait<false>(bar(B8_QFULL0 + qb), (phs >> 1) & 1, abort_at);
        if (!ok) break;
        tc_fence_after();
        if (elect_one()) {
#pragma unroll
          for (int a = 0; a < C::CTQ; ++a)
            tc_cp_32x128b_warpx4(tSFQ0 + 8 * qb + 4 * a, at(kDescSF, sbase + C8::OFF_QSF + qb * 1024 + 512 * a));
        }
        __syncwarp();
      }
      const int TM = TA > TB ? TA : TB;
      for (int s2 = 0; ok && s2 < TM; ++s2) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int kind = j ^ (s2 & 1);
          if (s2 >= (kind ? TB : TA)) continue;
          if ((int)(g & 1) != pr) { ++g; continue; }              // the other warp's step
          const int qb = (kind ? phs - 1 : phs) & 1;              // the Q buffer of the step's item
          ok = mbar_wait<false>(k_full(sq), phq, abort_at);
          if (ok) ok = mbar_wait<false>(bar(B8_SEMPTY0 + pr), (m & 1) ^ 1, abort_at);   // both teams have read the slot (a fresh barrier passes)
          if (!ok) break;
          tc_fence_after();
          const uint32_t tSFQ = tSFQ0 + 8 * qb;
          const uint64_t dQ0 = at(kDescQK, sbase + C8::OFF_Q + qb * C::Q_BYTES);
          const uint64_t dK0 = at(kDescQK, stq);
          if (elect_one()) {
#pragma unroll
            for (int a = 0; a < C::CTQ; ++a) tc_cp_32x128b_warpx4(tSFK + 4 * a, at(kDescSF, stq + C::K_BYTES + 512 * a));
            if (NV) {
              tc_mma_fp4_4x(tS, dQ0, dK0, kIdQK0, tSFQ, tSFK, 0);
              if (C::KBLK == 2) tc_mma_fp4_4x(tS, dQ0 + 2, dK0 + 2, kIdQK1, tSFQ + 4, tSFK + 4, 1);
            } else {
              tc_mma_fp4_2x(tS, dQ0, dK0, kIdQK0, tSFQ, tSFK, 0);
              if (C::KBLK == 2) tc_mma_fp4_2x(tS, dQ0 + 2, dK0 + 2, kIdQK1, tSFQ, tSFK, 1);
            }
            tc_commit(bar(B8_SFULL0 + pr));
            tc_commit(k_empty(sq));                               // K back to the producer
          }
          __syncwarp();
          ++g;
          ++m;
          stq += 2 * C8::KST_BYTES;
          if ((sq += 2) >= C8::KST) { sq = pr; phq ^= 1; stq = sbase + C8::OFF_K + pr * C8::KST_BYTES; }
        }
      }
      if (ok && phs >= 1) {                                       // this warp's products of item phs - 1 are issued: its Q buffer may take item phs + 1
        if (elect_one()) tc_commit(bar(B8_QFREE0 + ((phs - 1) & 1)));
        __syncwarp();
      }
    }
    if (*abortf && elect_one()) tc_commit(bar(pr ? B8_DRAIN2 : B8_DRAIN0));
    __syncwarp();
  } else if (warp == 2) {
    // ===================================================================== PV issuer (B-steps)
    constexpr uint32_t kIdPV = make_idesc_f8(BM, C::DN);
    const uint32_t tO = tmem + kColO;
    uint32_t g = 0;                                             // steps so far (both kinds): team pair of a step
    int sv = 0, phv = 0;
    uint32_t nb[2] = {0, 0};                                    // B-steps served so far, per team pair
    bool ok = true;
    for (int phs = 0; ok && phs <= n_my; ++phs) {
      int TA = 0, TB = 0;
      if (phs < n_my) TA = work(phs).T2;
      if (phs >= 1) TB = work(phs - 1).T2;
      if (phs >= 2) ok = mbar_wait<false>(bar(B8_OFREE), (phs - 2) & 1, abort_at);   // epilogue of item phs - 2 has read O
      const int TM = TA > TB ? TA : TB;
      for (int s2 = 0; ok && s2 < TM; ++s2) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int kind = j ^ (s2 & 1);
          if (s2 >= (kind ? TB : TA)) continue;
          if (kind == 0) { ++g; continue; }                       // an A-step: only its slot is counted
          const int pr = g & 1;
          ok = mbar_wait<false>(bar(B8_SMDONE0 + pr), (pr ? nb[1] : nb[0]) & 1, abort_at);   // bytes of both tiles are in tensor memory
          if (ok) ok = mbar_wait<false>(v_full(sv), phv, abort_at);
          if (!ok) break;
          if (pr) ++nb[1]; else ++nb[0];
          tc_fence_after();
          const uint64_t dV = at(kDescV, sbase + C8::OFF_V + sv * C8::VST_BYTES);
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)                         // 32 keys per product: 8 columns of P, 32 bytes along V8^T's rows
              tc_mma_f8_ta(tO, tmem + k8ColP + 32 * pr + 8 * kk, dV + 2 * kk, kIdPV, (s2 > 0 || kk > 0) ? 1u : 0u);
            tc_commit(v_empty(sv));                               // V back to the producer
            tc_commit(bar(B8_PFREE0 + pr));
            if (s2 == TB - 1) tc_commit(bar(B8_OFULL));
          }
          __syncwarp();
          ++g;
          if (++sv == C8::VST) { sv = 0; phv ^= 1; }
        }
      }
    }
    if (*abortf && elect_one()) tc_commit(bar(B8_DRAIN0 + 1));
    __syncwarp();
  } else if (warp < kFirstSoftmaxWarp) {
    // ===================================================================== epilogue warps
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;
    const uint32_t tO = tmem + ((uint32_t)(quarter * 32) << 16) + kColO;
    bool ok = true;
    for (int k = 0; ok && k < n_my; ++k) {
      const WorkItem wi = work(k);
      ok = mbar_wait<false>(bar(B8_OFULL), k & 1, abort_at);
      if (!ok) break;
      tc_fence_after();
      const int mu = reinterpret_cast<const volatile int*>(sgen + C8::OFF_MU)[(k % kMuSlots) * BM + row];
      float Lhw;
      {
        uint32_t r16[16];
        tmem_ld_32x32b_x16(tO + D, r16);
        tmem_wait_ld();
        Lhw = __uint_as_float(r16[0]);
      }
      const float inv = __frcp_rn(Lhw * __ldcg(pp.v_G + wi.kvh));
      if (lane == 0) bulk_wait_read_all();
      __syncwarp();
#pragma unroll
      for (int c0 = 0; c0 < D; c0 += 16) {
        uint32_t o[16];
        tmem_ld_32x32b_x16(tO + c0, o);
        tmem_wait_ld();
        if (c0 + 16 == D) {                                     // last read of O
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(B8_OFREE));
        }
        uint8_t* half = sgen + C8::OFF_OUT + (c0 >> 6) * (BM * 128) + row * 128;
#pragma unroll
        for (int c = 0; c < 16; c += 8) {
          uint32_t pk[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const __nv_bfloat162 hh = __floats2bfloat162_rn(__uint_as_float(o[c + 2 * q]) * inv, __uint_as_float(o[c + 2 * q + 1]) * inv);
            pk[q] = *reinterpret_cast<const uint32_t*>(&hh);
          }
          const int chunk = ((c0 & 63) + c) >> 3;
          *reinterpret_cast<uint4*>(half + ((chunk ^ (row & 7)) << 4)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        }
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
#pragma unroll
        for (int hf = 0; hf < D / 64; ++hf)
          tma_store_2d(&tmO, hf * 128, wi.qrow0 + quarter * 32, sbase + C8::OFF_OUT + hf * (BM * 128) + quarter * 32 * 128);
        bulk_commit_group();
      }
      if (p.LSE) p.LSE[(size_t)wi.qrow0 + row] = 0.69314718055994531f * ((float)mu - kP8Shift + log2f(Lhw));
    }
  } else {
    // ===================================================================== softmax teams
    const int team = (warp - kFirstSoftmaxWarp) >> 2;
    const int pr = team >> 1;                                   // the steps with g & 1 == pr are this pair's
    const int h = team & 1;                                     // which 64 keys of a stage
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;
    const uint32_t tS = tmem + ((uint32_t)(quarter * 32) << 16) + kColS + BN * team;
    const uint32_t sfull = bar(B8_SFULL0 + pr), sempty = bar(B8_SEMPTY0 + pr);
    const uint32_t smdone = bar(B8_SMDONE0 + pr), pfree = bar(B8_PFREE0 + pr);
    const uint32_t tP = tmem + ((uint32_t)(quarter * 32) << 16) + k8ColP + 32 * pr + 16 * h;
    uint64_t c2 = p.c_mx2;                                      // MXFP4: a kernel parameter, read from uniform registers
    if (NV) {
      const float c = __fdiv_rn(p.c_base, __fmul_rn(__ldcg(p.q_G), __ldcg(p.k_G)));
      c2 = pack2(c, c);
    }
    const float c32 = __uint_as_float((uint32_t)c2);
    bool ok = true;
    uint32_t g = 0;                                             // steps so far (both kinds, all pairs)
    uint32_t nbt = 0;                                           // B-visits of this team so far
    // keys of the team's tile that this row sees in an item's last stage, the masked one (causal: keys 0..i of row
    // i = qt * 128 + row; padded sequence: keys 0..len-1; both: the fewer)
    auto tile_keys = [&](const WorkItem& w) {
      const int seen = p.causal ? min(w.len, w.qt * BM + row + 1) : w.len;
      return seen - (w.T2 - 1) * BS - 64 * h;
    };
    float b = 0.f;                                              // 8 - mu of the item in its second sweep
    for (int phs = 0; ok && phs <= n_my; ++phs) {
      WorkItem wa = {}, wb = {};
      int TA = 0, TB = 0;
      if (phs < n_my) { wa = work(phs); TA = wa.T2; }
      if (phs >= 1) { wb = work(phs - 1); TB = wb.T2; }
      const int va = CAUSAL ? tile_keys(wa) : 64, vb = CAUSAL ? tile_keys(wb) : 64;
      float smax = -INFINITY;                                   // this team's share of the maxima of item phs
      auto first_sweep_step = [&](bool diag) {                  // scores of item phs: maxima only
        uint32_t sraw[32];
        tmem_ld_32x32b_x32(tS, sraw);
        tmem_wait_ld();
        if (diag) mask_scores(sraw, va);
        smax = fmaxf(smax, max32(sraw));
        tmem_ld_32x32b_x32(tS + 32, sraw);
        tmem_wait_ld();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(sempty);
        if (diag) mask_scores(sraw, va - 32);
        smax = fmaxf(smax, max32(sraw));
      };
      bool swept = false;                                       // the pair's next A-step is done already
      const int TM = TA > TB ? TA : TB;
      for (int s2 = 0; ok && s2 < TM; ++s2) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int kind = j ^ (s2 & 1);
          if (s2 >= (kind ? TB : TA)) continue;
          if ((int)(g & 1) != pr) { ++g; continue; }              // the other pair's step
          if (kind == 0 && swept) { swept = false; ++g; continue; }
          ok = mbar_wait<false>(sfull, (g >> 1) & 1, abort_at);
          if (!ok) break;
          tc_fence_after();
          if (kind == 0) {
            first_sweep_step(CAUSAL && s2 == TA - 1);
          } else {
            // ---- second sweep of item phs - 1: bytes against its final reference
            uint32_t sraw[32], w[8];
            const bool diag = CAUSAL && s2 == TB - 1;
            tmem_ld_32x32b_x32(tS, sraw);
            tmem_wait_ld();
            fp8_p_block(sraw, c2, b, w);
            if (diag) mask_bytes(w, vb);
            tmem_ld_32x32b_x32(tS + 32, sraw);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(sempty);
            // the pair's probability slot was last read by the PV product of this team's previous B-visit
            if (nbt > 0) ok = mbar_wait<false>(pfree, (nbt - 1) & 1, abort_at);
            if (!ok) break;
            tmem_st_32x32b_x8(tP, w);
            fp8_p_block(sraw, c2, b, w);
            if (diag) mask_bytes(w, vb - 32);
            // The pair's next step is an A-step, whose scores may be there by now: they are reduced first, so that the product
            // after them, which the pair then waits for (580 of the 3080 clocks of an A- and a B-visit), starts a tail of this
            // visit earlier: 686 -> 680 us, d=64 677 -> 646.  The first half's bytes are in tensor memory by then: with all
            // sixteen words held the unmasked kernels spill 28 bytes and take 734 us.
            if (s2 + 1 < min(TA, TB) && mbar_test(sfull, ((g >> 1) + 1) & 1)) {
              tc_fence_after();
              first_sweep_step(CAUSAL && s2 + 1 == TA - 1);
              swept = true;
            }
            tmem_st_32x32b_x8(tP + 8, w);
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smdone);
            ++nbt;
          }
          ++g;
        }
      }
      if (!ok) break;
      if (phs < n_my) {
        // ---- the sixteen softmax warps meet: mu of item phs = ceil(c * max over all its keys), on the FMA pipe
        float* rmax = reinterpret_cast<float*>(sgen + C8::OFF_RMAX) + (phs & 1) * 4 * BM;
        rmax[team * BM + row] = smax;                           // (-inf from a team that served none of the item's A-steps)
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(B8_MURDY0 + (phs & 1)));
        ok = mbar_wait<false>(bar(B8_MURDY0 + (phs & 1)), (phs >> 1) & 1, abort_at);
        if (!ok) break;
        const float mall = fmaxf(fmaxf(rmax[row], rmax[BM + row]), fmaxf(rmax[2 * BM + row], rmax[3 * BM + row]));
        const float ymax = fminf(fmaxf(__fmul_rn(mall, c32), -2097152.0f), 2097152.0f);
        const float tt = __fadd_ru(ymax, 12582912.0f);          // ceil, exact for |y| < 2^22
        b = __fsub_rn(kP8Shift, __fsub_rn(tt, 12582912.0f));
        if (h == 0) reinterpret_cast<volatile int*>(sgen + C8::OFF_MU)[(phs % kMuSlots) * BM + row] = (int)(__float_as_uint(tt) - 0x4B400000u);
      }
    }
  }
  if (warp >= 3 && warp < kFirstSoftmaxWarp && lane == 0) bulk_wait_all();
  __syncthreads();
  if (*abortf && threadIdx.x == 0 && p.status) *p.status = FP4ATTN_ERR_TIMEOUT;
  if (warp == 1) {
    if (*abortf && lane == 0) {
      for (int r = 0; r < 3; ++r)
        for (int spin = 0; spin < (1 << 14) && !mbar_try_wait(bar(r == 2 ? B8_DRAIN2 : B8_DRAIN0 + r), 0); ++spin) {}
    }
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

template <int D, int NV, bool CAUSAL>
static int launch_fp8(const fp4attn_operands* ops, int B, int H, int N, const Fp8Params& prm, cudaStream_t st) {
  using C8 = Cfg8<D, (NV != 0)>;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return FP4ATTN_ERR_CUDA;
  static std::atomic<bool> attr_set[kMaxDevices];
  if (dev < 0 || dev >= kMaxDevices) return FP4ATTN_ERR_CUDA;
  if (!attr_set[dev].load(std::memory_order_acquire)) {
    if (cudaFuncSetAttribute(attn_fwd_fp8pv_kernel<D, NV, CAUSAL>, cudaFuncAttributeMaxDynamicSharedMemorySize, C8::SMEM_BYTES) != cudaSuccess)
      return FP4ATTN_ERR_CUDA;
    attr_set[dev].store(true, std::memory_order_release);
  }
  const CUtensorMap* tm = attention_tensor_maps_fp8v(D, ops, prm.a.O, B, H, prm.a.Hkv, N);
  if (!tm) return FP4ATTN_ERR_CUDA;
  const unsigned grid = (unsigned)(prm.a.n_items < sms ? prm.a.n_items : sms);
  launch_overlapped(attn_fwd_fp8pv_kernel<D, NV, CAUSAL>, dim3(grid), kFp8Threads, C8::SMEM_BYTES, st, tm[0], tm[1], tm[2], tm[3], prm);
  return cudaGetLastError() == cudaSuccess ? FP4ATTN_OK : FP4ATTN_ERR_CUDA;
}

// Entry used by fp4attn_fwd for pv_fmt = FP4ATTN_PV_E4M3; `prm` is filled as for the one-query FP4 kernel.
int launch_attn_fp8pv(const fp4attn_operands* ops, int B, int H, int N, int d, AttnParams prm, cudaStream_t st) {
  if (!ops->v_G) return FP4ATTN_ERR_INVALID_ARG;
  if (ops->p_map != FP4ATTN_PMAP_IDEAL || ops->p_scale_rule != FP4ATTN_PSCALE_CEIL || ops->g_per_head ||
      ops->schedule == FP4ATTN_SCHEDULE_TWO_QUERY)
    return FP4ATTN_ERR_INVALID_ARG;                               // the code maps and block rules belong to the FP4 probability path
  Fp8Params pp{prm, ops->v_G};
  const bool nv = ops->qk_fmt == FP4ATTN_FMT_NVFP4;
  const int sel = (d == 128 ? 4 : 0) | (nv ? 2 : 0) | ((prm.causal || prm.seq_len) ? 1 : 0);   // masked instances
  switch (sel) {
    case 0: return launch_fp8<64, 0, false>(ops, B, H, N, pp, st);
    case 1: return launch_fp8<64, 0, true>(ops, B, H, N, pp, st);
    case 2: return launch_fp8<64, 1, false>(ops, B, H, N, pp, st);
    case 3: return launch_fp8<64, 1, true>(ops, B, H, N, pp, st);
    case 4: return launch_fp8<128, 0, false>(ops, B, H, N, pp, st);
    case 5: return launch_fp8<128, 0, true>(ops, B, H, N, pp, st);
    case 6: return launch_fp8<128, 1, false>(ops, B, H, N, pp, st);
    default: return launch_fp8<128, 1, true>(ops, B, H, N, pp, st);
  }
}

}  // namespace fp4attn
