// Operand quantizers: bf16 -> packed E2M1 + scale bytes in the 128x4 atom order.
// HBM-bound: 256-bit loads (128-bit ones from tensors on a 16-byte boundary, and cp.async into shared memory for V), block
// maxima by lane shuffles, 32- to 128-bit stores.  Loads are ld.global.cg: a kernel may have
// started before its inputs were written (programmatic dependent launch), which rules out the non-coherent path.
#include "common.cuh"

namespace fp4attn {

constexpr int kThreads = 256;
constexpr int kGroupsPerCta = 1024;          // 16-byte groups (eight elements) of a chunk: what a CTA takes at a time
constexpr int kLoads = kGroupsPerCta / 2 / kThreads;   // 32-byte loads of a thread and chunk
constexpr int kRowsCtas = 4;                  // CTAs of the rows kernels per SM
constexpr int kMaxPartials = 1024;           // NVFP4 amax pass: one partial maximum per block
constexpr int kPartialsPerHead = 32;         // the same, per (batch, head) unit, for per-head factors

// ---------------------------------------------------------------- MXFP4, blocks along d (Q, K)
// |bf16| bit patterns order like the magnitudes, so the block maximum is taken on packed 16-bit
// integers; 6 v / alpha = v * (1.5 * 2^(129-u)) is one exact fp32 multiply.
// E8M0 byte from the bf16 bit pattern of the block maximum a = (1 + m/128) 2^(e-127): the biased exponent
// e, plus one where the rule rounds the amplitude up (Eq. "mx-scale" allows either neighbouring power of
// two): ceiling - whenever a is not a power of two; threshold - alpha = 2^floor(log2(1.6 a)), i.e. when
// 1 + m/128 >= 1.25; floor - never.  Values above the amplitude saturate at code 6 in the conversion.
template <int RULE>
__device__ __forceinline__ uint32_t mx_scale_byte_bf16(uint32_t a16) {
  if (a16 == 0) return 0;
  const uint32_t m = a16 & 0x7Fu;
  const uint32_t up = RULE == FP4ATTN_QSCALE_CEIL ? (m != 0) : RULE == FP4ATTN_QSCALE_THR16 ? (m >= 32u) : 0u;
  return min(max((a16 >> 7) + up, 1u), 254u);
}
// two products per instruction
template <int N_>
__device__ __forceinline__ void scale_values(float* v, float f) {
#pragma unroll
  for (int i = 0; i < N_; i += 2)
    asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %4};\n\tmul.rn.f32x2 c, a, b;\n\tmov.b64 {%0, %1}, c;\n\t}"
        : "=f"(v[i]), "=f"(v[i + 1]) : "f"(v[i]), "f"(v[i + 1]), "f"(f));
}
// v[i] <- 6 v[i] / alpha for the amplitude of byte u: exact in fp32 (one multiply by 1.5 * 2^k)
template <int N_>
__device__ __forceinline__ void mx_scale_values(float* v, uint32_t u) {
  if (u >= 2u) {
    scale_values<N_>(v, __uint_as_float(((256u - u) << 23) | 0x400000u));   // 1.5 * 2^(129-u) = 6 / alpha
  } else {                                                              // alpha = 2^-126: 6/alpha overflows fp32
    const float inv = mx_inv_amplitude(u);
#pragma unroll
    for (int i = 0; i < N_; ++i) v[i] = (v[i] * inv) * 6.0f;
  }
}
__device__ __forceinline__ uint32_t mx_codes_x8(const uint4& raw, uint32_t u) {
  float v[8];
  bf16x8_to_f32(raw, v);
  mx_scale_values<8>(v, u);
  return cvt_e2m1x8(v);
}
// MSE rule, blocks along d: two eight-element groups of a block sit in a lane, the other two in its neighbour, so the
// group sums meet as (g0 + g1) + (g2 + g3) in both.  The floor's error is in units four times
// smaller than the ceiling's, hence the factor; the floor wins only if strictly better.  Returns the
// chosen byte, `word` gets this lane's codes under it.
__device__ __forceinline__ uint32_t mx_choose_mse_rows(const uint32_t* raw, uint32_t a16, uint32_t* words) {
  const uint32_t uf = mx_scale_byte_bf16<FP4ATTN_QSCALE_FLOOR>(a16), uc = mx_scale_byte_bf16<FP4ATTN_QSCALE_CEIL>(a16);
  uint32_t wf[2], wc[2];
  float ef[2], ec[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float tf[8], tc[8];
    bf16x8_to_f32(make_uint4(raw[4 * h], raw[4 * h + 1], raw[4 * h + 2], raw[4 * h + 3]), tf);
#pragma unroll
    for (int i = 0; i < 8; ++i) tc[i] = tf[i];
    mx_scale_values<8>(tf, uf);
    mx_scale_values<8>(tc, uc);
    wf[h] = cvt_e2m1x8(tf);
    wc[h] = cvt_e2m1x8(tc);
    ef[h] = mx_error_x8(tf, wf[h]);
    ec[h] = mx_error_x8(tc, wc[h]);
  }
  float f = __fadd_rn(ef[0], ef[1]), c = __fadd_rn(ec[0], ec[1]);
  f = __fadd_rn(f, __shfl_xor_sync(0xffffffffu, f, 1));
  c = __fadd_rn(c, __shfl_xor_sync(0xffffffffu, c, 1));
  const bool take_f = (uf != uc) && (f < __fmul_rn(4.0f, c));
  words[0] = take_f ? wf[0] : wc[0];
  words[1] = take_f ? wf[1] : wc[1];
  return take_f ? uf : uc;
}

// 32 bytes in one load (64 a thread and chunk, and the next chunk's in flight while this one is converted): sixteen elements
// of a row, so that half a 32-block, or a whole 16-block, needs no lane exchange and its scale is formed once, not twice.
// W32: the tensor starts on a 32-byte boundary; one that only starts on a 16-byte boundary takes two loads.
template <bool W32>
__device__ __forceinline__ void load_16(uint32_t* r, const uint4* p) {
  if (W32) {
    asm volatile("ld.global.cg.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "l"(p) : "memory");
  } else {
    const uint4 lo = __ldcg(p), hi = __ldcg(p + 1);
    r[0] = lo.x; r[1] = lo.y; r[2] = lo.z; r[3] = lo.w;
    r[4] = hi.x; r[5] = hi.y; r[6] = hi.z; r[7] = hi.w;
  }
}
__device__ __forceinline__ uint32_t absmax_bf16x16(const uint32_t* r) {
  uint32_t m = r[0] & 0x7FFF7FFFu;
#pragma unroll
  for (int i = 1; i < 8; ++i) m = __vmaxu2(m, r[i] & 0x7FFF7FFFu);
  return max(m & 0xFFFFu, m >> 16);
}

// Bound by HBM.  67 M elements back to back on one stream: 26.7 us, 6.37 TB/s (one CTA per chunk, 16-byte loads, byte stores
// of the scales, a plain launch: 30.8); 3 / 4 / 5 CTAs per SM 27.5 / 26.7 / 27.6.
// The rows of all units are one list (a unit is a whole number of 128-row atoms), cut into chunks of kGroupsPerCta groups.
// grid rows_grid(): persistent CTAs that walk the chunks
template <int D, int RULE, bool W32>
__global__ void __launch_bounds__(kThreads, RULE == FP4ATTN_QSCALE_MSE ? 3 : kRowsCtas)
quant_mx_rows_kernel(const uint4* __restrict__ x, uint2* __restrict__ packed, uint8_t* __restrict__ sf, uint32_t n_chunks) {
  constexpr uint32_t LPR = D / 16;                 // lanes per row
  launch_dependents();
  wait_prior_grids();
  const uint32_t seg = threadIdx.x % LPR;
  uint32_t chunk = blockIdx.x, raw[kLoads][8];
#pragma unroll
  for (int k = 0; k < kLoads; ++k) load_16<W32>(raw[k], x + (size_t)chunk * kGroupsPerCta + 2 * (threadIdx.x + k * kThreads));
  while (true) {
    const uint32_t next = chunk + gridDim.x;
    uint32_t ahead[kLoads][8];
    if (next < n_chunks) {
#pragma unroll
      for (int k = 0; k < kLoads; ++k) load_16<W32>(ahead[k], x + (size_t)next * kGroupsPerCta + 2 * (threadIdx.x + k * kThreads));
    }
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
      uint32_t a = absmax_bf16x16(raw[k]);
      a = max(a, __shfl_xor_sync(0xffffffffu, a, 1));
      uint32_t u, w[2];
      if (RULE == FP4ATTN_QSCALE_MSE) {
        u = mx_choose_mse_rows(raw[k], a, w);
      } else {
        u = mx_scale_byte_bf16<RULE>(a);
        w[0] = mx_codes_x8(make_uint4(raw[k][0], raw[k][1], raw[k][2], raw[k][3]), u);
        w[1] = mx_codes_x8(make_uint4(raw[k][4], raw[k][5], raw[k][6], raw[k][7]), u);
      }
      packed[(size_t)chunk * (kGroupsPerCta / 2) + threadIdx.x + k * kThreads] = make_uint2(w[0], w[1]);
      // the row's scale bytes as one word, from the lanes of its blocks (d = 64: two of them, and two columns of padding)
      u |= __shfl_xor_sync(0xffffffffu, u, 2) << 8;
      if (D == 128) u |= __shfl_xor_sync(0xffffffffu, u, 4) << 16;
      const uint32_t row = chunk * (kGroupsPerCta / 2 / LPR) + (threadIdx.x + k * kThreads) / LPR;
      if (seg == 0) *reinterpret_cast<uint32_t*>(sf + (size_t)(row >> 7) * 512 + (row & 31) * 16 + ((row & 127) >> 5) * 4) = u;
    }
    if (next >= n_chunks) return;
    chunk = next;
#pragma unroll
    for (int k = 0; k < kLoads; ++k)
#pragma unroll
      for (int i = 0; i < 8; ++i) raw[k][i] = ahead[k][i];
  }
}

// ---------------------------------------------------------------- MXFP4, blocks along keys (V), transposed out
// A [128 keys x D] tile (contiguous in memory) goes through shared memory; a thread owns two adjacent head-dim
// columns and one 32-key block, reads them as bf16x2 words and writes two 16-byte code groups.  A warp owns eight column
// pairs of all four key blocks, so that a column's four code groups leave as 64 contiguous bytes (two whole sectors) and its
// four scale bytes meet by lane exchange; 16-byte chunk c of a tile row sits at c ^ 2 (key block), which keeps the reads of
// the four blocks in different banks.  (One warp per key block, with half-sector stores and the scale bytes meeting in shared
// memory: 29.5 us for 67 M elements at d = 128; this way 29.0.)
// Registers are not capped: at 102 a thread two CTAs fit an SM and take 27.6 us (d = 64: 27.7); capped to 80, three with 29.1
// (30.5); three tile buffers 29.3, four 27.0 (31.0).
// Persistent CTAs walk the tiles with two tile buffers: the asynchronous copies (cp.async, 16 bytes per thread
// and copy, no registers in between) of the next tile are in flight while the current one is converted, so the
// memory system always has work although each tile passes through a load -> barrier -> convert sequence.
// grid min(tiles, CTAs that fit) , 2*D threads, dynamic shared memory two tiles
template <int D> constexpr int kVTileBytes = 128 * D * 2;
template <int D> __device__ __forceinline__ uint32_t v_swizzle(uint32_t key) { return 2 * ((key >> 5) & 3); }   // on the chunk index
__device__ __forceinline__ void cp_async_16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory"); }

template <int D, int RULE>
__global__ void __launch_bounds__(2 * D, 1)
quant_mx_v_kernel(const uint4* __restrict__ x, uint4* __restrict__ packed, uint8_t* __restrict__ sf, int N, int n_tiles) {
  constexpr int T = 2 * D;                         // threads: D/2 column pairs x 4 key blocks
  constexpr int LOADS = 128 * D / 8 / T;           // 16-byte copies per thread and tile: 8
  extern __shared__ __align__(16) uint8_t vsm[];
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(vsm);
  const int tiles_per_head = N / 128;
  const int cp = (threadIdx.x >> 5) * 8 + (threadIdx.x & 7);   // column pair: columns 2cp, 2cp+1
  const int kb = (threadIdx.x >> 3) & 3;           // key block 0..3
  auto issue = [&](int t, int buf) {               // tile t is contiguous: 128 keys x D bf16 starting at key 128 t of the flat [B*H*N] key space
    const uint4* src = x + (size_t)t * (128 * D / 8);
#pragma unroll
    for (int k = 0; k < LOADS; ++k) {
      const uint32_t j = threadIdx.x + k * T;      // 16-byte chunk of the tile, in row j / (D / 8)
      cp_async_16(sbase + buf * kVTileBytes<D> + (j ^ v_swizzle<D>(j / (D / 8))) * 16, src + j);
    }
    cp_async_commit();
  };
  int t = blockIdx.x, i = 0;
  launch_dependents();
  wait_prior_grids();
  if (t < n_tiles) issue(t, 0);
  for (; t < n_tiles; t += gridDim.x, ++i) {
    const int tn = t + gridDim.x;
    if (tn < n_tiles) { issue(tn, (i + 1) & 1); cp_async_wait<1>(); } else { cp_async_wait<0>(); }
    __syncthreads();
    const uint32_t* tile = reinterpret_cast<const uint32_t*>(vsm + (i & 1) * kVTileBytes<D>);
    const size_t bh = t / tiles_per_head;
    const int kt = t - (int)bh * tiles_per_head;     // 128-key tile within the head
    uint32_t w[32];
    uint32_t m = 0;
#pragma unroll
    for (int r = 0; r < 32; ++r) {
      w[r] = tile[(kb * 32 + r) * (D / 2) + (cp ^ (8 * kb))];
      m = __vmaxu2(m, w[r] & 0x7FFF7FFFu);
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {                    // low half = column 2cp, high half = column 2cp+1
      const uint32_t a16 = c ? (m >> 16) : (m & 0xFFFFu);
      uint32_t u = mx_scale_byte_bf16<RULE == FP4ATTN_QSCALE_MSE ? FP4ATTN_QSCALE_CEIL : RULE>(a16);
      float v[32];
#pragma unroll
      for (int r = 0; r < 32; ++r) v[r] = __uint_as_float(c ? (w[r] & 0xFFFF0000u) : (w[r] << 16));
      uint4 out;
      if (RULE == FP4ATTN_QSCALE_MSE) {
        // both amplitudes; group sums of eight consecutive keys combined as (g0 + g1) + (g2 + g3)
        const uint32_t uf = mx_scale_byte_bf16<FP4ATTN_QSCALE_FLOOR>(a16);
        float tf[32];
#pragma unroll
        for (int r = 0; r < 32; ++r) tf[r] = v[r];
        mx_scale_values<32>(tf, uf);
        mx_scale_values<32>(v, u);
        uint32_t wf[4], wc[4];
        float gf[4], gc[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          wf[j] = cvt_e2m1x8(tf + 8 * j);
          wc[j] = cvt_e2m1x8(v + 8 * j);
          gf[j] = mx_error_x8(tf + 8 * j, wf[j]);
          gc[j] = mx_error_x8(v + 8 * j, wc[j]);
        }
        const float ef = __fadd_rn(__fadd_rn(gf[0], gf[1]), __fadd_rn(gf[2], gf[3]));
        const float ec = __fadd_rn(__fadd_rn(gc[0], gc[1]), __fadd_rn(gc[2], gc[3]));
        const bool take_f = (uf != u) && (ef < __fmul_rn(4.0f, ec));
        out = take_f ? make_uint4(wf[0], wf[1], wf[2], wf[3]) : make_uint4(wc[0], wc[1], wc[2], wc[3]);
        u = take_f ? uf : u;
      } else {
        mx_scale_values<32>(v, u);
        out.x = cvt_e2m1x8(v);
        out.y = cvt_e2m1x8(v + 8);
        out.z = cvt_e2m1x8(v + 16);
        out.w = cvt_e2m1x8(v + 24);
      }
      const int col = 2 * cp + c;
      packed[((bh * D + col) * (size_t)(N / 2) + (size_t)kt * 64 + kb * 16) / 16] = out;
      u |= __shfl_xor_sync(0xffffffffu, u, 8) << 8;  // kb 0: bytes of blocks 0, 1 (kb 2: of 2, 3)
      u |= __shfl_xor_sync(0xffffffffu, u, 16) << 16;
      uint32_t* atom = reinterpret_cast<uint32_t*>(sf + (size_t)t * 512);   // row r at word (r % 32) * 4 + r / 32
      if (kb == 0) atom[(col & 31) * 4 + (col >> 5)] = u;
      if (D == 64 && kb == 1) atom[(col & 31) * 4 + 2 + (col >> 5)] = 0;    // rows from 64 on are padding
    }
    __syncthreads();                                 // the tile buffer is free again
  }
}

// ---- a unit's maximum within one thread-block cluster: every CTA reduces its share, the shares meet through distributed
// shared memory.  The second barrier (cluster_leave) keeps a CTA's share readable until every other CTA has read it.
__device__ __forceinline__ uint32_t cluster_size() { uint32_t n; asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(n)); return n; }
__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm("mov.u32 %0, %%cluster_ctaid.x;" : "=r"(r)); return r; }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// `m`: each thread's maximum; all threads of all CTAs of the cluster; THREADS threads per CTA
template <int THREADS>
__device__ __forceinline__ uint32_t cluster_max(uint32_t m) {
  __shared__ uint32_t wmax[THREADS / 32], share;
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = __reduce_max_sync(0xffffffffu, threadIdx.x < THREADS / 32 ? wmax[threadIdx.x] : 0u);
    if (threadIdx.x == 0) share = m;
  }
  cluster_arrive();
  cluster_wait();
  const uint32_t lane = threadIdx.x & 31;
  m = 0;
  if (lane < cluster_size()) {
    uint32_t remote;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"((uint32_t)__cvta_generic_to_shared(&share)), "r"(lane));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(m) : "r"(remote) : "memory");
  }
  m = __reduce_max_sync(0xffffffffu, m);
  cluster_arrive();
  return m;
}
__device__ __forceinline__ void cluster_leave() { cluster_wait(); }

// Encode factor of a tensor or unit from its partial maxima: fl32(top / max), 1 for an all-zero one.  Each kernel that needs
// the factor takes it so (at most 1024 partials, in L2) instead of waiting for a kernel of its own to form it.
// encode_factor_warp: every warp by itself, at most 32 partials; encode_factor_block: the whole block, with a barrier.
__device__ __forceinline__ float encode_factor_of(float amax, float top) { return amax == 0.f ? 1.0f : __fdiv_rn(top, amax); }
__device__ __forceinline__ float encode_factor_warp(const float* partials, int n_partials, float top) {
  const int lane = threadIdx.x & 31;
  float a = lane < n_partials ? __ldcg(partials + lane) : 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
  return encode_factor_of(a, top);
}
__device__ __forceinline__ float encode_factor_block(const float* partials, int n_partials, float top) {
  __shared__ float wmax[kThreads / 32];
  float a = 0.f;
  for (int i = threadIdx.x; i < n_partials; i += kThreads) a = fmaxf(a, __ldcg(partials + i));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = a;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kThreads / 32; ++i) a = fmaxf(a, wmax[i]);
  return encode_factor_of(a, top);
}

// ---------------------------------------------------------------- E4M3 V (FP8 P/V route), transposed out
// Same tile pipeline as the MXFP4 V kernel; a thread owns two adjacent head-dim columns and one 32-key block and
// writes 32 bytes per column: byte = Q_E4M3(fl32(v * G)), G the unit's encode factor (one per (batch, head)).
__device__ __forceinline__ uint32_t cvt_e4m3x4(float a, float b, float c, float d) {   // a in bits 0-7 ... d in bits 24-31
  uint32_t w;
  asm("{\n\t.reg .b16 lo, hi;\n\t"
      "cvt.rn.satfinite.e4m3x2.f32 lo, %2, %1;\n\t"
      "cvt.rn.satfinite.e4m3x2.f32 hi, %4, %3;\n\t"
      "mov.b32 %0, {lo, hi};\n\t}"
      : "=r"(w) : "f"(a), "f"(b), "f"(c), "f"(d));
  return w;
}
template <int D>
__global__ void __launch_bounds__(2 * D, D == 128 ? 3 : 6)
quant_e4m3_v_kernel(const uint4* __restrict__ x, uint4* __restrict__ bytes_out, const float* __restrict__ partials, int n_partials,
                    float* __restrict__ G_out, int N, int n_tiles) {
  constexpr int T = 2 * D;
  constexpr int LOADS = 128 * D / 8 / T;
  extern __shared__ __align__(16) uint8_t vsm[];
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(vsm);
  const int tiles_per_head = N / 128;
  const int cp = (threadIdx.x >> 5) * 8 + (threadIdx.x & 7);
  const int kb = (threadIdx.x >> 3) & 3;
  auto issue = [&](int t, int buf) {
    const uint4* src = x + (size_t)t * (128 * D / 8);
#pragma unroll
    for (int k = 0; k < LOADS; ++k) {
      const uint32_t j = threadIdx.x + k * T;      // 16-byte chunk of the tile, in row j / (D / 8)
      cp_async_16(sbase + buf * kVTileBytes<D> + (j ^ v_swizzle<D>(j / (D / 8))) * 16, src + j);
    }
    cp_async_commit();
  };
  int t = n_tiles - 1 - (int)blockIdx.x, i = 0;    // from the end of the tensor: the amax pass has read that last
  launch_dependents();
  wait_prior_grids();
  if (t >= 0) issue(t, 0);
  for (; t >= 0; t -= gridDim.x, ++i) {
    const int tn = t - (int)gridDim.x;
    if (tn >= 0) { issue(tn, (i + 1) & 1); cp_async_wait<1>(); } else { cp_async_wait<0>(); }
    __syncthreads();
    const uint32_t* tile = reinterpret_cast<const uint32_t*>(vsm + (i & 1) * kVTileBytes<D>);
    const size_t bh = t / tiles_per_head;
    const int kt = t - (int)bh * tiles_per_head;
    const float G = encode_factor_warp(partials + bh * n_partials, n_partials, 448.0f);
    if (kt == 0 && threadIdx.x == 0) G_out[bh] = G;
    uint32_t w[32];
#pragma unroll
    for (int r = 0; r < 32; ++r) w[r] = tile[(kb * 32 + r) * (D / 2) + (cp ^ (8 * kb))];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      uint32_t o[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        float v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
          v[e] = __fmul_rn(__uint_as_float(c ? (w[4 * j + e] & 0xFFFF0000u) : (w[4 * j + e] << 16)), G);
        o[j] = cvt_e4m3x4(v[0], v[1], v[2], v[3]);
      }
      const int col = 2 * cp + c;
      uint4* dst = bytes_out + ((bh * D + col) * (size_t)N + (size_t)kt * 128 + kb * 32) / 16;
      dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
      dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- NVFP4 pass 1: amax partials
// grid (P, U): U = 1 for the tensor-wide maximum, U = B*H for one maximum per (batch, head) unit; row y of
// the grid covers groups [y * n_groups, (y + 1) * n_groups) and writes partials[y * P .. y * P + P)
template <bool W32>
__global__ void __launch_bounds__(kThreads)
amax_partials_kernel(const uint4* __restrict__ x, size_t n_groups, float* __restrict__ partials) {
  x += (size_t)blockIdx.y * n_groups;
  partials += (size_t)blockIdx.y * gridDim.x;
  launch_dependents();
  wait_prior_grids();
  // |bf16| bit patterns order like the magnitudes: packed 16-bit maxima, two independent 32-byte loads per
  // trip (both NVFP4 passes over 67 M elements with 1 / 2 / 4 / 8 loads 49.9 / 48.9 / 50.5 / 50.9 us; a contiguous share per block
  // instead of interleaved ones 50.9)
  uint32_t m = 0;
  const size_t stride = (size_t)gridDim.x * kThreads;
  size_t g = (size_t)blockIdx.x * kThreads + threadIdx.x;
  n_groups /= 2;                                   // 32 bytes each
  for (; g + stride < n_groups; g += 2 * stride) {
    uint32_t r[2][8];
    load_16<W32>(r[0], x + 2 * g);
    load_16<W32>(r[1], x + 2 * (g + stride));
    m = max(m, max(absmax_bf16x16(r[0]), absmax_bf16x16(r[1])));
  }
  for (; g < n_groups; g += stride) {
    uint32_t r[8];
    load_16<W32>(r, x + 2 * g);
    m = max(m, absmax_bf16x16(r));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  __shared__ uint32_t wmax[kThreads / 32];
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < kThreads / 32; ++i) m = max(m, wmax[i]);
    partials[blockIdx.x] = __uint_as_float(m << 16);
  }
}

__device__ __forceinline__ uint32_t cvt_e4m3_byte(float t) {     // RNE, saturating at 448
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(0.f), "f"(t));
  return r & 0xFFu;
}
__device__ __forceinline__ float e4m3_byte_to_f32(uint32_t b) {
  uint32_t h2;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)b));
  return __half2float(__ushort_as_half((unsigned short)(h2 & 0xFFFFu)));
}

// fl32(x / 6), x >= 0: the rounded product with fl32(1/6) and one Newton step on its exact remainder (Markstein's theorem; every
// significand checked against the division), three instructions where the general division takes about ten and a branch.
// For x below 2^103; below 2^-100 the remainder may be subnormal and the result off by a unit, far under the smallest scale.
__device__ __forceinline__ float sixth(float x) {
  const float r = 0.16666667163372040f, q = __fmul_rn(x, r);
  return __fmaf_rn(__fmaf_rn(-6.0f, q, x), r, q);
}
// G / S for scale byte b, 0 for S = 0 (a zero block) and for a NaN
__device__ __forceinline__ float nv_ratio(uint32_t b, float G) {
  const float S = e4m3_byte_to_f32(b);
  return (S > 0.f) ? __fdiv_rn(G, S) : 0.f;
}
// The ratios of a tensor or unit by scale byte (bit 7 is never set but in a NaN): 128 divisions instead of one per block.
// Whole block; ends with a barrier.
__device__ __forceinline__ void nv_ratio_table(float* table, float G) {
  if (threadIdx.x < 128) table[threadIdx.x] = nv_ratio(threadIdx.x, G);
  __syncthreads();
}

// one chunk's codes and scale bytes from its bf16 words; `table`: nv_ratio_table, or null where the factor changes too often for one
template <int D>
__device__ __forceinline__ void nv_code_chunk(const uint32_t (&raw)[kLoads][8], float G, const float* table, uint32_t chunk, uint2* packed, uint8_t* sf) {
  constexpr uint32_t LPR = D / 16;                 // lanes per row
  constexpr uint32_t CT = (D / 16 + 3) / 4;
  const uint32_t seg = threadIdx.x % LPR;
  // a * G is at most about 2688 for any finite G.  An infinite one (tensors below 2^-116) makes it infinite, which the division
  // by 6 keeps and the remainder in sixth() would turn into a NaN.
  const bool plain = G < INFINITY;
#pragma unroll
  for (int k = 0; k < kLoads; ++k) {
    const float aG = __fmul_rn(__uint_as_float(absmax_bf16x16(raw[k]) << 16), G);
    uint32_t sb = cvt_e4m3_byte(plain ? sixth(aG) : __fdiv_rn(aG, 6.0f));
    const float r = table ? table[sb & 127u] : nv_ratio(sb, G);
    uint32_t w[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float v[8];
      bf16x8_to_f32(make_uint4(raw[k][4 * h], raw[k][4 * h + 1], raw[k][4 * h + 2], raw[k][4 * h + 3]), v);
      scale_values<8>(v, r);                                     // sign rides along; 0*r = 0 for zero blocks
      w[h] = cvt_e2m1x8(v);
    }
    packed[(size_t)chunk * (kGroupsPerCta / 2) + threadIdx.x + k * kThreads] = make_uint2(w[0], w[1]);
    sb |= __shfl_xor_sync(0xffffffffu, sb, 1) << 8;              // four columns' bytes as one word
    sb |= __shfl_xor_sync(0xffffffffu, sb, 2) << 16;
    const uint32_t row = chunk * (kGroupsPerCta / 2 / LPR) + (threadIdx.x + k * kThreads) / LPR;
    if ((seg & 3) == 0)
      *reinterpret_cast<uint32_t*>(sf + ((size_t)(row >> 7) * CT + (seg >> 2)) * 512 + (row & 31) * 16 + ((row & 127) >> 5) * 4) = sb;
  }
}

// ---------------------------------------------------------------- NVFP4 pass 2, blocks of 16 along d (Q, K)
// Bound by HBM (twice over the tensor, less what is left of it in L2); where L2 holds the tensor, by its instructions.  67 M
// elements, both passes: 48.9 us (two IEEE divisions per block: 49.5; with a kernel of its own for the factor, a block's scale
// formed in two lanes and plain launches 61.6), 8.4 M 9.0 (9.3).
// The chunks and the grid of quant_mx_rows_kernel, walked from the tensor's end (the amax pass has read that last).  A chunk
// lies within one unit; where units have factors of their own a CTA forms its unit's for every chunk.
// UNITS: one factor per unit.
template <int D, bool W32, bool UNITS>
__global__ void __launch_bounds__(kThreads, kRowsCtas)
quant_nv_rows_kernel(const uint4* __restrict__ x, uint2* __restrict__ packed, uint8_t* __restrict__ sf,
                     const float* __restrict__ partials, int n_partials, float* __restrict__ G_out, uint32_t n_chunks,
                     uint32_t chunks_per_unit) {
  launch_dependents();
  wait_prior_grids();
  uint32_t i = blockIdx.x, raw[kLoads][8];
#pragma unroll
  for (int k = 0; k < kLoads; ++k) load_16<W32>(raw[k], x + (size_t)(n_chunks - 1 - i) * kGroupsPerCta + 2 * (threadIdx.x + k * kThreads));
  __shared__ float ratio[128];
  float G = 0.f;
  if (!UNITS) {
    G = encode_factor_block(partials, n_partials, 2688.0f);
    if (blockIdx.x == 0 && threadIdx.x == 0) G_out[0] = G;
    nv_ratio_table(ratio, G);
  }
  while (true) {
    const uint32_t chunk = n_chunks - 1 - i;
    i += gridDim.x;
    uint32_t ahead[kLoads][8];
    if (i < n_chunks) {
#pragma unroll
      for (int k = 0; k < kLoads; ++k) load_16<W32>(ahead[k], x + (size_t)(n_chunks - 1 - i) * kGroupsPerCta + 2 * (threadIdx.x + k * kThreads));
    }
    if (UNITS) {
      const uint32_t unit = chunk / chunks_per_unit;
      G = encode_factor_warp(partials + (size_t)unit * n_partials, n_partials, 2688.0f);
      if (threadIdx.x == 0 && unit * chunks_per_unit == chunk) G_out[unit] = G;
    }
    nv_code_chunk<D>(raw, G, UNITS ? nullptr : ratio, chunk, packed, sf);
    if (i >= n_chunks) return;
#pragma unroll
    for (int k = 0; k < kLoads; ++k)
#pragma unroll
      for (int j = 0; j < 8; ++j) raw[k][j] = ahead[k][j];
  }
}

// Both passes over a unit with a factor of its own in one launch: a cluster takes the unit, its CTAs every cluster_size()-th
// chunk, and the second pass runs from the last chunk back.  Units of up to 1 MB are still in L2 then (the resident clusters
// hold 74 MB of them), so the tensor is read from memory once; of larger ones the part that is.  All resident clusters
// read, meet and write at about the same time, and the second half is bound by instructions: 64 units of 1 MB take 23.4 us (two
// divisions per block instead of a table of ratios and sixth(): 24.6), 3.7 TB/s of input and output.  (Held in shared memory for
// the second pass by one CTA of 512 threads per SM: 32.8 us, its sixteen warps are too few for the conversion's latency.)
template <int D, bool W32>
__global__ void __launch_bounds__(kThreads, kRowsCtas)
quant_nv_unit_kernel(const uint4* __restrict__ x, uint2* __restrict__ packed, uint8_t* __restrict__ sf, float* __restrict__ G_out,
                     int chunks_per_unit) {
  launch_dependents();
  wait_prior_grids();
  const int step = (int)cluster_size(), unit = blockIdx.x / step, first = unit * chunks_per_unit, rank = (int)cluster_rank();
  uint32_t raw[kLoads][8], m = 0;
  const int mine = (chunks_per_unit - rank + step - 1) / step;    // chunks first + rank, first + rank + step, ...
  auto load = [&](int k_chunk, uint32_t (&r)[kLoads][8]) {
    const uint4* src = x + (size_t)(first + rank + k_chunk * step) * kGroupsPerCta;
#pragma unroll
    for (int k = 0; k < kLoads; ++k) load_16<W32>(r[k], src + 2 * (threadIdx.x + k * kThreads));
  };
  if (mine > 0) load(0, raw);
  for (int c = 0; c < mine; ++c) {
    uint32_t ahead[kLoads][8];
    if (c + 1 < mine) load(c + 1, ahead);
#pragma unroll
    for (int k = 0; k < kLoads; ++k) m = max(m, absmax_bf16x16(raw[k]));
    if (c + 1 < mine) {
#pragma unroll
      for (int k = 0; k < kLoads; ++k)
#pragma unroll
        for (int j = 0; j < 8; ++j) raw[k][j] = ahead[k][j];
    }
  }
  const float G = encode_factor_of(__uint_as_float(cluster_max<kThreads>(m) << 16), 2688.0f);
  if (rank == 0 && threadIdx.x == 0) G_out[unit] = G;
  __shared__ float ratio[128];
  nv_ratio_table(ratio, G);
  for (int c = mine - 1; c >= 0; --c) {                           // the last chunk is still in registers
    uint32_t ahead[kLoads][8];
    if (c > 0) load(c - 1, ahead);
    nv_code_chunk<D>(raw, G, ratio, (uint32_t)(first + rank + c * step), packed, sf);
    if (c > 0) {
#pragma unroll
      for (int k = 0; k < kLoads; ++k)
#pragma unroll
        for (int j = 0; j < 8; ++j) raw[k][j] = ahead[k][j];
    }
  }
  cluster_leave();
}

}  // namespace fp4attn

using namespace fp4attn;

extern "C" size_t fp4attn_packed_bytes(int B, int H, int N, int d) {
  if (B <= 0 || H <= 0 || N <= 0 || d <= 0) return 0;
  return (size_t)B * H * N * d / 2;
}

static bool shape_ok(int B, int H, int N, int d) {
  return B > 0 && H > 0 && (d == 64 || d == 128) && N >= 128 && N % 128 == 0;
}

extern "C" size_t fp4attn_scale_bytes(int fmt, int role, int B, int H, int N, int d) {
  if (!shape_ok(B, H, N, d)) return 0;
  if (role == FP4ATTN_ROLE_V) {
    if (fmt != FP4ATTN_FMT_MXFP4) return 0;
    return (size_t)B * H * ((d + 127) / 128) * (N / 128) * 512;          // rows d, columns N/32
  }
  if (role != FP4ATTN_ROLE_Q && role != FP4ATTN_ROLE_K) return 0;
  if (fmt != FP4ATTN_FMT_MXFP4 && fmt != FP4ATTN_FMT_NVFP4) return 0;
  const int C = d / (fmt == FP4ATTN_FMT_MXFP4 ? 32 : 16);
  return (size_t)B * H * (N / 128) * ((C + 3) / 4) * 512;
}

extern "C" size_t fp4attn_quantize_workspace_bytes(int fmt, int role, int B, int H, int N, int d) {
  (void)role; (void)B; (void)H; (void)N; (void)d;
  return fmt == FP4ATTN_FMT_NVFP4 ? (size_t)kMaxPartials * sizeof(float) : 0;
}

namespace fp4attn {
// V kernel: persistent CTAs, as many as fit per SM with two tile buffers each (the opt-in to more than 48 KB of
// dynamic shared memory is set once per device and instance)
template <int D, int RULE>
static void launch_mx_v(const uint4* xs, int n_tiles, int N, void* packed, void* scales, cudaStream_t st) {
  static std::atomic<int> ctas[kMaxDevices];        // 0 unknown, else CTAs of the persistent grid
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return;   // the launch check below reports it
  int grid = ctas[dev].load(std::memory_order_acquire);
  if (!grid) {
    int sms = 0, per_sm = 0;
    if (cudaFuncSetAttribute(quant_mx_v_kernel<D, RULE>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kVTileBytes<D>) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, quant_mx_v_kernel<D, RULE>, 2 * D, 2 * kVTileBytes<D>) != cudaSuccess || per_sm < 1)
      return;
    grid = sms * per_sm;
    ctas[dev].store(grid, std::memory_order_release);
  }
  launch_overlapped(quant_mx_v_kernel<D, RULE>, dim3(n_tiles < grid ? n_tiles : grid), 2 * D, 2 * kVTileBytes<D>, st, xs, (uint4*)packed,
                    (uint8_t*)scales, N, n_tiles);
}

int device_sms() {
  static std::atomic<int> sm_count[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
  int sms = sm_count[dev].load(std::memory_order_acquire);
  if (!sms) {
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return 0;
    sm_count[dev].store(sms, std::memory_order_release);
  }
  return sms;
}

// Persistent CTAs of the rows kernels: at most what the device holds at once, each with the same number of chunks (within
// one).  One CTA per chunk would pay a CTA's start - its launch, the wait for the kernels before, the encode factor - every
// 16 KB.
static unsigned rows_grid(size_t n_chunks) {
  const int sms = device_sms();
  if (!sms) return (unsigned)n_chunks;
  const size_t resident = (size_t)kRowsCtas * sms, rounds = (n_chunks + resident - 1) / resident;
  return (unsigned)((n_chunks + rounds - 1) / rounds);
}

// Shared by fp4attn_quantize and the variants that bring their own scratch.
template <int RULE>
static void launch_mx(const uint4* xs, int role, int B, int H, int N, int d, void* packed, void* scales, cudaStream_t st) {
  if (role != FP4ATTN_ROLE_V) {
    const size_t n_chunks = (size_t)B * H * N * d / 8 / kGroupsPerCta;                     // N % 128 == 0 makes this exact
    const bool w32 = ((uintptr_t)xs & 31) == 0;
    launch_overlapped(d == 128 ? (w32 ? quant_mx_rows_kernel<128, RULE, true> : quant_mx_rows_kernel<128, RULE, false>)
                               : (w32 ? quant_mx_rows_kernel<64, RULE, true> : quant_mx_rows_kernel<64, RULE, false>), dim3(rows_grid(n_chunks)), kThreads, 0,
                      st, xs, (uint2*)packed, (uint8_t*)scales, (uint32_t)n_chunks);
  } else if (d == 128) {
    launch_mx_v<128, RULE>(xs, B * H * (N / 128), N, packed, scales, st);
  } else {
    launch_mx_v<64, RULE>(xs, B * H * (N / 128), N, packed, scales, st);
  }
}

// CTAs of the cluster that takes a unit of so many chunks: up to eight (the portable limit), but four for 8 to 15 chunks once
// clusters of eight would not all be resident: with one chunk a CTA (two at most) a wave brings too little for its start and
// its two meetings.  128 / 192 KB a unit, us for clusters of eight / four: 64 units 5.8 / 6.1, 7.5 / 8.0; 128 units 9.9 / 8.2,
// 12.3 / 10.7; 512 units 32.8 / 23.3, 39.7 / 34.2 (two launches 27.8, 42.1).
static unsigned cluster_for(size_t units, size_t chunks) {
  if (chunks >= 16 || (chunks >= 8 && units * 8 <= (size_t)kRowsCtas * device_sms())) return 8;
  return chunks >= 4 ? 4 : chunks >= 2 ? 2 : 1;
}
// One launch for both passes where the clusters make two CTAs an SM, or where every CTA has at most two chunks and the second
// launch costs more than it brings.  Below that two launches are faster, which give every CTA of the device a share.
// Microseconds from a graph, two launches against one: 1 / 4 / 16 / 32 units of 512 KB 3.4 / 4.7, 3.9 / 4.9, 6.4 / 8.4, 10.0 /
// 10.5; 4 / 8 of 1 MB 5.6 / 8.2, 7.1 / 11.1; 8 / 64 / 512 of 128 KB 3.6 / 2.8, 6.4 / 5.8, 27.8 / 23.3; 512 of 256 / 512 KB 54.6 / 45.6,
// 101 / 81; 64 of 1 / 2 / 4 / 8 MB 28.6 / 25.0, 55.1 / 50.4, 98.3 / 89.5, 192 / 179.
static bool nv_in_one_launch(size_t units, size_t chunks) {
  const unsigned cluster = cluster_for(units, chunks);
  return chunks <= 2 * cluster || units * cluster >= (size_t)2 * device_sms();
}

int launch_quantize(const void* x, int fmt, int role, int B, int H, int N, int d, void* packed, void* scales,
                    float* G_out, float* partials, cudaStream_t st, int mx_rule, bool per_head = false) {
  const size_t n_groups = (size_t)B * H * N * d / 8;
  const size_t n_chunks = n_groups / kGroupsPerCta, unit_chunks = (size_t)N * d / 8 / kGroupsPerCta;   // N % 128 == 0 makes these exact
  const uint4* xs = reinterpret_cast<const uint4*>(x);
  if (fmt == FP4ATTN_FMT_MXFP4) {
    if (mx_rule == FP4ATTN_QSCALE_THR16)      launch_mx<FP4ATTN_QSCALE_THR16>(xs, role, B, H, N, d, packed, scales, st);
    else if (mx_rule == FP4ATTN_QSCALE_FLOOR) launch_mx<FP4ATTN_QSCALE_FLOOR>(xs, role, B, H, N, d, packed, scales, st);
    else if (mx_rule == FP4ATTN_QSCALE_MSE)   launch_mx<FP4ATTN_QSCALE_MSE>(xs, role, B, H, N, d, packed, scales, st);
    else                                      launch_mx<FP4ATTN_QSCALE_CEIL>(xs, role, B, H, N, d, packed, scales, st);
  } else {
    const size_t units = per_head ? (size_t)B * H : 1, per_unit = per_head ? unit_chunks : n_chunks;
    if (nv_in_one_launch(units, per_unit)) {
      const bool w32u = ((uintptr_t)xs & 31) == 0;
      const unsigned cluster = cluster_for(units, per_unit);
      launch_overlapped_clusters(d == 128 ? (w32u ? quant_nv_unit_kernel<128, true> : quant_nv_unit_kernel<128, false>)
                                 : (w32u ? quant_nv_unit_kernel<64, true> : quant_nv_unit_kernel<64, false>),
                        dim3((unsigned)units * cluster), kThreads, 0, st, cluster, xs, (uint2*)packed, (uint8_t*)scales, G_out, (int)per_unit);
      return cudaGetLastError() == cudaSuccess ? FP4ATTN_OK : FP4ATTN_ERR_CUDA;
    }
    const unsigned most = per_head ? (unsigned)kPartialsPerHead : (unsigned)kMaxPartials;
    const size_t want = per_head ? unit_chunks : n_chunks;
    const int n_partials = (int)(want < most ? want : most);
    const bool w32 = ((uintptr_t)xs & 31) == 0;
    launch_overlapped(w32 ? amax_partials_kernel<true> : amax_partials_kernel<false>, per_head ? dim3(n_partials, B * H) : dim3(n_partials), kThreads, 0, st, xs,
                      per_head ? n_groups / ((size_t)B * H) : n_groups, partials);
    auto rows = per_head ? (d == 128 ? (w32 ? quant_nv_rows_kernel<128, true, true> : quant_nv_rows_kernel<128, false, true>)
                                     : (w32 ? quant_nv_rows_kernel<64, true, true> : quant_nv_rows_kernel<64, false, true>))
                         : (d == 128 ? (w32 ? quant_nv_rows_kernel<128, true, false> : quant_nv_rows_kernel<128, false, false>)
                                     : (w32 ? quant_nv_rows_kernel<64, true, false> : quant_nv_rows_kernel<64, false, false>));
    launch_overlapped(rows, dim3(rows_grid(n_chunks)), kThreads, 0, st, xs,
                      (uint2*)packed, (uint8_t*)scales, (const float*)partials, n_partials, G_out, (uint32_t)n_chunks,
                      (uint32_t)(per_head ? unit_chunks : 0));
  }
  return cudaGetLastError() == cudaSuccess ? FP4ATTN_OK : FP4ATTN_ERR_CUDA;
}

int validate_quantize(const void* x, int fmt, int role, int B, int H, int N, int d, const void* packed,
                      const void* scales, const float* G_out) {
  if (!x || !packed || !scales) return FP4ATTN_ERR_INVALID_ARG;
  if (fmt != FP4ATTN_FMT_MXFP4 && fmt != FP4ATTN_FMT_NVFP4) return FP4ATTN_ERR_INVALID_ARG;
  if (role != FP4ATTN_ROLE_Q && role != FP4ATTN_ROLE_K && role != FP4ATTN_ROLE_V) return FP4ATTN_ERR_INVALID_ARG;
  if (B <= 0 || H <= 0 || N <= 0 || d <= 0) return FP4ATTN_ERR_INVALID_ARG;
  if (!shape_ok(B, H, N, d)) return FP4ATTN_ERR_UNSUPPORTED_SHAPE;
  if (fmt == FP4ATTN_FMT_NVFP4 && role == FP4ATTN_ROLE_V) return FP4ATTN_ERR_INVALID_ARG;   // V is always MXFP4
  if (fmt == FP4ATTN_FMT_NVFP4 && !G_out) return FP4ATTN_ERR_INVALID_ARG;
  if (((uintptr_t)x | (uintptr_t)packed | (uintptr_t)scales) & 15) return FP4ATTN_ERR_ALIGNMENT;
  return FP4ATTN_OK;
}
}  // namespace fp4attn

extern "C" int fp4attn_quantize(const void* x, int fmt, int role, int B, int H, int N, int d, void* packed,
                                void* scales, float* G_out, void* workspace, size_t workspace_bytes,
                                fp4attn_stream_t stream) {
  int rc = validate_quantize(x, fmt, role, B, H, N, d, packed, scales, G_out);
  if (rc != FP4ATTN_OK) return rc;
  const size_t need = fp4attn_quantize_workspace_bytes(fmt, role, B, H, N, d);
  if (need && (!workspace || workspace_bytes < need)) return FP4ATTN_ERR_WORKSPACE;
  if (need && ((uintptr_t)workspace & 15)) return FP4ATTN_ERR_ALIGNMENT;
  rc = check_device_sm100();
  if (rc != FP4ATTN_OK) return rc;
  return launch_quantize(x, fmt, role, B, H, N, d, packed, scales, G_out, (float*)workspace, (cudaStream_t)stream,
                         FP4ATTN_QSCALE_CEIL);
}

extern "C" int fp4attn_quantize_mxfp4_rule(const void* x, int role, int scale_rule, int B, int H, int N, int d,
                                           void* packed, void* scales, fp4attn_stream_t stream) {
  if (scale_rule != FP4ATTN_QSCALE_CEIL && scale_rule != FP4ATTN_QSCALE_THR16 && scale_rule != FP4ATTN_QSCALE_FLOOR &&
      scale_rule != FP4ATTN_QSCALE_MSE)
    return FP4ATTN_ERR_INVALID_ARG;
  int rc = validate_quantize(x, FP4ATTN_FMT_MXFP4, role, B, H, N, d, packed, scales, nullptr);
  if (rc != FP4ATTN_OK) return rc;
  rc = check_device_sm100();
  if (rc != FP4ATTN_OK) return rc;
  return launch_quantize(x, FP4ATTN_FMT_MXFP4, role, B, H, N, d, packed, scales, nullptr, nullptr, (cudaStream_t)stream,
                         scale_rule);
}

extern "C" size_t fp4attn_quantize_nvfp4_per_head_workspace_bytes(int B, int H, int N, int d) {
  if (!shape_ok(B, H, N, d)) return 0;
  return (size_t)B * H * kPartialsPerHead * sizeof(float);
}

extern "C" int fp4attn_quantize_nvfp4_per_head(const void* x, int role, int B, int H, int N, int d, void* packed,
                                               void* scales, float* G_out, void* workspace, size_t workspace_bytes,
                                               fp4attn_stream_t stream) {
  int rc = validate_quantize(x, FP4ATTN_FMT_NVFP4, role, B, H, N, d, packed, scales, G_out);
  if (rc != FP4ATTN_OK) return rc;
  const size_t need = fp4attn_quantize_nvfp4_per_head_workspace_bytes(B, H, N, d);
  if (!workspace || workspace_bytes < need) return FP4ATTN_ERR_WORKSPACE;
  if ((uintptr_t)workspace & 15) return FP4ATTN_ERR_ALIGNMENT;
  rc = check_device_sm100();
  if (rc != FP4ATTN_OK) return rc;
  return launch_quantize(x, FP4ATTN_FMT_NVFP4, role, B, H, N, d, packed, scales, G_out, (float*)workspace,
                         (cudaStream_t)stream, FP4ATTN_QSCALE_CEIL, true);
}

// ---------------------------------------------------------------- allocation-free NVFP4 variant
// Scratch for the amax pass lives in the library image.  In host code the symbol below is only a
// handle; the device address is fetched once per device with cudaGetSymbolAddress.
static __device__ __align__(256) float g_noalloc_partials[kMaxPartials];

extern "C" int fp4attn_quantize_nvfp4_noalloc(const void* x, int role, int B, int H, int N, int d, void* packed,
                                              void* scales, float* G_out, fp4attn_stream_t stream) {
  int rc = validate_quantize(x, FP4ATTN_FMT_NVFP4, role, B, H, N, d, packed, scales, G_out);
  if (rc != FP4ATTN_OK) return rc;
  if ((unsigned long long)B * H * N * d > FP4ATTN_NOALLOC_MAX_ELEMENTS) return FP4ATTN_ERR_WORKSPACE;
  rc = check_device_sm100();
  if (rc != FP4ATTN_OK) return rc;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return FP4ATTN_ERR_CUDA;
  // per-device address of g_noalloc_partials; several host threads may make the first call on a device at
  // once (they all store the same address)
  static std::atomic<float*> scratch_addr[kMaxDevices];
  if (dev < 0 || dev >= kMaxDevices) return FP4ATTN_ERR_INVALID_ARG;
  float* scratch = scratch_addr[dev].load(std::memory_order_acquire);
  if (!scratch) {
    if (cudaGetSymbolAddress((void**)&scratch, g_noalloc_partials) != cudaSuccess || !scratch) return FP4ATTN_ERR_CUDA;
    scratch_addr[dev].store(scratch, std::memory_order_release);
  }
  return launch_quantize(x, FP4ATTN_FMT_NVFP4, role, B, H, N, d, packed, scales, G_out, scratch,
                         (cudaStream_t)stream, FP4ATTN_QSCALE_CEIL);
}

// ---------------------------------------------------------------- E4M3 V of the FP8 P/V route
extern "C" size_t fp4attn_quantize_v_e4m3_workspace_bytes(int B, int H, int N, int d) {
  if (!shape_ok(B, H, N, d)) return 0;
  return (size_t)B * H * kPartialsPerHead * sizeof(float);
}

template <int D>
static int launch_e4m3_v(const uint4* xs, int BH, int N, void* bytes_out, const float* partials, int n_partials, float* G, cudaStream_t st) {
  static std::atomic<int> ctas[kMaxDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return FP4ATTN_ERR_CUDA;
  int grid = ctas[dev].load(std::memory_order_acquire);
  if (!grid) {
    int sms = 0, per_sm = 0;
    if (cudaFuncSetAttribute(quant_e4m3_v_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kVTileBytes<D>) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, quant_e4m3_v_kernel<D>, 2 * D, 2 * kVTileBytes<D>) != cudaSuccess || per_sm < 1)
      return FP4ATTN_ERR_CUDA;
    grid = sms * per_sm;
    ctas[dev].store(grid, std::memory_order_release);
  }
  const int n_tiles = BH * (N / 128);
  launch_overlapped(quant_e4m3_v_kernel<D>, dim3(n_tiles < grid ? n_tiles : grid), 2 * D, 2 * kVTileBytes<D>, st, xs, (uint4*)bytes_out,
                    partials, n_partials, G, N, n_tiles);
  return FP4ATTN_OK;
}

extern "C" int fp4attn_quantize_v_e4m3(const void* x, int B, int H, int N, int d, void* bytes_out, float* G_out,
                                       void* workspace, size_t workspace_bytes, fp4attn_stream_t stream) {
  if (!x || !bytes_out || !G_out) return FP4ATTN_ERR_INVALID_ARG;
  if (B <= 0 || H <= 0 || N <= 0 || d <= 0) return FP4ATTN_ERR_INVALID_ARG;
  if (!shape_ok(B, H, N, d)) return FP4ATTN_ERR_UNSUPPORTED_SHAPE;
  if (((uintptr_t)x | (uintptr_t)bytes_out) & 15) return FP4ATTN_ERR_ALIGNMENT;
  const size_t need = fp4attn_quantize_v_e4m3_workspace_bytes(B, H, N, d);
  if (!workspace || workspace_bytes < need) return FP4ATTN_ERR_WORKSPACE;
  if ((uintptr_t)workspace & 15) return FP4ATTN_ERR_ALIGNMENT;
  int rc = check_device_sm100();
  if (rc != FP4ATTN_OK) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  const uint4* xs = reinterpret_cast<const uint4*>(x);
  const size_t groups_per_unit = (size_t)N * d / 8;
  const unsigned gx = (unsigned)(groups_per_unit / kGroupsPerCta);
  const int n_partials = (int)(gx < (unsigned)kPartialsPerHead ? gx : kPartialsPerHead);
  launch_overlapped(((uintptr_t)xs & 31) == 0 ? amax_partials_kernel<true> : amax_partials_kernel<false>, dim3(n_partials, B * H), kThreads, 0, st, xs, groups_per_unit, (float*)workspace);
  const float* partials = (const float*)workspace;
  rc = d == 128 ? launch_e4m3_v<128>(xs, B * H, N, bytes_out, partials, n_partials, G_out, st)
                : launch_e4m3_v<64>(xs, B * H, N, bytes_out, partials, n_partials, G_out, st);
  if (rc != FP4ATTN_OK) return rc;
  return cudaGetLastError() == cudaSuccess ? FP4ATTN_OK : FP4ATTN_ERR_CUDA;
}
