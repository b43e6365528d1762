// Shared device helpers for the fp4attn kernels (sm_100a only).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <string.h>

#include <atomic>
#include <mutex>

#include "../../include/fp4attn.h"

namespace fp4attn {

// Eight floats -> one 32-bit word of eight E2M1 codes (element k in nibble k).
__device__ __forceinline__ uint32_t cvt_e2m1x8(const float* v) {
  uint32_t w;
  asm("{\n\t.reg .b8 t0, t1, t2, t3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 t0, %2, %1;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 t1, %4, %3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 t2, %6, %5;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 t3, %8, %7;\n\t"
      "mov.b32 %0, {t0, t1, t2, t3};\n\t}"
      : "=r"(w)
      : "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]));
  return w;
}

// same, with negative inputs clamped to +0 by the conversion itself
__device__ __forceinline__ uint32_t cvt_e2m1x8_relu(const float* v) {
  uint32_t w;
  asm("{\n\t.reg .b8 t0, t1, t2, t3;\n\t"
      "cvt.rn.satfinite.relu.e2m1x2.f32 t0, %2, %1;\n\t"
      "cvt.rn.satfinite.relu.e2m1x2.f32 t1, %4, %3;\n\t"
      "cvt.rn.satfinite.relu.e2m1x2.f32 t2, %6, %5;\n\t"
      "cvt.rn.satfinite.relu.e2m1x2.f32 t3, %8, %7;\n\t"
      "mov.b32 %0, {t0, t1, t2, t3};\n\t}"
      : "=r"(w)
      : "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]));
  return w;
}

// the first six of eight elements; the last two get code 0
__device__ __forceinline__ uint32_t cvt_e2m1x6_relu(const float* v) {
  uint32_t w;
  asm("{\n\t.reg .b8 t0, t1, t2, t3;\n\tmov.b32 {t3, _, _, _}, 0;\n\t"
      "cvt.rn.satfinite.relu.e2m1x2.f32 t0, %2, %1;\n\t"
      "cvt.rn.satfinite.relu.e2m1x2.f32 t1, %4, %3;\n\t"
      "cvt.rn.satfinite.relu.e2m1x2.f32 t2, %6, %5;\n\t"
      "mov.b32 %0, {t0, t1, t2, t3};\n\t}"
      : "=r"(w)
      : "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]));
  return w;
}

// Squared error of eight scaled values t against their codes (one word), in code units: d = t - q exact,
// fl32(d * d) added left to right in fp32 - the order the MSE amplitude rule is defined with.
__device__ __forceinline__ float mx_error_x8(const float* t, uint32_t codes) {
  float acc = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    uint32_t h2;
    asm("{\n\t.reg .b8 b;\n\t.reg .b32 s;\n\tshr.b32 s, %1, %2;\n\tcvt.u8.u32 b, s;\n\tcvt.rn.f16x2.e2m1x2 %0, b;\n\t}"
        : "=r"(h2) : "r"(codes), "r"(8 * i));
    const float2 q = __half22float2(*reinterpret_cast<const __half2*>(&h2));
    const float d0 = __fsub_rn(t[2 * i], q.x), d1 = __fsub_rn(t[2 * i + 1], q.y);
    const float s0 = __fmul_rn(d0, d0), s1 = __fmul_rn(d1, d1);
    acc = (i == 0) ? s0 : __fadd_rn(acc, s0);
    acc = __fadd_rn(acc, s1);
  }
  return acc;
}
__device__ __forceinline__ void bf16x8_to_f32(const uint4& raw, float* v) {
  const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[2 * i] = __uint_as_float(w[i] << 16);
    v[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
  }
}

// 2^(127-u) for u in [0, 254] (u = 254 needs the subnormal 2^-127).
__device__ __forceinline__ float mx_inv_amplitude(uint32_t u) {
  return __uint_as_float(u == 254u ? 0x00400000u : ((254u - u) << 23));
}

// Programmatic dependent launch.  Every quantizer kernel lets its successor start when its own last blocks have
// (launch_dependents in each block's first instructions), and every kernel of the path touches global memory only after wait_prior_grids, which
// returns when all earlier kernels of the stream are complete and their writes visible.  What overlaps is a kernel's launch
// and its set-up with the tail of the one before: the 1.5-2.5 us between two kernels of a step (B=1, H=16, N=4096, affine map,
// whole step: 73.7 -> 64.0 us).  The attention kernels wait but do not announce: the next step's quantizer blocks, resident
// beside an attention block and waiting, cost it up to 3 % (B=32, H=16, N=1024: 242 against 228 us a step).
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_prior_grids() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... Params, class... Args>
cudaError_t launch_overlapped_clusters(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, unsigned cluster,
                                       Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2] = {};
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}
template <class... Params, class... Args>
cudaError_t launch_overlapped(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, Args&&... args) {
  return launch_overlapped_clusters(kernel, grid, threads, smem, st, 1u, static_cast<Args&&>(args)...);
}

constexpr int kMaxDevices = 64;      // per-device host-side caches are arrays of this length

int check_device_sm100();            // FP4ATTN_OK or FP4ATTN_ERR_UNSUPPORTED_ARCH / _CUDA
int device_sms();                    // SMs of the current device, kept per device; 0 if the runtime does not tell

}  // namespace fp4attn
