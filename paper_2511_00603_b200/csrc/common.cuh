// Small device helpers shared by the kernels.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include "desc.h"

namespace epara {

// Programmatic dependent launch.  Every kernel of a step is launched with programmatic stream
// serialisation: it may become resident while the kernel before it in the stream is still running,
// which hides launch latency and set-up.  pdl_wait() returns once all earlier kernels have completed and
// their writes are visible, and then lets the next kernel start launching.
// Rule: a kernel touches nothing that an earlier kernel of the stream writes or reads
// before its pdl_wait(); weights and the step's descriptors (uploaded by a copy that completes
// before the first kernel) may be read earlier.  Every kernel waits at least once, so completion
// is transitive along the stream.  (Launches `beside` another one wait at their end: see pdl_begin().)
//
// Why the trigger follows the wait: what a kernel does before its wait is mostly requests for weights.  With the trigger
// at the top of each kernel these piled up several kernels deep, while the kernels they were early for -- norms,
// attention, small projections, all bound by latency -- waited for memory behind them.  One kernel ahead is enough to keep
// HBM busy over a boundary (1B decoder: one request 972 -> 902 us a step, 27 requests 1385 -> 1331; one image through
// ViT-B 671 -> 635; steps of large kernels unchanged).
// A kernel that streams weights to its end takes the two halves apart: a block of it triggers when the first of its warps
// has nothing left to request.
__device__ __forceinline__ void pdl_wait_only() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// (one thread per block is enough; a block that exits counts as having triggered)
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { pdl_wait_only(); pdl_trigger(); }

// Launches of one wave work on different models (or on different rows) and do not need each other's results.  The first of
// them waits as above; the others run `beside` it: they do not wait at their start -- they could only be launched once every block
// of the kernel before had triggered, hence after all kernels before the wave were complete -- and one block of theirs waits
// at its end, so that completion stays transitive.  Without a wait a kernel's L1 may hold old lines: what earlier kernels wrote
// is read past L1 (TMA, cp.async.cg, ld.cg).  That such reads see it rests on the hardware, not on a written guarantee: the kernels
// before the wave were complete, their writes in L2, when the wave's first launch passed its own wait, and CUDA promises visibility only
// to a thread that has waited itself.  (512-token chunk beside 24 decode requests, 1B decoder: 2637 us a step with every
// launch waiting, 2519 like this; the saturated mix 13100 and 13040.)
__device__ __forceinline__ void pdl_begin(int beside) {
  if (!beside) pdl_wait_only();
  pdl_trigger();
}
__device__ __forceinline__ void pdl_end(int beside) {
  if (beside && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) pdl_wait_only();
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

__device__ __forceinline__ float bf2f(bf16 v) { return __bfloat162float(v); }
__device__ __forceinline__ bf16 f2bf(float v) { return __float2bfloat16_rn(v); }

// 8 bf16 packed in a uint4 -> 8 floats (bf16 is the top half of an fp32).
__device__ __forceinline__ void unpack8(const uint4& u, float* f) {
  f[0] = __uint_as_float(u.x << 16); f[1] = __uint_as_float(u.x & 0xffff0000u);
  f[2] = __uint_as_float(u.y << 16); f[3] = __uint_as_float(u.y & 0xffff0000u);
  f[4] = __uint_as_float(u.z << 16); f[5] = __uint_as_float(u.z & 0xffff0000u);
  f[6] = __uint_as_float(u.w << 16); f[7] = __uint_as_float(u.w & 0xffff0000u);
}

__device__ __forceinline__ unsigned pack2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<unsigned*>(&v);
}

// RoPE of one interleaved pair of bf16.  The roundings are spelled out: a key has the same bits wherever it is rotated.
__device__ __forceinline__ unsigned rotate_pair(unsigned u, float c, float s) {
  const float a = __uint_as_float(u << 16), b = __uint_as_float(u & 0xffff0000u);
  return pack2(__fmaf_rn(a, c, -__fmul_rn(b, s)), __fmaf_rn(a, s, __fmul_rn(b, c)));
}
__device__ __forceinline__ unsigned rotate_pair(unsigned u, float2 cs) { return rotate_pair(u, cs.x, cs.y); }

__device__ __forceinline__ unsigned long long pair_of(float v) {
  const unsigned long long u = __float_as_uint(v);
  return u << 32 | u;
}

// GELU in its erf form, 0.5 x (1 + erf(x / sqrt 2)), evaluated as 0.5 x (1 + tanh(x P(x^2))) with
// P(t) = a + b t + c t^2 fitted (minimax over |x| <= 8) so that tanh(x P(x^2)) follows erf(x / sqrt 2):
// the formula itself is within 2.6e-5 of the erf form everywhere.  t is clamped at 64, where the
// argument is already past saturation, because c < 0 would turn P around for |x| > 11.  tanh comes
// from the hardware approximation (relative error 2^-11 of tanh), which bounds the absolute error of
// the result by about 2.5e-4 |x|: below the rounding of the bf16 store for x > 0, and of the size of
// that rounding at the typical magnitude of the tensor for the small negative outputs.
// Seven FMA-pipe instructions and one special-function instruction per element.
__device__ __forceinline__ float gelu_erf(float x) {
  const float t = fminf(x * x, 64.0f);
  float p = fmaf(t, -3.51516781e-4f, 3.70056460e-2f);
  p = fmaf(t, p, 7.97507884e-1f);
  float th;
  asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(x * p));
  const float hx = 0.5f * x;
  return fmaf(hx, th, hx);
}
// The same for two values, two fp32 operations per instruction (the same roundings): the loops of an epilogue are bound by
// issue slots, 13 an element with a scalar form and 9 like this.
__device__ __forceinline__ void gelu_erf2(float& a, float& b) {
  asm("{\n\t.reg .b64 x, t, p, h;\n\t.reg .f32 t0, t1;\n\t"
      "mov.b64 x, {%0, %1};\n\t"
      "mul.rn.f32x2 t, x, x;\n\t"
      "mov.b64 {t0, t1}, t;\n\tmin.f32 t0, t0, 0f42800000;\n\tmin.f32 t1, t1, 0f42800000;\n\tmov.b64 t, {t0, t1};\n\t"
      "fma.rn.f32x2 p, t, %2, %3;\n\t"
      "fma.rn.f32x2 p, t, p, %4;\n\t"
      "mul.rn.f32x2 p, x, p;\n\t"
      "mov.b64 {t0, t1}, p;\n\ttanh.approx.f32 t0, t0;\n\ttanh.approx.f32 t1, t1;\n\tmov.b64 p, {t0, t1};\n\t"
      "mul.rn.f32x2 h, x, %5;\n\t"
      "fma.rn.f32x2 x, h, p, h;\n\t"
      "mov.b64 {%0, %1}, x;\n\t}"
      : "+f"(a), "+f"(b)
      : "l"(pair_of(-3.51516781e-4f)), "l"(pair_of(3.70056460e-2f)), "l"(pair_of(7.97507884e-1f)), "l"(pair_of(0.5f)));
}
// a, b plus the two bf16 in w
__device__ __forceinline__ void add_bias2(float& a, float& b, unsigned w) {
  asm("{\n\t.reg .b64 x, y;\n\t.reg .b32 lo, hi;\n\tshl.b32 lo, %2, 16;\n\tand.b32 hi, %2, 0xffff0000;\n\t"
      "mov.b64 x, {%0, %1};\n\tmov.b64 y, {lo, hi};\n\tadd.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}" : "+f"(a), "+f"(b) : "r"(w));
}
// x / (1 + e^-x) with the fast division (2 ulp; the denominator is at least 1, and an overflowed e^-x gives 0,
// the limit).  The IEEE division's special-case path, which a zero numerator takes, measured 3x slower in
// the epilogue loops.
__device__ __forceinline__ float silu_f(float x) { return __fdividef(x, 1.0f + __expf(-x)); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

}  // namespace epara
