// Small device helpers shared by the kernel translation units.
#pragma once
#include <atomic>

#include <cuda_runtime.h>

namespace tddft {

// Radix-stage passes (n = 8 and 12, and the FP64 inverse z transform of the local potential at every n):
// at 96, 384 threads give every butterfly loop (1152, 2304, 3072 butterflies) whole iterations.
template <int N> struct FFTThreads { static constexpr int value = (N >= 96) ? 384 : 256; };

// Minimum resident CTAs per SM requested of the register allocator for them: four in FP32, which fit
// without spills; FP64 variants keep their registers.
template <typename R> struct FFTMinBlocks { static constexpr int value = 1; };
template <> struct FFTMinBlocks<float> { static constexpr int value = 4; };

// Programmatic dependent launch: the kernel may be set up before its predecessor on the stream has
// ended, and calls pdl_wait() (which returns when it has, its writes visible) before it touches
// memory the predecessor writes or reads.  2 us less between two short dependent kernels.
//
// A pointer that a kernel gets as const __restrict__, and a load by __ldg, promise the compiler that
// nobody writes the data while the kernel lives; an unaliased pointer promises that pdl_wait() does
// not concern it.  Either lets a load move above the wait.  So a kernel launched by launch_pdl
// takes what any kernel of the chain writes through plain pointers and reads it by ordinary loads,
// which the wait's memory clobber keeps behind it; the qualifiers are for the tables written at
// creation only.  (Steps at 48^3, 64^3 and 96^3 measure the same within 0.4 % either way.)
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Opt in to a kernel's dynamic shared memory, once per device (the attribute calls cost more host time
// than the launch).
template <typename K> inline cudaError_t opt_in_smem(K kf, size_t smem, std::atomic<unsigned long long>& done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (done.load(std::memory_order_relaxed) & bit) return cudaSuccess;
  if ((e = cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
  e = cudaFuncSetAttribute(kf, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
  return e;
}

template <typename... K, typename... A>
inline cudaError_t launch_pdl(void (*kf)(K...), dim3 grid, int nt, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(nt);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kf, static_cast<K>(args)...);
}

template <int N> __device__ __forceinline__ int freq(int i) { return i < N / 2 ? i : i - N; }

// FP32 Chebyshev arithmetic with the series constants as float pairs hi + lo (see
// split_constants): (x - c p) / Delta with c = {hi, lo} and 1 / Delta = {hi, lo} ...
__device__ __forceinline__ float shifted_f(float x, float p, const float* c, const float* id) {
  const float d = (x - c[0] * p) - c[1] * p;
  return d * id[0] + d * id[1];
}
// ... and a z for the complex constant z = {re hi, im hi, re lo, im lo}.
__device__ __forceinline__ float2 cmul_split(float2 a, const float* z) {
  return make_float2((z[0] * a.x - z[1] * a.y) + (z[2] * a.x - z[3] * a.y),
                     (z[0] * a.y + z[1] * a.x) + (z[2] * a.y + z[3] * a.x));
}

// Accumulator updates acc += sum_j z_j t_j in float-float arithmetic, rounded to FP32 once.
// Rounding each product of FP32 data with a fixed FP32 constant (and each partial sum) is biased
// for a given constant: summed over a state the errors do not cancel, and the series output gains
// or loses ~1e-8 of its norm per series, every step in the same direction (an FP32 path drifted
// by ~6e-8 in norm per step).  Here every product is split exactly (p + pe = a b, by a fused
// multiply-add) and every sum is exact (hi + lo, Knuth's two-sum), so the update is the exact
// value rounded once.  __fmul_rn / __fadd_rn are never contracted into multiply-adds, which would
// break the splits.
__device__ __forceinline__ void ff_madd(float& hi, float& lo, float a, float b) {
  const float p = __fmul_rn(a, b);
  const float pe = fmaf(a, b, -p);
  const float s = __fadd_rn(hi, p);
  const float bb = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  hi = s;
  lo += e + pe;
}
// (hi, lo) += t z for the complex constant z = {re hi, im hi, re lo, im lo}.
__device__ __forceinline__ void ff_cmadd(float2& hi, float2& lo, float2 t, const float* z) {
  ff_madd(hi.x, lo.x, z[0], t.x);
  ff_madd(hi.x, lo.x, -z[1], t.y);
  ff_madd(hi.y, lo.y, z[0], t.y);
  ff_madd(hi.y, lo.y, z[1], t.x);
  lo.x += z[2] * t.x - z[3] * t.y;
  lo.y += z[2] * t.y + z[3] * t.x;
}

// (hi, lo) += s (-i)^i t up to the sign in s = {hi, lo}: the parts of t as they are (i even) or
// (t.y, -t.x) (i odd, swap).  Half the products of ff_cmadd.
__device__ __forceinline__ void ff_rmadd(float2& hi, float2& lo, float2 t, const float* s, bool swap) {
  const float a = swap ? t.y : t.x, b = swap ? -t.x : t.y;
  ff_madd(hi.x, lo.x, s[0], a);
  ff_madd(hi.y, lo.y, s[0], b);
  lo.x += s[1] * a;
  lo.y += s[1] * b;
}
// z (hi + lo) rounded to FP32 once, z = {re hi, im hi, re lo, im lo}.
__device__ __forceinline__ float2 ff_phase(float2 hi, float2 lo, const float* z) {
  float2 h = make_float2(0.f, 0.f), l = make_float2(0.f, 0.f);
  ff_cmadd(h, l, hi, z);
  l.x += z[0] * lo.x - z[1] * lo.y;
  l.y += z[0] * lo.y + z[1] * lo.x;
  return make_float2(h.x + l.x, h.y + l.y);
}

#define TDDFT_DISPATCH_N(N, CALL)          \
  switch (N) {                             \
    case 8: { constexpr int NN = 8; return CALL; }   \
    case 12: { constexpr int NN = 12; return CALL; } \
    case 16: { constexpr int NN = 16; return CALL; } \
    case 24: { constexpr int NN = 24; return CALL; } \
    case 32: { constexpr int NN = 32; return CALL; } \
    case 48: { constexpr int NN = 48; return CALL; } \
    case 64: { constexpr int NN = 64; return CALL; } \
    case 96: { constexpr int NN = 96; return CALL; } \
    default: return cudaErrorInvalidValue;           \
  }

template <typename R> __device__ __forceinline__ void sincos_r(R x, R* s, R* c);
template <> __device__ __forceinline__ void sincos_r<float>(float x, float* s, float* c) { sincosf(x, s, c); }
template <> __device__ __forceinline__ void sincos_r<double>(double x, double* s, double* c) { sincos(x, s, c); }

template <typename R>
__device__ __forceinline__ R warp_sum(R v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}


}  // namespace tddft
