// xy pass of the kinetic term with its planes brought into shared memory by the bulk
// asynchronous copy engine (FP32, two-factor sizes).
//
// The register-fed pass reads its plane from HBM into registers, so the bytes in flight are
// bounded by the warps resident on the SM.  Here each CTA is persistent and double-buffers whole
// planes: while it transforms plane j in one buffer, the row copies of plane j + grid
// (`cp.async.bulk`, one 16-byte-aligned row each, completion counted in bytes on an mbarrier)
// fill the other.  The first DFT stage reads the buffer in place; the rest of the transform is
// that of k_fft_xy2 (one exchange per axis, the last stage writing HBM from registers), so the
// results are the same bits.  (The z pass gains nothing from this form: with one exchange its
// register-fed kernel keeps more CTAs per SM busy than a double-buffered slab would leave.)
//
// Source and destination may be the same array: a CTA reads each plane (by the copy engine)
// before it writes it, and no other CTA touches it.
//
// Every mbarrier wait has an iteration limit: on expiry the CTA sets bit 2 of the error word,
// waits once more (again with a limit) for the copy in flight and carries on with what the
// buffer holds; every index stays in bounds, and the host reports the flag.
#include <cstdint>

#include "bulk.cuh"
#include "fft.cuh"
#include "impl.cuh"
#include "kcommon.cuh"

namespace tddft {

namespace {

// N rows of N complex values (row r at g + r * stride) into a buffer with row pitch P; called by
// the 32 lanes of warp 0.  Row bytes N * 8, the pitch P * 8 and the row addresses are
// multiples of 16 for every size used here (N even).
template <int N, int P>
__device__ __forceinline__ void issue_rows(const float2* g, size_t stride, float2* buf, uint32_t bar, int lane) {
  constexpr uint32_t ROW = N * sizeof(float2);
  if (lane == 0) bulk_expect(bar, ROW * N);
  __syncwarp();
  for (int row = lane; row < N; row += 32) bulk_copy(buf + row * P, g + (size_t)row * stride, ROW, bar);
}

// Row pitch of the two buffers (rows arrive as they are: no swizzle).
template <int N> struct TmaPitch { static constexpr int value = (N % 16 == 8) ? N : N + 8; };

// Resident CTAs asked of the register allocator; the two 36 KB buffers of a 64^2 plane allow three.
// At 96^2 the two 78 KB buffers would leave one CTA per SM: 96 takes the register-fed pass.
template <int N> struct XyTmaBlocks { static constexpr int value = 8; };
template <> struct XyTmaBlocks<64> { static constexpr int value = 3; };
template <> struct XyTmaBlocks<48> { static constexpr int value = 5; };

}  // namespace

// The transform is that of k_fft_xy2 (XYPlane) with its first side reading the buffer in place: the
// forward x A side rows by warp, the inverse y B side with every read of the plane before the first
// write.
template <int N, bool INV>
__global__ void __launch_bounds__(XYThreads<N>::value, XyTmaBlocks<N>::value)
k_fft_xy2_tma(const float2* src, float2* dst, const float2* __restrict__ twg, int nplanes, int* err) {
  using C = float2;
  constexpr int RS = TmaPitch<N>::value;
  using PL = XYPlane<C, N, RS, false>;
  constexpr int R1 = PL::R1, R2 = PL::R2, NT = PL::NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* buf0 = tw + N;
  C* buf1 = buf0 + N * RS;
  uint64_t* bars = reinterpret_cast<uint64_t*>(buf1 + N * RS);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bar0 = sm_addr(&bars[0]), bar1 = sm_addr(&bars[1]);
  if (threadIdx.x == 0) bulk_init(bar0, bar1);
  for (int i = threadIdx.x; i < N; i += NT) tw[i] = twg[i];
  pdl_wait();
  __syncthreads();
  int pl = blockIdx.x;
  if (pl < nplanes && warp == 0) issue_rows<N, RS>(src + (size_t)pl * N * N, N, buf0, bar0, lane);
  // Buffer schedule: at the start of plane j the copies of plane j + grid go to the other buffer,
  // whose last reader (plane j - grid) ended with the CTA barrier closing the previous step.
  for (int it = 0; pl < nplanes; ++it, pl += gridDim.x) {
    const int sb = it & 1;
    C* s = sb ? buf1 : buf0;
    const int nx = pl + gridDim.x;
    if (nx < nplanes && warp == 0) issue_rows<N, RS>(src + (size_t)nx * N * N, N, sb ? buf0 : buf1, sb ? bar0 : bar1, lane);
    bulk_wait(sb ? bar1 : bar0, (uint32_t)(it >> 1) & 1u, err, 2);
    C* o = dst + (size_t)pl * N * N;
    if constexpr (!INV) {
      PL::x_a_fwd(s, s, RS, tw, warp, lane);
      __syncwarp();
      PL::template x_b<false>(s, tw, warp, lane);
      __syncthreads();
      PL::template y_a<false>(s, tw);
      __syncthreads();
      PL::y_b_fwd(s, o, tw);
    } else {
      // y, B side in place: item (x, K0)
      C u[PL::YB][R1];
#pragma unroll
      for (int p = 0; p < PL::YB; ++p) {
        const int i = threadIdx.x + p * NT;
        if (N * R2 % NT == 0 || i < N * R2) {
          const int k0 = i / N, x = i - k0 * N;
#pragma unroll
          for (int k1 = 0; k1 < R1; ++k1) u[p][k1] = s[PL::col(k0 + R2 * k1, x)];
        }
      }
      __syncthreads();
#pragma unroll
      for (int p = 0; p < PL::YB; ++p) {
        const int i = threadIdx.x + p * NT;
        if (N * R2 % NT == 0 || i < N * R2) {
          const int k0 = i / N, x = i - k0 * N;
          TF<C, N, true>::b_side(u[p], k0, tw);
#pragma unroll
          for (int n0 = 0; n0 < R1; ++n0) s[PL::col(k0 * R1 + n0, x)] = u[p][n0];
        }
      }
      __syncthreads();
      PL::template y_a<true>(s, tw);
      __syncthreads();
      PL::template x_b<true>(s, tw, warp, lane);
      __syncwarp();
      PL::x_a_inv(s, o, tw, warp, lane);
    }
    __syncthreads();
  }
}

bool fft_xy_tma_supported(int N) { return N == 16 || N == 24 || N == 32 || N == 48 || N == 64; }

// CTAs of a full wave on the current device, asked once per device and kernel.
template <int N, bool INV>
static cudaError_t xy_tma_ni(cudaStream_t st, const void* src, void* dst, int nbatch, const void* tw, int* err) {
  const size_t smem = (size_t)(N + 2 * N * TmaPitch<N>::value) * sizeof(float2) + 2 * sizeof(uint64_t);
  auto kf = k_fft_xy2_tma<N, INV>;
  static std::atomic<unsigned long long> done{0};
  static std::atomic<int> wave[64];
  int dev = 0;
  cudaError_t e;
  if ((e = opt_in_smem(kf, smem, done)) != cudaSuccess || (e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  int ctas = wave[dev & 63].load(std::memory_order_relaxed);
  if (!ctas) {
    int sms = 0, per_sm = 0;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
        (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kf, XYThreads<N>::value, smem)) != cudaSuccess)
      return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    ctas = sms * per_sm;
    wave[dev & 63].store(ctas, std::memory_order_relaxed);
  }
  const int nplanes = N * nbatch;
  return launch_pdl(kf, dim3(std::min(nplanes, ctas)), XYThreads<N>::value, smem, st, (const float2*)src, (float2*)dst,
                    (const float2*)tw, nplanes, err);
}
template <int N>
static cudaError_t xy_tma_n(cudaStream_t st, const void* src, void* dst, int nbatch, const void* tw, bool inv,
                            int* err) {
  return inv ? xy_tma_ni<N, true>(st, src, dst, nbatch, tw, err) : xy_tma_ni<N, false>(st, src, dst, nbatch, tw, err);
}

cudaError_t launch_fft_xy_tma(cudaStream_t st, int N, const void* src, void* dst, int nbatch, const void* tw, bool inv,
                              int* err) {
  if (nbatch <= 0) return cudaSuccess;
  if (((uintptr_t)src & 15) != 0 || !err) return cudaErrorInvalidValue;
  switch (N) {
    case 16: return xy_tma_n<16>(st, src, dst, nbatch, tw, inv, err);
    case 24: return xy_tma_n<24>(st, src, dst, nbatch, tw, inv, err);
    case 32: return xy_tma_n<32>(st, src, dst, nbatch, tw, inv, err);
    case 48: return xy_tma_n<48>(st, src, dst, nbatch, tw, inv, err);
    case 64: return xy_tma_n<64>(st, src, dst, nbatch, tw, inv, err);
    default: return cudaErrorNotSupported;
  }
}


cudaError_t set_first_wait_fft(unsigned polls) { return cudaMemcpyToSymbol(g_first_wait, &polls, sizeof(polls)); }

}  // namespace tddft
