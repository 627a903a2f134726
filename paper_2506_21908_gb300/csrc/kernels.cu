// sm_103a kernels of the spinor propagation step.
//
//   k_fft_xy     one z-plane of one spinor component: 2D FFT along x then y in shared memory
//   k_fft_z      one y-slab of one component: FFT along z, multiply by 1/2|G+k+A|^2, inverse FFT
//                along z -- the kinetic term of Eq. HNC-SDFT (k_fft_xy2, k_fft_z2_kin: two-factor sizes)
//   k_proj_gather  c_{a,p,sigma} = sum_{r in S_a} beta~_p(r)^* psi_sigma(r) dV and D_a c
//                (the contraction of the separable projectors, Eq. Vps with the L.S block)
//   (k_epilogue, the pointwise Hamiltonian and Chebyshev update, is in epilogue.cu)
//   k_density    rho_v = sum_k w_k sum_i f_i {|u|^2, |d|^2, Re u d*, Im u d*}  (Eqs. rho1-rho3)
//   k_potential  locally collinear LSDA (Eqs. LC+ALDA2, LC+ALDA) and assembly of V_v
//   reductions   deterministic fixed-order block reductions for energies and norms
#include <algorithm>
#include <cstdint>

#include "fft.cuh"
#include "impl.cuh"
#include "kcommon.cuh"
#include "kepi.cuh"

namespace tddft {


// ============================================================================ FFT passes

template <typename R, int N, bool INV>
__global__ void __launch_bounds__(FFTThreads<N>::value, FFTMinBlocks<R>::value)
k_fft_xy(const typename CT<R>::type* src, typename CT<R>::type* dst, const typename CT<R>::type* __restrict__ twg) {
  using C = typename CT<R>::type;
  constexpr int NT = FFTThreads<N>::value;
  constexpr int RS = N + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* s = tw + N;
  const size_t base = ((size_t)blockIdx.y * N + blockIdx.x) * (size_t)(N * N);
  for (int i = threadIdx.x; i < N; i += NT) tw[i] = twg[i];
  plane_load<N, NT, RS>(s, src + base);
  __syncthreads();
  fft_pass<C, N, NT, INV>(s, RS, 1, tw);  // along x (rows: y)
  fft_pass<C, N, NT, INV>(s, 1, RS, tw);  // along y (rows: x)
  plane_store<N, NT, RS>(dst + base, s);
}


// Per-axis multiplier tables for the z pass: the kinetic factor 1/2 |G + s|^2 scale is
// tx[x] + ty[y] + tz[z] with ta[i] = 1/2 (g_a f(i) + s_a)^2 scale (computed in FP64, stored in R).
template <typename R, int N>
__device__ __forceinline__ void z_tables(R* tx, R* tz, R* ty, const ZParams& zp, int y, int k) {
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    const double qx = zp.gs[0] * freq<N>(i) + zp.shift[k][0];
    const double qz = zp.gs[2] * freq<N>(i) + zp.shift[k][2];
    tx[i] = (R)(0.5 * qx * qx * zp.scale);
    tz[i] = (R)(0.5 * qz * qz * zp.scale);
  }
  if (threadIdx.x == 0) {
    const double qy = zp.gs[1] * freq<N>(y) + zp.shift[k][1];
    *ty = (R)(0.5 * qy * qy * zp.scale);
  }
}

template <typename R, int N, int MODE>
__global__ void __launch_bounds__(FFTThreads<N>::value, FFTMinBlocks<R>::value)
k_fft_z(typename CT<R>::type* __restrict__ data, const typename CT<R>::type* __restrict__ twg, ZParams zp) {
  using C = typename CT<R>::type;
  constexpr int NT = FFTThreads<N>::value;
  // dense slab [z][x]: the z transforms run with x fastest across lanes, conflict-free at any pitch
  constexpr int RS = N;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* s = tw + N;
  R* tx = reinterpret_cast<R*>(s + N * RS);
  R* tz = tx + N;
  R* ty = tz + N;
  const int y = blockIdx.x;
  const int b = blockIdx.y;
  const size_t base = (size_t)b * N * N * N + (size_t)y * N;
  for (int i = threadIdx.x; i < N; i += NT) tw[i] = twg[i];
  if (MODE != Z_INV_ONLY) z_tables<R, N>(tx, tz, ty, zp, y, b / zp.comps_per_k);
  slab_load<N, NT, RS>(s, data + base, (size_t)N * N);
  __syncthreads();
  if (MODE != Z_INV_ONLY) {
    fft_pass<C, N, NT, false>(s, 1, RS, tw);  // along z (rows: x)
    const R tyv = *ty;
    for (int i = threadIdx.x; i < N * N; i += NT) {
      const int z = i / N, x = i - z * N;
      s[z * RS + x] = cscale(s[z * RS + x], tx[x] + tyv + tz[z]);
    }
    __syncthreads();
  }
  fft_pass<C, N, NT, true>(s, 1, RS, tw);
  slab_store<N, NT, RS>(data + base, s, (size_t)N * N);
}

// ---------------------------------------------------------------- two-factor passes (N = R1 R2)

// Resident CTAs per SM asked of the register allocator (FP32; what the dense planes and slabs
// allow).  FP64 is bound by its arithmetic and keeps its registers.
template <typename R, int N> struct XYBlocks { static constexpr int value = 1; };
template <> struct XYBlocks<float, 96> { static constexpr int value = 3; };
template <> struct XYBlocks<float, 64> { static constexpr int value = 5; };
template <> struct XYBlocks<float, 48> { static constexpr int value = 10; };
template <> struct XYBlocks<float, 32> { static constexpr int value = 8; };
template <> struct XYBlocks<float, 24> { static constexpr int value = 10; };
template <> struct XYBlocks<float, 16> { static constexpr int value = 16; };

// xy transform of one z-plane with one shared-memory exchange per axis: the x transform's A side
// reads global memory directly, the y transform's B side writes it directly (forward); the
// inverse runs the steps in the opposite order.  The x axis is warp-local and in place (XYPlane), so
// two CTA barriers remain, and the dense swizzled plane lets three CTAs of 96^2 share an SM.
template <typename R, int N, bool INV>
__global__ void __launch_bounds__(XYThreads<N>::value, XYBlocks<R, N>::value)
k_fft_xy2(const typename CT<R>::type* src, typename CT<R>::type* dst, const typename CT<R>::type* __restrict__ twg) {
  using C = typename CT<R>::type;
  using PL = XYPlane<C, N, N, sizeof(R) == 4 && N % 16 == 0>;
  constexpr int R1 = PL::R1, R2 = PL::R2, NT = PL::NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tw = reinterpret_cast<C*>(smem_raw);
  C* s = tw + N;
  const size_t base = ((size_t)blockIdx.y * N + blockIdx.x) * (size_t)(N * N);
  const C* g = src + base;
  C* o = dst + base;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < N; i += NT) tw[i] = twg[i];
  pdl_wait();
  __syncthreads();
  if constexpr (!INV) {
    PL::x_a_fwd(s, g, N, tw, warp, lane);
    __syncwarp();
    PL::template x_b<false>(s, tw, warp, lane);
    __syncthreads();
    PL::template y_a<false>(s, tw);
    __syncthreads();
    PL::y_b_fwd(s, o, tw);
  } else {
    // y, B side from global: item (x, K0)
#pragma unroll
    for (int p = 0; p < PL::YB; ++p) {
      const int i = threadIdx.x + p * NT;
      if (N * R2 % NT == 0 || i < N * R2) {
        const int k0 = i / N, x = i - k0 * N;
        C u[R1];
#pragma unroll
        for (int k1 = 0; k1 < R1; ++k1) u[k1] = g[(k0 + R2 * k1) * N + x];
        TF<C, N, true>::b_side(u, k0, tw);
#pragma unroll
        for (int n0 = 0; n0 < R1; ++n0) s[PL::col(k0 * R1 + n0, x)] = u[n0];
      }
    }
    __syncthreads();
    PL::template y_a<true>(s, tw);
    __syncthreads();
    PL::template x_b<true>(s, tw, warp, lane);
    __syncwarp();
    PL::x_a_inv(s, o, tw, warp, lane);
  }
}

// Columns, threads and CTAs per SM of the z pass: a column's transform touches no other column, so a
// CTA takes 32 columns (16, 24 or 48 at those sizes), few enough threads that the barriers of one
// CTA leave the others of the SM running.  FP64: 8 columns (128-byte rows) and one warp, so that few
// components still give every SM's FP64 pipe the same work (24^3 with 8 components: 192 CTAs of 24
// columns on 152 SMs took 17.5 us with the launch, 576 of 8 take 14.2).
template <typename R, int N> struct ZCols { static constexpr int value = sizeof(R) == 8 ? 8 : (N % 32 == 0 ? 32 : N); };
template <typename R, int N> struct ZThreads {
  static constexpr int value = sizeof(R) == 8 ? 32 : (N % 32 == 0 ? 128 : (N == 16 ? 64 : 96));
};
template <typename R, int N> struct ZBlocks { static constexpr int value = 1; };
template <> struct ZBlocks<float, 96> { static constexpr int value = 7; };
template <> struct ZBlocks<float, 64> { static constexpr int value = 8; };
template <> struct ZBlocks<float, 48> { static constexpr int value = 8; };
template <> struct ZBlocks<float, 32> { static constexpr int value = 8; };
template <> struct ZBlocks<float, 24> { static constexpr int value = 8; };
template <> struct ZBlocks<float, 16> { static constexpr int value = 16; };

// Kinetic factors 1/2 (g_a f + s_a)^2 scale of every k-point, per axis in the order of the passes (x by
// kx_at), [nk][3][N]: formed in FP64 once per A(t) (a CTA forming its own spent an eighth of the
// FP64 pipe on them).
template <typename R, int N>
__global__ void k_kin_tables(ZParams zp, R* __restrict__ out) {
  const int k = blockIdx.x;
  for (int i = threadIdx.x; i < 3 * N; i += blockDim.x) {
    const int a = i / N, j = i - a * N;
    const double q = zp.gs[a] * freq<N>(a == 0 ? kx_at<N>(j) : j) + zp.shift[k][a];
    out[(size_t)k * 3 * N + i] = (R)(0.5 * q * q * zp.scale);
  }
}

// z transform + kinetic multiply + inverse z transform of one slab (y, columns), one exchange each
// way: A side (x, n0) reads global memory along z, B side (x, K0) transforms, multiplies by
// tx[x] + ty[y] + tz[kz] and transforms back in registers, A side writes global memory.
template <typename R, int N>
__global__ void __launch_bounds__(ZThreads<R, N>::value, ZBlocks<R, N>::value)
k_fft_z2_kin(typename CT<R>::type* data, const typename CT<R>::type* __restrict__ twg, const R* tab, int comps_per_k) {
  using C = typename CT<R>::type;
  using TFW = TF<C, N, false>;
  using TIN = TF<C, N, true>;
  constexpr int NT = ZThreads<R, N>::value, CW = ZCols<R, N>::value;
  constexpr int R1 = TwoFactor<N>::R1, R2 = TwoFactor<N>::R2;
  constexpr int IA = CW * R1, IB = CW * R2;
  constexpr int PA = (IA + NT - 1) / NT, PB = (IB + NT - 1) / NT;
  static_assert(NT % CW == 0, "a thread's items share one column");
  __shared__ C tw[N];
  __shared__ R tz[N];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* s = reinterpret_cast<C*>(smem_raw);          // [K0 R1 + n0][x], dense
  const int y = blockIdx.x / (N / CW), x0 = (blockIdx.x - y * (N / CW)) * CW;
  const int b = blockIdx.y;
  C* g = data + (size_t)b * N * N * N + (size_t)y * N + x0;
  constexpr size_t ZS = (size_t)N * N;
  for (int i = threadIdx.x; i < N; i += NT) tw[i] = twg[i];
  pdl_wait();
  C v[PA][R2];
#pragma unroll
  for (int p = 0; p < PA; ++p) {
    const int i = threadIdx.x + p * NT;
    if (IA % NT == 0 || i < IA) {
      const int n0 = i / CW, x = i - n0 * CW;
#pragma unroll
      for (int q = 0; q < R2; ++q) v[p][q] = g[(size_t)(n0 + R1 * q) * ZS + x];
    }
  }
  const R* tk = tab + (size_t)(b / comps_per_k) * 3 * N;
  for (int i = threadIdx.x; i < N; i += NT) tz[i] = tk[2 * N + i];
  const R txy = tk[x0 + threadIdx.x % CW] + tk[N + y];
  __syncthreads();  // tables
#pragma unroll
  for (int p = 0; p < PA; ++p) {
    const int i = threadIdx.x + p * NT;
    if (IA % NT == 0 || i < IA) {
      const int n0 = i / CW, x = i - n0 * CW;
      TFW::a_side(v[p], n0, tw);
#pragma unroll
      for (int k0 = 0; k0 < R2; ++k0) s[(k0 * R1 + n0) * CW + x] = v[p][k0];
    }
  }
  __syncthreads();
#pragma unroll
  for (int p = 0; p < PB; ++p) {
    const int i = threadIdx.x + p * NT;
    if (IB % NT == 0 || i < IB) {
      const int k0 = i / CW, x = i - k0 * CW;
      C u[R1];
#pragma unroll
      for (int n0 = 0; n0 < R1; ++n0) u[n0] = s[(k0 * R1 + n0) * CW + x];
      TFW::b_side(u, k0, tw);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) u[k1] = cscale(u[k1], txy + tz[k0 + R2 * k1]);
      TIN::b_side(u, k0, tw);
#pragma unroll
      for (int n0 = 0; n0 < R1; ++n0) s[(k0 * R1 + n0) * CW + x] = u[n0];
    }
  }
  __syncthreads();
#pragma unroll
  for (int p = 0; p < PA; ++p) {
    const int i = threadIdx.x + p * NT;
    if (IA % NT == 0 || i < IA) {
      const int n0 = i / CW, x = i - n0 * CW;
      C w[R2];
#pragma unroll
      for (int k0 = 0; k0 < R2; ++k0) w[k0] = s[(k0 * R1 + n0) * CW + x];
      TIN::a_side(w, n0, tw);
#pragma unroll
      for (int n1 = 0; n1 < R2; ++n1) g[(size_t)(n0 + R1 * n1) * ZS + x] = w[n1];
    }
  }
}

// Kinetic energy of one slab by Parseval: z transform of the xy transform (read only), then
// sum |psi(G)|^2 1/2 |G + k + A|^2 scale over the slab's G, in the working precision over a work
// item's R1 values and in FP64 above, to part[b][slab].  Half the passes of the kinetic operator
// and its product with psi.
template <typename R, int N>
__global__ void __launch_bounds__(ZThreads<R, N>::value)
k_fft_z2_energy(const typename CT<R>::type* __restrict__ data, const typename CT<R>::type* __restrict__ twg,
                const R* __restrict__ tab, int comps_per_k, double* __restrict__ part) {
  using C = typename CT<R>::type;
  using TFW = TF<C, N, false>;
  constexpr int NT = ZThreads<R, N>::value, CW = ZCols<R, N>::value;
  constexpr int R1 = TwoFactor<N>::R1, R2 = TwoFactor<N>::R2;
  constexpr int IA = CW * R1, IB = CW * R2;
  constexpr int PA = (IA + NT - 1) / NT, PB = (IB + NT - 1) / NT;
  __shared__ C tw[N];
  __shared__ R tz[N];
  __shared__ double red[NT / 32];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* s = reinterpret_cast<C*>(smem_raw);  // [K0 R1 + n0][x], dense
  const int y = blockIdx.x / (N / CW), x0 = (blockIdx.x - y * (N / CW)) * CW;
  const int b = blockIdx.y;
  const C* g = data + (size_t)b * N * N * N + (size_t)y * N + x0;
  constexpr size_t ZS = (size_t)N * N;
  const R* tk = tab + (size_t)(b / comps_per_k) * 3 * N;
  for (int i = threadIdx.x; i < N; i += NT) {
    tw[i] = twg[i];
    tz[i] = tk[2 * N + i];
  }
  const R tyv = tk[N + y];
  __syncthreads();  // tables
#pragma unroll
  for (int p = 0; p < PA; ++p) {
    const int i = threadIdx.x + p * NT;
    if (IA % NT == 0 || i < IA) {
      const int n0 = i / CW, x = i - n0 * CW;
      C v[R2];
#pragma unroll
      for (int q = 0; q < R2; ++q) v[q] = g[(size_t)(n0 + R1 * q) * ZS + x];
      TFW::a_side(v, n0, tw);
#pragma unroll
      for (int k0 = 0; k0 < R2; ++k0) s[(k0 * R1 + n0) * CW + x] = v[k0];
    }
  }
  __syncthreads();
  double e = 0.0;
#pragma unroll
  for (int p = 0; p < PB; ++p) {
    const int i = threadIdx.x + p * NT;
    if (IB % NT == 0 || i < IB) {
      const int k0 = i / CW, x = i - k0 * CW;
      C u[R1];
#pragma unroll
      for (int n0 = 0; n0 < R1; ++n0) u[n0] = s[(k0 * R1 + n0) * CW + x];
      TFW::b_side(u, k0, tw);
      const R txy = tk[x0 + x] + tyv;
      R t = (R)0;
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) t += (u[k1].x * u[k1].x + u[k1].y * u[k1].y) * (txy + tz[k0 + R2 * k1]);
      e += (double)t;
    }
  }
  e = warp_sum(e);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = e;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < NT / 32; ++w) t += red[w];
    part[(size_t)b * gridDim.x + blockIdx.x] = t;
  }
}

template <typename R, int N, bool INV>
static cudaError_t fft_xy_ni(cudaStream_t st, const void* src, void* data, int nbatch, const void* tw) {
  using C = typename CT<R>::type;
  static std::atomic<unsigned long long> done{0};
  cudaError_t e;
  if constexpr (TwoFactor<N>::ok) {
    const size_t smem = (size_t)(N + N * N) * sizeof(C);
    auto kf = k_fft_xy2<R, N, INV>;
    if ((e = opt_in_smem(kf, smem, done)) != cudaSuccess) return e;
    return launch_pdl(kf, dim3(N, nbatch), XYThreads<N>::value, smem, st, (const C*)src, (C*)data, (const C*)tw);
  } else {
    const size_t smem = (size_t)(N + N * (N + 1)) * sizeof(C);
    auto kf = k_fft_xy<R, N, INV>;
    if ((e = opt_in_smem(kf, smem, done)) != cudaSuccess) return e;
    kf<<<dim3(N, nbatch), FFTThreads<N>::value, smem, st>>>((const C*)src, (C*)data, (const C*)tw);
  }
  return cudaGetLastError();
}
template <typename R, int N>
static cudaError_t fft_xy_n(cudaStream_t st, const void* src, void* data, int nbatch, const void* tw, bool inv) {
  return inv ? fft_xy_ni<R, N, true>(st, src, data, nbatch, tw) : fft_xy_ni<R, N, false>(st, src, data, nbatch, tw);
}

template <typename R, int N, int MODE>
static cudaError_t fft_z_nm(cudaStream_t st, void* data, int nbatch, const void* tw, const void* tab, const ZParams& zp) {
  using C = typename CT<R>::type;
  static std::atomic<unsigned long long> done{0};
  cudaError_t e;
  if constexpr (MODE == Z_KIN && TwoFactor<N>::ok) {
    constexpr int CW = ZCols<R, N>::value;
    const size_t smem = (size_t)N * CW * sizeof(C);
    auto kf = k_fft_z2_kin<R, N>;
    if ((e = opt_in_smem(kf, smem, done)) != cudaSuccess) return e;
    return launch_pdl(kf, dim3(N * (N / CW), nbatch), ZThreads<R, N>::value, smem, st, (C*)data, (const C*)tw,
                      (const R*)tab, zp.comps_per_k);
  } else {
    const size_t smem = (size_t)(N + N * N) * sizeof(C) + (2 * N + 2) * sizeof(R);
    auto kf = k_fft_z<R, N, MODE>;
    if ((e = opt_in_smem(kf, smem, done)) != cudaSuccess) return e;
    kf<<<dim3(N, nbatch), FFTThreads<N>::value, smem, st>>>((C*)data, (const C*)tw, zp);
  }
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_fft_xy(cudaStream_t st, int N, const void* src, void* data, int nbatch, const void* tw, bool inv) {
  TDDFT_DISPATCH_N(N, (fft_xy_n<R, NN>(st, src, data, nbatch, tw, inv)));
}
template <typename R>
cudaError_t launch_fft_z_kinetic(cudaStream_t st, int N, void* data, int nbatch, const void* tw, const void* tab,
                                 const ZParams& zp) {
  TDDFT_DISPATCH_N(N, (fft_z_nm<R, NN, Z_KIN>(st, data, nbatch, tw, tab, zp)));
}
// Slabs per component of the energy pass (0: no such pass at this size).
template <typename R> int fft_z_energy_parts(int N) {
  switch (N) {
    case 16: return 16 * (16 / ZCols<R, 16>::value);
    case 24: return 24 * (24 / ZCols<R, 24>::value);
    case 32: return 32 * (32 / ZCols<R, 32>::value);
    case 48: return 48 * (48 / ZCols<R, 48>::value);
    case 64: return 64 * (64 / ZCols<R, 64>::value);
    case 96: return 96 * (96 / ZCols<R, 96>::value);
    default: return 0;
  }
}
template <typename R, int N>
static cudaError_t fft_z_energy_n(cudaStream_t st, const void* data, int nbatch, const void* tw, const void* tab,
                                  const ZParams& zp, double* part) {
  if constexpr (TwoFactor<N>::ok) {
    using C = typename CT<R>::type;
    static std::atomic<unsigned long long> done{0};
    constexpr int CW = ZCols<R, N>::value;
    const size_t smem = (size_t)N * CW * sizeof(C);
    auto kf = k_fft_z2_energy<R, N>;
    cudaError_t e = opt_in_smem(kf, smem, done);
    if (e != cudaSuccess) return e;
    kf<<<dim3(N * (N / CW), nbatch), ZThreads<R, N>::value, smem, st>>>((const C*)data, (const C*)tw, (const R*)tab,
                                                                     zp.comps_per_k, part);
    return cudaGetLastError();
  } else {
    return cudaErrorInvalidValue;
  }
}
// out2[band] = {sum of the band's per_band partials, 0}: one warp per band.
__global__ void k_energy_sum(int nbands, int per_band, const double* __restrict__ part, double* __restrict__ out2) {
  const int band = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (band >= nbands) return;
  double t = 0.0;
  for (int i = lane; i < per_band; i += 32) t += part[(size_t)band * per_band + i];
  t = warp_sum(t);
  if (lane == 0) {
    out2[2 * band] = t;
    out2[2 * band + 1] = 0.0;
  }
}
template <typename R>
static cudaError_t fft_z_energy(cudaStream_t st, int N, const void* data, int nbatch, const void* tw, const void* tab,
                                const ZParams& zp, double* part) {
  TDDFT_DISPATCH_N(N, (fft_z_energy_n<R, NN>(st, data, nbatch, tw, tab, zp, part)));
}
template <typename R>
cudaError_t launch_fft_z_energy(cudaStream_t st, int N, const void* data, int nbands, const void* tw, const void* tab,
                                const ZParams& zp, double* part, double* out2) {
  cudaError_t e = fft_z_energy<R>(st, N, data, 2 * nbands, tw, tab, zp, part);
  if (e != cudaSuccess) return e;
  k_energy_sum<<<(nbands + 3) / 4, 128, 0, st>>>(nbands, 2 * fft_z_energy_parts<R>(N), part, out2);
  return cudaGetLastError();
}
cudaError_t launch_fft_z_inverse(cudaStream_t st, int N, double2* data, int nbatch, const double2* tw) {
  const ZParams zp{};
  TDDFT_DISPATCH_N(N, (fft_z_nm<double, NN, Z_INV_ONLY>(st, data, nbatch, tw, nullptr, zp)));
}
template <typename R, int N> static cudaError_t kin_tables_n(cudaStream_t st, int nk, const ZParams& zp, void* out) {
  k_kin_tables<R, N><<<nk, 128, 0, st>>>(zp, (R*)out);
  return cudaGetLastError();
}
template <typename R> cudaError_t launch_kin_tables(cudaStream_t st, int N, int nk, const ZParams& zp, void* out) {
  TDDFT_DISPATCH_N(N, (kin_tables_n<R, NN>(st, nk, zp, out)));
}

// ============================================================================ projectors

// exp(i s.d) of every entry, per k-point: evaluated once per A(t) instead of once per entry, spinor
// and Chebyshev term (in FP64 the sine and cosine were 110 of the 181 FP64 instructions an entry
// cost the gather, whose bound is the FP64 pipe).
template <typename R>
__global__ void __launch_bounds__(256)
k_phase_table(size_t nent, const R* __restrict__ rows, EpiParams ep, typename CT<R>::type* out) {
  using C = typename CT<R>::type;
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nent) return;
  const int k = blockIdx.y;
  R t[4];
  load_row<R, 4>(rows + e * 4, t);
  R sn, cs;
  sincos_r<R>((R)ep.shift[k][0] * t[0] + (R)ep.shift[k][1] * t[1] + (R)ep.shift[k][2] * t[2], &sn, &cs);
  pdl_wait();
  out[(size_t)k * nent + e] = cmake<C>(cs, sn);
}
template <typename R>
cudaError_t launch_phase_table(cudaStream_t st, size_t nent, int nk, const R* rows, const EpiParams& ep, void* out) {
  if (nent == 0) return cudaSuccess;
  return launch_pdl(k_phase_table<R>, dim3((unsigned)((nent + 255) / 256), nk), 256, 0, st, nent, rows, ep,
                    (typename CT<R>::type*)out);
}

// Projector values of every entry (once, at creation).
template <typename R, int NLM>
__global__ void __launch_bounds__(256)
k_beta_table(size_t nent, const R* __restrict__ rows, const int* __restrict__ atom, ProjTables<R> pt, R* __restrict__ out) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= nent) return;
  int a = 0;
  if (atom) a = atom[e];
  else
    while (a + 1 < pt.natoms && (size_t)pt.g_ptr[a + 1] <= e) ++a;
  R t[4], nl[4], b[NLM];
  load_row<R, 4>(rows + e * 4, t);
  load_row<R, 4>(pt.nrm + (size_t)a * 4, nl);
  beta_values<R, NLM>(t[0], t[1], t[2], t[3], nl, pt.yc, b);
  R* o = out + e * beta_pitch(NLM);
#pragma unroll
  for (int p = 0; p < beta_pitch(NLM); ++p) o[p] = p < NLM ? b[p] : (R)0;
}
template <typename R>
cudaError_t launch_beta_table(cudaStream_t st, size_t nent, const R* rows, const int* atom, const ProjTables<R>& pt,
                              R* out) {
  if (nent == 0) return cudaSuccess;
  const unsigned grid = (unsigned)((nent + 255) / 256);
  switch (pt.nlm) {
    case 1: k_beta_table<R, 1><<<grid, 256, 0, st>>>(nent, rows, atom, pt, out); break;
    case 4: k_beta_table<R, 4><<<grid, 256, 0, st>>>(nent, rows, atom, pt, out); break;
    case 9: k_beta_table<R, 9><<<grid, 256, 0, st>>>(nent, rows, atom, pt, out); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// Sum of v[0..NV) over the lanes of a warp, NV values at once: each of the five steps exchanges
// half of the values a lane still holds, so it takes about NV additions where NV separate
// butterflies take 5 NV (FP64 additions are the bound of a small gather).  On return the lane
// holds the sums of the values lane_sum_index(j) in v[j]; indices out of range are negative.
__host__ __device__ constexpr int lane_sum_count(int nv) {
  for (int o = 0; o < 5; ++o) nv = (nv + 1) / 2;
  return nv;
}
template <int N, int O, typename R>
__device__ __forceinline__ void lane_sums(R* v, int lane) {
  constexpr int H = (N + 1) / 2;
  const bool up = (lane & O) != 0;
#pragma unroll
  for (int i = 0; i < H; ++i) {
    const R hi = (i + H < N) ? v[i + H] : (R)0;
    const R mine = up ? hi : v[i], other = up ? v[i] : hi;
    v[i] = mine + __shfl_xor_sync(0xffffffffu, other, O);
  }
  if constexpr (O > 1) lane_sums<H, O / 2>(v, lane);
}
// Index of the sum that slot j holds after lane_sums<N, O> (negative: none).
template <int N, int O>
__device__ __forceinline__ int lane_sum_index(int j, int lane) {
  constexpr int H = (N + 1) / 2;
  int pos = j;
  if constexpr (O > 1) pos = lane_sum_index<H, O / 2>(j, lane);
  if (pos < 0) return -1;
  if (lane & O) pos += H;
  return pos < N ? pos : -1;
}

// CTA (atom, chunk; spinor group): c[p][sigma] = sum_e beta_p exp(+i s.d) psi_sigma(r_e) dV over the
// chunk's entries, SPN spinors of one k-point per thread (they share the entry's tables); with
// several chunks the last CTA of the group to finish adds the partial sums in chunk order (the
// result does not depend on which one that is), then D c.
//
// Bound by the FP64 pipe in FP64 (44 instructions an entry and spinor with the phases and projector
// values read from tables, 181 when they were evaluated here) and by the latency of the entry ->
// psi loads in FP32; one CTA per (atom, spinor) left the chip idle for few of either (4 CTAs,
// 126 us, at 24^3 with one atom and four spinors).
constexpr int PG_NT = 128;
template <typename R> struct GatherMinBlocks { static constexpr int value = 3; };
template <> struct GatherMinBlocks<float> { static constexpr int value = 4; };

template <typename R, int NLM, int SPN>
__global__ void __launch_bounds__(PG_NT, GatherMinBlocks<R>::value)
k_proj_gather(const typename CT<R>::type* psi, size_t N3, ProjTables<R> pt, R dV, int nstates, int chunks, R* part,
              int* counters, typename CT<R>::type* c_out, typename CT<R>::type* dc_out) {
  using C = typename CT<R>::type;
  constexpr int NS = 4 * NLM;    // reals per spinor: (re, im) x (up, dn) x NLM
  constexpr int NV = SPN * NS;
  const int a = blockIdx.x / chunks, ch = blockIdx.x - a * chunks;
  const int kb = blockIdx.y * SPN;
  const int k = kb / nstates;
  const C* up = psi + (size_t)(2 * kb) * N3;
  const C* ph = reinterpret_cast<const C*>(pt.g_ph) + (size_t)k * pt.nent;
  R acc[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) acc[i] = (R)0;
  const int g0 = pt.g_ptr[a], ng = pt.g_ptr[a + 1] - g0;
  const int e0 = g0 + (int)((long long)ng * ch / chunks), e1 = g0 + (int)((long long)ng * (ch + 1) / chunks);
  // Software pipeline over this thread's entries e, e + PG_NT, ...: the grid index of the entry
  // after next, and the psi values and phase of the next entry, are requested before the current
  // entry is processed, so two dependent load chains are in flight at a time.
  const C zc = cmake<C>((R)0, (R)0);
  int e = e0 + threadIdx.x;
  int r1 = (e + PG_NT < e1) ? pt.g_idx[e + PG_NT] : 0;  // index of the next entry
  C pc = zc, w[2 * SPN];
#pragma unroll
  for (int j = 0; j < 2 * SPN; ++j) w[j] = zc;
  const int r0 = (e < e1) ? pt.g_idx[e] : 0;
  pdl_wait();
  if (e < e1) {
    pc = ph[e];
#pragma unroll
    for (int j = 0; j < 2 * SPN; ++j) w[j] = up[(size_t)j * N3 + r0];
  }
  for (; e < e1; e += PG_NT) {
    C pn = zc, wn[2 * SPN];
    int r2 = 0;
#pragma unroll
    for (int j = 0; j < 2 * SPN; ++j) wn[j] = zc;
    if (e + PG_NT < e1) {
      pn = ph[e + PG_NT];
#pragma unroll
      for (int j = 0; j < 2 * SPN; ++j) wn[j] = up[(size_t)j * N3 + r1];
      if (e + 2 * PG_NT < e1) r2 = pt.g_idx[e + 2 * PG_NT];
    }
    R bt[beta_pitch(NLM)];
    entry_beta<R, NLM>(e, a, pt.g_row, pt.g_beta, pt, bt);
#pragma unroll
    for (int s = 0; s < SPN; ++s) {
      const C u = cmul(w[2 * s], pc), d = cmul(w[2 * s + 1], pc);  // psi exp(+i arg)
#pragma unroll
      for (int p = 0; p < NLM; ++p) {
        acc[s * NS + 4 * p + 0] += bt[p] * u.x;
        acc[s * NS + 4 * p + 1] += bt[p] * u.y;
        acc[s * NS + 4 * p + 2] += bt[p] * d.x;
        acc[s * NS + 4 * p + 3] += bt[p] * d.y;
      }
    }
    pc = pn;
#pragma unroll
    for (int j = 0; j < 2 * SPN; ++j) w[j] = wn[j];
    r1 = r2;
  }
  __shared__ R red[PG_NT / 32][NV];
  __shared__ C cv[SPN * 2 * NLM];
  __shared__ int last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  lane_sums<NV, 16>(acc, lane);
#pragma unroll
  for (int j = 0; j < lane_sum_count(NV); ++j) {
    const int i = lane_sum_index<NV, 16>(j, lane);
    if (i >= 0) red[warp][i] = acc[j];
  }
  __syncthreads();
  const size_t grp = (size_t)blockIdx.y * pt.natoms + a;
  if (threadIdx.x < NV) {
    R s = red[0][threadIdx.x];
#pragma unroll
    for (int v = 1; v < PG_NT / 32; ++v) s += red[v][threadIdx.x];
    if (chunks == 1) red[0][threadIdx.x] = s;
    else part[(grp * chunks + ch) * NV + threadIdx.x] = s;
  }
  if (chunks > 1) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      last = atomicAdd(counters + grp, 1) == chunks - 1;
      if (last) counters[grp] = 0;  // for the next launch
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (threadIdx.x < NV) {
      R s = (R)0;
      for (int i = 0; i < chunks; ++i) s += __ldcg(part + (grp * chunks + i) * NV + threadIdx.x);
      red[0][threadIdx.x] = s;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < SPN * 2 * NLM; i += PG_NT) {
    const C c = cmake<C>(red[0][2 * i] * dV, red[0][2 * i + 1] * dV);
    cv[i] = c;
    const int s = i / (2 * NLM), q = i - s * 2 * NLM;
    c_out[((size_t)(kb + s) * pt.natoms + a) * 2 * NLM + q] = c;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < SPN * 2 * NLM; i += PG_NT) {
    const int s = i / (2 * NLM), q = i - s * 2 * NLM;
    const R* D = pt.Dmat + ((size_t)a * 2 * NLM + q) * 2 * NLM * 2;
    R re = 0, im = 0;
    for (int u = 0; u < 2 * NLM; ++u) {
      const R dr = D[2 * u], di = D[2 * u + 1];
      const C c = cv[s * 2 * NLM + u];
      re += dr * c.x - di * c.y;
      im += dr * c.y + di * c.x;
    }
    dc_out[((size_t)(kb + s) * pt.natoms + a) * 2 * NLM + q] = cmake<C>(re, im);
  }
}

// Spinors per thread: two in FP32 where a k-point's states pair up, else one (FP64: registers).
static int gather_spn(size_t rsize, int nstates) { return rsize == 4 && nstates % 2 == 0 ? 2 : 1; }

// Enough CTAs for four per SM (608 on this chip) of at least 256 entries each (two per thread); the
// FP32 gather, whose CTAs wait for memory, goes on to four times as many of at least 2048 entries,
// because the last, partly filled wave costs as much as a full one (64^3 x 104 spinors: 676 CTAs of
// one chunk 107 us, 2704 of four 80 us; at 32^3 with 14 spinors chunks of 256 take 13.5 us with
// 630 CTAs and 18.6 us with 1974).  The FP64 pipe stays busy with fewer.
int proj_chunks(int natoms, int ngroups, size_t nent, size_t rsize) {
  const long long have = (long long)natoms * ngroups;
  if (have <= 0) return 1;
  const long long per_atom = (long long)(nent / (size_t)natoms);
  const long long fill = std::min((608 + have - 1) / have, per_atom / 256);
  const long long waves = rsize == 4 ? std::min((2432 + have - 1) / have, per_atom / 2048) : 1;
  return (int)std::max(1LL, std::min(64LL, std::max(fill, waves)));
}
size_t proj_gather_part_bytes(int natoms, int nlm, int nk, int nstates, size_t nent, size_t rsize) {
  const int spn = gather_spn(rsize, nstates), groups = nk * nstates / spn;
  return (size_t)groups * natoms * proj_chunks(natoms, groups, nent, rsize) * spn * 4 * nlm * rsize;
}
size_t proj_gather_counters(int natoms, int nk, int nstates) { return (size_t)natoms * nk * nstates; }

template <typename R>
cudaError_t launch_proj_gather(cudaStream_t st, int N, const void* psi, int nkb, const ProjTables<R>& pt,
                               double dV, const EpiParams& ep, void* part, int* counters, void* c_out, void* dc_out) {
  using C = typename CT<R>::type;
  if (pt.natoms == 0) return cudaSuccess;
  const int spn = gather_spn(sizeof(R), ep.nstates), groups = nkb / spn;
  const int chunks = proj_chunks(pt.natoms, groups, pt.nent, sizeof(R));
  dim3 grid(pt.natoms * chunks, groups);
  const size_t N3 = (size_t)N * N * N;
#define PG_ARGS (const C*)psi, N3, pt, (R)dV, ep.nstates, chunks, (R*)part, counters, (C*)c_out, (C*)dc_out
#define PG_CASE(NLM)                                                                         \
  if constexpr (sizeof(R) == 4) {                                                            \
    if (spn == 2) return launch_pdl(k_proj_gather<R, NLM, 2>, grid, PG_NT, 0, st, PG_ARGS);  \
  }                                                                                          \
  return launch_pdl(k_proj_gather<R, NLM, 1>, grid, PG_NT, 0, st, PG_ARGS)
  switch (pt.nlm) {
    case 1: PG_CASE(1);
    case 4: PG_CASE(4);
    case 9: PG_CASE(9);
    default: return cudaErrorInvalidValue;
  }
#undef PG_CASE
#undef PG_ARGS
}


// ============================================================================ density

// Band group g = blockIdx.y sums bands [kb0, kb1) for two neighbouring points per thread and
// writes its partial 4-vector; with one group it writes rho directly.  The groups are then
// added in a fixed order (deterministic result).
template <typename R>
__global__ void __launch_bounds__(256)
k_density(const typename CT<R>::type* psi, size_t N3, int nkb, int ngroups, const double* __restrict__ wf, double* out) {
  const size_t r = 2 * ((size_t)blockIdx.x * blockDim.x + threadIdx.x);
  if (r >= N3) return;
  const int g = blockIdx.y;
  const int kb0 = (int)(((long long)nkb * g) / ngroups), kb1 = (int)(((long long)nkb * (g + 1)) / ngroups);
  double s[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};
  pdl_wait();
  // FP32 spinors: bilinears of up to 8 bands are summed in FP32 (the inputs' own precision) and
  // each such partial sum is added to the FP64 accumulators; FP64 spinors: FP64 throughout
  constexpr int CH = sizeof(R) == 4 ? 8 : 1;
  for (int kc = kb0; kc < kb1; kc += CH) {
    R p[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};
    const int kend = min(kb1, kc + CH);
#pragma unroll 1
    for (int kb = kc; kb < kend; ++kb) {
      const Pair<typename CT<R>::type> u = ld2(psi + (size_t)(2 * kb) * N3 + r);
      const Pair<typename CT<R>::type> d = ld2(psi + (size_t)(2 * kb + 1) * N3 + r);
      const R w = (R)wf[kb];
      const R ux[2] = {u.a.x, u.b.x}, uy[2] = {u.a.y, u.b.y};
      const R dx[2] = {d.a.x, d.b.x}, dy[2] = {d.a.y, d.b.y};
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        p[j][0] += w * (ux[j] * ux[j] + uy[j] * uy[j]);
        p[j][1] += w * (dx[j] * dx[j] + dy[j] * dy[j]);
        p[j][2] += w * (ux[j] * dx[j] + uy[j] * dy[j]);  // Re(u conj d)
        p[j][3] += w * (uy[j] * dx[j] - ux[j] * dy[j]);  // Im(u conj d)
      }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int c = 0; c < 4; ++c) s[j][c] += (double)p[j][c];
  }
  double* o = out + (size_t)g * 4 * N3;
#pragma unroll
  for (int c = 0; c < 4; ++c) *reinterpret_cast<double2*>(o + c * N3 + r) = make_double2(s[0][c], s[1][c]);
}

__global__ void k_density_reduce(size_t n, int ngroups, const double* part, double* rho) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  pdl_wait();
  double t = 0.0;
  for (int g = 0; g < ngroups; ++g) t += part[(size_t)g * n + i];
  rho[i] = t;
}

int density_groups(size_t N3, int nkb) {
  // enough resident threads to hide the load latency: about 6e5 threads
  const size_t per = N3 / 2;
  int g = (int)((600000 + per - 1) / per);
  if (g > nkb) g = nkb;
  if (g > 16) g = 16;
  return g < 1 ? 1 : g;
}

template <typename R>
cudaError_t launch_density(cudaStream_t st, size_t N3, const void* psi, int nkb, const double* wf, double* rho,
                           double* part) {
  const int G = part ? density_groups(N3, nkb) : 1;
  const size_t nthreads = N3 / 2;
  dim3 grid((unsigned)((nthreads + 255) / 256), G);
  cudaError_t e = launch_pdl(k_density<R>, grid, 256, 0, st, (const typename CT<R>::type*)psi, N3, nkb, G, wf,
                             G == 1 ? rho : part);
  if (e != cudaSuccess || G == 1) return e;
  return launch_pdl(k_density_reduce, dim3((unsigned)((4 * N3 + 255) / 256)), 256, 0, st, 4 * N3, G, part, rho);
}

// ============================================================================ XC and potential

// PW92 interpolation G(rs) and dG/drs for one parameter row (A, a1, b1, b2, b3, b4), p = 1;
// sr = sqrt(rs) and isr = 1 / sr are shared by the three rows.
__device__ __forceinline__ void pw92_g(double rs, double sr, double isr, double A, double a1, double b1, double b2,
                                       double b3, double b4, double* g, double* dg) {
  const double q0 = -2.0 * A * (1.0 + a1 * rs);
  const double q1 = 2.0 * A * sr * (b1 + sr * (b2 + sr * (b3 + sr * b4)));
  const double q1p = A * (b1 * isr + 2.0 * b2 + 3.0 * b3 * sr + 4.0 * b4 * rs);
  const double r = 1.0 / (q1 * (q1 + 1.0));  // one division: 1 / q1 = (q1 + 1) r
  const double lg = log1p((q1 + 1.0) * r);
  *g = q0 * lg;
  *dg = -2.0 * A * a1 * lg - q0 * q1p * r;
}

// Slater exchange with spin scaling plus PW92 correlation on (nu, nd): energy density, v_up, v_dn.
// Three cube roots per point: with c = n^(1/3), rs = (3 / 4 pi)^(1/3) / c and
// (1 +- zeta)^(1/3) = 2^(1/3) n_up,dn^(1/3) / c (nu, nd >= 0, so |zeta| <= 1).
__device__ void lsda_point(double nu, double nd, double* e, double* vu, double* vd) {
  const double c6 = 1.240700981798800033;    // (6 / pi)^(1/3)
  const double crs = 0.6203504908994000167;  // (3 / (4 pi))^(1/3)
  const double c2 = 1.259921049894873165;    // 2^(1/3)
  const double fden = 1.923661050931536320;  // 1 / (2^(4/3) - 2)
  const double cbu = cbrt(nu), cbd = cbrt(nd);
  const double ex = -0.75 * c6 * (nu * cbu + nd * cbd);
  const double vxu = -c6 * cbu, vxd = -c6 * cbd;
  const double n = nu + nd;
  const double icn = 1.0 / cbrt(n);
  const double rs = crs * icn;
  double z = (nu - nd) / n;
  z = fmin(1.0, fmax(-1.0, z));
  const double sr = sqrt(rs), isr = 1.0 / sr;
  double ec0, d0, ec1, d1, mac, dmac;
  pw92_g(rs, sr, isr, 0.031091, 0.21370, 7.5957, 3.5876, 1.6382, 0.49294, &ec0, &d0);
  pw92_g(rs, sr, isr, 0.015545, 0.20548, 14.1189, 6.1977, 3.3662, 0.62517, &ec1, &d1);
  pw92_g(rs, sr, isr, 0.016887, 0.11125, 10.357, 3.6231, 0.88026, 0.49671, &mac, &dmac);
  const double ac = -mac, dac = -dmac;
  const double opz = 1.0 + z, omz = 1.0 - z;
  const double cpz = c2 * cbu * icn, cmz = c2 * cbd * icn;
  const double f = (opz * cpz + omz * cmz - 2.0) * fden;
  const double fp = (4.0 / 3.0) * (cpz - cmz) * fden;
  const double fpp0 = 1.709921;
  const double z3 = z * z * z, z4 = z3 * z;
  const double ec = ec0 + ac * f * (1.0 - z4) / fpp0 + (ec1 - ec0) * f * z4;
  const double drs = d0 + dac * f * (1.0 - z4) / fpp0 + (d1 - d0) * f * z4;
  const double dz = ac / fpp0 * (fp * (1.0 - z4) - 4.0 * z3 * f) + (ec1 - ec0) * (fp * z4 + 4.0 * z3 * f);
  const double common = ec - rs / 3.0 * drs;
  *e = ex + n * ec;
  *vu = vxu + common - (z - 1.0) * dz;
  *vd = vxd + common - (z + 1.0) * dz;
}

// Bound by the FP64 pipe (some 600 instructions a point); small CTAs spread a small grid over the
// SMs (24^3: 30 us on 54 CTAs of 256).
constexpr int kPotThreads = 64;
__global__ void __launch_bounds__(kPotThreads) k_potential(size_t N3, const double* rho, const double* vH, const double* __restrict__ vloc, double Bx, double By,
                            double Bz, int xc, int mode, double* V, float* Vf, double* exc, double* vxc4) {
  const size_t r = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= N3) return;
  pdl_wait();
  const double r0 = rho[r], r1 = rho[N3 + r], r2 = rho[2 * N3 + r], r3 = rho[3 * N3 + r];
  const double n = r0 + r1, mx = 2.0 * r2, my = -2.0 * r3, mz = r0 - r1;
  double e = 0.0, vbar = 0.0, bx = 0.0, by = 0.0, bz = 0.0;
  if (xc && n >= 1e-14 && mode == TDDFT_SPIN_COLLINEAR) {
    // Eq. HSDFT: LSDA on the channel densities, field along the quantisation axis
    double vu, vd;
    lsda_point(r0, r1, &e, &vu, &vd);
    vbar = 0.5 * (vu + vd);
    bz = 0.5 * (vu - vd);
  } else if (xc && n >= 1e-14 && mode == TDDFT_SPIN_UNPOLARISED) {
    double vu, vd;
    lsda_point(0.5 * n, 0.5 * n, &e, &vu, &vd);
    vbar = vu;
  } else if (xc && n >= 1e-14) {
    const double mag = sqrt(mx * mx + my * my + mz * mz);
    const double s = fmin(mag, n);
    double vu, vd;
    lsda_point(0.5 * (n + s), 0.5 * (n - s), &e, &vu, &vd);
    vbar = 0.5 * (vu + vd);
    if (mag > 1e-14) {
      const double bm = 0.5 * (vu - vd) / mag;
      bx = bm * mx; by = bm * my; bz = bm * mz;
    }
  }
  const double v = vloc[r] + vH[r] + vbar;
  const double tx = bx + 0.5 * Bx, ty = by + 0.5 * By, tz = bz + 0.5 * Bz;  // mu_B = 1/2
  const double V0 = v + tz, V1 = v - tz, V2 = 2.0 * tx, V3 = -2.0 * ty;
  V[r] = V0; V[N3 + r] = V1; V[2 * N3 + r] = V2; V[3 * N3 + r] = V3;
  if (Vf) {
    Vf[r] = (float)V0; Vf[N3 + r] = (float)V1; Vf[2 * N3 + r] = (float)V2; Vf[3 * N3 + r] = (float)V3;
  }
  exc[r] = e;
  vxc4[r] = vbar + bz; vxc4[N3 + r] = vbar - bz; vxc4[2 * N3 + r] = 2.0 * bx; vxc4[3 * N3 + r] = -2.0 * by;
}

cudaError_t launch_potential(cudaStream_t st, size_t N3, const double* rho, const double* vH, const double* vloc,
                             const double* B, int xc, int mode, double* V, float* Vf, double* exc, double* vxc4) {
  return launch_pdl(k_potential, dim3((unsigned)((N3 + kPotThreads - 1) / kPotThreads)), kPotThreads, 0, st, N3, rho, vH, vloc, B[0], B[1], B[2],
                    xc, mode, V, Vf, exc, vxc4);
}

__global__ void k_complex_real_part(size_t n, const double2* in, double* out, double scale) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = in[i].x * scale;
}
cudaError_t launch_complex_real_part(cudaStream_t st, size_t N3, const double2* in, double* out, double scale) {
  k_complex_real_part<<<(unsigned)((N3 + 255) / 256), 256, 0, st>>>(N3, in, out, scale);
  return cudaGetLastError();
}

// V_loc(G) = sum_a [-4 pi Z / G^2 exp(-G^2 rc^2 / 4) exp(-i G.R_a)] / Omega, G = 0: sum_a pi Z rc^2 / Omega.
template <int N>
__global__ void k_vloc_G(double gx0, double gy0, double gz0, int natoms, const double* __restrict__ pos,
                         const double* __restrict__ Zr, double omega, double2* __restrict__ out) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t N3 = (size_t)N * N * N;
  if (i >= N3) return;
  const int x = (int)(i % N), y = (int)((i / N) % N), z = (int)(i / ((size_t)N * N));
  const double gx = gx0 * freq<N>(kx_at<N>(x)), gy = gy0 * freq<N>(y), gz = gz0 * freq<N>(z);  // order of the xy pass
  const double g2 = gx * gx + gy * gy + gz * gz;
  const double kPi = 3.14159265358979323846;
  double re = 0.0, im = 0.0;
  for (int a = 0; a < natoms; ++a) {
    const double Z = Zr[2 * a], rc = Zr[2 * a + 1];
    const double t = g2 > 0.0 ? -4.0 * kPi * Z / g2 * exp(-g2 * rc * rc * 0.25) : kPi * Z * rc * rc;
    double sn, cs;
    sincos(gx * pos[3 * a] + gy * pos[3 * a + 1] + gz * pos[3 * a + 2], &sn, &cs);
    re += t * cs;
    im -= t * sn;
  }
  out[i] = make_double2(re / omega, im / omega);
}
template <int N>
static cudaError_t vloc_G_n(cudaStream_t st, const double* L, int natoms, const double* pos, const double* Zr,
                            double omega, double2* out) {
  const double kPi = 3.14159265358979323846;
  k_vloc_G<N><<<(unsigned)(((size_t)N * N * N + 255) / 256), 256, 0, st>>>(2 * kPi / L[0], 2 * kPi / L[1], 2 * kPi / L[2],
                                                                           natoms, pos, Zr, omega, out);
  return cudaGetLastError();
}
cudaError_t launch_vloc_G(cudaStream_t st, int N, const double* L, int natoms, const double* pos, const double* Zr,
                          double omega, double2* out) {
  TDDFT_DISPATCH_N(N, (vloc_G_n<NN>(st, L, natoms, pos, Zr, omega, out)));
}

// ============================================================================ conversions

// Precision conversion of spinor arrays.  The source or destination may be page-locked host
// memory read or written through its mapped address (over the CPU-GPU link), where the rate
// depends on the requests in flight: each warp moves 8 x 32 consecutive elements, eight
// independent 16-byte loads per thread, every load instruction covering 512 contiguous bytes.
constexpr int kConvPerThread = 8;

template <typename R>
__global__ void __launch_bounds__(256) k_convert_in(size_t n, const double2* __restrict__ in, typename CT<R>::type* __restrict__ out) {
  using C = typename CT<R>::type;
  const size_t base = (((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (32 * kConvPerThread) + (threadIdx.x & 31);
  double2 v[kConvPerThread];
#pragma unroll
  for (int q = 0; q < kConvPerThread; ++q) {
    const size_t i = base + 32 * q;
    if (i < n) v[q] = in[i];
  }
#pragma unroll
  for (int q = 0; q < kConvPerThread; ++q) {
    const size_t i = base + 32 * q;
    if (i < n) out[i] = cmake<C>((R)v[q].x, (R)v[q].y);
  }
}
template <typename R>
__global__ void __launch_bounds__(256) k_convert_out(size_t n, const typename CT<R>::type* __restrict__ in, double2* __restrict__ out) {
  using C = typename CT<R>::type;
  const size_t base = (((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * (32 * kConvPerThread) + (threadIdx.x & 31);
  C v[kConvPerThread];
#pragma unroll
  for (int q = 0; q < kConvPerThread; ++q) {
    const size_t i = base + 32 * q;
    if (i < n) v[q] = in[i];
  }
#pragma unroll
  for (int q = 0; q < kConvPerThread; ++q) {
    const size_t i = base + 32 * q;
    if (i < n) out[i] = make_double2((double)v[q].x, (double)v[q].y);
  }
}
template <typename R>
cudaError_t launch_convert_in(cudaStream_t st, size_t n, const double2* in, void* out) {
  if (n == 0) return cudaSuccess;
  const size_t per_cta = 256 * kConvPerThread;
  k_convert_in<R><<<(unsigned)((n + per_cta - 1) / per_cta), 256, 0, st>>>(n, in, (typename CT<R>::type*)out);
  return cudaGetLastError();
}
template <typename R>
cudaError_t launch_convert_out(cudaStream_t st, size_t n, const void* in, double2* out) {
  if (n == 0) return cudaSuccess;
  const size_t per_cta = 256 * kConvPerThread;
  k_convert_out<R><<<(unsigned)((n + per_cta - 1) / per_cta), 256, 0, st>>>(n, (const typename CT<R>::type*)in, out);
  return cudaGetLastError();
}

// ============================================================================ reductions (fixed order)

template <int NT>
__device__ double block_sum(double v, double* sh) {
  v = warp_sum(v);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) sh[warp] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < NT / 32; ++w) t += sh[w];
  return t;  // valid in thread 0
}

// out[i] = sum over parts of part[parts][nval]: one warp per value, lanes stride over the parts (a
// single thread per value waits for one load after the other: 50 us for 304 parts).
__global__ void k_parts_total(int nparts, int nval, const double* __restrict__ part, double* __restrict__ out) {
  const int i = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (i >= nval) return;
  double s = 0.0;
  for (int b = lane; b < nparts; b += 32) s += part[(size_t)b * nval + i];
  s = warp_sum(s);
  if (lane == 0) out[i] = s;
}

// out2[band] = sum over npts of conj(a) b (complex, double accumulation) in two passes: CTA
// (chunk, band) sums a fixed range of points, then one warp per band adds the chunks in a fixed
// order (deterministic, and every SM busy).
constexpr int kDotChunks = 64;
template <typename R>
__global__ void __launch_bounds__(256) k_band_dot_part(size_t npts, const typename CT<R>::type* __restrict__ a,
                                                       const typename CT<R>::type* __restrict__ b, double* part) {
  __shared__ double sh[8];
  const size_t off = (size_t)blockIdx.y * npts;
  const size_t len = (npts + kDotChunks - 1) / kDotChunks;
  const size_t lo = (size_t)blockIdx.x * len, hi = lo + len < npts ? lo + len : npts;
  // groups of kDotGroup products are summed in R before entering the FP64 sum (FP64 arithmetic
  // is scarce on this part; in FP64 mode R is double and nothing changes)
  constexpr int kDotGroup = 8;
  double re = 0.0, im = 0.0;
  for (size_t i0 = lo + threadIdx.x; i0 < hi; i0 += (size_t)256 * kDotGroup) {
    R gr = (R)0, gi = (R)0;
#pragma unroll
    for (int j = 0; j < kDotGroup; ++j) {
      const size_t i = i0 + (size_t)j * 256;
      if (i < hi) {
        const auto x = a[off + i], y = b[off + i];
        gr += x.x * y.x + x.y * y.y;
        gi += x.x * y.y - x.y * y.x;
      }
    }
    re += (double)gr;
    im += (double)gi;
  }
  const double tr = block_sum<256>(re, sh);
  const double ti = block_sum<256>(im, sh);
  if (threadIdx.x == 0) {
    const size_t o = ((size_t)blockIdx.y * kDotChunks + blockIdx.x) * 2;
    part[o] = tr;
    part[o + 1] = ti;
  }
}
__global__ void k_band_dot_sum(int nbands, const double* __restrict__ part, double* out2) {
  const int band = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (band >= nbands) return;
  double re = 0.0, im = 0.0;
  for (int ch = lane; ch < kDotChunks; ch += 32) {
    re += part[((size_t)band * kDotChunks + ch) * 2];
    im += part[((size_t)band * kDotChunks + ch) * 2 + 1];
  }
  re = warp_sum(re);
  im = warp_sum(im);
  if (lane == 0) {
    out2[2 * band] = re;
    out2[2 * band + 1] = im;
  }
}
template <typename R>
cudaError_t launch_band_dot(cudaStream_t st, size_t npts, int nbands, const void* a, const void* b, double* out2,
                            double* part) {
  using C = typename CT<R>::type;
  k_band_dot_part<R><<<dim3(kDotChunks, nbands), 256, 0, st>>>(npts, (const C*)a, (const C*)b, part);
  k_band_dot_sum<<<(nbands + 3) / 4, 128, 0, st>>>(nbands, part, out2);
  return cudaGetLastError();
}
size_t band_dot_part_doubles(int nbands) { return (size_t)nbands * kDotChunks * 2; }

// out[kb] = Re sum conj(c) dc over atoms, projectors and spins.
template <typename R>
__global__ void k_nl_energy(int ncoef, const typename CT<R>::type* __restrict__ c,
                            const typename CT<R>::type* __restrict__ dc, double* out) {
  __shared__ double sh[8];
  const size_t off = (size_t)blockIdx.x * ncoef;
  double s = 0.0;
  for (int i = threadIdx.x; i < ncoef; i += 256) s += (double)c[off + i].x * dc[off + i].x + (double)c[off + i].y * dc[off + i].y;
  const double t = block_sum<256>(s, sh);
  if (threadIdx.x == 0) out[blockIdx.x] = t;
}
template <typename R>
cudaError_t launch_nl_energy(cudaStream_t st, int nkb, int ncoef, const void* c, const void* dc, double* out) {
  using C = typename CT<R>::type;
  k_nl_energy<R><<<nkb, 256, 0, st>>>(ncoef, (const C*)c, (const C*)dc, out);
  return cudaGetLastError();
}

// Spin-orbit torque of one spinor (block kb): sum over atoms and components i of
// Re c^dagger T^i c, the rows (atom, i, r) spread over the threads, fixed-order block sums.
template <typename R>
__global__ void __launch_bounds__(256)
k_soc_torque(int natoms, int M, const typename CT<R>::type* __restrict__ c, const double2* __restrict__ T,
             double* out) {
  __shared__ double sh[8];
  const typename CT<R>::type* ck = c + (size_t)blockIdx.x * natoms * M;
  double acc[3] = {0.0, 0.0, 0.0};
  const int rows = natoms * M;
  for (int i = 0; i < 3; ++i) {
    for (int t = threadIdx.x; t < rows; t += 256) {
      const int a = t / M, r = t - a * M;
      const double2* Tr = T + (((size_t)a * 3 + i) * M + r) * M;
      const typename CT<R>::type* ca = ck + (size_t)a * M;
      double re = 0.0, im = 0.0;  // (T c)_r
      for (int q = 0; q < M; ++q) {
        const double cr = (double)ca[q].x, ci = (double)ca[q].y;
        re += Tr[q].x * cr - Tr[q].y * ci;
        im += Tr[q].x * ci + Tr[q].y * cr;
      }
      acc[i] += (double)ca[r].x * re + (double)ca[r].y * im;  // Re conj(c_r) (T c)_r
    }
  }
  for (int i = 0; i < 3; ++i) {
    const double v = block_sum<256>(acc[i], sh);
    if (threadIdx.x == 0) out[(size_t)blockIdx.x * 3 + i] = v;
  }
}
template <typename R>
cudaError_t launch_soc_torque(cudaStream_t st, int nkb, int natoms, int M, const void* c, const double2* T,
                              double* out) {
  k_soc_torque<R><<<nkb, 256, 0, st>>>(natoms, M, (const typename CT<R>::type*)c, T, out);
  return cudaGetLastError();
}

// Field integrals (without dV): [0] v_loc n, [1] v_H n, [2] e_xc, [3..5] m, [6] n, [7] B.m,
// [8] <rho_v, V_v^xc>, [9] count of non-finite rho values.  Two passes: each of kFieldBlocks
// CTAs sums a fixed range of points, then one CTA adds the block partials in a fixed order.
constexpr int kFieldBlocks = 304;
__global__ void __launch_bounds__(256)
k_field_sums_part(size_t N3, const double* __restrict__ rho, const double* __restrict__ vloc, const double* __restrict__ vH,
                  const double* __restrict__ exc, const double* __restrict__ vxc4, double Bx, double By, double Bz,
                  double* part) {
  __shared__ double sh[8];
  double acc[10];
  for (int i = 0; i < 10; ++i) acc[i] = 0.0;
  const size_t len = (N3 + kFieldBlocks - 1) / kFieldBlocks;
  const size_t lo = (size_t)blockIdx.x * len, hi = lo + len < N3 ? lo + len : N3;
  for (size_t r = lo + threadIdx.x; r < hi; r += 256) {
    const double r0 = rho[r], r1 = rho[N3 + r], r2 = rho[2 * N3 + r], r3 = rho[3 * N3 + r];
    const double n = r0 + r1, mx = 2.0 * r2, my = -2.0 * r3, mz = r0 - r1;
    acc[0] += vloc[r] * n;
    acc[1] += vH[r] * n;
    acc[2] += exc[r];
    acc[3] += mx; acc[4] += my; acc[5] += mz;
    acc[6] += n;
    acc[7] += Bx * mx + By * my + Bz * mz;
    acc[8] += r0 * vxc4[r] + r1 * vxc4[N3 + r] + r2 * vxc4[2 * N3 + r] + r3 * vxc4[3 * N3 + r];
    acc[9] += (isfinite(r0) && isfinite(r1) && isfinite(r2) && isfinite(r3)) ? 0.0 : 1.0;
  }
  for (int i = 0; i < 10; ++i) {
    const double t = block_sum<256>(acc[i], sh);
    if (threadIdx.x == 0) part[(size_t)blockIdx.x * 10 + i] = t;
  }
}
cudaError_t launch_field_sums(cudaStream_t st, size_t N3, const double* rho, const double* vloc, const double* vH,
                              const double* exc, const double* vxc4, const double* /*V*/, const double* B, double* out,
                              double* part) {
  k_field_sums_part<<<kFieldBlocks, 256, 0, st>>>(N3, rho, vloc, vH, exc, vxc4, B[0], B[1], B[2], part);
  k_parts_total<<<1, 320, 0, st>>>(kFieldBlocks, 10, part, out);
  return cudaGetLastError();
}
size_t field_sums_part_doubles() { return (size_t)kFieldBlocks * 10; }

// int b_xc x m and int m (without dV) from rho_v and the XC 4-vector [vbar + b_z, vbar - b_z,
// 2 b_x, -2 b_y], in the two passes of the field sums.  (One CTA over all points took most of a
// report's reductions: 1.1 ms at 64^3.)
__global__ void __launch_bounds__(256)
k_xc_torque_part(size_t N3, const double* __restrict__ rho, const double* __restrict__ vxc4, double* part) {
  __shared__ double sh[8];
  double acc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  const size_t len = (N3 + kFieldBlocks - 1) / kFieldBlocks;
  const size_t lo = (size_t)blockIdx.x * len, hi = lo + len < N3 ? lo + len : N3;
  for (size_t r = lo + threadIdx.x; r < hi; r += 256) {
    const double r0 = rho[r], r1 = rho[N3 + r], r2 = rho[2 * N3 + r], r3 = rho[3 * N3 + r];
    const double mx = 2.0 * r2, my = -2.0 * r3, mz = r0 - r1;
    const double bz = 0.5 * (vxc4[r] - vxc4[N3 + r]), bx = 0.5 * vxc4[2 * N3 + r], by = -0.5 * vxc4[3 * N3 + r];
    acc[0] += by * mz - bz * my;
    acc[1] += bz * mx - bx * mz;
    acc[2] += bx * my - by * mx;
    acc[3] += mx; acc[4] += my; acc[5] += mz;
  }
  for (int i = 0; i < 6; ++i) {
    const double t = block_sum<256>(acc[i], sh);
    if (threadIdx.x == 0) part[(size_t)blockIdx.x * 6 + i] = t;
  }
}
cudaError_t launch_xc_torque(cudaStream_t st, size_t N3, const double* rho, const double* vxc4, double* out6,
                             double* part) {
  k_xc_torque_part<<<kFieldBlocks, 256, 0, st>>>(N3, rho, vxc4, part);
  k_parts_total<<<1, 192, 0, st>>>(kFieldBlocks, 6, part, out6);
  return cudaGetLastError();
}

// Sums of the three N3-fields of g, the same two passes.
__global__ void __launch_bounds__(256) k_sum3_part(size_t N3, const double* __restrict__ g, double* part) {
  __shared__ double sh[8];
  const size_t len = (N3 + kFieldBlocks - 1) / kFieldBlocks;
  const size_t lo = (size_t)blockIdx.x * len, hi = lo + len < N3 ? lo + len : N3;
  double acc[3] = {0.0, 0.0, 0.0};
  for (size_t r = lo + threadIdx.x; r < hi; r += 256)
    for (int a = 0; a < 3; ++a) acc[a] += g[a * N3 + r];
  for (int a = 0; a < 3; ++a) {
    const double t = block_sum<256>(acc[a], sh);
    if (threadIdx.x == 0) part[(size_t)blockIdx.x * 3 + a] = t;
  }
}
cudaError_t launch_sum3(cudaStream_t st, size_t N3, const double* g, double* out, double* part) {
  k_sum3_part<<<kFieldBlocks, 256, 0, st>>>(N3, g, part);
  k_parts_total<<<1, 96, 0, st>>>(kFieldBlocks, 3, part, out);
  return cudaGetLastError();
}

__global__ void __launch_bounds__(256) k_max_abs_diff(size_t n, const double* a, const double* b, double* part) {
  __shared__ double sh[8];
  double m = 0.0;
  for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (size_t)gridDim.x * 256)
    m = fmax(m, fabs(a[i] - b[i]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t = fmax(t, sh[w]);
    part[blockIdx.x] = t;
  }
}
__global__ void k_max_total(int nparts, const double* __restrict__ part, double* out) {
  double m = 0.0;
  for (int i = threadIdx.x; i < nparts; i += 32) m = fmax(m, part[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
  if (threadIdx.x == 0) *out = m;
}
cudaError_t launch_max_abs_diff(cudaStream_t st, size_t n, const double* a, const double* b, double* out, double* part) {
  k_max_abs_diff<<<kFieldBlocks, 256, 0, st>>>(n, a, b, part);
  k_max_total<<<1, 32, 0, st>>>(kFieldBlocks, part, out);
  return cudaGetLastError();
}

// Sets *flag when the local potential leaves [lo, hi] given the kinetic maximum and projector bound.
__global__ void k_check_window(size_t N3, const double* V, double lo, double hi, double kin_max, double nl_bound,
                               int* flag) {
  const size_t r = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= N3) return;
  pdl_wait();
  const double v = 0.5 * (V[r] + V[N3 + r]);
  const double bz = 0.5 * (V[r] - V[N3 + r]), bx = 0.5 * V[2 * N3 + r], by = 0.5 * V[3 * N3 + r];
  const double b = sqrt(bx * bx + by * by + bz * bz);
  const bool bad = !(v - b - nl_bound >= lo) || !(v + b + nl_bound + kin_max <= hi);
  if (bad) atomicOr(flag, 1);
}
cudaError_t launch_check_window(cudaStream_t st, size_t N3, const double* V, double lo, double hi, double kin_max,
                                double nl_bound, int* flag) {
  return launch_pdl(k_check_window, dim3((unsigned)((N3 + 255) / 256)), 256, 0, st, N3, V, lo, hi, kin_max, nl_bound, flag);
}

// n = rho_uu + rho_dd and m = (2 Re rho_ud, -2 Im rho_ud, rho_uu - rho_dd) from rho_v, into
// nm[0 .. N3) (n) and nm[N3 .. 4 N3) (m_x, m_y, m_z).
__global__ void k_nm_from_rho(size_t N3, const double* __restrict__ rho, double* __restrict__ nm) {
  const size_t r = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= N3) return;
  const double r0 = rho[r], r1 = rho[N3 + r], r2 = rho[2 * N3 + r], r3 = rho[3 * N3 + r];
  nm[r] = r0 + r1;
  nm[N3 + r] = 2.0 * r2;
  nm[2 * N3 + r] = -2.0 * r3;
  nm[3 * N3 + r] = r0 - r1;
}
cudaError_t launch_nm_from_rho(cudaStream_t st, size_t N3, const double* rho, double* nm) {
  k_nm_from_rho<<<(unsigned)((N3 + 255) / 256), 256, 0, st>>>(N3, rho, nm);
  return cudaGetLastError();
}

// Extrema of the local potential for the automatic spectral window: min and max of
// v = (V_0 + V_1)/2 and max of |b| = |(V_2, V_3, V_0 - V_1)|/2 over the grid.  Products and sums
// are rounded one by one (no fused multiply-add), as in a plain IEEE evaluation; min and max do
// not depend on the order, so the result is exact.  Partials per block, then one block.
__global__ void __launch_bounds__(256) k_window_part(size_t N3, const double* __restrict__ V, double* part) {
  __shared__ double sh[3][8];
  double vmin = 1e300, vmax = -1e300, bmax = 0.0;
  for (size_t r = (size_t)blockIdx.x * blockDim.x + threadIdx.x; r < N3; r += (size_t)gridDim.x * blockDim.x) {
    const double v = __dmul_rn(0.5, __dadd_rn(V[r], V[N3 + r]));
    const double bz = __dmul_rn(0.5, __dsub_rn(V[r], V[N3 + r]));
    const double bx = __dmul_rn(0.5, V[2 * N3 + r]), by = __dmul_rn(0.5, V[3 * N3 + r]);
    const double b = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(bx, bx), __dmul_rn(by, by)), __dmul_rn(bz, bz)));
    vmin = fmin(vmin, v);
    vmax = fmax(vmax, v);
    bmax = fmax(bmax, b);
  }
  for (int o = 16; o > 0; o >>= 1) {
    vmin = fmin(vmin, __shfl_xor_sync(0xffffffffu, vmin, o));
    vmax = fmax(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
    bmax = fmax(bmax, __shfl_xor_sync(0xffffffffu, bmax, o));
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) { sh[0][warp] = vmin; sh[1][warp] = vmax; sh[2][warp] = bmax; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) {
      vmin = fmin(vmin, sh[0][w]);
      vmax = fmax(vmax, sh[1][w]);
      bmax = fmax(bmax, sh[2][w]);
    }
    part[3 * blockIdx.x] = vmin;
    part[3 * blockIdx.x + 1] = vmax;
    part[3 * blockIdx.x + 2] = bmax;
  }
}
__global__ void k_window_total(int nparts, const double* __restrict__ part, double* out) {
  double vmin = 1e300, vmax = -1e300, bmax = 0.0;
  for (int i = threadIdx.x; i < nparts; i += 32) {
    vmin = fmin(vmin, part[3 * i]);
    vmax = fmax(vmax, part[3 * i + 1]);
    bmax = fmax(bmax, part[3 * i + 2]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    vmin = fmin(vmin, __shfl_down_sync(0xffffffffu, vmin, o));
    vmax = fmax(vmax, __shfl_down_sync(0xffffffffu, vmax, o));
    bmax = fmax(bmax, __shfl_down_sync(0xffffffffu, bmax, o));
  }
  if (threadIdx.x != 0) return;
  out[0] = vmin;
  out[1] = vmax;
  out[2] = bmax;
}
cudaError_t launch_window_extrema(cudaStream_t st, size_t N3, const double* V, double* part, double* out3) {
  k_window_part<<<kFieldBlocks, 256, 0, st>>>(N3, V, part);
  k_window_total<<<1, 32, 0, st>>>(kFieldBlocks, part, out3);
  return cudaGetLastError();
}

// ============================================================================ per-atom moments
// Nearest atom of every grid point (minimum image), Algorithm 1's NearestAtom rule; equal
// distances go to the lowest atom index.  Every operation is explicitly rounded (no fused
// multiply-add) so that ties resolve the same way as in a plain IEEE evaluation of
// d = x h - R, d -= L rint(d / L), |d|^2 = (dx^2 + dy^2) + dz^2.
__global__ void k_voronoi_owner(int N, double hx, double hy, double hz, double Lx, double Ly, double Lz, int natoms,
                                const double* __restrict__ pos, int* __restrict__ owner) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const size_t N3 = (size_t)N * N * N;
  if (i >= N3) return;
  const int x = (int)(i % N), y = (int)((i / N) % N), z = (int)(i / ((size_t)N * N));
  const double rx = __dmul_rn((double)x, hx), ry = __dmul_rn((double)y, hy), rz = __dmul_rn((double)z, hz);
  double best = 1e300;
  int own = 0;
  for (int a = 0; a < natoms; ++a) {
    double dx = __dsub_rn(rx, pos[3 * a]), dy = __dsub_rn(ry, pos[3 * a + 1]), dz = __dsub_rn(rz, pos[3 * a + 2]);
    dx = __dsub_rn(dx, __dmul_rn(Lx, rint(__ddiv_rn(dx, Lx))));
    dy = __dsub_rn(dy, __dmul_rn(Ly, rint(__ddiv_rn(dy, Ly))));
    dz = __dsub_rn(dz, __dmul_rn(Lz, rint(__ddiv_rn(dz, Lz))));
    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    if (d2 < best) {
      best = d2;
      own = a;
    }
  }
  owner[i] = own;
}
cudaError_t launch_voronoi_owner(cudaStream_t st, int N, const double* L, int natoms, const double* pos, int* owner) {
  const size_t N3 = (size_t)N * N * N;
  k_voronoi_owner<<<(unsigned)((N3 + 255) / 256), 256, 0, st>>>(N, L[0] / N, L[1] / N, L[2] / N, L[0], L[1], L[2],
                                                               natoms, pos, owner);
  return cudaGetLastError();
}

// out[a] = {sum m_x, sum m_y, sum m_z, sum n} over the points owned by atom a (fixed order; multiply
// by dV on the host): kAtomChunks CTAs per atom each scan a range of the grid's owners (one CTA per
// atom over the whole grid left the chip idle), then one warp per atom adds their sums.
constexpr int kAtomChunks = 32;
__global__ void __launch_bounds__(256) k_atom_sums(size_t N3, const double* __restrict__ rho,
                                                   const int* __restrict__ owner, double* __restrict__ part) {
  __shared__ double sh[8];
  const int a = blockIdx.x;
  const size_t len = (N3 + kAtomChunks - 1) / kAtomChunks;
  const size_t lo = (size_t)blockIdx.y * len, hi = lo + len < N3 ? lo + len : N3;
  double acc[4] = {0, 0, 0, 0};
  for (size_t r = lo + threadIdx.x; r < hi; r += 256) {
    if (owner[r] != a) continue;
    const double r0 = rho[r], r1 = rho[N3 + r], r2 = rho[2 * N3 + r], r3 = rho[3 * N3 + r];
    acc[0] += 2.0 * r2;
    acc[1] += -2.0 * r3;
    acc[2] += r0 - r1;
    acc[3] += r0 + r1;
  }
  for (int c = 0; c < 4; ++c) {
    const double t = block_sum<256>(acc[c], sh);
    if (threadIdx.x == 0) part[((size_t)a * kAtomChunks + blockIdx.y) * 4 + c] = t;
    __syncthreads();
  }
}
__global__ void k_atom_sums_total(int natoms, const double* __restrict__ part, double* __restrict__ out) {
  const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;  // (atom, value)
  if (i >= 4 * natoms) return;
  const double s = warp_sum(part[((size_t)(i >> 2) * kAtomChunks + lane) * 4 + (i & 3)]);
  if (lane == 0) out[i] = s;
}
size_t atom_sums_part_doubles(int natoms) { return (size_t)natoms * kAtomChunks * 4; }
cudaError_t launch_atom_sums(cudaStream_t st, size_t N3, int natoms, const double* rho, const int* owner, double* out,
                             double* part) {
  static_assert(kAtomChunks == 32, "one lane per chunk");
  k_atom_sums<<<dim3(natoms, kAtomChunks), 256, 0, st>>>(N3, rho, owner, part);
  k_atom_sums_total<<<natoms, 128, 0, st>>>(natoms, part, out);
  return cudaGetLastError();
}

// ============================================================================ instantiations
#define TDDFT_INST(R)                                                                                           \
  template cudaError_t launch_fft_xy<R>(cudaStream_t, int, const void*, void*, int, const void*, bool);                       \
  template cudaError_t launch_fft_z_kinetic<R>(cudaStream_t, int, void*, int, const void*, const void*,          \
                                               const ZParams&);                                                 \
  template int fft_z_energy_parts<R>(int);                                                                      \
  template cudaError_t launch_fft_z_energy<R>(cudaStream_t, int, const void*, int, const void*, const void*,       \
                                              const ZParams&, double*, double*);                                \
  template cudaError_t launch_kin_tables<R>(cudaStream_t, int, int, const ZParams&, void*);                      \
  template cudaError_t launch_phase_table<R>(cudaStream_t, size_t, int, const R*, const EpiParams&, void*);      \
  template cudaError_t launch_beta_table<R>(cudaStream_t, size_t, const R*, const int*, const ProjTables<R>&,    \
                                            R*);                                                                \
  template cudaError_t launch_proj_gather<R>(cudaStream_t, int, const void*, int, const ProjTables<R>&, double,  \
                                             const EpiParams&, void*, int*, void*, void*);                      \
  template cudaError_t launch_density<R>(cudaStream_t, size_t, const void*, int, const double*, double*,         \
                                         double*);                                                                \
  template cudaError_t launch_convert_in<R>(cudaStream_t, size_t, const double2*, void*);                        \
  template cudaError_t launch_convert_out<R>(cudaStream_t, size_t, const void*, double2*);                       \
  template cudaError_t launch_band_dot<R>(cudaStream_t, size_t, int, const void*, const void*, double*, double*); \
  template cudaError_t launch_nl_energy<R>(cudaStream_t, int, int, const void*, const void*, double*);          \
  template cudaError_t launch_soc_torque<R>(cudaStream_t, int, int, int, const void*, const double2*, double*);

TDDFT_INST(float)
TDDFT_INST(double)

}  // namespace tddft
