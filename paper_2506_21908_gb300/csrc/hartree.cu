// Poisson solve v_H(G) = 4 pi n(G) / |G|^2 (G = 0 dropped) of a real FP64 field, the Hartree term
// of Eq. HNC-SDFT.
//
// The field is real, so planes z and z + N/2 are packed as one complex plane: every xy transform
// runs on N/2 planes, and in the z pass the column (ky, kx) together with its mirror (-ky, -kx)
// gives back both planes' spectra; one column of each mirror pair is transformed, the other
// follows by conjugation.  Half the work of the complex transform.
//
// Five passes (x, y, z with the multiplication, inverse y, inverse x), each over whole lines cut
// into tiles of TX lines per CTA.  The solve is one small field, bound by the FP64 pipe of the SMs
// it occupies and by launch latency: with one CTA per plane (N CTAs on 152 SMs) it took 110 us at
// 48^3.  Tiles of 8 lines give N^2 / 16 CTAs per pass, and each pass is set up while the one before
// drains (programmatic dependent launch; every kernel waits for its predecessor before it touches
// memory): 40 us at 48^3 and 47 us at 64^3, 51 and 58 us with plain launches.  With its data requested
// before the twiddles that it waits for with them, 39 and 46 us.  Letting a pass start its CTAs as
// soon as its predecessor's have started (an early trigger) is slower, 78 and 156 us.
#include "fft.cuh"
#include "impl.cuh"
#include "kcommon.cuh"

namespace tddft {

namespace {

using C = double2;

// Factors of every supported size (8 and 12 have no two-factor plane pass, only these lines).
template <int N> struct LineFactor { static constexpr int R1 = TwoFactor<N>::R1, R2 = TwoFactor<N>::R2; };
template <> struct LineFactor<8> { static constexpr int R1 = 4, R2 = 2; };
template <> struct LineFactor<12> { static constexpr int R1 = 4, R2 = 3; };

template <int N> struct LineTile {
  static constexpr int TX = (N % 8 == 0) ? 8 : 4;  // lines per CTA
  static constexpr int R1 = LineFactor<N>::R1, R2 = LineFactor<N>::R2;
  static constexpr int NT = TX * (R1 > R2 ? R1 : R2);  // one item per thread and side
};


// exp(-2 pi i t / N): from the table, or formed here when there is none (tw_out then receives it from
// the first CTA for the passes that follow).
template <int N>
__device__ __forceinline__ void twiddles(C* tw, const C* twg, C* tw_out) {
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    if (twg) {
      tw[i] = twg[i];
    } else {
      double s, c;
      sincospi(-2.0 * (double)i / (double)N, &s, &c);
      tw[i] = make_double2(c, s);
      if (tw_out && blockIdx.x == 0) tw_out[i] = tw[i];
    }
  }
}

// Two-factor line transform in two steps around one exchange s[(k0 R1 + n0) TX + line]; see
// fft.cuh.  Forward: A side (n0) from x[n0 + R1 q], B side (k0) to X[k0 + R2 k1]; inverse backwards.
template <int N> __device__ __forceinline__ void fwd_a(C* v, int n0, int line, C* s, const C* tw) {
  using L = LineTile<N>;
  SmallDFT<C, L::R2, false>::run(v);
#pragma unroll
  for (int k0 = 0; k0 < L::R2; ++k0) s[(k0 * L::R1 + n0) * L::TX + line] = k0 ? cmul(v[k0], tw[k0 * n0]) : v[k0];
}
template <int N> __device__ __forceinline__ void fwd_b(C* u, int k0, int line, const C* s) {
  using L = LineTile<N>;
#pragma unroll
  for (int n0 = 0; n0 < L::R1; ++n0) u[n0] = s[(k0 * L::R1 + n0) * L::TX + line];
  SmallDFT<C, L::R1, false>::run(u);
}
template <int N> __device__ __forceinline__ void inv_b(C* u, int k0, int line, C* s, const C* tw) {
  using L = LineTile<N>;
  SmallDFT<C, L::R1, true>::run(u);
#pragma unroll
  for (int n0 = 0; n0 < L::R1; ++n0) s[(k0 * L::R1 + n0) * L::TX + line] = n0 ? cmulc(u[n0], tw[k0 * n0]) : u[n0];
}
template <int N> __device__ __forceinline__ void inv_a(C* v, int n0, int line, const C* s) {
  using L = LineTile<N>;
#pragma unroll
  for (int k0 = 0; k0 < L::R2; ++k0) v[k0] = s[(k0 * L::R1 + n0) * L::TX + line];
  SmallDFT<C, L::R2, true>::run(v);
}

// x lines: TX rows of the packed planes.  Forward: f(z) + i f(z + N/2), f = in (+ in2), into g;
// inverse: real and imaginary parts of g back to the two planes of out.
template <int N, bool INV>
__global__ void __launch_bounds__(LineTile<N>::NT)
k_poisson_x(const double* in, const double* in2, C* g, double* out, const C* twg, C* tw_out) {
  using L = LineTile<N>;
  constexpr int R1 = L::R1, R2 = L::R2, TX = L::TX;
  constexpr size_t HALF = (size_t)N * N * N / 2;
  __shared__ C tw[N], s[N * TX];
  if (!twg) twiddles<N>(tw, nullptr, nullptr);
  pdl_wait();
  // every pass requests its data before the twiddles that it waits for with it
  const size_t base = (size_t)blockIdx.x * TX * N;  // row (z, y) = blockIdx.x TX + line of the packed planes
  const int line = threadIdx.x / (INV ? R2 : R1), j = threadIdx.x - line * (INV ? R2 : R1);  // k0 or n0
  C v[R2], u[R1];
  if constexpr (!INV) {
    if (line < TX) {
#pragma unroll
      for (int q = 0; q < R2; ++q) {
        const size_t i = base + line * N + j + R1 * q;
        v[q] = make_double2(in[i], in[i + HALF]);
        if (in2) v[q] = make_double2(v[q].x + in2[i], v[q].y + in2[i + HALF]);
      }
    }
  } else {
    if (line < TX) {
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) u[k1] = g[base + line * N + j + R2 * k1];
    }
  }
  if (twg) twiddles<N>(tw, twg, nullptr);
  else if (tw_out && blockIdx.x == 0)
    for (int i = threadIdx.x; i < N; i += blockDim.x) tw_out[i] = tw[i];
  __syncthreads();
  if constexpr (!INV) {
    if (line < TX) fwd_a<N>(v, j, line, s, tw);
    __syncthreads();
    if (threadIdx.x < TX * R2) {
      const int lb = threadIdx.x / R2, k0 = threadIdx.x - lb * R2;
      fwd_b<N>(u, k0, lb, s);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) g[base + lb * N + k0 + R2 * k1] = u[k1];
    }
  } else {
    if (line < TX) inv_b<N>(u, j, line, s, tw);
    __syncthreads();
    if (threadIdx.x < TX * R1) {
      const int la = threadIdx.x / R1, n0 = threadIdx.x - la * R1;
      inv_a<N>(v, n0, la, s);
#pragma unroll
      for (int q = 0; q < R2; ++q) {
        const size_t i = base + la * N + n0 + R1 * q;
        out[i] = v[q].x;
        out[i + HALF] = v[q].y;
      }
    }
  }
}

// y lines in place: TX neighbouring x of one packed plane (blockIdx.y).
template <int N, bool INV>
__global__ void __launch_bounds__(LineTile<N>::NT) k_poisson_y(C* g, const C* twg) {
  using L = LineTile<N>;
  constexpr int R1 = L::R1, R2 = L::R2, TX = L::TX;
  __shared__ C tw[N], s[N * TX];
  pdl_wait();
  C* p = g + (size_t)blockIdx.y * N * N + blockIdx.x * TX;
  const int line = threadIdx.x % TX, j = threadIdx.x / TX;  // n0 (A side) or k0 (B side)
  C v[R2], u[R1];
  if (!INV && j < R1) {
#pragma unroll
    for (int q = 0; q < R2; ++q) v[q] = p[(size_t)(j + R1 * q) * N + line];
  }
  if (INV && j < R2) {
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) u[k1] = p[(size_t)(j + R2 * k1) * N + line];
  }
  twiddles<N>(tw, twg, nullptr);
  __syncthreads();
  if constexpr (!INV) {
    if (j < R1) fwd_a<N>(v, j, line, s, tw);
    __syncthreads();
    if (j < R2) {
      fwd_b<N>(u, j, line, s);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) p[(size_t)(j + R2 * k1) * N + line] = u[k1];
    }
  } else {
    if (j < R2) inv_b<N>(u, j, line, s, tw);
    __syncthreads();
    if (j < R1) {
      inv_a<N>(v, j, line, s);
#pragma unroll
      for (int q = 0; q < R2; ++q) p[(size_t)(j + R1 * q) * N + line] = v[q];
    }
  }
}

// z lines: column k = (ky, kx) and its mirror -k.  With G_j the packed planes' spectra and b_j =
// conj G_j(-k), plane j has the spectrum (G_j + b_j) / 2 and plane j + N/2 has (G_j - b_j) / 2i; the
// solved columns V go back as G_j(k) = V_j + i V_{j+N/2}, G_j(-k) = conj V_j + i conj V_{j+N/2}.
// CTA: TX columns kx of the row ky = blockIdx.y <= N/2; rows 0 and N/2 mirror onto themselves, so
// only their columns kx <= N/2 are taken (every mirror pair belongs to one line).
template <int N>
__global__ void __launch_bounds__(LineTile<N>::NT) k_poisson_z(C* g, const C* twg, ZParams zp) {
  using L = LineTile<N>;
  constexpr int R1 = L::R1, R2 = L::R2, TX = L::TX, H = N / 2;
  constexpr size_t P = (size_t)N * N;
  __shared__ C tw[N], s[N * TX];
  const int ky = blockIdx.y, x0 = blockIdx.x * TX;
  const bool self_row = ky == 0 || ky == H;
  pdl_wait();
  if (self_row && x0 > H) return;
  const int line = threadIdx.x % TX, j = threadIdx.x / TX;
  const int kx = x0 + line, mx = (N - kx) % N, my = (N - ky) % N;
  const bool on = !self_row || kx <= H;
  C* gk = g + (size_t)ky * N + kx;
  C* gm = g + (size_t)my * N + mx;
  C v[R2];
  if (on && j < R1) {
#pragma unroll
    for (int q = 0; q < R2; ++q) {
      const int z = j + R1 * q, jz = z < H ? z : z - H;
      const C a = gk[jz * P], b = gm[jz * P];  // b_j = (b.x, -b.y)
      v[q] = z < H ? make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y)) : make_double2(0.5 * (a.y + b.y), 0.5 * (b.x - a.x));
    }
  }
  twiddles<N>(tw, twg, nullptr);
  __syncthreads();
  if (on && j < R1) fwd_a<N>(v, j, line, s, tw);
  __syncthreads();
  C u[R1];
  if (on && j < R2) {
    fwd_b<N>(u, j, line, s);
    const double gx = zp.gs[0] * freq<N>(kx), gy = zp.gs[1] * freq<N>(ky);
    const double gxy = gx * gx + gy * gy;
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) {
      const double gz = zp.gs[2] * freq<N>(j + R2 * k1);
      const double g2 = gxy + gz * gz;
      u[k1] = cscale(u[k1], g2 > 0.0 ? 4.0 * 3.14159265358979323846 / g2 * zp.scale : 0.0);
    }
    inv_b<N>(u, j, line, s, tw);  // writes the cells of s that this thread read
  }
  __syncthreads();
  C w[R2];
  if (on && j < R1) inv_a<N>(w, j, line, s);
  __syncthreads();
  if (on && j < R1) {
#pragma unroll
    for (int q = 0; q < R2; ++q) s[(j + R1 * q) * TX + line] = w[q];
  }
  __syncthreads();
  if (on)
    for (int z = j; z < H; z += L::NT / TX) {
      const C a = s[z * TX + line], b = s[(z + H) * TX + line];
      gk[z * P] = make_double2(a.x - b.y, a.y + b.x);
      if (gm != gk) gm[z * P] = make_double2(a.x + b.y, b.x - a.y);
    }
}

template <int N>
cudaError_t poisson_n(cudaStream_t st, const double* in, const double* in2, double* out, double2* g, const double2* tw,
                      double2* tw_out, const ZParams& zp) {
  using L = LineTile<N>;
  constexpr int rows = N * N / 2 / L::TX;
  const dim3 lines(N / L::TX, N / 2);
  const double2* twp = tw ? tw : tw_out;
  cudaError_t e;
  if ((e = launch_pdl(k_poisson_x<N, false>, dim3(rows), L::NT, 0, st, in, in2, g, nullptr, tw, tw_out)) != cudaSuccess ||
      (e = launch_pdl(k_poisson_y<N, false>, lines, L::NT, 0, st, g, twp)) != cudaSuccess ||
      (e = launch_pdl(k_poisson_z<N>, dim3(N / L::TX, N / 2 + 1), L::NT, 0, st, g, twp, zp)) != cudaSuccess ||
      (e = launch_pdl(k_poisson_y<N, true>, lines, L::NT, 0, st, g, twp)) != cudaSuccess)
    return e;
  return launch_pdl(k_poisson_x<N, true>, dim3(rows), L::NT, 0, st, nullptr, nullptr, g, out, twp, nullptr);
}

}  // namespace

cudaError_t launch_poisson(cudaStream_t st, int N, const double* in, const double* in2, double* out, double2* g,
                           const double2* tw, double2* tw_out, const double* L) {
  ZParams zp{};
  const double pi = 3.14159265358979323846;
  for (int a = 0; a < 3; ++a) zp.gs[a] = 2.0 * pi / L[a];
  zp.scale = 1.0 / ((double)N * N * N);
  TDDFT_DISPATCH_N(N, (poisson_n<NN>(st, in, in2, out, g, tw, tw_out, zp)));
}

}  // namespace tddft
