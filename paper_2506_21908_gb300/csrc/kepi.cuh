// Point-wise Hamiltonian helpers shared by the epilogue kernels: the 2x2 spin-matrix local
// potential [[v + b_z, b_x - i b_y], [b_x + i b_y, v - b_z]] from the 4-vector
// V_v = [v + b_z, v - b_z, 2 b_x, -2 b_y] (Eq. potential4) and the projector scatter
// sum_a sum_p beta_p(d) exp(-i (k+A).d) (D c)_p (Eq. Vps with the L.S blocks).
#pragma once
#include "fft.cuh"
#include "impl.cuh"
#include "kcommon.cuh"

namespace tddft {

template <typename C> struct Pair { C a, b; };
__device__ __forceinline__ Pair<float2> ld2(const float2* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ void st2(float2* p, float2 a, float2 b) {
  *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ Pair<double2> ld2(const double2* p) { return {p[0], p[1]}; }
__device__ __forceinline__ void st2(double2* p, double2 a, double2 b) { p[0] = a; p[1] = b; }

// One row of a projector table (3 + NLM values: d, beta).  Rows whose size is a multiple of
// 16 bytes start on 16-byte boundaries (the table is one allocation) and are read as vectors.
template <typename R, int TAB>
__device__ __forceinline__ void load_row(const R* __restrict__ t, R* v) {
  if constexpr (sizeof(R) == 4 && TAB % 4 == 0) {
    const float4* t4 = reinterpret_cast<const float4*>(t);
#pragma unroll
    for (int i = 0; i < TAB / 4; ++i) {
      const float4 q = __ldg(t4 + i);
      v[4 * i] = q.x; v[4 * i + 1] = q.y; v[4 * i + 2] = q.z; v[4 * i + 3] = q.w;
    }
  } else if constexpr (sizeof(R) == 8 && TAB % 2 == 0) {
    const double2* t2 = reinterpret_cast<const double2*>(t);
#pragma unroll
    for (int i = 0; i < TAB / 2; ++i) {
      const double2 q = __ldg(t2 + i);
      v[2 * i] = q.x; v[2 * i + 1] = q.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < TAB; ++i) v[i] = __ldg(t + i);
  }
}

// Projector values beta_p(d) = N_l g S_lm(d), p = l^2 + l + mu, from a compact row (d, g): the
// real solid harmonics r^l Y_lm for l <= 2 in the order of the tables (1; y, z, x; xy, yz,
// 3z^2 - r^2, xz, x^2 - y^2), nl = N_0, N_1, N_2 of the atom, yc the harmonic constants.
template <typename R, int NLM>
__device__ __forceinline__ void beta_values(R x, R y, R z, R g, const R* nl, const R* yc, R* b) {
  b[0] = nl[0] * g * yc[0];
  if constexpr (NLM > 1) {
    const R s1 = nl[1] * g * yc[1];
    b[1] = s1 * y; b[2] = s1 * z; b[3] = s1 * x;
  }
  if constexpr (NLM > 4) {
    const R s2 = nl[2] * g * yc[2], s0 = nl[2] * g * yc[3];
    b[4] = s2 * (x * y); b[5] = s2 * (y * z);
    b[6] = s0 * ((R)2 * z * z - x * x - y * y);
    b[7] = s2 * (x * z); b[8] = (R)0.5 * s2 * (x * x - y * y);
  }
}

// Projector values of entry e: FP64 reads its table row, FP32 evaluates them from the compact row.
template <typename R, int NLM>
__device__ __forceinline__ void entry_beta(size_t e, int a, const R* rows, const R* beta, const ProjTables<R>& pt, R* bt) {
  if constexpr (sizeof(R) == 8) {
    load_row<R, beta_pitch(NLM)>(beta + e * beta_pitch(NLM), bt);
  } else {
    R t[4], nl[4];
    load_row<R, 4>(rows + e * 4, t);
    load_row<R, 4>(pt.nrm + (size_t)a * 4, nl);
    beta_values<R, NLM>(t[0], t[1], t[2], t[3], nl, pt.yc, bt);
  }
}

// The projector entries of a thread's point(s) in scatter order, one entry ahead: the table row, phase
// and atom of the next entry are requested before the current one is used (FP32, whose scatter is
// bound by these dependent loads; FP64 is bound by its arithmetic and reads its longer rows in
// place).  The first entry's loads are issued together with the spinors' (start).
template <typename R, int NLM> struct EntryStream {
  using C = typename CT<R>::type;
  const ProjTables<R>& pt;
  const C* ph;
  int e, end, a;
  C pe;
  float4 row;
  __device__ __forceinline__ EntryStream(const ProjTables<R>& t, const C* p, int e0, int e1)
      : pt(t), ph(p), e(e0), end(e1), a(0), pe(cmake<C>((R)0, (R)0)), row(make_float4(0.f, 0.f, 0.f, 0.f)) {}
  __device__ __forceinline__ void start() {
    if (sizeof(R) == 4 && e < end) fetch();
  }
  __device__ __forceinline__ void fetch() {
    a = pt.s_atom[e];
    pe = ph[e];
    if constexpr (sizeof(R) == 4) row = __ldg(reinterpret_cast<const float4*>(pt.s_row) + e);
  }
  // projector values, phase and atom of the current entry; moves on to the next
  __device__ __forceinline__ void next(R* bt, C& phase, int& atom) {
    if constexpr (sizeof(R) == 8) {
      fetch();
      entry_beta<R, NLM>(e, a, pt.s_row, pt.s_beta, pt, bt);
      phase = pe;
      atom = a;
      ++e;
    } else {
      const float4 t = row;
      phase = pe;
      atom = a;
      ++e;
      if (e < end) fetch();
      R nl[4];
      load_row<R, 4>(pt.nrm + (size_t)atom * 4, nl);
      beta_values<R, NLM>(t.x, t.y, t.z, t.w, nl, pt.yc, bt);
    }
  }
};

// Local part of H at one point: (hu, hd) holds the kinetic part on entry; the 2x2 potential is added.
template <typename R, typename C>
__device__ __forceinline__ void h_local(C& hu, C& hd, C pu, C pd, R V0, R V1, R hx, R hy) {
  hu = cmake<C>(hu.x + V0 * pu.x + hx * pd.x - hy * pd.y, hu.y + V0 * pu.y + hx * pd.y + hy * pd.x);
  hd = cmake<C>(hd.x + V1 * pd.x + hx * pu.x + hy * pu.y, hd.y + V1 * pd.y + hx * pu.y - hy * pu.x);
}

// Projector scatter at one point for both spinor components: the entries of the stream before e1.
template <typename R, int NLM>
__device__ __forceinline__ void h_scatter(typename CT<R>::type& hu, typename CT<R>::type& hd, EntryStream<R, NLM>& es,
                                          int e1, const typename CT<R>::type* dcb) {
  using C = typename CT<R>::type;
  while (es.e < e1) {
    R bt[beta_pitch(NLM)];
    C pe;
    int a;
    es.next(bt, pe, a);
    const C* dca = dcb + (size_t)a * 2 * NLM;  // this spinor's D c of atom a, (up, dn) per p
    R vux = 0, vuy = 0, vdx = 0, vdy = 0;
#pragma unroll
    for (int p = 0; p < NLM; ++p) {
      const R bp = bt[p];
      const Pair<C> cc = ld2(dca + 2 * p);
      vux += bp * cc.a.x; vuy += bp * cc.a.y;
      vdx += bp * cc.b.x; vdy += bp * cc.b.y;
    }
    const R cs = pe.x, sn = pe.y;
    hu.x += vux * cs + vuy * sn; hu.y += vuy * cs - vux * sn;
    hd.x += vdx * cs + vdy * sn; hd.y += vdy * cs - vdx * sn;
  }
}

// The same for one point of two spinors of one k-point (index g = 0, 1): the projector entries
// of the point, their beta values and phases are evaluated once for both spinors.
template <typename R, int NLM>
__device__ __forceinline__ void h_scatter_2sp(typename CT<R>::type (&hu)[2], typename CT<R>::type (&hd)[2],
                                              EntryStream<R, NLM>& es, const typename CT<R>::type* dcb0,
                                              const typename CT<R>::type* dcb1) {
  using C = typename CT<R>::type;
  while (es.e < es.end) {
    R bt[beta_pitch(NLM)];
    C pe;
    int a;
    es.next(bt, pe, a);
    const R cs = pe.x, sn = pe.y;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const C* dca = (g ? dcb1 : dcb0) + (size_t)a * 2 * NLM;
      R vux = 0, vuy = 0, vdx = 0, vdy = 0;
#pragma unroll
      for (int p = 0; p < NLM; ++p) {
        const R bp = bt[p];
        const Pair<C> cc = ld2(dca + 2 * p);
        vux += bp * cc.a.x; vuy += bp * cc.a.y;
        vdx += bp * cc.b.x; vdy += bp * cc.b.y;
      }
      hu[g].x += vux * cs + vuy * sn; hu[g].y += vuy * cs - vux * sn;
      hd[g].x += vdx * cs + vdy * sn; hd[g].y += vdy * cs - vdx * sn;
    }
  }
}

}  // namespace tddft
