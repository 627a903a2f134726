// Tile-centric projector contraction on the tensor cores (tcgen05), FP32-mixed path.
//
// The grid is cut into bricks of BX x 8 x 8 points (BX = 32 or 16).  For one brick b, every atom
// image whose projector sphere reaches into the brick is a "slot" (at most 256 / nlm of them).
// With q = k + A(t) and the brick origin r_b, the projector phase of Eq. Vps in velocity gauge
// factorises as exp(i q.d) = exp(i q.(r - r_b)) exp(i q.delta), delta = r_b - R_image, so with the
// real projector values beta_{slot,p}(r) (zero outside the sphere):
//
//   gather   c[s,a,p] = dV sum_{b, slot of a} exp(i q.delta) sum_{r in b} beta_{slot,p}(r) psi'_s(r),
//            psi'_s(r) = exp(i q.(r - r_b)) psi_s(r);
//   scatter  (V_NL psi)_s(r) = exp(-i q.(r - r_b)) sum_{slot,p} beta_{slot,p}(r) X_s[slot,p],
//            X_s[slot,p] = exp(-i q.delta) (D c)[s, a_slot, p].
//
// Both inner sums are dense real products over one brick: the gather is [64 components x (re, im)]
// x [brick points] x [slots x nlm], read psi once per brick; the scatter is [128 points] x
// [slots x nlm] x [components x (re, im)].  The real projector values of every brick are built
// once at creation in FP64 and stored in the operand layout of the tensor cores (K-major, rows of
// 128 bytes with the 128-byte swizzle), as one rounded part (TF32) or as hi + lo parts (TF32 x3,
// BF16 x3, FP16 x3: hi*hi + hi*lo + lo*hi with FP32 accumulation, the split-precision product).
//
// Each CTA: worker warps (8 in the gather, 16 in the scatter) stage psi (phase, split, swizzled
// stores) or X and drain the tensor memory, one warp issues the MMAs (one elected thread), one the
// bulk copies of the projector tables; two shared-memory stages between them, full / empty mbarriers.  Every
// mbarrier wait has an iteration limit: on expiry the CTA sets bit 1 of the error word, stops
// issuing work, waits (with a limit) for its copies and MMAs in flight and frees its tensor memory.
#include <cstdint>
#include <type_traits>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "bulk.cuh"
#include "fft.cuh"
#include "impl.cuh"
#include "kcommon.cuh"

namespace tddft {

namespace {

constexpr int PT_ROWB = 128;        // bytes per operand row
constexpr int PT_PART = 128 * PT_ROWB;  // one 128-row operand part (16 KB)
constexpr unsigned PT_WAIT_LIMIT = 1u << 22;

__device__ __forceinline__ uint32_t sw128(uint32_t off) { return off ^ (((off >> 7) & 7u) << 4); }

// K-major operand, rows of 128 bytes with the 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;            // leading byte offset (not used by swizzled K-major operands)
  d |= (uint64_t)(1024 >> 4) << 32;  // stride byte offset between 8-row groups
  d |= (uint64_t)1 << 46;            // descriptor version of this architecture family
  d |= (uint64_t)2 << 61;            // 128-byte swizzle
  return d;
}

// Element kinds: bytes per element, instruction descriptor type code.
template <int EK> struct Elt;
template <> struct Elt<TILE_TF32> { static constexpr int bytes = 4, code = 2; };
template <> struct Elt<TILE_BF16> { static constexpr int bytes = 2, code = 1; };
template <> struct Elt<TILE_F16> { static constexpr int bytes = 2, code = 0; };

// D = F32, A = B of kind EK, both K-major, M = 128, N.
template <int EK> __device__ __forceinline__ uint32_t idesc(int n) {
  return (1u << 4) | ((uint32_t)Elt<EK>::code << 7) | ((uint32_t)Elt<EK>::code << 10) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

template <int EK>
__device__ __forceinline__ void mma(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t id, uint32_t acc) {
  if constexpr (EK == TILE_TF32)
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(id), "r"(acc));
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(id), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool pt_wait(uint32_t bar, uint32_t parity) {
  for (unsigned it = 0; it < PT_WAIT_LIMIT; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

__device__ __forceinline__ void pt_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

// Split x into the rounded part(s) of kind EK (hi, and lo = x - hi for the split product).
__device__ __forceinline__ float tf32_rna(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}
template <int EK> struct Split;
template <> struct Split<TILE_TF32> {
  __device__ __forceinline__ static void two(float x, uint32_t& hi, uint32_t& lo) {
    const float h = tf32_rna(x);
    hi = __float_as_uint(h);
    lo = __float_as_uint(tf32_rna(x - h));
  }
};
template <> struct Split<TILE_BF16> {
  __device__ __forceinline__ static void two(float x, uint32_t& hi, uint32_t& lo) {
    const __nv_bfloat16 h = __float2bfloat16_rn(x);
    hi = __bfloat16_as_ushort(h);
    lo = __bfloat16_as_ushort(__float2bfloat16_rn(x - __bfloat162float(h)));
  }
};
template <> struct Split<TILE_F16> {
  __device__ __forceinline__ static void two(float x, uint32_t& hi, uint32_t& lo) {
    const __half h = __float2half_rn(x);
    hi = __half_as_ushort(h);
    lo = __half_as_ushort(__float2half_rn(x - __half2float(h)));
  }
};

// Store element k of row `row` of a swizzled operand part (k within the 128-byte row).
template <int EK> __device__ __forceinline__ void put(unsigned char* part, int row, int k, uint32_t v) {
  const uint32_t off = sw128((uint32_t)row * PT_ROWB + (uint32_t)(k * Elt<EK>::bytes));
  if constexpr (Elt<EK>::bytes == 4) *reinterpret_cast<uint32_t*>(part + off) = v;
  else *reinterpret_cast<uint16_t*>(part + off) = (uint16_t)v;
}

// 16 consecutive columns of the thread's lane, without the wait for completion.
__device__ __forceinline__ void tmem_ld16_async(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld8_async(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld4_async(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
// W = 4 or 8 columns; tmem_regs_ready as above.
template <int W> __device__ __forceinline__ void tmem_ld_async(uint32_t taddr, uint32_t* r) {
  if constexpr (W == 4) tmem_ld4_async(taddr, r);
  else tmem_ld8_async(taddr, r);
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// After tmem_wait_ld: ties the loaded registers to a point after the wait, so that no use of them
// is scheduled before it.
__device__ __forceinline__ void tmem_regs_ready(uint32_t* r) {
  asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
               "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]));
}
template <int W> __device__ __forceinline__ void tmem_regs_ready_n(uint32_t* r) {
  asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]));
  if constexpr (W == 8) asm volatile("" : "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]));
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16};" ::"r"(taddr),
      "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]),
      "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15])
      : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Per-axis phase tables exp(+i q_a l h_a) of one brick (l = 0 .. extent-1).
__device__ __forceinline__ void phase_tables(float2* px, float2* py, float2* pz, int BX, const TileDev& td,
                                             const double* q) {
  for (int i = threadIdx.x; i < BX + 16; i += blockDim.x) {
    float s, c;
    if (i < BX) {
      sincosf((float)(q[0] * td.h[0] * i), &s, &c);
      px[i] = make_float2(c, s);
    } else if (i < BX + 8) {
      sincosf((float)(q[1] * td.h[1] * (i - BX)), &s, &c);
      py[i - BX] = make_float2(c, s);
    } else {
      sincosf((float)(q[2] * td.h[2] * (i - BX - 8)), &s, &c);
      pz[i - BX - 8] = make_float2(c, s);
    }
  }
}

__device__ __forceinline__ float2 cm(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }

}  // namespace

// Two neighbouring values a, b (elements k, k + 1) as packed 16-bit hi and lo pairs.
template <int EK> struct Split2;
template <> struct Split2<TILE_F16> {
  __device__ __forceinline__ static void two(float a, float b, uint32_t& hi, uint32_t& lo) {
    const __half2 h = __floats2half2_rn(a, b);
    const float2 f = __half22float2(h);
    const __half2 l = __floats2half2_rn(a - f.x, b - f.y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
  }
};
template <> struct Split2<TILE_BF16> {
  __device__ __forceinline__ static void two(float a, float b, uint32_t& hi, uint32_t& lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    const float2 f = __bfloat1622float2(h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(a - f.x, b - f.y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
  }
};

constexpr int PT_WARPS = 8;                   // worker warps
constexpr int PT_NT = 32 * (PT_WARPS + 2);    // + MMA warp + copy warp
constexpr int PT_MMA_WARP = PT_WARPS, PT_COPY_WARP = PT_WARPS + 1;

// ============================================================================ gather

// Chunks per accumulation group of the gather.  The tensor cores add each product into the FP32
// accumulator with a rounding that is biased toward zero, so one accumulator that takes every
// chunk of a brick (hundreds of MMAs) loses a relative 1e-5 of every partial sum, the same sign
// everywhere.  The accumulation therefore restarts from zero every CPG chunks: group 0 accumulates
// in the running sum R (tensor-memory columns 256..511), every later group in P (columns 0..255),
// and the worker warps add P into R on the CUDA cores (round to nearest) between groups; the bias
// falls with the length of a group.
template <int TERMS> struct GatherGroups { static constexpr int CPG = (TERMS == 3) ? 4 : 8; };

// Spinors, read once by a CTA: ordinary loads past L1, in program order with the waits (asm volatile),
// since pdl_wait() has to precede them.  Requested after the arrival that the MMAs of the staged chunk
// wait for, they take the gather from 615 to 600 us (96^3, 128 atoms, 128 spinors) and from 651 to
// 632 us (48^3 x 1024) against read-only loads through L1; before that arrival 603 and 637 us.
__device__ __forceinline__ void ld_stream(float4& v, const void* p) {
  asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
}
__device__ __forceinline__ void ld_stream(float2& v, const void* p) {
  asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
}

// CTA (kg, item): 64 components (group g of k-point k) against the slots of one brick.
template <int EK, int TERMS>
__global__ void __launch_bounds__(PT_NT, 1)
k_tile_gather(const float2* psi, int N, int comps_per_k, int groups, TileDev td, EpiParams ep, float* part, int* err) {
  constexpr int EPR = PT_ROWB / Elt<EK>::bytes;  // points per chunk (K elements per row)
  constexpr int NPART = (TERMS == 3) ? 2 : 1;
  constexpr int BPART = 256 * PT_ROWB;          // largest B part (N <= 256)
  constexpr int STAGE = NPART * (PT_PART + BPART);
  constexpr int CPW = 64 / PT_WARPS;            // components per worker warp
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  constexpr int CPG = GatherGroups<TERMS>::CPG;
  __shared__ uint64_t bar_full[2], bar_empty[2], bar_acc, bar_grp, bar_drain;
  __shared__ uint32_t tmem_base;
  __shared__ volatile int abort_flag;
  __shared__ float2 px[32], py[8], pz[8];

  // after a failed wait anywhere in the launch the remaining CTAs do nothing (the call reports it)
  if (*reinterpret_cast<volatile int*>(err) & 1) {
    pdl_wait();  // a launch never ends before its predecessor, even if all its CTAs skip their work
    return;
  }
  const int kg = blockIdx.x, it = blockIdx.y;
  const int k = kg / groups, comp0 = (kg % groups) * 64;
  const int nslot = td.it_nslot[it], npad = td.it_npad[it];
  if (nslot == 0) {  // a brick no projector sphere reaches
    pdl_wait();
    return;
  }
  const int BX = td.BX;
  const int brick = td.it_brick[it];
  const int bx = brick % td.nbx, by = (brick / td.nbx) % td.nby, bz = brick / (td.nbx * td.nby);
  const int x0 = bx * BX, y0 = by * 8, z0 = bz * 8;
  const int nch = BX * 64 / EPR;
  const int ngrp = nch / CPG;  // nch is a multiple of 16 and of CPG, so ngrp >= 2
  const size_t N3 = (size_t)N * N * N;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto stageA = [&](int s, int q) { return smem + (size_t)s * STAGE + (size_t)q * PT_PART; };
  auto stageB = [&](int s, int q) { return smem + (size_t)s * STAGE + (size_t)NPART * PT_PART + (size_t)q * BPART; };

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < 2; ++s) {
      bar_init(sm_addr(&bar_full[s]), 32 * PT_WARPS + 1);
      bar_init(sm_addr(&bar_empty[s]), 1);
    }
    bar_init(sm_addr(&bar_acc), 1);
    bar_init(sm_addr(&bar_grp), 1);
    bar_init(sm_addr(&bar_drain), 32 * PT_WARPS);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // Worker warps: each lane's point(s) of a chunk and the spinor components [warp CPW, + CPW) of the
  // group there; the first two chunks are requested before the CTA's set-up.  Byte offsets of the
  // group's components fit 32 bits, a lane's x and the rows of its chunks need no division, and two
  // register sets alternate.  The kernel is bound by the chain MMA -> stage free -> conversion and
  // copy -> MMA of its two stages, and by the MMAs' wait for P between groups: adding P into R before
  // the next conversion instead of after it took 677 to 614 us (96^3, 128 atoms, 128 spinors) and 688
  // to 650 us (48^3 x 1024).  (16 worker warps: 876 us.)
  constexpr int PPL = (EPR == 64) ? 2 : 1;  // points per lane
  using V = typename std::conditional<PPL == 2, float4, float2>::type;
  const int bsh = BX == 32 ? 5 : 4, kk = lane * PPL, lx = kk & (BX - 1);
  const int rpc = EPR >> bsh, row0 = kk >> bsh;  // grid rows per chunk, this lane's row in one
  const char* gbase = reinterpret_cast<const char*>(psi + ((size_t)k * comps_per_k + comp0) * N3);
  const uint32_t n3b = (uint32_t)N3 * (uint32_t)sizeof(float2);  // at most 64 n3b = 453 MB to a group
  const uint32_t o0 = (uint32_t)warp * CPW * n3b + (uint32_t)((z0 * N + y0) * N + x0 + lx) * (uint32_t)sizeof(float2);
  const int nvalid = min(CPW, comps_per_k - comp0 - warp * CPW);
  auto load = [&](int c, V* w) {
    const int row = c * rpc + row0;
    const uint32_t o = o0 + (uint32_t)(((row >> 3) * N + (row & 7)) * N) * (uint32_t)sizeof(float2);
#pragma unroll
    for (int j = 0; j < CPW; ++j) {
      V v;
      if constexpr (PPL == 2) v = make_float4(0.f, 0.f, 0.f, 0.f);
      else v = make_float2(0.f, 0.f);
      if (j < nvalid) ld_stream(v, gbase + (o + (uint32_t)j * n3b));
      w[j] = v;
    }
  };
  V wa[CPW], wb[CPW];
  if (warp < PT_WARPS) {
    pdl_wait();
    load(0, wa);
    load(1, wb);
  }
  phase_tables(px, py, pz, BX, td, ep.shift[k]);
  if (warp == PT_MMA_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sm_addr(&tmem_base)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base;
  const uint32_t accP = tmem, accR = tmem + 256u;
  // worker warp: lane quarter of the accumulator, and the first of the blocks of 16 columns it takes
  // (every CSTEP columns)
  constexpr int CSTEP = 16 * (PT_WARPS / 4);
  const int quarter = warp & 3, cfirst = 16 * (warp >> 2);
  const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;

  if (warp < PT_WARPS) {
    // ---- psi' = exp(i q.(r - r_b)) psi, split, into rows cl (re) and 64 + cl (im) of stage A
    const float2 px0 = px[lx], px1 = px[PPL == 2 ? lx + 1 : lx];
    // one chunk from w; then the chunk after next is requested into w.  False: give up.
    auto chunk = [&](int c, V* w) -> bool {
      // group g (1 <= g <= ngrp - 2) ended with chunk c - 2: add P into R first of all, since the MMAs of
      // chunk c - 1 (group g + 1), staged already, wait to reuse P (the votes keep the warp together
      // for the tensor-memory accesses)
      const int gd = (c - 1) / CPG;
      if ((c - 1) % CPG == 0 && gd >= 2 && gd <= ngrp - 1) {
        if (!pt_wait(sm_addr(&bar_grp), (gd - 2) & 1)) abort_flag = 1;
        if (__any_sync(0xffffffffu, abort_flag != 0)) return false;
        asm volatile("tcgen05.fence::after_thread_sync;");
        for (int c0 = cfirst; c0 < npad; c0 += 2 * CSTEP) {  // two blocks of 16 columns at a time
          const bool two = c0 + CSTEP < npad;
          uint32_t pv[2][16], rv[2][16];
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (h == 0 || two) {
              tmem_ld16_async(accP + lane_off + (uint32_t)(c0 + h * CSTEP), pv[h]);
              tmem_ld16_async(accR + lane_off + (uint32_t)(c0 + h * CSTEP), rv[h]);
            }
          tmem_wait_ld();
#pragma unroll
          for (int h = 0; h < 2; ++h)
            if (h == 0 || two) {
              tmem_regs_ready(pv[h]);
              tmem_regs_ready(rv[h]);
              float sum[16];
#pragma unroll
              for (int j = 0; j < 16; ++j) sum[j] = __uint_as_float(rv[h][j]) + __uint_as_float(pv[h][j]);
              tmem_st16(accR + lane_off + (uint32_t)(c0 + h * CSTEP), sum);
            }
        }
        tmem_wait_st();
        asm volatile("tcgen05.fence::before_thread_sync;");
        pt_arrive(sm_addr(&bar_drain));
      }
      const int s = c & 1;
      if (c >= 2 && !pt_wait(sm_addr(&bar_empty[s]), ((c >> 1) - 1) & 1)) abort_flag = 1;
      if (__any_sync(0xffffffffu, abort_flag != 0)) return false;
      const int row = c * rpc + row0;
      const float2 pyz = cm(py[row & 7], pz[row >> 3]);
      const float2 ph0 = cm(px0, pyz), ph1 = PPL == 2 ? cm(px1, pyz) : ph0;
      unsigned char* a0 = stageA(s, 0) + (warp * CPW) * PT_ROWB;
#pragma unroll
      for (int j = 0; j < CPW; ++j) {
        // row j of this warp's eight: its swizzle is j
        unsigned char* q = a0 + j * PT_ROWB + ((lane * 4) ^ (j << 4));
        const float2 v0 = cm(make_float2(w[j].x, w[j].y), ph0);
        uint32_t rh, rl, ih, il;
        if constexpr (PPL == 2) {
          const float2 v1 = cm(make_float2(w[j].z, w[j].w), ph1);
          Split2<EK>::two(v0.x, v1.x, rh, rl);
          Split2<EK>::two(v0.y, v1.y, ih, il);
        } else {
          Split<EK>::two(v0.x, rh, rl);
          Split<EK>::two(v0.y, ih, il);
        }
        *reinterpret_cast<uint32_t*>(q) = rh;
        *reinterpret_cast<uint32_t*>(q + 64 * PT_ROWB) = ih;
        if constexpr (TERMS == 3) {
          *reinterpret_cast<uint32_t*>(q + PT_PART) = rl;
          *reinterpret_cast<uint32_t*>(q + PT_PART + 64 * PT_ROWB) = il;
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      pt_arrive(sm_addr(&bar_full[s]));
      if (c + 2 < nch) load(c + 2, w);
      return true;
    };
    for (int c = 0; c < nch; c += 2)  // nch is even
      if (!chunk(c, wa) || !chunk(c + 1, wb)) break;
  } else if (warp == PT_COPY_WARP) {
    if (lane == 0) {
      // ---- projector values of the brick, chunk by chunk
      const unsigned char* src = td.g_tab + td.it_goff[it];
      const uint32_t pbytes = (uint32_t)npad * PT_ROWB;
      int issued = 0;
      for (int c = 0; c < nch; ++c) {
        const int s = c & 1;
        if (c >= 2 && !pt_wait(sm_addr(&bar_empty[s]), ((c >> 1) - 1) & 1)) abort_flag = 1;
        if (abort_flag) break;
        bulk_expect(sm_addr(&bar_full[s]), NPART * pbytes);
        for (int q = 0; q < NPART; ++q)
          bulk_copy(stageB(s, q), src + ((size_t)c * NPART + q) * pbytes, pbytes, sm_addr(&bar_full[s]));
        issued = c + 1;
      }
      // every copy issued has landed before the CTA moves on
      for (int c = (issued > 2 ? issued - 2 : 0); c < issued; ++c)
        if (!pt_wait(sm_addr(&bar_full[c & 1]), (c >> 1) & 1)) atomicOr(err, 1);
    }
  } else {
    if (lane == 0) {
      const uint32_t id = idesc<EK>(npad);
      for (int c = 0; c < nch; ++c) {
        const int s = c & 1, g = c / CPG, cg = c % CPG;
        // the first wait may be shortened by the testing hook: on expiry the error bit is set and
        // the wait is retried with the full limit
        if (c == 0 && !bulk_first_try(sm_addr(&bar_full[s]), 0)) atomicOr(err, 1);
        // P holds group g - 1 until the worker warps have added it into R
        if (cg == 0 && g >= 2 && !pt_wait(sm_addr(&bar_drain), (g - 2) & 1)) abort_flag = 1;
        if (!abort_flag && !pt_wait(sm_addr(&bar_full[s]), (c >> 1) & 1)) abort_flag = 1;
        if (abort_flag) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t dst = (g == 0) ? accR : accP;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          const uint32_t off = (uint32_t)ks * 32;
          const uint64_t ah = desc_sw128(sm_addr(stageA(s, 0)) + off), bh = desc_sw128(sm_addr(stageB(s, 0)) + off);
          mma<EK>(dst, ah, bh, id, (cg | ks) ? 1u : 0u);
          if constexpr (TERMS == 3) {
            const uint64_t al = desc_sw128(sm_addr(stageA(s, 1)) + off), bl = desc_sw128(sm_addr(stageB(s, 1)) + off);
            mma<EK>(dst, ah, bl, id, 1u);
            mma<EK>(dst, al, bh, id, 1u);
          }
        }
        mma_commit(sm_addr(&bar_empty[s]));
        // groups 1 .. ngrp - 2 are added into R by the worker warps; the last one at the end
        if (cg == CPG - 1 && g >= 1 && g <= ngrp - 2) mma_commit(sm_addr(&bar_grp));
      }
      // also after an abort: every MMA issued completes before the accumulator is read or freed
      mma_commit(sm_addr(&bar_acc));
      if (!pt_wait(sm_addr(&bar_acc), 0)) atomicOr(err, 1);
    }
  }
  // ---- R + P (the last group) (rows: component re / im; columns: slot x nlm) -> partial sums;
  // the warps of a lane quarter take alternate blocks of 16 columns
  if (warp < PT_WARPS) {
    const bool ok = __all_sync(0xffffffffu, pt_wait(sm_addr(&bar_acc), 0));
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (!ok || __any_sync(0xffffffffu, abort_flag != 0)) {
      if (lane == 0) atomicOr(err, 1);
    } else {
      const int row = quarter * 32 + lane;
      const int ncol = td.nlm * nslot;
      float* dst = part + (size_t)kg * td.part_layer + td.it_poff[it];
      for (int c0 = cfirst; c0 < npad; c0 += CSTEP) {
        uint32_t pv[16], rv[16];
        tmem_ld16_async(accP + lane_off + (uint32_t)c0, pv);
        tmem_ld16_async(accR + lane_off + (uint32_t)c0, rv);
        tmem_wait_ld();
        tmem_regs_ready(pv);
        tmem_regs_ready(rv);
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (c0 + j < ncol) dst[(size_t)(c0 + j) * 128 + row] = __uint_as_float(rv[j]) + __uint_as_float(pv[j]);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == PT_MMA_WARP)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// Sum the partial products of every (brick, slot) of atom a in a fixed order with the phase
// exp(i q.delta), times dV: c[kb][a][2p + sigma]; then D c with the atom's block.  Thread (p, t):
// projector p of component t, so a CTA has 64 nlm threads; the phases of up to kRedPh pairs at a
// time are formed once per CTA, and four pairs' partial products are requested before the first
// is used.  Bound by the latency of those loads: with one thread per component looping over the
// projectors (64 threads, one pair at a time, 3 % of the warp slots) it took 241 us at the large
// supercell with 32 spinors and 107 us at 64^3 with 48; gather and reduction together went from
// 869 to 677 us per launch at the large supercell with 128 spinors (614 us with the gather's
// groups added ahead of the conversion).
constexpr int kRedPh = 256;
__global__ void __launch_bounds__(64 * kMaxNLM)
k_tile_reduce(const float* part, TileDev td, int groups, int comps_per_k, int nstates, int natoms, float dV,
              EpiParams ep, const float* __restrict__ Dmat, float2* c_out, float2* dc_out) {
  const int a = blockIdx.x, kg = blockIdx.y;
  const int k = kg / groups, comp0 = (kg % groups) * 64;
  const int nlm = td.nlm;
  const int t = threadIdx.x & 63, p = threadIdx.x >> 6;
  __shared__ float2 cs[64][kMaxNLM];
  __shared__ float2 ph[kRedPh];
  __shared__ long long so[kRedPh];
  const double* q = ep.shift[k];
  const int e0 = td.a_ptr[a], e1 = td.a_ptr[a + 1];
  const float* base = part + (size_t)kg * td.part_layer + (size_t)p * 128 + t;
  float2 acc = make_float2(0.f, 0.f);
  pdl_wait();
  for (int b0 = e0; b0 < e1; b0 += kRedPh) {
    const int nb = min(kRedPh, e1 - b0);
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
      const int it = td.a_item[b0 + i], sl = td.a_slot[b0 + i];
      const float4 dl = td.slot_delta[(size_t)it * td.smax + sl];
      float sn, cs_;
      sincosf((float)(q[0] * dl.x + q[1] * dl.y + q[2] * dl.z), &sn, &cs_);
      ph[i] = make_float2(cs_, sn);
      so[i] = td.it_poff[it] + (long long)sl * nlm * 128;
    }
    __syncthreads();
    for (int i = 0; i < nb; i += 4) {
      float re[4], im[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        re[j] = im[j] = 0.f;
        if (i + j < nb) {
          const float* src = base + so[i + j];
          re[j] = src[0];
          im[j] = src[64];
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (i + j < nb) {
          acc.x += re[j] * ph[i + j].x - im[j] * ph[i + j].y;
          acc.y += re[j] * ph[i + j].y + im[j] * ph[i + j].x;
        }
    }
  }
  cs[t][p] = make_float2(acc.x * dV, acc.y * dV);
  __syncthreads();
  const int comp = comp0 + t;
  if (comp >= comps_per_k) return;
  const int sp = comp >> 1, sig = comp & 1;     // spinor within k, spin component
  const int pair = t & ~1;                      // the spinor's two components in cs
  const size_t kb = (size_t)k * nstates + sp;
  const int M = 2 * nlm;
  const float* D = Dmat + (size_t)a * M * M * 2;
  const int row = 2 * p + sig;
  float re = 0.f, im = 0.f;
  for (int u = 0; u < M; ++u) {
    const float2 cu = cs[pair + (u & 1)][u >> 1];
    const float dr = D[(row * M + u) * 2], di = D[(row * M + u) * 2 + 1];
    re += dr * cu.x - di * cu.y;
    im += dr * cu.y + di * cu.x;
  }
  const size_t o = (kb * natoms + a) * M + row;
  c_out[o] = cs[t][p];
  dc_out[o] = make_float2(re, im);
}

// ============================================================================ scatter

// CTA (kg, brick): SC components (X, the B operand, resident) against the brick's points in
// tiles of 128 (the A operand, streamed).  AK < 0: out = exp(-i q.(r - r_b)) (beta^T X) at every
// point of a brick with projectors (the points of other bricks are never written and keep their
// zeros).  AK >= 0: the drain runs the Chebyshev epilogue of every point of the brick itself
// (kinetic part from io.kin, V_NL from the tensor memory, the 2x2 local potential, T_{k+1} and the
// accumulators) with the arithmetic of k_epilogue, so V_NL never crosses HBM; bricks without
// projectors take the same path with V_NL = 0.  AK as in k_epilogue: 0 no accumulator, 1 and 2
// real coefficients on one or both, 3 complex coefficients with run-time flags.
//
// Bound by HBM as long as enough loads are in flight: one CTA holds the SM (its 512
// tensor-memory columns), so 16 worker warps drain it, four to each lane quarter of the tensor
// memory, inputs are requested before the wait for the tile's products, and the projector table
// and the next tiles' rows (into L2) are on their way while X is built.
// At the large supercell with 128 spinors the mean launch went from 2676 us (3.2 TB/s, 8 warps,
// complex coefficients) to 1927 us (4.5 TB/s).
constexpr int ST_WARPS = 16;                  // worker warps
constexpr int ST_NT = 32 * (ST_WARPS + 3);    // + MMA warp + copy warp + prefetch warp
constexpr int ST_MMA_WARP = ST_WARPS, ST_COPY_WARP = ST_WARPS + 1, ST_PF_WARP = ST_WARPS + 2;

__device__ __forceinline__ void prefetch_l2_line(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

template <int EK, int TERMS, int AK>
__global__ void __launch_bounds__(ST_NT, 1)
k_tile_scatter(float2* out, int N, int comps_per_k, int sgroups, int nstates, int natoms, TileDev td, EpiParams ep,
               const float2* dc, int* err, EpiIO io) {
  constexpr int EPR = PT_ROWB / Elt<EK>::bytes;    // projector indices per K chunk
  constexpr int SC = (Elt<EK>::bytes == 4) ? 32 : 64;  // components per CTA
  constexpr int NPART = (TERMS == 3) ? 2 : 1;
  constexpr int XPART = 2 * SC * PT_ROWB;          // one K chunk of X (2 SC rows)
  constexpr int STAGE = NPART * PT_PART;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  __shared__ uint64_t bar_full[2], bar_empty[2], bar_accf[2], bar_acce[2], bar_x, bar_fin;
  __shared__ volatile int progress;  // tile the first drain warp is at (paces the prefetches)
  __shared__ uint32_t tmem_base;
  __shared__ volatile int abort_flag;
  __shared__ float2 px[32], py[8], pz[8];
  __shared__ float2 sph[256];  // exp(-i q.delta) per slot (at most 256 / nlm slots)

  if (*reinterpret_cast<volatile int*>(err) & 1) {
    pdl_wait();  // a launch never ends before its predecessor
    return;
  }
  const int kg = blockIdx.x, it = blockIdx.y;
  const int k = kg / sgroups, comp0 = (kg % sgroups) * SC;
  const int nslot = td.it_nslot[it], kch = td.it_kch[it];
  if (AK < 0 && nslot == 0) {  // nothing to add at this brick
    pdl_wait();
    return;
  }
  const bool has_nl = nslot > 0;
  const int BX = td.BX;
  const int brick = td.it_brick[it];
  const int bx = brick % td.nbx, by = (brick / td.nbx) % td.nby, bz = brick / (td.nbx * td.nby);
  const int x0 = bx * BX, y0 = by * 8, z0 = bz * 8;
  // this CTA's share of the brick's tiles (gridDim.z shares): t0 + 0 .. ntile - 1
  const int t0 = (BX * 64 / 128) / gridDim.z * blockIdx.z, ntile = (BX * 64 / 128) / gridDim.z;
  const size_t N3 = (size_t)N * N * N;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nlm = td.nlm;
  unsigned char* X = smem;                                          // [kch][NPART][XPART]
  unsigned char* A = smem + (size_t)kch * NPART * XPART;             // [2][NPART][PT_PART]
  auto xpart = [&](int kc, int q) { return X + ((size_t)kc * NPART + q) * XPART; };
  auto apart = [&](int s, int q) { return A + (size_t)s * STAGE + (size_t)q * PT_PART; };

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < 2; ++s) {
      bar_init(sm_addr(&bar_full[s]), 1);
      bar_init(sm_addr(&bar_empty[s]), 1);
      bar_init(sm_addr(&bar_accf[s]), 1);
      bar_init(sm_addr(&bar_acce[s]), 32 * ST_WARPS);
    }
    bar_init(sm_addr(&bar_x), 32 * ST_WARPS);
    bar_init(sm_addr(&bar_fin), 1);
    progress = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  phase_tables(px, py, pz, BX, td, ep.shift[k]);
  const double* q = ep.shift[k];
  for (int s = threadIdx.x; s < nslot; s += blockDim.x) {
    const float4 dl = td.slot_delta[(size_t)it * td.smax + s];
    float sn, c;
    sincosf((float)(q[0] * dl.x + q[1] * dl.y + q[2] * dl.z), &sn, &c);
    sph[s] = make_float2(c, -sn);
  }
  // tensor memory: two accumulators of 2 SC columns (tiles alternate); with three products the
  // hi x lo and lo x hi products go to a second pair at column 256, so the rounding of the tensor
  // cores' accumulation (biased toward zero) sees a third of the MMAs at full magnitude
  constexpr uint32_t TMEM_COLS = (TERMS == 3) ? 512u : 256u;
  if (warp == ST_MMA_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sm_addr(&tmem_base)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base;

  // ---- X: rows cl (re) and SC + cl (im), K element j = slot * nlm + p.  One 16-byte load of D c
  // gives both spin components of one spinor at one projector (index 2 p + sigma).
  if (warp < ST_WARPS) {
    const int tid = threadIdx.x;
    pdl_wait();
    constexpr int SPG = SC / 2;                    // spinors per CTA
    const int total = nslot * SPG * nlm;
    const float4* dc4 = reinterpret_cast<const float4*>(dc);
    for (int b0 = 0; b0 < total; b0 += 4 * 32 * ST_WARPS) {
      float4 f[4];
      int ee[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = b0 + u * 32 * ST_WARPS + tid;
        ee[u] = e;
        f[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (e < total) {
          const int p = e % nlm, sp = (e / nlm) % SPG, sl = e / (nlm * SPG);
          const int comp = comp0 + 2 * sp;
          if (comp < comps_per_k) {
            const int a = td.slot_atom[(size_t)it * td.smax + sl];
            const size_t kb = (size_t)k * nstates + (comp >> 1);
            f[u] = dc4[(kb * natoms + a) * nlm + p];
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = ee[u];
        if (e >= total) continue;
        const int p = e % nlm, sp = (e / nlm) % SPG, sl = e / (nlm * SPG);
        const int j = sl * nlm + p, kc = j / EPR, el = j % EPR;
        const float2 x0v = cm(make_float2(f[u].x, f[u].y), sph[sl]);
        const float2 x1v = cm(make_float2(f[u].z, f[u].w), sph[sl]);
        const float vals[4] = {x0v.x, x0v.y, x1v.x, x1v.y};
        const int rows[4] = {2 * sp, SC + 2 * sp, 2 * sp + 1, SC + 2 * sp + 1};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          uint32_t hi, lo;
          Split<EK>::two(vals[r], hi, lo);
          put<EK>(xpart(kc, 0), rows[r], el, hi);
          if constexpr (TERMS == 3) put<EK>(xpart(kc, 1), rows[r], el, lo);
        }
      }
    }
    // padding of the last K chunk
    const int j0 = nslot * nlm, pad = kch * EPR - j0;
    for (int i = tid; i < pad * 2 * SC; i += 32 * ST_WARPS) {
      const int row = i % (2 * SC), j = j0 + i / (2 * SC);
      put<EK>(xpart(j / EPR, 0), row, j % EPR, 0u);
      if constexpr (TERMS == 3) put<EK>(xpart(j / EPR, 1), row, j % EPR, 0u);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    pt_arrive(sm_addr(&bar_x));
  }

  const int nchunk = ntile * kch;
  if (warp == ST_COPY_WARP) {
    if (lane == 0 && has_nl) {
      const unsigned char* src = td.s_tab + td.it_soff[it] + (size_t)t0 * kch * NPART * PT_PART;
      int issued = 0;
      for (int j = 0; j < nchunk; ++j) {
        const int s = j & 1;
        if (j >= 2 && !pt_wait(sm_addr(&bar_empty[s]), ((j >> 1) - 1) & 1)) abort_flag = 1;
        if (abort_flag) break;
        bulk_expect(sm_addr(&bar_full[s]), NPART * PT_PART);
        for (int qq = 0; qq < NPART; ++qq)
          bulk_copy(apart(s, qq), src + ((size_t)j * NPART + qq) * PT_PART, PT_PART, sm_addr(&bar_full[s]));
        issued = j + 1;
      }
      for (int j = (issued > 2 ? issued - 2 : 0); j < issued; ++j)
        if (!pt_wait(sm_addr(&bar_full[j & 1]), (j >> 1) & 1)) atomicOr(err, 1);
    }
  } else if (warp == ST_MMA_WARP) {
    if (lane == 0 && has_nl) {
      const uint32_t id = idesc<EK>(2 * SC);
      if (!pt_wait(sm_addr(&bar_x), 0)) abort_flag = 1;
      for (int t = 0; t < ntile && !abort_flag; ++t) {
        const int acc = t & 1;
        if (t >= 2 && !pt_wait(sm_addr(&bar_acce[acc]), ((t >> 1) - 1) & 1)) { abort_flag = 1; break; }
        const uint32_t dtm = tmem + (uint32_t)(acc * 2 * SC), dlo = dtm + 256u;
        for (int kc = 0; kc < kch; ++kc) {
          const int j = t * kch + kc, s = j & 1;
          if (!pt_wait(sm_addr(&bar_full[s]), (j >> 1) & 1)) { abort_flag = 1; break; }
          asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) {
            const uint32_t off = (uint32_t)ks * 32;
            const uint64_t ah = desc_sw128(sm_addr(apart(s, 0)) + off), bh = desc_sw128(sm_addr(xpart(kc, 0)) + off);
            mma<EK>(dtm, ah, bh, id, (kc | ks) ? 1u : 0u);
            if constexpr (TERMS == 3) {
              const uint64_t al = desc_sw128(sm_addr(apart(s, 1)) + off), bl = desc_sw128(sm_addr(xpart(kc, 1)) + off);
              mma<EK>(dlo, ah, bl, id, (kc | ks) ? 1u : 0u);
              mma<EK>(dlo, al, bh, id, 1u);
            }
          }
          mma_commit(sm_addr(&bar_empty[s]));
        }
        if (abort_flag) break;
        mma_commit(sm_addr(&bar_accf[acc]));
      }
      // every MMA issued has completed before the tensor memory is released
      mma_commit(sm_addr(&bar_fin));
      if (!pt_wait(sm_addr(&bar_fin), 0)) atomicOr(err, 1);
    }
  } else if (warp == ST_PF_WARP) {
    if constexpr (AK == 0 || AK == 1) {
      // ---- the spinor rows of the tiles ahead of the drain, into L2: two tiles before the X build has
      // finished, then one tile ahead.  The drain's loads then wait for L2 and not for HBM, and HBM is
      // busy while the CTA starts.  Only a pace: nothing waits for this warp.  (With both accumulators
      // the rows of two tiles of every SM no longer stay in L2, and the form is faster without.)
      const bool rec = ep.mode == EPI_RECUR;
      const float2* arr[4] = {io.Tk, io.kin, rec ? io.Tkm1 : nullptr, AK == 1 && !ep.init1 ? io.acc1 : nullptr};
      // one 128-byte line (16 points) per lane; a row of BX points is one or two lines
      const int lpr = BX / 16, lines = 8;  // lines per row, lines per tile and component
      pdl_wait();
      const int total = min(SC, comps_per_k - comp0) * lines;
      for (int t = 0; t < ntile; ++t) {
        for (int poll = 0; poll < (1 << 14) && progress < t - 1 && !abort_flag; ++poll) __nanosleep(200);
        for (int i = lane; i < total; i += 32) {
          const int comp = i >> 3, l = i & 7, row = (t0 + t) * (lines / lpr) + l / lpr;
          const size_t o = ((size_t)k * comps_per_k + comp0 + comp) * N3 +
                           ((size_t)(z0 + (row >> 3)) * N + (y0 + (row & 7))) * N + x0 + (l % lpr) * 16;
#pragma unroll
          for (int a = 0; a < 4; ++a)
            if (arr[a]) prefetch_l2_line(arr[a] + o);
        }
      }
    }
  } else {
    // ---- drain: thread = point of the tile (lane quarter of the warp); the four warps of a
    // quarter take a fourth of the components each, eight (four spinors) at a time;
    // V_NL = exp(-i q.(r - r_b)) (re + i im)
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;
    const int cbeg = (warp >> 2) * (SC / 4), cend = cbeg + SC / 4;
    // epilogue constants (Chebyshev term k: T_{k+1} = f (H - c) T_k / Delta - T_{k-1}, f = 1 or 2)
    const bool rec = ep.mode == EPI_RECUR;
    const bool use1 = AK >= 1 && ep.use_acc1, use2 = AK >= 2 && ep.use_acc2;
    const bool ld1 = use1 && !ep.init1, ld2 = use2 && !ep.init2;
    // Without accumulators a step takes four spinors, requested together (the first of a tile before
    // the wait for its products).  The accumulator forms have registers for two: their steps take
    // one, and the inputs of the next step, over the end of the tile, are requested before this one
    // is computed (two register sets; a pair of steps reads its V_NL together).  At 48^3 x 1024
    // spinors: 1.40 ms without accumulators (1.56 ms in the paired form), 3.45 ms with two
    // (3.76 ms two at a time).
    constexpr bool PAIRED = AK >= 1;
    constexpr int NB = PAIRED ? 1 : 4;
    constexpr int W = PAIRED ? 4 : 8;  // components whose V_NL is read together
    const float2 z2 = make_float2(0.f, 0.f);
    struct In {
      float2 pu[NB], pd[NB], ku[NB], kd[NB], qu[NB], qd[NB], au[NB], ad[NB], bu[NB], bd[NB];
    } in0, in1;
    auto point = [&](int t) -> size_t {
      const int p = (t0 + t) * 128 + row;
      const int lx = p % BX, ly = (p / BX) & 7, lz = p / (BX * 8);
      return ((size_t)(z0 + lz) * N + (y0 + ly)) * N + (x0 + lx);
    };
    const size_t group = ((size_t)k * comps_per_k + comp0) * N3;
    // every input of NB spinors from component cu0 on, at point idx
    auto load = [&](In& f, size_t idx, int cu0) {
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        const int cu = cu0 + 2 * j;
        f.pu[j] = f.pd[j] = f.ku[j] = f.kd[j] = f.qu[j] = f.qd[j] = f.au[j] = f.ad[j] = f.bu[j] = f.bd[j] = z2;
        if (comp0 + cu < comps_per_k) {
          const size_t ou = group + idx + (size_t)cu * N3, od = ou + N3;
          f.pu[j] = io.Tk[ou]; f.pd[j] = io.Tk[od];
          f.ku[j] = io.kin[ou]; f.kd[j] = io.kin[od];
          if (rec) { f.qu[j] = io.Tkm1[ou]; f.qd[j] = io.Tkm1[od]; }
          if (ld1) { f.au[j] = io.acc1[ou]; f.ad[j] = io.acc1[od]; }
          if (ld2) { f.bu[j] = io.acc2[ou]; f.bd[j] = io.acc2[od]; }
        }
      }
    };
    auto load_v = [&](size_t idx) { return make_float4(io.V[idx], io.V[N3 + idx], io.V[2 * N3 + idx], io.V[3 * N3 + idx]); };
    float4 vn = make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (PAIRED) {
      load(in0, point(0), cbeg);
      vn = load_v(point(0));
    }
    for (int t = 0; t < ntile; ++t) {
      const int acc = t & 1;
      if (AK >= 0 && threadIdx.x == 0) progress = t;
      const int p = (t0 + t) * 128 + row;
      const int lx = p % BX, ly = (p / BX) & 7, lz = p / (BX * 8);
      const size_t idx = point(t);
      const uint32_t tb = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * 2 * SC);
      const size_t base = group + idx;  // component comp0 at this point
      if constexpr (AK == 0) {
        load(in0, idx, cbeg);
        vn = load_v(idx);
      }
      const float V0 = vn.x, V1 = vn.y, hx = 0.5f * vn.z, hy = 0.5f * vn.w;
      const float2 ph = cm(cm(px[lx], py[ly]), pz[lz]);
      const float2 phc = make_float2(ph.x, -ph.y);
      // one step: the Chebyshev epilogue of spinor components cu0 .. at this point, V_NL in re, im
      auto step = [&](const In& f, int cu0, const float* re, const float* im) {
#pragma unroll
        for (int j = 0; j < NB; ++j) {
          const int cu = cu0 + 2 * j;
          if (comp0 + cu >= comps_per_k) continue;
          const size_t ou = base + (size_t)cu * N3, od = ou + N3;
          const float2 vu = cm(make_float2(re[2 * j], im[2 * j]), phc);
          const float2 vd = cm(make_float2(re[2 * j + 1], im[2 * j + 1]), phc);
          float2 hu = make_float2(f.ku[j].x + vu.x, f.ku[j].y + vu.y);
          float2 hd = make_float2(f.kd[j].x + vd.x, f.kd[j].y + vd.y);
          const float2 u = f.pu[j], d = f.pd[j], qu = f.qu[j], qd = f.qd[j];
          hu = make_float2(hu.x + V0 * u.x + hx * d.x - hy * d.y, hu.y + V0 * u.y + hx * d.y + hy * d.x);
          hd = make_float2(hd.x + V1 * d.x + hx * u.x + hy * u.y, hd.y + V1 * d.y + hx * u.y - hy * u.x);
          // the series constants as float pairs (split_constants); T_1 without the factor 2 and
          // without T_{-1} (zero here)
          const float c2 = rec ? 2.f : 1.f;
          const float2 tu = make_float2(c2 * shifted_f(hu.x, u.x, ep.f_c, ep.f_id) - qu.x,
                                        c2 * shifted_f(hu.y, u.y, ep.f_c, ep.f_id) - qu.y);
          const float2 td = make_float2(c2 * shifted_f(hd.x, d.x, ep.f_c, ep.f_id) - qd.x,
                                        c2 * shifted_f(hd.y, d.y, ep.f_c, ep.f_id) - qd.y);
          io.Tout[ou] = tu;
          io.Tout[od] = td;
          // accumulators: up to three terms (T_{k-1}, T_k, T_{k+1}) at once in float-float
          // arithmetic, rounded once, as in k_epilogue
          auto upd = [&](float2* accp, int init, int fin, float2 xu, float2 xd, const float* cmf, const float* c0f,
                         const float* c1f, const float* rf, const float* phf) {
            if (init) xu = xd = z2;
            float2 lu = z2, ld = z2;
            if constexpr (AK < 3) {
              const bool odd = ep.odd;
              ff_rmadd(xu, lu, tu, rf + 4, !odd);
              ff_rmadd(xd, ld, td, rf + 4, !odd);
              ff_rmadd(xu, lu, u, rf + 2, odd);
              ff_rmadd(xd, ld, d, rf + 2, odd);
              if (rec) {
                ff_rmadd(xu, lu, qu, rf, !odd);
                ff_rmadd(xd, ld, qd, rf, !odd);
              }
              if (fin) {
                accp[ou] = ff_phase(xu, lu, phf);
                accp[od] = ff_phase(xd, ld, phf);
                return;
              }
            } else {
              ff_cmadd(xu, lu, tu, c1f);
              ff_cmadd(xd, ld, td, c1f);
              ff_cmadd(xu, lu, u, c0f);
              ff_cmadd(xd, ld, d, c0f);
              if (rec) {
                ff_cmadd(xu, lu, qu, cmf);
                ff_cmadd(xd, ld, qd, cmf);
              }
            }
            accp[ou] = make_float2(xu.x + lu.x, xu.y + lu.y);
            accp[od] = make_float2(xd.x + ld.x, xd.y + ld.y);
          };
          if (use1) upd(io.acc1, ep.init1, ep.fin1, f.au[j], f.ad[j], ep.f_am, ep.f_a0, ep.f_a1, ep.f_ra, ep.f_ph1);
          if (use2) upd(io.acc2, ep.init2, ep.fin2, f.bu[j], f.bd[j], ep.f_bm, ep.f_b0, ep.f_b1, ep.f_rb, ep.f_ph2);
        }
      };
      if (has_nl) {
        if (!pt_wait(sm_addr(&bar_accf[acc]), (t >> 1) & 1)) abort_flag = 1;
        if (__any_sync(0xffffffffu, abort_flag != 0)) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
      }
#pragma unroll 1
      for (int c0 = cbeg; c0 < cend; c0 += W) {
        if constexpr (PAIRED) load(in1, idx, c0 + W / 2);
        float re[W], im[W];
        if (has_nl) {
          auto part = [&](uint32_t col, float* o) {
            uint32_t h[W];
            tmem_ld_async<W>(tb + col, h);
            if constexpr (TERMS == 3) {
              uint32_t l[W];
              tmem_ld_async<W>(tb + 256u + col, l);
              tmem_wait_ld();
              tmem_regs_ready_n<W>(h);
              tmem_regs_ready_n<W>(l);
#pragma unroll
              for (int j = 0; j < W; ++j) o[j] = __uint_as_float(h[j]) + __uint_as_float(l[j]);
            } else {
              tmem_wait_ld();
              tmem_regs_ready_n<W>(h);
#pragma unroll
              for (int j = 0; j < W; ++j) o[j] = __uint_as_float(h[j]);
            }
          };
          part((uint32_t)c0, re);
          part((uint32_t)(SC + c0), im);
          if (c0 + W >= cend) {
            asm volatile("tcgen05.fence::before_thread_sync;");
            pt_arrive(sm_addr(&bar_acce[acc]));
          }
        } else {
#pragma unroll
          for (int j = 0; j < W; ++j) re[j] = im[j] = 0.f;
        }
        if constexpr (AK < 0) {
#pragma unroll
          for (int j = 0; j < W; ++j)
            if (comp0 + c0 + j < comps_per_k) out[base + (size_t)(c0 + j) * N3] = cm(make_float2(re[j], im[j]), phc);
        } else if constexpr (!PAIRED) {
          if (c0 != cbeg) load(in0, idx, c0);
          step(in0, c0, re, im);
        } else {
          step(in0, c0, re, im);
          if (c0 + W < cend) {
            load(in0, idx, c0 + W);
          } else if (t + 1 < ntile) {
            const size_t nidx = point(t + 1);
            load(in0, nidx, cbeg);
            vn = load_v(nidx);
          }
          step(in1, c0 + W / 2, re + W / 2, im + W / 2);
        }
      }
    }
    if (abort_flag && lane == 0) atomicOr(err, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == ST_MMA_WARP)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
}

// ============================================================================ launchers

// At least 120 KB, so that one CTA (holding all 512 tensor-memory columns) runs per SM.
size_t tile_gather_smem(int terms) {
  const size_t need = (size_t)((terms == 3) ? 2 : 1) * (PT_PART + 256 * PT_ROWB) * 2 + 1024;
  return need > 120 * 1024 ? need : 120 * 1024;
}
// With three products, at least 120 KB, so that one CTA (holding all 512 tensor-memory columns)
// runs per SM.
size_t tile_scatter_smem(int ek, int terms, int kch_max) {
  const int sc = (ek == TILE_TF32) ? 32 : 64;
  const size_t np = (terms == 3) ? 2 : 1;
  const size_t need = (size_t)kch_max * np * 2 * sc * PT_ROWB + 2 * np * PT_PART + 1024;
  return (terms == 3 && need < 120 * 1024) ? 120 * 1024 : need;
}

template <int EK, int TERMS>
static cudaError_t gather_et(cudaStream_t st, int N, const void* psi, int nk, int nstates, const TileDev& td,
                             double dV, const EpiParams& ep, const float* Dmat, float* part, void* c_out,
                             void* dc_out, int* err) {
  const int comps_per_k = 2 * nstates;
  const int groups = (comps_per_k + 63) / 64;
  const size_t smem = tile_gather_smem(TERMS);
  auto kf = k_tile_gather<EK, TERMS>;
  static std::atomic<unsigned long long> done{0};
  cudaError_t e = opt_in_smem(kf, smem, done);
  if (e != cudaSuccess) return e;
  e = launch_pdl(kf, dim3(nk * groups, td.nitems), PT_NT, smem, st, (const float2*)psi, N, comps_per_k,
                             groups, td, ep, part, err);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_tile_reduce, dim3(td.natoms, nk * groups), 64 * td.nlm, 0, st, part, td, groups, comps_per_k,
                    nstates, td.natoms, (float)dV, ep, Dmat, (float2*)c_out, (float2*)dc_out);
}

template <int EK, int TERMS, int AK>
static cudaError_t scatter_et(cudaStream_t st, int N, void* out, int nk, int nstates, const TileDev& td,
                              const EpiParams& ep, const void* dc, int* err, const EpiIO& io) {
  constexpr int SC = (Elt<EK>::bytes == 4) ? 32 : 64;
  const int comps_per_k = 2 * nstates;
  const int sgroups = (comps_per_k + SC - 1) / SC;
  const size_t smem = tile_scatter_smem(EK, TERMS, td.kch_max);
  if (smem > 224 * 1024) return cudaErrorInvalidConfiguration;
  auto kf = k_tile_scatter<EK, TERMS, AK>;
  static std::atomic<unsigned long long> done{0};
  if (cudaError_t e = opt_in_smem(kf, 224 * 1024, done)) return e;  // any handle's kch_max (at most 193 KB)
  // One CTA runs per SM: with few of them the last wave is a large part of the launch, so a brick's
  // tiles are then shared by two CTAs, each building X for itself.  Up to four waves (152 SMs) of
  // whole bricks two shares are faster (64^3 x 104 spinors, 3.4 waves: 441 -> 412 us per launch); four
  // shares of 1.4 waves are slower than one (48^3 x 27: 80 -> 87 us).
  const int ctas = nk * sgroups * td.nitems;
  const int shares = ctas <= 608 ? 2 : 1;
  return launch_pdl(kf, dim3(nk * sgroups, td.nitems, shares), ST_NT, smem, st, (float2*)out, N, comps_per_k, sgroups, nstates,
                    td.natoms, td, ep, (const float2*)dc, err, io);
}

template <int AK>
static cudaError_t scatter_dispatch(cudaStream_t st, int N, void* out, int nk, int nstates, const TileDev& td,
                                    const EpiParams& ep, const void* dc, int* err, const EpiIO& io) {
  switch (td.ek * 4 + td.terms) {
    case TILE_TF32 * 4 + 1: return scatter_et<TILE_TF32, 1, AK>(st, N, out, nk, nstates, td, ep, dc, err, io);
    case TILE_TF32 * 4 + 3: return scatter_et<TILE_TF32, 3, AK>(st, N, out, nk, nstates, td, ep, dc, err, io);
    case TILE_BF16 * 4 + 3: return scatter_et<TILE_BF16, 3, AK>(st, N, out, nk, nstates, td, ep, dc, err, io);
    case TILE_F16 * 4 + 3: return scatter_et<TILE_F16, 3, AK>(st, N, out, nk, nstates, td, ep, dc, err, io);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_tile_gather(cudaStream_t st, int N, const void* psi, int nk, int nstates, const TileDev& td,
                               double dV, const EpiParams& ep, const float* Dmat, float* part, void* c_out,
                               void* dc_out, int* err) {
  if (td.nitems == 0) return cudaSuccess;
  switch (td.ek * 4 + td.terms) {
    case TILE_TF32 * 4 + 1: return gather_et<TILE_TF32, 1>(st, N, psi, nk, nstates, td, dV, ep, Dmat, part, c_out, dc_out, err);
    case TILE_TF32 * 4 + 3: return gather_et<TILE_TF32, 3>(st, N, psi, nk, nstates, td, dV, ep, Dmat, part, c_out, dc_out, err);
    case TILE_BF16 * 4 + 3: return gather_et<TILE_BF16, 3>(st, N, psi, nk, nstates, td, dV, ep, Dmat, part, c_out, dc_out, err);
    case TILE_F16 * 4 + 3: return gather_et<TILE_F16, 3>(st, N, psi, nk, nstates, td, dV, ep, Dmat, part, c_out, dc_out, err);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_tile_scatter(cudaStream_t st, int N, void* out, int nk, int nstates, const TileDev& td,
                                const EpiParams& ep, const void* dc, int* err) {
  if (td.nitems == 0) return cudaSuccess;
  return scatter_dispatch<-1>(st, N, out, nk, nstates, td, ep, dc, err, EpiIO{});
}

cudaError_t launch_tile_epilogue(cudaStream_t st, int N, int nk, int nstates, const TileDev& td, const EpiParams& ep,
                                 const void* dc, int* err, const EpiIO& io) {
  if (ep.mode != EPI_FIRST && ep.mode != EPI_RECUR) return cudaErrorInvalidValue;
  if (td.nitems == 0) return cudaSuccess;
  EpiParams epx = ep;
  split_constants(epx);
  if (!ep.use_acc1 && !ep.use_acc2) return scatter_dispatch<0>(st, N, nullptr, nk, nstates, td, epx, dc, err, io);
  if (!ep.real_coef) return scatter_dispatch<3>(st, N, nullptr, nk, nstates, td, epx, dc, err, io);
  if (!ep.use_acc2) return scatter_dispatch<1>(st, N, nullptr, nk, nstates, td, epx, dc, err, io);
  return scatter_dispatch<2>(st, N, nullptr, nk, nstates, td, epx, dc, err, io);
}

cudaError_t set_first_wait_tile(unsigned polls) { return cudaMemcpyToSymbol(g_first_wait, &polls, sizeof(polls)); }

}  // namespace tddft
