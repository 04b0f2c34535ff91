// dwf_hop2.cuh -- the tuned hopping pass and the site-local 5th-dimension kernels for
// the even Ls of tuned_ls() (sm_103a).
//
// Work split: one thread per (4D site, pair of 5th-dimension slices s0 = 2t,
// s1 = 2t + 1), G = Ls / 2 threads per site; a CTA of nt threads (a multiple of 32,
// at most 128) takes nt / G sites, and the nt mod G threads left over help with the
// 5th-dimension operators only.
//   * the half-fields store each spinor component of a slice pair as
//     (re s0, re s1, im s0, im s1) (dwf_fields.cuh), so one vector load gives a
//     thread both slices of a component in lane order, and the projection,
//     SU(3) multiply and reconstruction of the two slices run as paired FP32
//     instructions (FFMA2 / FADD2 / FMUL2 of sm_100+, one link entry feeding
//     both lanes); FP64 runs the same code on scalar lanes;
//   * one link load and one neighbour-table entry serve both slices; the
//     boundary sign of a hop (and the per-site scale of 16-bit storage) rides
//     on the FMAs of the reconstruction;
//   * the B pre-multiplication of D_bb pass A (cyclic bidiagonal per chirality,
//     Eq. mobius1 with D_w -> 1) is applied to the neighbour spinor before the
//     projection: (B v)+(s) = d+ v+(s) + o+ v+(s-1), (B v)-(s) = d- v-(s) + o- v-(s+1).
//     v+ of the pair below and v- of the pair above come from the registers of the
//     neighbouring threads by shuffles: a warp then takes 32 / G whole sites (FP16,
//     24^3x48, Ls = 12: pass A 343 us, 411 with the pairs loaded in addition);
//   * the 5th-dimension post operators (I^-1, K = B I^-1, K^T, B^T) run as
//     O(Ls) recurrences on register-resident chains after a transpose through
//     shared memory: every cyclic bidiagonal matrix of the construction, put in
//     "lower" form by reversing the slice order where needed, is either
//     multiplied (y_k = a_k v_k + b_k v_{k-1}) or solved with one forward sweep
//     for the unknown first element and one back-substitution sweep.
#pragma once

#include <algorithm>
#include <atomic>
#include <cstdlib>

#include <cudaTypedefs.h>

#include "dwf_fields.cuh"

namespace dwf {
namespace hop2 {

// Chain coefficient block: [op][chirality][kChainStride(Ls)] in the compute type,
// op = 0 B (mult), 1 B^T (mult), 2 I (mult), 3 I (solve), 4 I^T (solve).  Step k of
// a sweep (lower form, sweep order) reads one 4-vector at 4k:
// mult:  (diagonal, off-diagonal, 0, 0)
// solve: (1/D_k, O_k/D_k, beta_k, 0); then (G, O_0, 0, 0) at 4 Ls.
enum { OP_B = 0, OP_BT = 1, OP_I = 2, OP_ISOLVE = 3, OP_ITSOLVE = 4, NOPS = 5 };
__host__ __device__ constexpr int chain_stride(int Ls) { return 4 * Ls + 4; }
__host__ __device__ constexpr int chain_block(int Ls) { return NOPS * 2 * chain_stride(Ls); }
// op is transposed -> reversed sweep order for chirality 0, else for chirality 1
__host__ __device__ constexpr bool op_transposed(int op) { return op == OP_BT || op == OP_ITSOLVE; }

// Programs (sequence of ops) used as post / local operators.
enum { PR_NONE = 0, PR_K = 1, PR_IINV = 2, PR_KT = 3, PR_BT = 4, PR_I = 5, PR_ITINV = 6, PR_B = 7 };
__host__ __device__ constexpr int prog_len(int p) { return p == PR_K || p == PR_KT ? 2 : (p ? 1 : 0); }
__host__ __device__ constexpr int prog_op(int p, int i) {
  return p == PR_K ? (i == 0 ? OP_ISOLVE : OP_B)
       : p == PR_IINV ? OP_ISOLVE
       : p == PR_KT ? (i == 0 ? OP_BT : OP_ITSOLVE)
       : p == PR_BT ? OP_BT
       : p == PR_I ? OP_I
       : p == PR_ITINV ? OP_ITSOLVE
       : p == PR_B ? OP_B : -1;
}
// elements of the coefficients of a program's ops, in the order of its ops
__host__ __device__ constexpr int prog_coefs(int Ls, int p) { return prog_len(p) * 2 * chain_stride(Ls); }
__host__ __device__ constexpr bool op_is_solve(int op) { return op == OP_ISOLVE || op == OP_ITSOLVE; }

// Shared-memory layout of one 4D site for the 5th-dimension programs, per chirality in
// the sweep order of the program (the slices of a chirality whose sweep is reversed are
// stored last slice first): slices 2k, 2k + 1 of the sweep at k * kPairStride, real
// component R = 2c + (0 re | 1 im) at 2R as (even slice, odd slice).  A sweep then
// reads two slices of a component by one 8-byte (FP64: 16-byte) access at constant
// offsets.  52 = 20 mod 32 spreads the 16-byte stores of a quarter warp over the banks
// (two-way conflicts at G = 3, 4, 5), and sites 24 = 12 * 2 words apart modulo 32 make the
// accesses of consecutive sweeps (12 of a chirality per site) conflict-free.
constexpr int kPairStride = 52;
__host__ __device__ constexpr int site_stride(int Ls) {
  return (Ls / 2) * kPairStride + ((24 - ((Ls / 2) * kPairStride) % 32) + 32) % 32;
}

// ---------------------------------------------------------------------------
// Lane-pair arithmetic: lane x = slice s0, lane y = slice s1.
// ---------------------------------------------------------------------------
template <typename T>
struct Pr;
template <>
struct Pr<float> {
  using V = float2;
  static __device__ __forceinline__ V fma(V a, V b, V c) { return __ffma2_rn(a, b, c); }
  static __device__ __forceinline__ V mul(V a, V b) { return __fmul2_rn(a, b); }
  static __device__ __forceinline__ V add(V a, V b) { return __fadd2_rn(a, b); }
  static __device__ __forceinline__ V sub(V a, V b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
  static __device__ __forceinline__ V neg(V a) { return make_float2(-a.x, -a.y); }
  static __device__ __forceinline__ V dup(float v) { return make_float2(v, v); }
  static __device__ __forceinline__ V mk(float x, float y) { return make_float2(x, y); }
};
template <>
struct Pr<double> {
  using V = double2;
  static __device__ __forceinline__ V fma(V a, V b, V c) {
    return make_double2(::fma(a.x, b.x, c.x), ::fma(a.y, b.y, c.y));
  }
  static __device__ __forceinline__ V mul(V a, V b) { return make_double2(a.x * b.x, a.y * b.y); }
  static __device__ __forceinline__ V add(V a, V b) { return make_double2(a.x + b.x, a.y + b.y); }
  static __device__ __forceinline__ V sub(V a, V b) { return make_double2(a.x - b.x, a.y - b.y); }
  static __device__ __forceinline__ V neg(V a) { return make_double2(-a.x, -a.y); }
  static __device__ __forceinline__ V dup(double v) { return make_double2(v, v); }
  static __device__ __forceinline__ V mk(double x, double y) { return make_double2(x, y); }
};

// 6 complex lane pairs: one chirality (2 spins x 3 colours), index spin * 3 + colour
template <typename V>
struct HalfP {
  V re[6], im[6];
};
// 12 complex lane pairs: a full spinor for the two slices
template <typename V>
struct SpinP {
  V re[12], im[12];
};

// ---------------------------------------------------------------------------
// Pair access to the half-field layouts of dwf_fields.cuh (pair m, NP pairs).
// load6: components c0 .. c0 + 5 (c0 = 0: P_+ spins, 6: P_- spins), unscaled.
// Ordinary loads (see load_pair there): these kernels may start ahead of the end of the one before.
// ---------------------------------------------------------------------------
template <class SP>
struct PairIO;

template <>
struct PairIO<Store32> {
  using V = float2;
  static __device__ __forceinline__ void load6(const void* base, size_t m, size_t NP, int c0, V* re,
                                               V* im) {
    const float4* p = reinterpret_cast<const float4*>(base) + (size_t)c0 * NP + m;
#pragma unroll
    for (int k = 0; k < 6; k++) {
      const float4 v = p[(size_t)k * NP];
      re[k] = make_float2(v.x, v.y);
      im[k] = make_float2(v.z, v.w);
    }
  }
  static __device__ __forceinline__ V scale(const void*, size_t, size_t) { return make_float2(1.f, 1.f); }
  static __device__ __forceinline__ void quantize(SpinP<V>&) {}
  static __device__ __forceinline__ void store(void* base, size_t m, size_t NP, const SpinP<V>& a) {
    float4* p = reinterpret_cast<float4*>(base) + m;
#pragma unroll
    for (int c = 0; c < 12; c++)
      p[(size_t)c * NP] = make_float4(a.re[c].x, a.re[c].y, a.im[c].x, a.im[c].y);
  }
};

template <>
struct PairIO<Store64> {
  using V = double2;
  static __device__ __forceinline__ void load6(const void* base, size_t m, size_t NP, int c0, V* re,
                                               V* im) {
    const double2* p = reinterpret_cast<const double2*>(base) + ((size_t)c0 * NP + m) * 2;
#pragma unroll
    for (int k = 0; k < 6; k++) {
      re[k] = p[(size_t)k * NP * 2];
      im[k] = p[(size_t)k * NP * 2 + 1];
    }
  }
  static __device__ __forceinline__ V scale(const void*, size_t, size_t) { return make_double2(1.0, 1.0); }
  static __device__ __forceinline__ void quantize(SpinP<V>&) {}
  static __device__ __forceinline__ void store(void* base, size_t m, size_t NP, const SpinP<V>& a) {
    double2* p = reinterpret_cast<double2*>(base) + m * 2;
#pragma unroll
    for (int c = 0; c < 12; c++) {
      p[(size_t)c * NP * 2] = a.re[c];
      p[(size_t)c * NP * 2 + 1] = a.im[c];
    }
  }
};

template <bool BF>
struct PairIO<Store16<BF>> {
  using V = float2;
  using S = Store16<BF>;
  static __device__ __forceinline__ void load6(const void* base, size_t m, size_t NP, int c0, V* re,
                                               V* im) {
    const uint4* p = reinterpret_cast<const uint4*>(base) + (size_t)(c0 >> 1) * NP + m;
#pragma unroll
    for (int j = 0; j < 3; j++) {
      const uint4 v = p[(size_t)j * NP];
      re[2 * j] = S::to_f2(v.x);
      im[2 * j] = S::to_f2(v.y);
      re[2 * j + 1] = S::to_f2(v.z);
      im[2 * j + 1] = S::to_f2(v.w);
    }
  }
  static __device__ __forceinline__ V scale(const void* base, size_t m, size_t NP) {
    return reinterpret_cast<const float2*>(reinterpret_cast<const uint4*>(base) + 6 * NP)[m];
  }
  static __device__ __forceinline__ float2 scales_of(const SpinP<V>& a) {
    float mx = 0.f, my = 0.f;
#pragma unroll
    for (int c = 0; c < 12; c++) {
      mx = fmaxf(mx, fmaxf(fabsf(a.re[c].x), fabsf(a.im[c].x)));
      my = fmaxf(my, fmaxf(fabsf(a.re[c].y), fabsf(a.im[c].y)));
    }
    return make_float2(S::scale_of(mx), S::scale_of(my));
  }
  // a <- what store() followed by a load gives back, in registers (a kernel must
  // not re-read through the non-coherent path what it wrote itself)
  static __device__ __forceinline__ void quantize(SpinP<V>& a) {
    const float2 sc = scales_of(a);
    const float2 inv = make_float2(1.f / sc.x, 1.f / sc.y);
#pragma unroll
    for (int c = 0; c < 12; c++) {
      a.re[c] = __fmul2_rn(S::to_f2(S::from_f2(__fmul2_rn(a.re[c], inv))), sc);
      a.im[c] = __fmul2_rn(S::to_f2(S::from_f2(__fmul2_rn(a.im[c], inv))), sc);
    }
  }
  static __device__ __forceinline__ void store(void* base, size_t m, size_t NP, const SpinP<V>& a) {
    float mx = 0.f, my = 0.f;
#pragma unroll
    for (int c = 0; c < 12; c++) {
      mx = fmaxf(mx, fmaxf(fabsf(a.re[c].x), fabsf(a.im[c].x)));
      my = fmaxf(my, fmaxf(fabsf(a.re[c].y), fabsf(a.im[c].y)));
    }
    const float sx = S::scale_of(mx), sy = S::scale_of(my);
    const float2 inv = make_float2(1.f / sx, 1.f / sy);
    uint4* p = reinterpret_cast<uint4*>(base) + m;
#pragma unroll
    for (int j = 0; j < 6; j++)
      p[(size_t)j * NP] = make_uint4(S::from_f2(__fmul2_rn(a.re[2 * j], inv)),
                                     S::from_f2(__fmul2_rn(a.im[2 * j], inv)),
                                     S::from_f2(__fmul2_rn(a.re[2 * j + 1], inv)),
                                     S::from_f2(__fmul2_rn(a.im[2 * j + 1], inv)));
    reinterpret_cast<float2*>(reinterpret_cast<uint4*>(base) + 6 * NP)[m] = make_float2(sx, sy);
  }
};

// full spinor pair (scaled for 16-bit storage)
template <class SP>
__device__ __forceinline__ void load_spin(const void* base, size_t m, size_t NP,
                                          SpinP<typename Pr<typename SP::T>::V>& a) {
  using IO = PairIO<SP>;
  IO::load6(base, m, NP, 0, a.re, a.im);
  IO::load6(base, m, NP, 6, a.re + 6, a.im + 6);
  if constexpr (SP::kScaled) {
    const float2 sc = IO::scale(base, m, NP);
#pragma unroll
    for (int c = 0; c < 12; c++) {
      a.re[c] = __fmul2_rn(a.re[c], sc);
      a.im[c] = __fmul2_rn(a.im[c], sc);
    }
  }
}

// ---------------------------------------------------------------------------
// Spin structure in the chiral basis: (1 - dir gamma_mu) psi = (h, -dir A^+ h),
// h = psi_+ - dir A psi_-, A_x = -i sigma_1, A_y = -i sigma_2, A_z = -i sigma_3,
// A_t = 1.  Row k of h is P_k + cf (i) M_pk; row k of the lower half is
// rs (i) chi_pk, with pk the partner row and (i) present for x and z.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int partner(int mu, int k) { return mu <= 1 ? 1 - k : k; }
__host__ __device__ constexpr bool imag_mu(int mu) { return mu == 0 || mu == 2; }
__host__ __device__ constexpr int proj_sign(int mu, int dir, int k) {
  return mu == 0 ? dir : (mu == 3 ? -dir : (k == 0 ? dir : -dir));
}
__host__ __device__ constexpr int recon_sign(int mu, int dir, int k) {
  return mu == 0 || mu == 3 ? -dir : (k == 0 ? -dir : dir);
}

template <typename T>
struct Args {
  void* out;
  const void* v;
  const void* w;
  size_t stride;
  const void* gauge_p;
  const void* gauge_q;
  const int4* nbr;      // [Vh][2] int4 of output parity: x+ x- y+ y- | z+ z- t+ t- (bit 31: sign)
  const T* bdiag;       // [2][Ls] B diagonal (PRE_B)
  const T* boff;        // [2][Ls] B off-diagonal (PRE_B)
  const T* chain;       // chain coefficient block (programs)
  T c_hop, c_loc;
  Reduce red;
  size_t cstride;       // elements between right-hand sides of bdiag, boff, chain
  const int* active;    // per right-hand side: 0 skips it (nullptr: all active)
  int* err;             // set to 1 when a bounded wait gives up (staged variant)
  // EX_HAT: out2 = I^-T gamma5 out.  EX_RUPD: r = out2 is updated, r -= a out, a = *num / den
  // (stored to a_out, one per right-hand side sstride apart), and out itself is not stored.
  void* out2;
  const double* num;
  SumIn den;
  double* a_out;
  int sstride;
  bin_t* zero[2];       // bins that the right-hand side's first block sets to zero
};

template <typename T>
__device__ __forceinline__ void zero_bins(const Args<T>& a, int rhs, int tid, int nth) {
  if (blockIdx.x == 0)
#pragma unroll
    for (int i = 0; i < 2; i++)
      if (a.zero[i])
        for (int k = tid; k < kBins; k += nth) a.zero[i][(size_t)rhs * kBins + k] = 0ull;
}

// h = P_+ - dir A P_- in place into P: the half spinor of (1 - DIR gamma_mu).
template <typename T, int MU, int DIR>
__device__ __forceinline__ void project_half(HalfP<typename Pr<T>::V>& P, const HalfP<typename Pr<T>::V>& M) {
  using A = Pr<T>;
  using V = typename A::V;
#pragma unroll
  for (int k = 0; k < 2; k++) {
    const int pk = partner(MU, k);
    const int cs = proj_sign(MU, DIR, k);
#pragma unroll
    for (int a = 0; a < 3; a++) {
      const V pr = P.re[3 * k + a], pi = P.im[3 * k + a];
      const V mr = M.re[3 * pk + a], mi = M.im[3 * pk + a];
      if (imag_mu(MU)) {  // P + cs i M
        P.re[3 * k + a] = cs > 0 ? A::sub(pr, mi) : A::add(pr, mi);
        P.im[3 * k + a] = cs > 0 ? A::add(pi, mr) : A::sub(pi, mr);
      } else {            // P + cs M
        P.re[3 * k + a] = cs > 0 ? A::add(pr, mr) : A::sub(pr, mr);
        P.im[3 * k + a] = cs > 0 ? A::add(pi, mi) : A::sub(pi, mi);
      }
    }
  }
}

// Component a of chi_k = U' h_k for the half spinor h = P; U' = U (dir > 0) or U^+ (dir < 0).
template <typename T, int DIR>
__device__ __forceinline__ void link_row(const HalfP<typename Pr<T>::V>& P, const Link<T>& U, int k, int a,
                                         typename Pr<T>::V& cr, typename Pr<T>::V& ci) {
  using A = Pr<T>;
  using V = typename A::V;
#pragma unroll
  for (int b = 0; b < 3; b++) {
    const cplx<T> u = DIR > 0 ? U.u[3 * a + b] : U.u[3 * b + a];
    const V ur = A::dup(u.re);
    const V ui = A::dup(DIR > 0 ? u.im : -u.im);
    const V hr = P.re[3 * k + b], hi = P.im[3 * k + b];
    if (b == 0) {
      cr = A::mul(ur, hr);
      ci = A::mul(ur, hi);
    } else {
      cr = A::fma(ur, hr, cr);
      ci = A::fma(ur, hi, ci);
    }
    cr = A::fma(A::neg(ui), hi, cr);
    ci = A::fma(ui, hr, ci);
  }
}

// chi_k = U' h_k, acc_upper(k) += f chi_k, acc_lower(pk) += f rs (i) chi_k.
template <class SP, int MU, int DIR>
__device__ __forceinline__ void mul_acc(const HalfP<typename Pr<typename SP::T>::V>& P,
                                        const Link<typename SP::T>& U,
                                        typename Pr<typename SP::T>::V f,
                                        SpinP<typename Pr<typename SP::T>::V>& acc) {
  using T = typename SP::T;
  using A = Pr<T>;
  using V = typename A::V;
  const V fn = A::neg(f);
#pragma unroll
  for (int k = 0; k < 2; k++) {
    const int q = partner(MU, k);  // lower row fed by chi_k
    const int rs = recon_sign(MU, DIR, q);
#pragma unroll
    for (int a = 0; a < 3; a++) {
      V cr, ci;
      link_row<T, DIR>(P, U, k, a, cr, ci);
      acc.re[3 * k + a] = A::fma(f, cr, acc.re[3 * k + a]);
      acc.im[3 * k + a] = A::fma(f, ci, acc.im[3 * k + a]);
      const int l = 6 + 3 * q + a;
      if (imag_mu(MU)) {  // += rs i chi: re -= rs chi_im, im += rs chi_re
        acc.re[l] = A::fma(rs > 0 ? fn : f, ci, acc.re[l]);
        acc.im[l] = A::fma(rs > 0 ? f : fn, cr, acc.im[l]);
      } else {            // += rs chi
        acc.re[l] = A::fma(rs > 0 ? f : fn, cr, acc.re[l]);
        acc.im[l] = A::fma(rs > 0 ? f : fn, ci, acc.im[l]);
      }
    }
  }
}

// 32 / G sites fill a warp.
__host__ __device__ constexpr bool warp_groups(int Ls) { return 32 % (Ls / 2) == 0; }

// v or -v by its sign bit (the FP64 pipe takes no part)
__device__ __forceinline__ float signed_by(bool neg, float v) {
  return __uint_as_float(__float_as_uint(v) ^ (neg ? 0x80000000u : 0u));
}
__device__ __forceinline__ double signed_by(bool neg, double v) {
  return __hiloint2double(__double2hiint(v) ^ (neg ? (int)0x80000000u : 0), __double2loint(v));
}

__device__ __forceinline__ float lane_of(float v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ double lane_of(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }

// Where a hop's neighbour spinor pair, its scale and its link come from.
// Memory: pair m of field v, link mu of half-site hl in the parity's links.
template <class SP>
struct MemSrc {
  using V = typename Pr<typename SP::T>::V;
  const void* v;
  size_t m, NP;
  const void* links;
  int hl;
  __device__ __forceinline__ void load6(int c0, V* re, V* im) const { PairIO<SP>::load6(v, m, NP, c0, re, im); }
  __device__ __forceinline__ V scale() const { return PairIO<SP>::scale(v, m, NP); }
  template <int MU>
  __device__ __forceinline__ void link(Link<typename SP::T>& U) const {
    GaugeOf<SP>::type::load(links, hl, MU, U);
  }
};

// acc += f (1 - dir gamma_mu) U' v'(x +- mu) for the two slices of a thread,
// U' = U_mu(x) (dir > 0) or U_mu(x - mu)^+ (dir < 0).  With PRE_B the G threads of a site
// are neighbouring lanes and every thread of the warp calls it.  With CHI the hop's f chi
// goes to components 0 .. 5 (dir > 0) or 6 .. 11 of acc instead of being added up.
template <class SP, int LS, int PRE, int MU, int DIR, bool CHI, class Src>
__device__ __forceinline__ void hop_from(const Src& src, bool neg, int t, const typename SP::T (&bd)[2][2],
                                         const typename SP::T (&bo)[2][2],
                                         SpinP<typename Pr<typename SP::T>::V>& acc) {
  using T = typename SP::T;
  using A = Pr<T>;
  using V = typename A::V;
  constexpr int HALF = LS / 2;
  HalfP<V> P, M;
  src.load6(0, P.re, P.im);
  src.load6(6, M.re, M.im);
  V f = A::dup(neg ? (T)-1 : (T)1);  // boundary sign of the hop
  if constexpr (PRE == PRE_B) {
    // (B v)+ needs v+(s0 - 1) = lane y of the pair below (cyclic in s),
    // (B v)- needs v-(s1 + 1) = lane x of the pair above.
    const int tb = t == 0 ? HALF - 1 : t - 1, ta = t + 1 == HALF ? 0 : t + 1;
    const int base = (threadIdx.x & 31) - t;
    T a1 = bd[0][0], a2 = bo[0][0], a3 = bd[0][1], a4 = bo[0][1];
    T b1 = bd[1][0], b2 = bo[1][0], b3 = bd[1][1], b4 = bo[1][1];
    if constexpr (SP::kScaled) {
      const V sc = src.scale();
      const T sb = lane_of(sc.y, base + tb), sa = lane_of(sc.x, base + ta);
      a1 *= sc.x; a2 *= sb; a3 *= sc.y; a4 *= sc.x;
      b1 *= sc.x; b2 *= sc.y; b3 *= sc.y; b4 *= sa;
    }
#pragma unroll
    for (int k = 0; k < 6; k++) {
      const T pr = lane_of(P.re[k].y, base + tb), pi = lane_of(P.im[k].y, base + tb);
      const T mr = lane_of(M.re[k].x, base + ta), mi = lane_of(M.im[k].x, base + ta);
      P.re[k] = A::mk(::fma(a2, pr, a1 * P.re[k].x), ::fma(a4, P.re[k].x, a3 * P.re[k].y));
      P.im[k] = A::mk(::fma(a2, pi, a1 * P.im[k].x), ::fma(a4, P.im[k].x, a3 * P.im[k].y));
      M.re[k] = A::mk(::fma(b2, M.re[k].y, b1 * M.re[k].x), ::fma(b4, mr, b3 * M.re[k].y));
      M.im[k] = A::mk(::fma(b2, M.im[k].y, b1 * M.im[k].x), ::fma(b4, mi, b3 * M.im[k].y));
    }
  } else if constexpr (SP::kScaled) {
    f = A::mul(f, src.scale());  // per-slice scale of the neighbour site
  }
  Link<T> U;
  src.template link<MU>(U);
  project_half<T, MU, DIR>(P, M);
  if constexpr (CHI) {
    static_assert(!SP::kScaled, "f is a sign here");
#pragma unroll
    for (int k = 0; k < 2; k++)
#pragma unroll
      for (int a = 0; a < 3; a++) {
        V cr, ci;
        link_row<T, DIR>(P, U, k, a, cr, ci);
        const int c = (DIR > 0 ? 0 : 6) + 3 * k + a;
        acc.re[c] = A::mk(signed_by(neg, cr.x), signed_by(neg, cr.y));
        acc.im[c] = A::mk(signed_by(neg, ci.x), signed_by(neg, ci.y));
      }
  } else {
    mul_acc<SP, MU, DIR>(P, U, f, acc);
  }
}

// The same from memory: neighbour entry nb of site h.
template <class SP, int LS, int PRE, int MU, int DIR, bool CHI = false>
__device__ __forceinline__ void hop_dir(int nb, int h, int t, size_t NP,
                                        const typename SP::T (&bd)[2][2],
                                        const typename SP::T (&bo)[2][2], const void* v,
                                        const void* gp, const void* gq,
                                        SpinP<typename Pr<typename SP::T>::V>& acc) {
  const int hn = nb & 0x7fffffff;
  const MemSrc<SP> src{v, (size_t)hn * (LS / 2) + t, NP, DIR > 0 ? gp : gq, DIR > 0 ? h : hn};
  hop_from<SP, LS, PRE, MU, DIR, CHI>(src, nb < 0, t, bd, bo, acc);
}

// One step's coefficients (4-vector) of a sweep.
template <typename T>
struct Coef4 {
  T a, b, c, d;
};
__device__ __forceinline__ Coef4<float> coef4(const float* p) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  return Coef4<float>{v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ Coef4<double> coef4(const double* p) {
  const double2 v = *reinterpret_cast<const double2*>(p), w = *reinterpret_cast<const double2*>(p + 2);
  return Coef4<double>{v.x, v.y, w.x, w.y};
}

// Lower-form cyclic bidiagonal multiply: y_k = a_k v_k + b_k v_{k-1 mod L}.
template <typename T, int LS, int NIT>
__device__ __forceinline__ void chain_mult(T (&V)[NIT][LS], const T* c) {
  T last[NIT];
#pragma unroll
  for (int q = 0; q < NIT; q++) last[q] = V[q][LS - 1];
#pragma unroll
  for (int k = LS - 1; k >= 1; k--) {
    const Coef4<T> e = coef4(c + 4 * k);
#pragma unroll
    for (int q = 0; q < NIT; q++) V[q][k] = fma(e.b, V[q][k - 1], e.a * V[q][k]);
  }
  const Coef4<T> e = coef4(c);
#pragma unroll
  for (int q = 0; q < NIT; q++) V[q][0] = fma(e.b, last[q], e.a * V[q][0]);
}

// Lower-form cyclic bidiagonal solve D_k y_k + O_k y_{k-1 mod L} = v_k:
// y_k = alpha_k + beta_k t with t = y_0 from the row-0 equation.
template <typename T, int LS, int NIT>
__device__ __forceinline__ void chain_solve(T (&V)[NIT][LS], const T* c) {
  T h0[NIT], prev[NIT];
#pragma unroll
  for (int q = 0; q < NIT; q++) {
    h0[q] = V[q][0];
    prev[q] = (T)0;
  }
#pragma unroll
  for (int k = 1; k < LS; k++) {
    const Coef4<T> e = coef4(c + 4 * k);
#pragma unroll
    for (int q = 0; q < NIT; q++) {
      prev[q] = fma(-e.b, prev[q], e.a * V[q][k]);
      V[q][k] = prev[q];
    }
  }
  const Coef4<T> e = coef4(c + 4 * LS);  // (G, O_0)
#pragma unroll
  for (int q = 0; q < NIT; q++) {
    const T t = fma(-e.b, prev[q], h0[q]) * e.a;
    V[q][0] = t;
    prev[q] = t;
  }
#pragma unroll
  for (int k = 1; k < LS; k++) {
    const T bc = c[4 * k + 2];
#pragma unroll
    for (int q = 0; q < NIT; q++) V[q][k] = fma(bc, prev[q], V[q][k]);
  }
}

// Coefficients of the ops of PROG (both chiralities) into shared memory, 16 bytes at a time.
template <typename T, int LS, int PROG>
__device__ __forceinline__ void load_coefs(T* coef, const T* chain, int tid, int nth) {
  constexpr int n = 2 * chain_stride(LS) * (int)sizeof(T) / 16;
#pragma unroll
  for (int i = 0; i < prog_len(PROG); i++) {
    const uint4* src = reinterpret_cast<const uint4*>(chain + prog_op(PROG, i) * 2 * chain_stride(LS));
    uint4* dst = reinterpret_cast<uint4*>(coef) + i * n;
    for (int k = tid; k < n; k += nth) dst[k] = __ldg(src + k);
  }
}

// Chirality ch of PROG sweeps the slices last to first.
__host__ __device__ constexpr bool prog_reversed(int prog, int ch) {
  return (ch == 1) != op_transposed(prog_op(prog, 0));
}

__device__ __forceinline__ float2 pair_at(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ double2 pair_at(const double* p) { return *reinterpret_cast<const double2*>(p); }

// Run program PROG on the sites of a CTA in shared memory (nsites blocks of
// site_stride(LS)), by nth threads: one half of them takes the sweeps of chirality 0,
// the other those of chirality 1 (12 real components each per site), so that a
// coefficient is one broadcast load for all sweeps of a thread.
template <typename T, int LS, int PROG>
__device__ __forceinline__ void run_prog(T* sbuf, const T* coef, int tid, int nth, int nsites) {
  constexpr int NIT = (48 + LS - 1) / LS;  // sweeps per thread: 24 nsites / nth <= 48 / LS
  constexpr bool EXACT = 48 % LS == 0 && 32 % (LS / 2) == 0;
  const int half = nth >> 1, ch = tid >= half ? 1 : 0;
  T* p[NIT];
  bool ok[NIT];
  T V[NIT][LS];
#pragma unroll
  for (int q = 0; q < NIT; q++) {
    const int i = tid - ch * half + q * half;
    ok[q] = EXACT || i < 12 * nsites;
    const int site = i / 12;
    p[q] = sbuf + site * site_stride(LS) + 24 * ch + 2 * (i - 12 * site);
#pragma unroll
    for (int k = 0; k < LS / 2; k++) {
      if (ok[q]) {
        const auto v = pair_at(p[q] + k * kPairStride);
        V[q][2 * k] = v.x;
        V[q][2 * k + 1] = v.y;
      } else {
        V[q][2 * k] = V[q][2 * k + 1] = (T)0;
      }
    }
  }
#pragma unroll
  for (int i = 0; i < prog_len(PROG); i++) {
    const T* c = coef + (2 * i + ch) * chain_stride(LS);
    if (op_is_solve(prog_op(PROG, i))) chain_solve<T, LS, NIT>(V, c);
    else chain_mult<T, LS, NIT>(V, c);
  }
#pragma unroll
  for (int q = 0; q < NIT; q++)
    if (ok[q]) {
#pragma unroll
      for (int k = 0; k < LS / 2; k++) {
        using V2 = typename Pr<T>::V;
        *reinterpret_cast<V2*>(p[q] + k * kPairStride) = Pr<T>::mk(V[q][2 * k], V[q][2 * k + 1]);
      }
    }
}

// Slice pair t of a site <-> shared memory, in the sweep order of PROG.
__device__ __forceinline__ void put4(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void put4(double* p, double a, double b, double c, double d) {
  reinterpret_cast<double2*>(p)[0] = make_double2(a, b);
  reinterpret_cast<double2*>(p)[1] = make_double2(c, d);
}
template <typename T, int LS, int PROG>
__device__ __forceinline__ void put(T* site, int t, const SpinP<typename Pr<T>::V>& a) {
#pragma unroll
  for (int ch = 0; ch < 2; ch++) {
    constexpr bool R[2] = {prog_reversed(PROG, 0), prog_reversed(PROG, 1)};
    T* p = site + (R[ch] ? LS / 2 - 1 - t : t) * kPairStride;
#pragma unroll
    for (int c = 6 * ch; c < 6 * ch + 6; c++) {
      if (R[ch]) put4(p + 4 * c, a.re[c].y, a.re[c].x, a.im[c].y, a.im[c].x);
      else put4(p + 4 * c, a.re[c].x, a.re[c].y, a.im[c].x, a.im[c].y);
    }
  }
}
template <typename T, int LS, int PROG>
__device__ __forceinline__ void get(const T* site, int t, SpinP<typename Pr<T>::V>& a) {
  using A = Pr<T>;
#pragma unroll
  for (int ch = 0; ch < 2; ch++) {
    constexpr bool R[2] = {prog_reversed(PROG, 0), prog_reversed(PROG, 1)};
    const T* p = site + (R[ch] ? LS / 2 - 1 - t : t) * kPairStride;
#pragma unroll
    for (int c = 6 * ch; c < 6 * ch + 6; c++) {
      const Coef4<T> v = coef4(p + 4 * c);
      a.re[c] = R[ch] ? A::mk(v.b, v.a) : A::mk(v.a, v.b);
      a.im[c] = R[ch] ? A::mk(v.d, v.c) : A::mk(v.c, v.d);
    }
  }
}

// squares of the two slices
template <typename V>
__device__ __forceinline__ V sqr(const SpinP<V>& a) {
  using A = Pr<decltype(a.re[0].x)>;
  V r = A::mul(a.re[0], a.re[0]);
  r = A::fma(a.im[0], a.im[0], r);
#pragma unroll
  for (int c = 1; c < 12; c++) {
    r = A::fma(a.re[c], a.re[c], r);
    r = A::fma(a.im[c], a.im[c], r);
  }
  return r;
}

template <typename V>
__device__ __forceinline__ void zero(SpinP<V>& a) {
#pragma unroll
  for (int c = 0; c < 12; c++) {
    a.re[c].x = 0;
    a.re[c].y = 0;
    a.im[c].x = 0;
    a.im[c].y = 0;
  }
}

template <typename T>
constexpr int min_blocks() { return sizeof(T) == 8 ? 2 : 4; }

// The step a = *num / den of EX_RUPD, computed by the first warp of a CTA at its start
// (later barriers of the kernel make it visible).
template <typename T>
__device__ __forceinline__ T& rupd_scalar() {
  __shared__ T a;
  return a;
}
template <typename T>
__device__ __forceinline__ void start_rupd(const Args<T>& a, int rhs, int tid) {
  if (tid < 32) {
    const bool first = blockIdx.x == 0;
    const double ad = a.num[(size_t)rhs * a.sstride] / sum_in(a.den, rhs, first);
    if (tid == 0) {
      rupd_scalar<T>() = (T)ad;
      if (first) a.a_out[(size_t)rhs * a.sstride] = ad;
    }
  }
}

// Steps of the CG on D_bb^+ D_bb that end a hopping pass (HopLaunch.extra).
enum { EX_NONE = 0, EX_HAT = 1, EX_RUPD = 2 };

// Common tail of the hopping kernels: 5th-dimension post program, scaling,
// optional gamma5, local term (c_loc = 1), store and fused norm.  Every thread of the
// CTA calls it (it contains __syncthreads); the nth threads with tid < nth run the
// program, threads with part = false (no site of their own) store nothing.  With EX_HAT
// the result also goes through PR_ITINV (coefficients after those of POST); with EX_RUPD
// it updates the residual, whose norm is the fused one.
template <class SP, int LS, int POST, int LOC, bool G5, bool NORM, int EX = EX_NONE>
__device__ __forceinline__ void epilogue_g(const Args<typename SP::T>& a, const typename SP::T* coef,
                                           typename SP::T* sbuf, int tid, int nth, int nsites, size_t NP,
                                           int h, int j, int t, bool active, bool part, int rhs,
                                           SpinP<typename Pr<typename SP::T>::V>& acc) {
  using T = typename SP::T;
  using A = Pr<T>;
  using V = typename A::V;
  if constexpr (POST != PR_NONE) {
    T* site = sbuf + j * site_stride(LS);
    if (part) put<T, LS, POST>(site, t, acc);
    __syncthreads();
    if (tid < nth) run_prog<T, LS, POST>(sbuf, coef, tid, nth, nsites);
    __syncthreads();
    if (part) get<T, LS, POST>(site, t, acc);
  }
  const V ch = A::dup(a.c_hop);
  const size_t off = rhs * a.stride;
  const size_t m = (size_t)h * (LS / 2) + t;
  if (LOC == LOC_ID) {
    if (active) {
      SpinP<V> w;
      load_spin<SP>(reinterpret_cast<const char*>(a.w) + off, m, NP, w);
#pragma unroll
      for (int c = 0; c < 12; c++) {
        const V f = (G5 && c >= 6) ? A::neg(ch) : ch;
        acc.re[c] = A::fma(f, acc.re[c], w.re[c]);
        acc.im[c] = A::fma(f, acc.im[c], w.im[c]);
      }
    }
  } else if (G5 || a.c_hop != (T)1) {
#pragma unroll
    for (int c = 0; c < 12; c++) {
      const V f = (G5 && c >= 6) ? A::neg(ch) : ch;
      acc.re[c] = A::mul(f, acc.re[c]);
      acc.im[c] = A::mul(f, acc.im[c]);
    }
  }
  if constexpr (EX == EX_RUPD) {
    if (active) {
      const V na = A::dup(-rupd_scalar<T>());
      char* r = reinterpret_cast<char*>(a.out2) + off;
      SpinP<V> x;
      load_spin<SP>(r, m, NP, x);
#pragma unroll
      for (int c = 0; c < 12; c++) {
        acc.re[c] = A::fma(na, acc.re[c], x.re[c]);
        acc.im[c] = A::fma(na, acc.im[c], x.im[c]);
      }
      PairIO<SP>::store(r, m, NP, acc);
    }
  } else {
    if (active) PairIO<SP>::store(reinterpret_cast<char*>(a.out) + off, m, NP, acc);
  }
  if constexpr (EX == EX_HAT) {
    static_assert(!SP::kScaled && NORM, "the fused hat is for FP32 and FP64 fields");
    const V nrm = active ? sqr(acc) : A::dup((T)0);
#pragma unroll
    for (int c = 6; c < 12; c++) {
      acc.re[c] = A::neg(acc.re[c]);
      acc.im[c] = A::neg(acc.im[c]);
    }
    T* site = sbuf + j * site_stride(LS);
    __syncthreads();
    if (part) put<T, LS, PR_ITINV>(site, t, acc);
    __syncthreads();
    if (tid < nth) run_prog<T, LS, PR_ITINV>(sbuf, coef + prog_coefs(LS, POST), tid, nth, nsites);
    __syncthreads();
    if (active) {
      get<T, LS, PR_ITINV>(site, t, acc);
      PairIO<SP>::store(reinterpret_cast<char*>(a.out2) + off, m, NP, acc);
    }
    block_sum_pair(nrm, a.red, rhs, gridDim.x, blockIdx.x);
  } else if (NORM) {
    V v = A::dup((T)0);
    if (active) {
      if constexpr (SP::kScaled) {
        // 16-bit storage rounds: the norm follows the stored values
        SpinP<V> q = acc;
        PairIO<SP>::quantize(q);
        v = sqr(q);
      } else {
        v = sqr(acc);
      }
    }
    block_sum_pair(v, a.red, rhs, gridDim.x, blockIdx.x);
  }
}

// Sites per CTA of nth threads: 32 / G per warp where a site's threads exchange registers,
// else as many as the threads have room for.
template <int LS, int PRE>
__host__ __device__ constexpr int cta_sites(int nth) {
  return PRE == PRE_B ? nth / 32 * (32 / (LS / 2)) : nth / (LS / 2);
}

// out = c_hop G post(H v') + loc(w), two 5th-dimension slices per thread.
template <class SP, int LS, int PRE, int POST, int LOC, bool G5, bool NORM, int MINB, int EX = EX_NONE>
__global__ void __launch_bounds__(128, MINB) hop_kernel(const Geom g, const Args<typename SP::T> a) {
  using T = typename SP::T;
  using V = typename Pr<T>::V;
  constexpr int G = LS / 2;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* coef = reinterpret_cast<T*>(smem_raw);
  T* sbuf = coef + prog_coefs(LS, POST) + (EX == EX_HAT ? prog_coefs(LS, PR_ITINV) : 0);
  constexpr bool BYWARP = PRE == PRE_B;  // a site's threads in one warp
  const int tid = threadIdx.x, nth = blockDim.x;
  const int S = cta_sites<LS, PRE>(nth);
  const int first = BYWARP ? tid >> 5 : 0, lane = BYWARP ? tid & 31 : tid;
  const int jl = lane / G, t = lane - jl * G, j = first * (32 / G) + jl;
  const int h = blockIdx.x * S + j;
  const bool part = warp_groups(LS) || (BYWARP ? jl < 32 / G : j < S);
  const bool active = part && h < g.Vh;
  const int rhs = blockIdx.z;
  ahead_trigger();
  if (a.active && !a.active[rhs]) return;
  const size_t co = (size_t)rhs * a.cstride;
  const size_t NP = (size_t)g.N5 >> 1;
  const int s0 = 2 * t;
  load_coefs<T, LS, POST>(coef, a.chain + co, tid, nth);
  if (EX == EX_HAT) load_coefs<T, LS, PR_ITINV>(coef + prog_coefs(LS, POST), a.chain + co, tid, nth);
  const int hl = BYWARP ? min(h, g.Vh - 1) : (active ? h : 0);
  const int4 nb0 = __ldg(a.nbr + 2 * hl), nb1 = __ldg(a.nbr + 2 * hl + 1);
  ahead_wait();
  zero_bins(a, rhs, tid, nth);
  if (EX == EX_RUPD) start_rupd(a, rhs, tid);
  const char* vb = reinterpret_cast<const char*>(a.v) + rhs * a.stride;
  SpinP<V> acc;
  zero(acc);
  // whole warps take part in the shuffles of the B pre-multiplication: threads past the
  // last site compute it again and store nothing
  if (BYWARP || active) {
    T bd[2][2] = {{0, 0}, {0, 0}}, bo[2][2] = {{0, 0}, {0, 0}};
    if (PRE == PRE_B) {
#pragma unroll
      for (int c = 0; c < 2; c++)
#pragma unroll
        for (int k = 0; k < 2; k++) {
          bd[c][k] = __ldg(a.bdiag + co + c * LS + s0 + k);
          bo[c][k] = __ldg(a.boff + co + c * LS + s0 + k);
        }
    }
    const int nb[8] = {nb0.x, nb0.y, nb0.z, nb0.w, nb1.x, nb1.y, nb1.z, nb1.w};
    hop_dir<SP, LS, PRE, 0, +1>(nb[0], hl, t, NP, bd, bo, vb, a.gauge_p, a.gauge_q, acc);
    hop_dir<SP, LS, PRE, 0, -1>(nb[1], hl, t, NP, bd, bo, vb, a.gauge_p, a.gauge_q, acc);
    hop_dir<SP, LS, PRE, 1, +1>(nb[2], hl, t, NP, bd, bo, vb, a.gauge_p, a.gauge_q, acc);
    hop_dir<SP, LS, PRE, 1, -1>(nb[3], hl, t, NP, bd, bo, vb, a.gauge_p, a.gauge_q, acc);
    hop_dir<SP, LS, PRE, 2, +1>(nb[4], hl, t, NP, bd, bo, vb, a.gauge_p, a.gauge_q, acc);
    hop_dir<SP, LS, PRE, 2, -1>(nb[5], hl, t, NP, bd, bo, vb, a.gauge_p, a.gauge_q, acc);
    hop_dir<SP, LS, PRE, 3, +1>(nb[6], hl, t, NP, bd, bo, vb, a.gauge_p, a.gauge_q, acc);
    hop_dir<SP, LS, PRE, 3, -1>(nb[7], hl, t, NP, bd, bo, vb, a.gauge_p, a.gauge_q, acc);
  }
  epilogue_g<SP, LS, POST, LOC, G5, NORM, EX>(a, coef, sbuf, tid, nth, S, NP, h, j, t, active, part, rhs, acc);
}

// --- small lattices: the directions of a site on four warps ---------------------------

// One component of a slice pair (FP32 and FP64 fields).
__device__ __forceinline__ void load_comp(const float* base, size_t m, size_t NP, int c, float2& re, float2& im) {
  const float4 v = reinterpret_cast<const float4*>(base)[(size_t)c * NP + m];
  re = make_float2(v.x, v.y);
  im = make_float2(v.z, v.w);
}
__device__ __forceinline__ void load_comp(const double* base, size_t m, size_t NP, int c, double2& re, double2& im) {
  const double2* p = reinterpret_cast<const double2*>(base) + ((size_t)c * NP + m) * 2;
  re = p[0];
  im = p[1];
}
__device__ __forceinline__ void store_comp(float* base, size_t m, size_t NP, int c, float2 re, float2 im) {
  reinterpret_cast<float4*>(base)[(size_t)c * NP + m] = make_float4(re.x, re.y, im.x, im.y);
}
__device__ __forceinline__ void store_comp(double* base, size_t m, size_t NP, int c, double2 re, double2 im) {
  double2* p = reinterpret_cast<double2*>(base) + ((size_t)c * NP + m) * 2;
  p[0] = re;
  p[1] = im;
}

// Where hop_split_kernel adds up the hops of a site.  FP32: on the way into the sweeps, direction
// x's warp having added up its own two (they come first in the order of the sum), which leaves
// one block less to read.  FP64 (sum_lanes): by the lanes of all four warps in a step of its own,
// 96 additions a thread; the sweeps fill few lanes (Ls = 32: 24 of 64), and an instruction of the
// FP64 pipe costs the same however many lanes are on.  D_bb + D_bb^+ (CUDA graph), by lanes / on
// the way into the sweeps, both with an access to each hop: FP64 4^3x8, Ls = 32 115 / 132 us,
// 8x4x4x8, Ls = 10 105 / 110; FP32 8^3x16, Ls = 8 30.7 / 25.8, 8^4, Ls = 16 26.2 / 25.0.  With the
// two hops of a direction in one access (put_hops): 112, 103, 25.0 and 25.1.
template <typename T>
__host__ __device__ constexpr bool sums_in_sweeps() { return sizeof(T) == 4; }

// Shared memory of the hops: direction x's block has the layout of put (site_stride); the other
// directions' follow.  FP32 sites are 16 words apart modulo 32 there: the 16-byte accesses of
// consecutive sweeps (12 of a site, one behind the other) are then conflict-free.
template <typename T>
__host__ __device__ constexpr int hop_site_stride(int Ls) {
  return sizeof(T) == 8 ? site_stride(Ls) : (Ls / 2) * kPairStride + ((16 - ((Ls / 2) * kPairStride) % 32) + 32) % 32;
}
template <typename T, int LS>
__device__ __forceinline__ T* hop_block(T* sbuf, int mu, int site) {
  constexpr int S = 32 / (LS / 2);
  return mu == 0 ? sbuf + site * site_stride(LS)
                 : sbuf + S * site_stride(LS) + ((mu - 1) * S + site) * hop_site_stride<T>(LS);
}

// The sweep of component R of chirality CH from what the four warps left of the eight hops of a
// site (hop_block: direction x's sum as put leaves it, then put_hops of the others).  The hops
// are added up one after the other as hop_kernel does, so that both kernels give the same bits:
// the upper rows of (1 -+ gamma_mu) U' v' are chi, the lower ones rs (i) chi of the partner row
// (mul_acc).
template <typename T, int LS, int CH>
__device__ __forceinline__ void sum_hops(T (&V)[LS], T* sbuf, int site, int R) {
  using A = Pr<T>;
  constexpr int G = LS / 2;
  const int row = R / 6, col = R - 6 * row;  // spin row, 2 colour + (re | im)
  const T* at[4];
  T sg[4];
#pragma unroll
  for (int mu = 1; mu < 4; mu++) {
    const int rs = row == 0 ? recon_sign(mu, +1, 0) : recon_sign(mu, +1, 1);
    // += rs i chi: re takes -rs im, im takes rs re
    sg[mu] = (T)(imag_mu(mu) && !(col & 1) ? -rs : rs);
    at[mu] = hop_block<T, LS>(sbuf, mu, site) + 4 * (CH == 0 ? R : 6 * partner(mu, row) + (imag_mu(mu) ? col ^ 1 : col));
  }
#pragma unroll
  for (int k = 0; k < G; k++) {
    const int o = (CH == 0 ? k : G - 1 - k) * kPairStride;
    const auto x = pair_at(hop_block<T, LS>(sbuf, 0, site) + 24 * CH + 2 * R + k * kPairStride);
    auto v = CH == 0 ? x : A::mk(x.y, x.x);
#pragma unroll
    for (int mu = 1; mu < 4; mu++) {
      const Coef4<T> h = coef4(at[mu] + o);
      const auto f = A::mk(h.a, h.b), b = A::mk(h.c, h.d);
      v = CH == 0 ? A::add(v, f) : A::fma(A::dup(sg[mu]), f, v);
      v = CH == 0 ? A::add(v, b) : A::fma(A::dup(-sg[mu]), b, v);
    }
    V[2 * k] = CH == 0 ? v.x : v.y;
    V[2 * k + 1] = CH == 0 ? v.y : v.x;
  }
}

// run_prog for 128 threads on nsites <= 32 / (LS / 2) sites, with HOPS on the sums of sum_hops.
// The result goes to the first block, in the layout of put.
template <typename T, int LS, int PROG, bool HOPS>
__device__ __forceinline__ void run_prog_split(T* sbuf, const T* coef, int tid, int nsites) {
  using A = Pr<T>;
  constexpr int G = LS / 2;
  constexpr int NIT = (12 * (32 / G) + 63) / 64;
  const int ch = tid >> 6;
  T V[NIT][LS];
#pragma unroll
  for (int q = 0; q < NIT; q++) {
    const int i = (tid & 63) + 64 * q, site = i / 12, R = i - 12 * site;
    if (i >= 12 * nsites) {
#pragma unroll
      for (int k = 0; k < LS; k++) V[q][k] = (T)0;
    } else if (!HOPS) {
#pragma unroll
      for (int k = 0; k < G; k++) {
        const auto v = pair_at(sbuf + site * site_stride(LS) + 24 * ch + 2 * R + k * kPairStride);
        V[q][2 * k] = v.x;
        V[q][2 * k + 1] = v.y;
      }
    } else if (ch == 0) {
      sum_hops<T, LS, 0>(V[q], sbuf, site, R);
    } else {
      sum_hops<T, LS, 1>(V[q], sbuf, site, R);
    }
  }
  // the result overwrites the first block, where a thread has read only what it writes
#pragma unroll
  for (int i = 0; i < prog_len(PROG); i++) {
    const T* c = coef + (2 * i + ch) * chain_stride(LS);
    if (op_is_solve(prog_op(PROG, i))) chain_solve<T, LS, NIT>(V, c);
    else chain_mult<T, LS, NIT>(V, c);
  }
#pragma unroll
  for (int q = 0; q < NIT; q++) {
    const int i = (tid & 63) + 64 * q, site = i / 12;
    T* p = sbuf + site * site_stride(LS) + 24 * ch + 2 * (i - 12 * site);
    if (i < 12 * nsites)
#pragma unroll
      for (int k = 0; k < G; k++)
        *reinterpret_cast<typename A::V*>(p + k * kPairStride) = A::mk(V[q][2 * k], V[q][2 * k + 1]);
  }
}

// f chi of a direction's two hops (components 0 .. 5 of a: to x + mu, 6 .. 11: to x - mu) of slice
// pair t into shared memory, in the sweep order of PROG's chirality 0: real component R of both, as
// (x + mu, x - mu) pairs, at 4 R.
template <typename T, int LS, int PROG>
__device__ __forceinline__ void put_hops(T* site, int t, const SpinP<typename Pr<T>::V>& a) {
  static_assert(prog_reversed(PROG, 0) != prog_reversed(PROG, 1), "one chirality sweeps the slices last to first");
  constexpr bool R = prog_reversed(PROG, 0);
  T* p = site + (R ? LS / 2 - 1 - t : t) * kPairStride;
#pragma unroll
  for (int c = 0; c < 6; c++) {
    if (R) {
      put4(p + 8 * c, a.re[c].y, a.re[c].x, a.re[6 + c].y, a.re[6 + c].x);
      put4(p + 8 * c + 4, a.im[c].y, a.im[c].x, a.im[6 + c].y, a.im[6 + c].x);
    } else {
      put4(p + 8 * c, a.re[c].x, a.re[c].y, a.re[6 + c].x, a.re[6 + c].y);
      put4(p + 8 * c + 4, a.im[c].x, a.im[c].y, a.im[6 + c].x, a.im[6 + c].y);
    }
  }
}

// Components 3 w .. 3 w + 2 of slice pair t summed over the eight hops that put_hops left, in the
// same order as sum_hops (w: the warp).
template <typename T, int LS, int PROG>
__device__ __forceinline__ void sum_lanes(T* sbuf, int site, int t, int w, typename Pr<T>::V (&re)[3],
                                          typename Pr<T>::V (&im)[3]) {
  using A = Pr<T>;
  using V = typename A::V;
  constexpr bool R = prog_reversed(PROG, 0);
  const int o = (R ? LS / 2 - 1 - t : t) * kPairStride, row = w & 1;
#pragma unroll
  for (int a = 0; a < 3; a++) re[a] = im[a] = A::dup((T)0);
#pragma unroll
  for (int mu = 0; mu < 4; mu++)
#pragma unroll
    for (int a = 0; a < 3; a++) {
      const T* p = hop_block<T, LS>(sbuf, mu, site) + o + 8 * (3 * (w < 2 ? row : partner(mu, row)) + a);
      const Coef4<T> x = coef4(p), y = coef4(p + 4);  // re, im: (to x + mu, to x - mu)
      if (w < 2) {
        re[a] = A::add(A::add(re[a], A::mk(x.a, x.b)), A::mk(x.c, x.d));
        im[a] = A::add(A::add(im[a], A::mk(y.a, y.b)), A::mk(y.c, y.d));
      } else {  // += rs chi or rs i chi, rs turned around for the hop to x - mu
        const V s = A::dup((T)(row == 0 ? recon_sign(mu, +1, 0) : recon_sign(mu, +1, 1))), n = A::neg(s);
        const Coef4<T>& u = imag_mu(mu) ? y : x;
        const Coef4<T>& v = imag_mu(mu) ? x : y;
        re[a] = A::fma(imag_mu(mu) ? n : s, A::mk(u.a, u.b), re[a]);
        re[a] = A::fma(imag_mu(mu) ? s : n, A::mk(u.c, u.d), re[a]);
        im[a] = A::fma(s, A::mk(v.a, v.b), im[a]);
        im[a] = A::fma(n, A::mk(v.c, v.d), im[a]);
      }
    }
  if (R) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
      re[a] = A::mk(re[a].y, re[a].x);
      im[a] = A::mk(im[a].y, im[a].x);
    }
  }
}

// hop_kernel with the four directions mu of a site on the four warps of a CTA (two hops
// each) and 32 / G sites per CTA; the hops are added up on the way into the
// 5th-dimension program, and each warp finishes three of the twelve components.
// For lattices that leave SM sub-partitions without a warp: a warp alone is bound by its
// own chain (FP64: one instruction per 64 cycles of its sub-partition's pipe; FP32: eight
// gathers one after the other), which this cuts to a quarter.
template <class SP, int LS, int PRE, int POST, int LOC, bool G5, bool NORM, int MINB, int EX = EX_NONE>
__global__ void __launch_bounds__(128, MINB) hop_split_kernel(const Geom g, const Args<typename SP::T> a) {
  using T = typename SP::T;
  using A = Pr<T>;
  using V = typename A::V;
  constexpr int G = LS / 2, S = 32 / G, SST = site_stride(LS);
  constexpr bool XSUM = sums_in_sweeps<T>();
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* coef = reinterpret_cast<T*>(smem_raw);
  T* sbuf = coef + prog_coefs(LS, POST) + (EX == EX_HAT ? prog_coefs(LS, PR_ITINV) : 0);
  const int tid = threadIdx.x, mu = tid >> 5, lane = tid & 31;
  const int j = lane / G, t = lane - j * G;
  const int h = blockIdx.x * S + j;
  const bool part = warp_groups(LS) || j < S;
  const bool active = part && h < g.Vh;
  const int rhs = blockIdx.z;
  ahead_trigger();
  if (a.active && !a.active[rhs]) return;
  const size_t co = (size_t)rhs * a.cstride;
  const size_t NP = (size_t)g.N5 >> 1;
  load_coefs<T, LS, POST>(coef, a.chain + co, tid, 128);
  if (EX == EX_HAT) load_coefs<T, LS, PR_ITINV>(coef + prog_coefs(LS, POST), a.chain + co, tid, 128);
  constexpr bool WHOLE = PRE == PRE_B;  // its shuffles need whole warps
  const int hl = WHOLE ? min(h, g.Vh - 1) : (active ? h : 0);
  const int2 nb = __ldg(reinterpret_cast<const int2*>(a.nbr) + (size_t)hl * 4 + mu);
  ahead_wait();
  zero_bins(a, rhs, tid, 128);
  if (EX == EX_RUPD) start_rupd(a, rhs, tid);
  const char* vb = reinterpret_cast<const char*>(a.v) + rhs * a.stride;
  SpinP<V> acc;
  zero(acc);
  if (WHOLE || active) {
    T bd[2][2] = {{0, 0}, {0, 0}}, bo[2][2] = {{0, 0}, {0, 0}};
    if (PRE == PRE_B) {
#pragma unroll
      for (int c = 0; c < 2; c++)
#pragma unroll
        for (int k = 0; k < 2; k++) {
          bd[c][k] = __ldg(a.bdiag + co + c * LS + 2 * t + k);
          bo[c][k] = __ldg(a.boff + co + c * LS + 2 * t + k);
        }
    }
#define DWF_SPLIT_MU(MU)                                                                          \
  case MU:                                                                                        \
    hop_dir<SP, LS, PRE, MU, +1, !(MU == 0 && XSUM)>(nb.x, hl, t, NP, bd, bo, vb, a.gauge_p, a.gauge_q, acc); \
    hop_dir<SP, LS, PRE, MU, -1, !(MU == 0 && XSUM)>(nb.y, hl, t, NP, bd, bo, vb, a.gauge_p, a.gauge_q, acc); \
    break;
    switch (mu) {
      DWF_SPLIT_MU(0)
      DWF_SPLIT_MU(1)
      DWF_SPLIT_MU(2)
      DWF_SPLIT_MU(3)
    }
#undef DWF_SPLIT_MU
  }
  // this warp's components of the result: 3 mu .. 3 mu + 2, all of chirality mu / 2
  const size_t off = rhs * a.stride, m = (size_t)h * G + t;
  const int c0 = 3 * mu, chir = mu >> 1;
  const T* other = reinterpret_cast<const T*>(
      (EX == EX_RUPD ? reinterpret_cast<const char*>(a.out2) : reinterpret_cast<const char*>(a.w)) + off);
  V wr[3], wi[3], xr[3], xi[3];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    wr[k] = wi[k] = xr[k] = xi[k] = A::dup((T)0);
    if (LOC == LOC_ID && active)
      load_comp(reinterpret_cast<const T*>(reinterpret_cast<const char*>(a.w) + off), m, NP, c0 + k, wr[k], wi[k]);
    if (EX == EX_RUPD && active) load_comp(other, m, NP, c0 + k, xr[k], xi[k]);
  }
  if (part) {
    if (XSUM && mu == 0) put<T, LS, POST>(sbuf + j * SST, t, acc);
    else put_hops<T, LS, POST>(hop_block<T, LS>(sbuf, mu, j), t, acc);
  }
  __syncthreads();
  const bool rev = prog_reversed(POST, 1) == (chir == 1);  // one of the chiralities is reversed
  T* p = sbuf + j * SST + (rev ? G - 1 - t : t) * kPairStride + 4 * c0;
  if constexpr (!XSUM) {
    V sr[3], si[3];
    if (part) sum_lanes<T, LS, POST>(sbuf, j, t, mu, sr, si);
    __syncthreads();  // the sums overwrite the first block
    if (part) {
#pragma unroll
      for (int k = 0; k < 3; k++) {
        if (rev) put4(p + 4 * k, sr[k].y, sr[k].x, si[k].y, si[k].x);
        else put4(p + 4 * k, sr[k].x, sr[k].y, si[k].x, si[k].y);
      }
    }
    __syncthreads();
  }
  run_prog_split<T, LS, POST, XSUM>(sbuf, coef, tid, S);
  __syncthreads();
  const T f = G5 && chir == 1 ? -a.c_hop : a.c_hop;
  V re[3], im[3];
  const T na = EX == EX_RUPD ? -rupd_scalar<T>() : (T)0;
  V n2 = A::dup((T)0);
  if (active) {
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const Coef4<T> v = coef4(p + 4 * k);
      re[k] = rev ? A::mk(v.b, v.a) : A::mk(v.a, v.b);
      im[k] = rev ? A::mk(v.d, v.c) : A::mk(v.c, v.d);
      re[k] = LOC == LOC_ID ? A::fma(A::dup(f), re[k], wr[k]) : A::mul(A::dup(f), re[k]);
      im[k] = LOC == LOC_ID ? A::fma(A::dup(f), im[k], wi[k]) : A::mul(A::dup(f), im[k]);
      if (EX == EX_RUPD) {
        re[k] = A::fma(A::dup(na), re[k], xr[k]);
        im[k] = A::fma(A::dup(na), im[k], xi[k]);
      }
      store_comp(reinterpret_cast<T*>(reinterpret_cast<char*>(EX == EX_RUPD ? a.out2 : a.out) + off), m, NP,
                 c0 + k, re[k], im[k]);
      n2 = A::fma(re[k], re[k], n2);
      n2 = A::fma(im[k], im[k], n2);
    }
  }
  if (EX == EX_HAT) {
    const bool hrev = prog_reversed(PR_ITINV, 1) == (chir == 1);
    T* q = sbuf + j * SST + (hrev ? G - 1 - t : t) * kPairStride + 4 * c0;
    __syncthreads();
    if (active) {
#pragma unroll
      for (int k = 0; k < 3; k++) {
        if (chir == 1) {
          re[k] = A::neg(re[k]);
          im[k] = A::neg(im[k]);
        }
        if (hrev) put4(q + 4 * k, re[k].y, re[k].x, im[k].y, im[k].x);
        else put4(q + 4 * k, re[k].x, re[k].y, im[k].x, im[k].y);
      }
    }
    __syncthreads();
    run_prog_split<T, LS, PR_ITINV, false>(sbuf, coef + prog_coefs(LS, POST), tid, S);
    __syncthreads();
    if (active) {
#pragma unroll
      for (int k = 0; k < 3; k++) {
        const Coef4<T> v = coef4(q + 4 * k);
        store_comp(reinterpret_cast<T*>(reinterpret_cast<char*>(a.out2) + off), m, NP, c0 + k,
                   hrev ? A::mk(v.b, v.a) : A::mk(v.a, v.b), hrev ? A::mk(v.d, v.c) : A::mk(v.c, v.d));
      }
    }
  }
  if (NORM) block_sum_pair(n2, a.red, rhs, gridDim.x, blockIdx.x);
}

// out = c * PROG(gamma5^g5in in), site-local, two slices per thread.
template <class SP, int LS, int PROG>
__global__ void __launch_bounds__(128) local_kernel(const Geom g, void* out, const void* in,
                                                    size_t stride, const typename SP::T* chain,
                                                    typename SP::T c, int g5in, size_t cstride,
                                                    const int* rhs_on) {
  using T = typename SP::T;
  using A = Pr<T>;
  using V = typename A::V;
  constexpr int G = LS / 2;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* coef = reinterpret_cast<T*>(smem_raw);
  T* sbuf = coef + prog_coefs(LS, PROG);
  const int tid = threadIdx.x, nth = blockDim.x;
  const int S = nth / G, j = tid / G, t = tid - j * G;
  const int h = blockIdx.x * S + j;
  const bool active = j < S && h < g.Vh;
  const int rhs = blockIdx.z;
  if (rhs_on && !rhs_on[rhs]) return;
  const size_t NP = (size_t)g.N5 >> 1;
  load_coefs<T, LS, PROG>(coef, chain + (size_t)rhs * cstride, tid, nth);
  const size_t off = rhs * stride;
  const size_t m = (size_t)h * G + t;
  SpinP<V> x;
  zero(x);
  if (active) load_spin<SP>(reinterpret_cast<const char*>(in) + off, m, NP, x);
  if (c != (T)1) {
#pragma unroll
    for (int k = 0; k < 12; k++) {
      x.re[k] = A::mul(A::dup(c), x.re[k]);
      x.im[k] = A::mul(A::dup(c), x.im[k]);
    }
  }
  if (g5in) {
#pragma unroll
    for (int k = 6; k < 12; k++) {
      x.re[k] = A::neg(x.re[k]);
      x.im[k] = A::neg(x.im[k]);
    }
  }
  T* site = sbuf + j * site_stride(LS);
  if (j < S) put<T, LS, PROG>(site, t, x);
  __syncthreads();
  run_prog<T, LS, PROG>(sbuf, coef, tid, nth, S);
  __syncthreads();
  if (!active) return;
  get<T, LS, PROG>(site, t, x);
  PairIO<SP>::store(reinterpret_cast<char*>(out) + off, m, NP, x);
}

}  // namespace hop2
}  // namespace dwf

#include "dwf_hop_tma.cuh"

namespace dwf {
namespace hop2 {

// Threads per CTA (HopLaunch.block_threads; 0: by this rule).
// FP32 and 16-bit: 128 threads, or 64 where a site's threads straddle warps and the CTA's
// tail of unused lanes counts (FP32, Ls = 12, 12^2x8x12, D_bb + D_bb^+, CUDA graph: 43.0 us at
// 64, 46.6 at 128); CTAs of one warp load the coefficients and pass the barriers once per
// warp (BF16, Ls = 16, 8^2x4^2: 30.8 us at 32, 28.6 at 64, 26.2 at 128).
// FP64: the largest CTA that still gives every SM eight of them: its pipe wants the warps
// spread evenly over the sub-partitions (Ls = 8, 12^2x8x12: 439 us at 64, 548 at 128).
// All of them give the same fields; the fused norms of FP64 fields and the sums of the tree are
// rounded CTA by CTA, so the size counts rule_nrhs right-hand sides and is never timed.
inline int tile_threads(int Ls, int Vh, int nrhs, bool f64) {
  if (!f64) return warp_groups(Ls) ? 128 : 64;
  for (int nt : {128, 64}) {
    const int S = nt / (Ls / 2);
    const long long blocks = (long long)((Vh + S - 1) / S) * nrhs;
    if (blocks >= 152 * 8 * 128 / nt) return nt;
  }
  return 32;
}

template <typename T>
constexpr size_t split_smem(int Ls, int prog, int extra) {
  return sizeof(T) * ((size_t)prog_coefs(Ls, prog) + (extra == EX_HAT ? prog_coefs(Ls, PR_ITINV) : 0) +
                      (size_t)(32 / (Ls / 2)) * (site_stride(Ls) + 3 * hop_site_stride<T>(Ls)));
}

inline size_t smem_bytes(int Ls, int S, size_t ts, int prog, int extra = EX_NONE) {
  const int coefs = prog_coefs(Ls, prog) + (extra == EX_HAT ? prog_coefs(Ls, PR_ITINV) : 0);
  return prog == PR_NONE ? 0 : ts * ((size_t)coefs + (size_t)S * site_stride(Ls));
}

// hop_split_kernel instead of hop_kernel while the warps of hop_kernel do not fill the 608
// SM sub-partitions once (FP32); FP64 up to a line between the sizes where it was seen to win
// (432 warps) and to lose (512).  Both give the same bits (sum_hops).  D_bb + D_bb^+ at Ls = 16,
// us with / without (CUDA graph): FP32 4^4 15.3 / 26.3, 8^4 (512 warps) 25.1 / 28.8, FP64 4^4
// 99 / 276, 8^3x4 (256) 167 / 277, 12^2x8x12 at Ls = 4 (432) 234 / 290; above the lines (with
// sums by direction, 2-8% faster in FP32): FP32 12 right-hand sides of 8^2x4^2 (1536 warps)
// 49.4 / 42.4, FP64 8^4 (512) 326 / 296.
inline bool split_directions(int Ls, int Vh, int nrhs, bool f64) {
  const int S = 32 / (Ls / 2);
  return (long long)((Vh + S - 1) / S) * nrhs <= (f64 ? 456 : 608);
}

// Raises a kernel's dynamic shared-memory limit once per process; safe when
// several host threads launch through different handles at the same time.
template <class K>
cudaError_t smem_limit_once(K k, size_t smem, std::atomic<bool>& done) {
  if (done.load(std::memory_order_acquire)) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) done.store(true, std::memory_order_release);
  return e;
}

// Tensor map of a half-field (nrhs fields back to back) as 32-bit words:
// dim 0 the slice pairs of one row (component or 16-byte chunk row), dim 1 the
// rows, dim 2 the right-hand sides; the box is one site (Ls/2 pairs) x all rows.
template <class SP, int LS>
cudaError_t encode_field_map(CUtensorMap* map, const Geom& g, const void* base, size_t stride,
                             int nrhs) {
  using ST = Stage<SP, LS>;
  static std::atomic<PFN_cuTensorMapEncodeTiled_v12000> enc_fn{nullptr};
  PFN_cuTensorMapEncodeTiled_v12000 enc = enc_fn.load(std::memory_order_acquire);
  if (!enc) {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                     cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
    enc = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    enc_fn.store(enc, std::memory_order_release);
  }
  const size_t NP = (size_t)g.N5 / 2;
  const cuuint64_t dims[3] = {(cuuint64_t)NP * ST::kWpp, (cuuint64_t)ST::kRows, (cuuint64_t)nrhs};
  const cuuint64_t row = (cuuint64_t)NP * ST::kWpp * 4;
  const cuuint64_t strides[2] = {row, (cuuint64_t)(stride ? stride : row * ST::kRows)};
  const cuuint32_t box[3] = {(cuuint32_t)(LS / 2 * ST::kWpp), (cuuint32_t)ST::kRows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 3, const_cast<void*>(base), dims, strides, box,
                   estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <class SP, int LS>
constexpr int tma_stages() { return 2; }

template <class SP, int LS, int PRE, int POST, int LOC, bool G5, bool NORM>
cudaError_t run_tma(const Geom& g, const HopLaunch& L, const Args<typename SP::T>& a, cudaStream_t st) {
  constexpr int NST = tma_stages<SP, LS>();
  constexpr int S = kTmaConsumers / (LS / 2);
  CUtensorMap map;
  cudaError_t e = encode_field_map<SP, LS>(&map, g, L.v, L.stride, L.nrhs);
  if (e != cudaSuccess) return e;
  const size_t smem = tma_smem_bytes<SP, LS, NST, POST>();
  auto k = hop_tma_kernel<SP, LS, PRE, POST, LOC, G5, NORM, NST, 1>;
  static std::atomic<bool> attr{false};
  e = smem_limit_once(k, smem, attr);
  if (e != cudaSuccess) return e;
  dim3 grid((g.Vh + S - 1) / S, 1, L.nrhs);
  int skip = -1;
  if (L.skip_hop && *L.skip_hop >= 0) {
    skip = *L.skip_hop;
    *L.skip_hop = -1;
  }
  k<<<grid, kTmaThreads, smem, st>>>(g, a, map, L.wait_budget > 0 ? L.wait_budget : (1LL << 31), skip);
  return cudaGetLastError();
}

template <class SP, int LS, int PRE, int POST, int LOC, bool G5, bool NORM, int EX = EX_NONE>
cudaError_t run(const Geom& g, const HopLaunch& L, cudaStream_t st) {
  using T = typename SP::T;
  Args<T> a;
  a.out = L.out;
  a.v = L.v;
  a.w = L.w;
  a.stride = L.stride;
  const char* gb = reinterpret_cast<const char*>(L.gauge);
  a.gauge_p = gb + (size_t)L.p * L.gauge_parity_bytes;
  a.gauge_q = gb + (size_t)(1 - L.p) * L.gauge_parity_bytes;
  a.nbr = reinterpret_cast<const int4*>(L.nbr) + (size_t)L.p * g.Vh * 2;
  a.bdiag = reinterpret_cast<const T*>(L.pre_diag);
  a.boff = reinterpret_cast<const T*>(L.pre_off);
  a.chain = reinterpret_cast<const T*>(L.chain);
  a.c_hop = (T)L.c_hop;
  a.c_loc = (T)L.c_loc;
  a.red = L.red ? *L.red : Reduce{};
  a.cstride = L.cstride;
  a.active = L.active;
  a.err = L.err;
  a.out2 = L.out2;
  a.num = L.num;
  a.den = L.den;
  a.a_out = L.a_out;
  a.sstride = L.sstride;
  a.zero[0] = L.zero[0];
  a.zero[1] = L.zero[1];
  if constexpr (tma_ls(LS) && POST != PR_NONE && EX == EX_NONE) {
    if (L.use_tma) {
      const cudaError_t e = run_tma<SP, LS, PRE, POST, LOC, G5, NORM>(g, L, a, st);
      if (e != cudaErrorNotSupported) return e;  // no tensor map to be had: direct loads
    }
  }
  if constexpr (!SP::kScaled) {
    if (L.block_threads == 0 && split_directions(LS, g.Vh, std::max(L.nrhs, L.rule_nrhs), sizeof(T) == 8)) {
      constexpr int S = 32 / (LS / 2);
      constexpr size_t smem = split_smem<T>(LS, POST, EX);
      auto k = hop_split_kernel<SP, LS, PRE, POST, LOC, G5, NORM, min_blocks<T>(), EX>;
      static std::atomic<bool> attr{false};
      cudaError_t e = smem_limit_once(k, smem, attr);
      if (e != cudaSuccess) return e;
      return launch_ahead(L.ahead, k, dim3((g.Vh + S - 1) / S, 1, L.nrhs), 128, smem, st, g, a);
    }
  }
  const int nt =
      L.block_threads ? L.block_threads : tile_threads(LS, g.Vh, std::max(L.nrhs, L.rule_nrhs), sizeof(T) == 8);
  const int S = cta_sites<LS, PRE>(nt);
  const auto smem_of = [](int n) { return smem_bytes(LS, cta_sites<LS, PRE>(n), sizeof(T), POST, EX); };
  dim3 grid((g.Vh + S - 1) / S, 1, L.nrhs);
  auto k = hop_kernel<SP, LS, PRE, POST, LOC, G5, NORM, min_blocks<T>(), EX>;
  static std::atomic<bool> attr{false};
  cudaError_t e = smem_limit_once(k, smem_of(128), attr);
  if (e != cudaSuccess) return e;
  return launch_ahead(L.ahead, k, grid, nt, smem_of(nt), st, g, a);
}

// The hot combinations of the CG; anything else returns cudaErrorNotSupported
// and the caller falls back to the generic kernel.
template <class SP, int LS>
cudaError_t dispatch_ls(const Geom& g, const HopLaunch& L, cudaStream_t st) {
  const bool norm = L.red != nullptr;
  if (L.loc == LOC_DENSE || (L.loc == LOC_ID && L.c_loc != 1.0)) return cudaErrorNotSupported;
  if constexpr (!SP::kScaled) {
    if (L.extra == EX_HAT && L.pre == PRE_NONE && L.post_prog == PR_IINV && L.loc == LOC_ID && !L.g5out && norm)
      return run<SP, LS, PRE_NONE, PR_IINV, LOC_ID, false, true, EX_HAT>(g, L, st);
    if (L.extra == EX_RUPD && L.pre == PRE_NONE && L.post_prog == PR_BT && L.loc == LOC_ID && L.g5out && norm)
      return run<SP, LS, PRE_NONE, PR_BT, LOC_ID, true, true, EX_RUPD>(g, L, st);
  }
  if (L.extra != EX_NONE) return cudaErrorNotSupported;
  // FP64 is bound by the FP64 pipe: its callers form B v once (PR_B) and hop that
  if constexpr (SP::kPrec != P64) {
    if (L.pre == PRE_B && L.post_prog == PR_K && L.loc == LOC_NONE && !L.g5out && !norm)
      return run<SP, LS, PRE_B, PR_K, LOC_NONE, false, false>(g, L, st);
  }
  if constexpr (SP::kPrec == P64) {  // D_alpha, the Schur right-hand side, the red solution
    if (L.pre == PRE_NONE && L.post_prog == PR_NONE && !L.post && L.loc == LOC_ID && !L.g5out && !norm)
      return run<SP, LS, PRE_NONE, PR_NONE, LOC_ID, false, false>(g, L, st);
  }
  if (L.pre == PRE_NONE && L.post_prog == PR_K && L.loc == LOC_NONE && !L.g5out && !norm)
    return run<SP, LS, PRE_NONE, PR_K, LOC_NONE, false, false>(g, L, st);
  if (L.pre == PRE_NONE && L.post_prog == PR_IINV && L.loc == LOC_ID && !L.g5out)
    return norm ? run<SP, LS, PRE_NONE, PR_IINV, LOC_ID, false, true>(g, L, st)
                : run<SP, LS, PRE_NONE, PR_IINV, LOC_ID, false, false>(g, L, st);
  if (L.pre == PRE_NONE && L.post_prog == PR_KT && L.loc == LOC_NONE && !L.g5out && !norm)
    return run<SP, LS, PRE_NONE, PR_KT, LOC_NONE, false, false>(g, L, st);
  if (L.pre == PRE_NONE && L.post_prog == PR_BT && L.loc == LOC_ID && L.g5out)
    return norm ? run<SP, LS, PRE_NONE, PR_BT, LOC_ID, true, true>(g, L, st)
                : run<SP, LS, PRE_NONE, PR_BT, LOC_ID, true, false>(g, L, st);
  return cudaErrorNotSupported;
}

template <class SP, int LS, int PROG>
cudaError_t run_local(const Geom& g, const LocalLaunch& L, cudaStream_t st) {
  using T = typename SP::T;
  const int nt = tile_threads(LS, g.Vh, L.nrhs, sizeof(T) == 8), S = nt / (LS / 2);
  const size_t smem = smem_bytes(LS, S, sizeof(T), PROG);
  auto k = local_kernel<SP, LS, PROG>;
  static std::atomic<bool> attr{false};
  cudaError_t e = smem_limit_once(k, smem_bytes(LS, 128 / (LS / 2), sizeof(T), PROG), attr);
  if (e != cudaSuccess) return e;
  dim3 grid((g.Vh + S - 1) / S, 1, L.nrhs);
  k<<<grid, nt, smem, st>>>(g, L.out, L.in, L.stride, reinterpret_cast<const T*>(L.chain), (T)L.c,
                            L.g5in, L.cstride, L.active);
  return cudaGetLastError();
}

// CALL(Ls) for the compiled Ls of the translation unit's group.
#define DWF_LS_CASE(LS, CALL)                                 \
  case LS:                                                    \
    if constexpr (ls_group(LS) == GROUP && tuned_ls(LS, SP::kScaled)) return CALL(LS); \
    break;
#define DWF_TUNED_LS(Ls, CALL)                                                              \
  switch (Ls) {                                                                             \
    DWF_LS_CASE(4, CALL) DWF_LS_CASE(6, CALL) DWF_LS_CASE(8, CALL) DWF_LS_CASE(10, CALL)    \
    DWF_LS_CASE(12, CALL) DWF_LS_CASE(16, CALL) DWF_LS_CASE(20, CALL) DWF_LS_CASE(24, CALL) \
    DWF_LS_CASE(32, CALL)                                                                   \
  }                                                                                         \
  return cudaErrorNotSupported;

template <class SP, int GROUP>
cudaError_t dispatch(const Geom& g, const HopLaunch& L, cudaStream_t st) {
  if (L.chain == nullptr || L.nbr == nullptr) return cudaErrorNotSupported;
#define DWF_CALL(LS) dispatch_ls<SP, LS>(g, L, st)
  DWF_TUNED_LS(g.Ls, DWF_CALL)
#undef DWF_CALL
}

template <class SP, int LS>
cudaError_t dispatch_local_ls(const Geom& g, const LocalLaunch& L, cudaStream_t st) {
  if (L.prog == PR_ITINV) return run_local<SP, LS, PR_ITINV>(g, L, st);
  if constexpr (SP::kPrec == P64) {
    if (L.prog == PR_B) return run_local<SP, LS, PR_B>(g, L, st);
    if (L.prog == PR_I) return run_local<SP, LS, PR_I>(g, L, st);
    if (L.prog == PR_K) return run_local<SP, LS, PR_K>(g, L, st);
    if (L.prog == PR_IINV) return run_local<SP, LS, PR_IINV>(g, L, st);
  }
  return cudaErrorNotSupported;
}

template <class SP, int GROUP>
cudaError_t dispatch(const Geom& g, const LocalLaunch& L, cudaStream_t st) {
  if (L.chain == nullptr || L.red != nullptr) return cudaErrorNotSupported;
#define DWF_CALL(LS) dispatch_local_ls<SP, LS>(g, L, st)
  DWF_TUNED_LS(g.Ls, DWF_CALL)
#undef DWF_CALL
}


// Fused CG residual update: r -= a w with a = num / den, |r|^2, and
// r^ = I^-T gamma5 r (the input of the next D_bb^+ pass A), two slices per
// thread; a is also stored to a_out (read by the next p/x update).
template <class SP, int LS>
__global__ void __launch_bounds__(128) rupdate_kernel(const Geom g, void* r, void* rhat,
                                                      const void* w, size_t stride,
                                                      const typename SP::T* chain, size_t cstride,
                                                      const double* num, const SumIn den,
                                                      double* a_out, int sstride, Reduce red,
                                                      const int* rhs_on) {
  using T = typename SP::T;
  using A = Pr<T>;
  using V = typename A::V;
  constexpr int G = LS / 2;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* coef = reinterpret_cast<T*>(smem_raw);
  T* sbuf = coef + prog_coefs(LS, PR_ITINV);
  const int tid = threadIdx.x, nth = blockDim.x;
  const int S = nth / G, j = tid / G, t = tid - j * G;
  const int h = blockIdx.x * S + j;
  const bool active = j < S && h < g.Vh;
  const int rhs = blockIdx.z;
  ahead_trigger();
  if (rhs_on && !rhs_on[rhs]) return;
  const size_t NP = (size_t)g.N5 >> 1;
  load_coefs<T, LS, PR_ITINV>(coef, chain + (size_t)rhs * cstride, tid, nth);
  ahead_wait();
  const size_t off = rhs * stride;
  const size_t m = (size_t)h * G + t;
  SpinP<V> x;
  zero(x);
  V nrm = A::dup((T)0);
  SpinP<V> wv;
  zero(wv);
  if (active) {
    load_spin<SP>(reinterpret_cast<const char*>(r) + off, m, NP, x);
    load_spin<SP>(reinterpret_cast<const char*>(w) + off, m, NP, wv);
  }
  // a by one warp, while the loads are on their way
  __shared__ T a_sh;
  if (tid < 32) {
    const double ad = num[(size_t)rhs * sstride] / sum_in(den, rhs, blockIdx.x == 0);
    if (tid == 0) {
      a_sh = (T)ad;
      if (blockIdx.x == 0) a_out[(size_t)rhs * sstride] = ad;
    }
  }
  __syncthreads();
  const V na = A::dup(-a_sh);
  if (active) {
#pragma unroll
    for (int k = 0; k < 12; k++) {
      x.re[k] = A::fma(na, wv.re[k], x.re[k]);
      x.im[k] = A::fma(na, wv.im[k], x.im[k]);
    }
    PairIO<SP>::store(reinterpret_cast<char*>(r) + off, m, NP, x);
    // 16-bit storage rounds: r^ and |r|^2 follow the stored residual
    PairIO<SP>::quantize(x);
    nrm = sqr(x);
  }
#pragma unroll
  for (int k = 6; k < 12; k++) {
    x.re[k] = A::neg(x.re[k]);
    x.im[k] = A::neg(x.im[k]);
  }
  T* site = sbuf + j * site_stride(LS);
  if (j < S) put<T, LS, PR_ITINV>(site, t, x);
  __syncthreads();
  run_prog<T, LS, PR_ITINV>(sbuf, coef, tid, nth, S);
  __syncthreads();
  if (active) {
    get<T, LS, PR_ITINV>(site, t, x);
    PairIO<SP>::store(reinterpret_cast<char*>(rhat) + off, m, NP, x);
  }
  block_sum_pair(nrm, red, rhs, gridDim.x, blockIdx.x);
}

template <class SP, int LS>
cudaError_t run_rupdate(const Geom& g, const RUpdateLaunch& L, cudaStream_t st) {
  using T = typename SP::T;
  const int nt = tile_threads(LS, g.Vh, std::max(L.nrhs, L.rule_nrhs), sizeof(T) == 8), S = nt / (LS / 2);
  auto k = rupdate_kernel<SP, LS>;
  static std::atomic<bool> attr{false};
  cudaError_t e = smem_limit_once(k, smem_bytes(LS, 128 / (LS / 2), sizeof(T), PR_ITINV), attr);
  if (e != cudaSuccess) return e;
  dim3 grid((g.Vh + S - 1) / S, 1, L.nrhs);
  return launch_ahead(L.ahead, k, grid, nt, smem_bytes(LS, S, sizeof(T), PR_ITINV), st, g, L.r, L.rhat, L.w,
                      L.stride, reinterpret_cast<const T*>(L.chain), L.cstride, L.num, L.den, L.a_out, L.sstride,
                      *L.red, L.active);
}

template <class SP, int GROUP>
cudaError_t dispatch(const Geom& g, const RUpdateLaunch& L, cudaStream_t st) {
#define DWF_CALL(LS) run_rupdate<SP, LS>(g, L, st)
  DWF_TUNED_LS(g.Ls, DWF_CALL)
#undef DWF_CALL
}
}  // namespace hop2
}  // namespace dwf
