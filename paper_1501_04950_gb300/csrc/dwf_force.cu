// dwf_force.cu -- fermion force of S = phi^+ (D_bb^+ D_bb)^-1 phi (sm_103a).
//
// With X = (D^+ D)^-1 phi and Y = D_bb X, the variation of S under a change of
// the links is dS = -2 Re[Y^+ dD_bb X].  Only the hopping blocks of Eq. redblack
// depend on U (D_rb = -1/2 H_rb B, D_br = -1/2 H_br B), which gives
//   dS = 2 Re[eta1^+ dD_br xi1] + 2 Re[eta2^+ dD_rb xi2],
//   eta1 = I^-T Y (black),  xi1 = I^-1 D_rb X (red),
//   eta2 = I^-T D_br^+ eta1 = -1/2 K^T gamma5 H_rb gamma5 eta1 (red),  xi2 = X (black).
// Each term is -1/2 sum_s over the hops of Eq. wilson that contain U_mu(x):
//   forward  x <- x+mu:  eta(x)^+ (1 - gamma_mu) dU w(x+mu)
//   backward x+mu <- x:  eta(x+mu)^+ (1 + gamma_mu) dU^+ w(x),      w = B xi.
// With the convention G_ij = dS/dRe U_ij + i dS/dIm U_ij a term Re[a^+ dU b]
// contributes a b^+, and sum_spin a_spin (P b)_spin^+ for P = 1 -+ gamma_mu
// reduces to the two rows of the projected half spinors: sum_k h(a)_k h(b)_k^+.
//
// The applies that lead here leave every factor in memory: W = B X on black sites and
// W = K H_rb B X = -2 B xi1 on red ones (the input and the result of pass A of Y = D_bb X),
// E = gamma5 eta1 on black and E = K^T H_rb gamma5 eta1 = -2 gamma5 eta2 on red ones
// (the hat and pass A of D_bb^+ Y).  gamma5 turns the projector of E around, so that for
// every link, with h-+ the half spinors of (1 -+ gamma_mu),
//   G_mu(x) = s/2 sum_slices [ h+(E(x)) h-(W(x+mu))^+ + h+(W(x)) h-(E(x+mu))^+ ]
// where s is the antiperiodic sign of the hop.
#include <algorithm>

#include "dwf_fields.cuh"
#include "dwf_hop2.cuh"

namespace dwf {

namespace {

using hop2::HalfP;
using hop2::PairIO;

struct ForceArgs {
  const void* E[2];  // by parity
  const void* W[2];
  const int4* nbr;   // [2][Vh][2] neighbour table, bit 31: antiperiodic sign
  const void* g64;   // internal FP64 gauge (both parities)
  size_t gpar;       // bytes per parity
  double* out;       // canonical [V][4][3][3] complex
  int projected;
};

// Components c0 .. c0 + 5 of slices 2t, 2t + 1 of site h (odd Ls: no slice past the last).
template <bool EVEN>
__device__ __forceinline__ void load6(const Geom& g, const void* f, int h, int t, int c0, double2* re,
                                      double2* im) {
  if constexpr (EVEN) {
    const int G = g.Ls >> 1;
    PairIO<Store64>::load6(f, (size_t)h * G + t, (size_t)g.N5 >> 1, c0, re, im);
  } else {
    const int n = site5(h, 2 * t, g.Ls);
    const bool two = 2 * t + 1 < g.Ls;
#pragma unroll
    for (int k = 0; k < 6; k++) {
      const double* a = Store64::at(f, c0 + k, n, g.N5);
      const double* b = Store64::at(f, c0 + k, two ? n + 1 : n, g.N5);
      re[k] = make_double2(__ldg(a), two ? __ldg(b) : 0.0);
      im[k] = make_double2(__ldg(a + 2), two ? __ldg(b + 2) : 0.0);
    }
  }
}

// Half spinors of (1 - DIR gamma_mu) f for the two slices.
template <bool EVEN, int MU, int DIR>
__device__ __forceinline__ void load_half(const Geom& g, const void* f, int h, int t, HalfP<double2>& P) {
  HalfP<double2> M;
  load6<EVEN>(g, f, h, t, 0, P.re, P.im);
  load6<EVEN>(g, f, h, t, 6, M.re, M.im);
  hop2::project_half<double, MU, DIR>(P, M);
}

// G_ij += sum over rows and slices of a_i conj(b_j)
__device__ __forceinline__ void outer_add(cplx<double> (&G)[9], const HalfP<double2>& a,
                                          const HalfP<double2>& b) {
#pragma unroll
  for (int k = 0; k < 2; k++)
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
      for (int j = 0; j < 3; j++) {
        const double2 ar = a.re[3 * k + i], ai = a.im[3 * k + i], br = b.re[3 * k + j], bi = b.im[3 * k + j];
        cplx<double>& c = G[3 * i + j];
        c.re = fma(ar.x, br.x, fma(ai.x, bi.x, fma(ar.y, br.y, fma(ai.y, bi.y, c.re))));
        c.im = fma(ai.x, br.x, fma(-ar.x, bi.x, fma(ai.y, br.y, fma(-ar.y, bi.y, c.im))));
      }
}

template <bool EVEN, int MU>
__device__ __forceinline__ void link_sum(const Geom& g, const ForceArgs& a, int p, int h, int hn, int t0,
                                         int step, cplx<double> (&G)[9]) {
  const int slots = (g.Ls + 1) >> 1;
  for (int t = t0; t < slots; t += step) {
    HalfP<double2> u, v;
    load_half<EVEN, MU, -1>(g, a.E[p], h, t, u);
    load_half<EVEN, MU, +1>(g, a.W[1 - p], hn, t, v);
    outer_add(G, u, v);
    load_half<EVEN, MU, -1>(g, a.W[p], h, t, u);
    load_half<EVEN, MU, +1>(g, a.E[1 - p], hn, t, v);
    outer_add(G, u, v);
  }
}

// One warp per direction mu (threadIdx.y) and 32 / PARTS sites of one parity (blockIdx.y);
// the PARTS lanes of a site share its slices.  Bound by the FP64 pipe: 2 x (24 + 72)
// operations per link and slice.  mu is the same for a whole warp, so that no lane waits
// for another direction's projection; the four warps of a CTA read the same sites.
// 16^3x32, Ls = 8: the whole force 8.91 -> 4.63 ms, this kernel 4.09 ms before (one
// thread per link with the four directions of a site in one warp, B folded in again per link).
template <bool EVEN, int PARTS>
__global__ void __launch_bounds__(128) force_kernel(const Geom g, const ForceArgs a) {
  constexpr int SITES = 32 / PARTS;
  const int mu = threadIdx.y, p = blockIdx.y;
  const int part = threadIdx.x / SITES;
  const int h = blockIdx.x * SITES + threadIdx.x % SITES;
  const bool active = h < g.Vh;
  cplx<double> G[9];
#pragma unroll
  for (int k = 0; k < 9; k++) G[k] = cmake(0.0, 0.0);
  double sign = 0.5;
  if (active) {
    const int4 q = __ldg(a.nbr + ((size_t)p * g.Vh + h) * 2 + (mu >> 1));
    const int nb = mu & 1 ? q.z : q.x;
    const int hn = nb & 0x7fffffff;
    if (nb < 0) sign = -0.5;
    switch (mu) {
      case 0: link_sum<EVEN, 0>(g, a, p, h, hn, part, PARTS, G); break;
      case 1: link_sum<EVEN, 1>(g, a, p, h, hn, part, PARTS, G); break;
      case 2: link_sum<EVEN, 2>(g, a, p, h, hn, part, PARTS, G); break;
      default: link_sum<EVEN, 3>(g, a, p, h, hn, part, PARTS, G); break;
    }
  }
  if (PARTS > 1) {
#pragma unroll
    for (int k = 0; k < 9; k++)
#pragma unroll
      for (int o = SITES; o < 32; o <<= 1) {
        G[k].re += __shfl_xor_sync(0xffffffffu, G[k].re, o);
        G[k].im += __shfl_xor_sync(0xffffffffu, G[k].im, o);
      }
  }
  if (!active || part > 0) return;
#pragma unroll
  for (int k = 0; k < 9; k++) G[k] = cmake(sign * G[k].re, sign * G[k].im);
  // canonical site index: x = 2 (h mod Lx/2) + parity offset of the row
  const Coords c = site_coords(g, h, p);
  const size_t link = ((size_t)c.x + (size_t)g.L[0] * (c.y + (size_t)g.L[1] * (c.z + (size_t)g.L[2] * c.t))) * 4 + mu;
  double2* o = reinterpret_cast<double2*>(a.out) + link * 9;
  if (!a.projected) {
#pragma unroll
    for (int k = 0; k < 9; k++) o[k] = make_double2(G[k].re, G[k].im);
    return;
  }
  // F = TA(U G^+), TA(M) = (M - M^+)/2 - tr(M - M^+)/6
  const double2* u = reinterpret_cast<const double2*>(reinterpret_cast<const char*>(a.g64) + (size_t)p * a.gpar) +
                     ((size_t)h * 4 + mu) * 9;
  cplx<double> M[9];
#pragma unroll
  for (int r = 0; r < 3; r++)
#pragma unroll
    for (int cc = 0; cc < 3; cc++) {
      cplx<double> acc = cmake(0.0, 0.0);
#pragma unroll
      for (int k = 0; k < 3; k++) {
        const double2 uu = u[3 * r + k];
        const cplx<double> gg = G[3 * cc + k];  // (G^+)_{k,cc} = conj(G_{cc,k})
        acc.re += uu.x * gg.re + uu.y * gg.im;
        acc.im += uu.y * gg.re - uu.x * gg.im;
      }
      M[3 * r + cc] = acc;
    }
  cplx<double> F[9];
#pragma unroll
  for (int r = 0; r < 3; r++)
#pragma unroll
    for (int cc = 0; cc < 3; cc++) {
      const cplx<double> m1 = M[3 * r + cc], m2 = M[3 * cc + r];
      F[3 * r + cc] = cmake(0.5 * (m1.re - m2.re), 0.5 * (m1.im + m2.im));
    }
  const double tr_im = F[0].im + F[4].im + F[8].im;
  F[0].im -= tr_im / 3.0;
  F[4].im -= tr_im / 3.0;
  F[8].im -= tr_im / 3.0;
#pragma unroll
  for (int k = 0; k < 9; k++) o[k] = make_double2(F[k].re, F[k].im);
}

template <bool EVEN, int PARTS>
void run_force(const Geom& g, const ForceArgs& a, cudaStream_t s) {
  constexpr int SITES = 32 / PARTS;
  const dim3 grid((g.Vh + SITES - 1) / SITES, 2), block(32, 4);
  force_kernel<EVEN, PARTS><<<grid, block, 0, s>>>(g, a);
}

}  // namespace

cudaError_t launch_force(const Geom& g, double* out, const void* e_black, const void* w_black,
                         const void* e_red, const void* w_red, const int* nbr, const void* g64,
                         size_t gpar, int black, int projected, cudaStream_t s) {
  ForceArgs a;
  a.E[black] = e_black;
  a.E[1 - black] = e_red;
  a.W[black] = w_black;
  a.W[1 - black] = w_red;
  a.nbr = reinterpret_cast<const int4*>(nbr);
  a.g64 = g64;
  a.gpar = gpar;
  a.out = out;
  a.projected = projected;
  // With fewer than 4 CTAs of 32 sites per SM the slices of a site are shared by 4 lanes:
  // the FP64 pipes of idle SMs then take part (the sum over lanes adds 36 operations per
  // link to ~190 per slice).
  const bool split = 2 * ((size_t)g.Vh + 31) / 32 < 4 * 152;
  if (g.Ls % 2 == 0) {
    if (split) run_force<true, 4>(g, a, s);
    else run_force<true, 1>(g, a, s);
  } else {
    if (split) run_force<false, 4>(g, a, s);
    else run_force<false, 1>(g, a, s);
  }
  return cudaGetLastError();
}

}  // namespace dwf
