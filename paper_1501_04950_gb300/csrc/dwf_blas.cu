// dwf_blas.cu -- layout conversions, sources, propagator extraction and the
// fused BLAS-1 kernels of the CG on the normal equations (sm_103a).
#include <algorithm>

#include "dwf_fields.cuh"

namespace dwf {

namespace {

constexpr int kBlasThreads = 256;

template <typename T>
__device__ __forceinline__ double sqd(const Spinor<T>& a) {
  T r = 0;
#pragma unroll
  for (int k = 0; k < 12; k++) r += a.c[k].re * a.c[k].re + a.c[k].im * a.c[k].im;
  return (double)r;
}

template <typename TD, typename TS>
__device__ __forceinline__ void cvt(Spinor<TD>& d, const Spinor<TS>& s) {
#pragma unroll
  for (int k = 0; k < 12; k++) d.c[k] = cmake((TD)s.c[k].re, (TD)s.c[k].im);
}

// ---- conversions --------------------------------------------------------------
// Canonical fields keep the 12 components of a 5D site together and the sites of a
// slice in a row; the half-fields keep the slice pairs of a site together, one row per
// component.  A CTA takes kTile-sized blocks of sites with all their slices through
// shared memory, so that both sides move whole lines: runs of (sites x 192) bytes on
// the canonical side, of (sites x Ls/2) pairs on the other.  Bound by HBM; one thread
// per 5D site, with 192-byte strides between the lanes on one side and Ls-strided
// scattered words on the other, moved 16^3x32, Ls = 16 at a sixth of that.
// 16^3x32, Ls = 16, FP32: a new gauge field, pack and unpack 550 -> 161 us (the bytes
// alone at the copy rate: 106).

// Tile element (site hl of the tile, slice s) at (hl Ls + s) kTileStride; real component
// R = 2c + (0 re | 1 im).  26 = 24 + 2: 8-byte accesses to consecutive 5D sites spread
// over the banks.
constexpr int kTileStride = 26;

// sites per tile: the largest power of two with at most 32 KB of tile (one tile per
// parity of the full fields: nfields = 2)
int tile_sites(int Ls, size_t ts, int nfields) {
  int n = 16;
  while (n > 2 && (size_t)n * Ls * kTileStride * ts * nfields > 32768) n /= 2;
  return n;
}
size_t tile_bytes(int Ls, int sites, size_t ts, int nfields) {
  // the tile(s), and one scale per 5D site of 16-bit storage
  return (size_t)sites * Ls * (kTileStride * ts + sizeof(float)) * nfields;
}

// 16 bytes of an internal field by one access (WIDE), or by accesses of one element for a
// caller's field that does not start on a 16-byte boundary.
template <bool WIDE>
__device__ __forceinline__ void put16(void* p, uint4 v) {
  if (WIDE) {
    *reinterpret_cast<uint4*>(p) = v;
  } else {
    uint32_t* q = reinterpret_cast<uint32_t*>(p);
    q[0] = v.x; q[1] = v.y; q[2] = v.z; q[3] = v.w;
  }
}
template <bool WIDE>
__device__ __forceinline__ void put16(void* p, double2 v) {
  if (WIDE) {
    *reinterpret_cast<double2*>(p) = v;
  } else {
    reinterpret_cast<double*>(p)[0] = v.x;
    reinterpret_cast<double*>(p)[1] = v.y;
  }
}
template <bool WIDE>
__device__ __forceinline__ uint4 get16(const uint4* p) {
  if (WIDE) return __ldg(p);
  const uint32_t* q = reinterpret_cast<const uint32_t*>(p);
  return make_uint4(__ldg(q), __ldg(q + 1), __ldg(q + 2), __ldg(q + 3));
}
template <bool WIDE>
__device__ __forceinline__ double2 get16(const double2* p) {
  if (WIDE) return __ldg(p);
  const double* q = reinterpret_cast<const double*>(p);
  return make_double2(__ldg(q), __ldg(q + 1));
}

// Tile -> internal half-field (n5 = 5D sites of the tile, first one at n0; both even).
template <class SP, bool WIDE>
__device__ __forceinline__ void tile_store(void* dst, const typename SP::T* tile, float* scale, int n0,
                                           int n5, int N5, int tid, int nth) {
  using T = typename SP::T;
  const size_t NP = (size_t)N5 >> 1, m0 = (size_t)n0 >> 1;
  const int np = n5 >> 1;
  if constexpr (SP::kScaled) {
    for (int n = tid; n < n5; n += nth) {
      float mx = 0.f;
#pragma unroll
      for (int k = 0; k < 24; k++) mx = fmaxf(mx, fabsf(tile[n * kTileStride + k]));
      scale[n] = SP::scale_of(mx);
    }
    __syncthreads();
    for (int i = tid; i < 6 * np; i += nth) {
      const int j = i / np, m = i - j * np;
      const T* a = tile + 2 * m * kTileStride + 4 * j;
      const T* b = a + kTileStride;
      const float ia = 1.f / scale[2 * m], ib = 1.f / scale[2 * m + 1];
      put16<WIDE>(reinterpret_cast<uint4*>(dst) + j * NP + m0 + m,
                  make_uint4(SP::from_f2(make_float2(a[0] * ia, b[0] * ib)), SP::from_f2(make_float2(a[1] * ia, b[1] * ib)),
                             SP::from_f2(make_float2(a[2] * ia, b[2] * ib)), SP::from_f2(make_float2(a[3] * ia, b[3] * ib))));
    }
    for (int n = tid; n < n5; n += nth) const_cast<float*>(SP::scales(dst, N5))[n0 + n] = scale[n];
  } else {
    for (int i = tid; i < 12 * np; i += nth) {
      const int c = i / np, m = i - c * np;
      const T* a = tile + 2 * m * kTileStride + 2 * c;
      const T* b = a + kTileStride;
      if constexpr (sizeof(T) == 8) {
        double2* o = reinterpret_cast<double2*>(dst) + (c * NP + m0 + m) * 2;
        put16<WIDE>(o, make_double2(a[0], b[0]));
        put16<WIDE>(o + 1, make_double2(a[1], b[1]));
      } else {
        put16<WIDE>(reinterpret_cast<uint4*>(dst) + c * NP + m0 + m,
                    make_uint4(__float_as_uint(a[0]), __float_as_uint(b[0]), __float_as_uint(a[1]), __float_as_uint(b[1])));
      }
    }
  }
}

// Internal half-field -> tile.
template <class SP, bool WIDE>
__device__ __forceinline__ void tile_load(typename SP::T* tile, const void* src, int n0, int n5, int N5,
                                          int tid, int nth) {
  using T = typename SP::T;
  const size_t NP = (size_t)N5 >> 1, m0 = (size_t)n0 >> 1;
  const int np = n5 >> 1;
  if constexpr (SP::kScaled) {
    for (int i = tid; i < 6 * np; i += nth) {
      const int j = i / np, m = i - j * np;
      const uint4 v = get16<WIDE>(reinterpret_cast<const uint4*>(src) + j * NP + m0 + m);
      const float* sc = SP::scales(src, N5) + n0 + 2 * m;
      const float sa = __ldg(sc), sb = __ldg(sc + 1);
      T* a = tile + 2 * m * kTileStride + 4 * j;
      T* b = a + kTileStride;
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const float2 q = SP::to_f2(w[k]);
        a[k] = sa * q.x;
        b[k] = sb * q.y;
      }
    }
  } else {
    for (int i = tid; i < 12 * np; i += nth) {
      const int c = i / np, m = i - c * np;
      T* a = tile + 2 * m * kTileStride + 2 * c;
      T* b = a + kTileStride;
      if constexpr (sizeof(T) == 8) {
        const double2* q = reinterpret_cast<const double2*>(src) + (c * NP + m0 + m) * 2;
        const double2 re = get16<WIDE>(q), im = get16<WIDE>(q + 1);
        a[0] = re.x; b[0] = re.y; a[1] = im.x; b[1] = im.y;
      } else {
        const uint4 v = get16<WIDE>(reinterpret_cast<const uint4*>(src) + c * NP + m0 + m);
        a[0] = __uint_as_float(v.x); b[0] = __uint_as_float(v.y); a[1] = __uint_as_float(v.z); b[1] = __uint_as_float(v.w);
      }
    }
  }
}

// Canonical half-field(s) [nrhs][Ls][Vh][12] <-> internal, `sites` sites per CTA.
template <class SP, bool PACK, bool WIDE>
__global__ void __launch_bounds__(kBlasThreads) half_kernel(const Geom g, void* field, double* canon,
                                                            size_t stride, int sites, int tiles) {
  using T = typename SP::T;
  extern __shared__ __align__(16) unsigned char tile_raw[];
  T* tile = reinterpret_cast<T*>(tile_raw);
  float* scale = reinterpret_cast<float*>(tile + (size_t)sites * g.Ls * kTileStride);
  const int tid = threadIdx.x, nth = blockDim.x, rhs = blockIdx.x / tiles;
  const int h0 = (blockIdx.x - rhs * tiles) * sites, nh = min(sites, g.Vh - h0);
  char* f = reinterpret_cast<char*>(field) + (size_t)rhs * stride;
  double2* c = reinterpret_cast<double2*>(canon) + (size_t)rhs * g.N5 * 12;
  const int run = nh * 12;  // components of one slice of the tile
  if (!PACK) {
    tile_load<SP, WIDE>(tile, f, h0 * g.Ls, nh * g.Ls, g.N5, tid, nth);
    __syncthreads();
  }
  for (int i = tid; i < run * g.Ls; i += nth) {
    const int s = i / run, r = i - s * run, hl = r / 12, k = r - 12 * hl;
    double2* q = c + ((size_t)s * g.Vh + h0) * 12 + r;
    T* e = tile + (hl * g.Ls + s) * kTileStride + 2 * k;
    if (PACK) {
      const double2 v = *q;
      e[0] = (T)v.x;
      e[1] = (T)v.y;
    } else {
      *q = make_double2((double)e[0], (double)e[1]);
    }
  }
  if (PACK) {
    __syncthreads();
    tile_store<SP, WIDE>(f, tile, scale, h0 * g.Ls, nh * g.Ls, g.N5, tid, nth);
  }
}

// Parity of the even-x site of half index h (sites 2h and 2h + 1 have both parities).
__device__ __forceinline__ int row_parity(const Geom& g, int h) {
  int r = h / g.Lxh;
  const int y = r % g.L[1];
  r /= g.L[1];
  return (y + r % g.L[2] + r / g.L[2]) & 1;
}

// full canonical [Ls][V][4][3] <-> FP64 internal halves, 2 x `sites` sites per CTA
template <bool SPLIT>
__global__ void __launch_bounds__(kBlasThreads) full_kernel(const Geom g, void* p0, void* p1, double* full,
                                                            int sites) {
  extern __shared__ __align__(16) unsigned char tile_raw[];
  double* tile = reinterpret_cast<double*>(tile_raw);
  const int tid = threadIdx.x, nth = blockDim.x;
  const int h0 = blockIdx.x * sites, nh = min(sites, g.Vh - h0);
  const int per = sites * g.Ls * kTileStride;  // tile of parity 1 after that of parity 0
  const int run = 2 * nh * 12;
  const size_t V = (size_t)g.Vh * 2;
  if (!SPLIT) {
    tile_load<Store64, true>(tile, p0, h0 * g.Ls, nh * g.Ls, g.N5, tid, nth);
    tile_load<Store64, true>(tile + per, p1, h0 * g.Ls, nh * g.Ls, g.N5, tid, nth);
    __syncthreads();
  }
  for (int i = tid; i < run * g.Ls; i += nth) {
    const int s = i / run, r = i - s * run, site = r / 12, k = r - 12 * site, hl = site >> 1;
    const int par = row_parity(g, h0 + hl) ^ (site & 1);
    double2* q = reinterpret_cast<double2*>(full) + (s * V + 2 * (size_t)h0) * 12 + r;
    double* e = tile + par * per + (hl * g.Ls + s) * kTileStride + 2 * k;
    if (SPLIT) {
      const double2 v = *q;
      e[0] = v.x;
      e[1] = v.y;
    } else {
      *q = make_double2(e[0], e[1]);
    }
  }
  if (SPLIT) {
    __syncthreads();
    tile_store<Store64, true>(p0, tile, nullptr, h0 * g.Ls, nh * g.Ls, g.N5, tid, nth);
    tile_store<Store64, true>(p1, tile + per, nullptr, h0 * g.Ls, nh * g.Ls, g.N5, tid, nth);
  }
}

// Links U[t][z][y][x][mu][3][3] -> the per-parity FP64, FP32 and FP16 layouts.  A CTA
// takes the 4 links of kGaugeSites neighbouring sites through shared memory: the links
// of the sites of one parity are a contiguous run of every output.  HBM bound, like the
// field conversions.
constexpr int kGaugeSites = 32;
__global__ void __launch_bounds__(kBlasThreads) gauge_convert_kernel(const Geom g, const double* U, double2* g64,
                                                                     float4* g32, uint4* g16) {
  __shared__ double2 tile[2][kGaugeSites / 2 * 36];
  const int tid = threadIdx.x, nth = blockDim.x;
  const int h0 = blockIdx.x * (kGaugeSites / 2), nh = min(kGaugeSites / 2, g.Vh - h0);
  const double2* u = reinterpret_cast<const double2*>(U) + (size_t)h0 * 72;
  for (int i = tid; i < nh * 72; i += nth) {
    const int site = i / 36, hl = site >> 1;
    tile[row_parity(g, h0 + hl) ^ (site & 1)][hl * 36 + (i - site * 36)] = u[i];
  }
  __syncthreads();
#pragma unroll
  for (int p = 0; p < 2; p++) {
    const size_t slot = ((size_t)p * g.Vh + h0) * 4;  // first link of the run
    for (int i = tid; i < nh * 36; i += nth) g64[slot * 9 + i] = tile[p][i];
    for (int i = tid; i < nh * 20; i += nth) {
      const int l = i / 5, k = 2 * (i - 5 * l);
      const double2 a = tile[p][l * 9 + k], b = k < 8 ? tile[p][l * 9 + k + 1] : make_double2(0.0, 0.0);
      g32[slot * 5 + i] = make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
    }
    for (int i = tid; i < nh * 12; i += nth) {
      const int l = i / 3, k = 4 * (i - 3 * l);
      uint32_t w[4];
#pragma unroll
      for (int q = 0; q < 4; q++) {
        w[q] = 0u;
        if (k + q < 9) {
          const double2 v = tile[p][l * 9 + k + q];
          w[q] = (uint32_t)__half_as_ushort(__float2half_rn((float)v.x)) |
                 ((uint32_t)__half_as_ushort(__float2half_rn((float)v.y)) << 16);
        }
      }
      g16[slot * 3 + i] = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// (Pb)_1 = P_- b_1 (spins 2,3), (Pb)_Ls = P_+ b_1 (spins 0,1); zero elsewhere.  One
// thread per slice pair m of either half (blockIdx.y), whose stores are whole lines.
__global__ void source_pb_kernel(const Geom g, void* p0, void* p1, const double* src) {
  const int NP = g.N5 >> 1, par = blockIdx.y;
  void* half = par ? p1 : p0;
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < NP; m += gridDim.x * blockDim.x) {
    Spinor<double> a[2];
#pragma unroll
    for (int l = 0; l < 2; l++) {
      const int n = 2 * m + l, h = n / g.Ls, s = n - h * g.Ls;
#pragma unroll
      for (int k = 0; k < 12; k++) a[l].c[k] = cmake(0.0, 0.0);
      if (s == 0 || s == g.Ls - 1) {
        const int site = 2 * h + (row_parity(g, h) ^ par);
        const double2* b = reinterpret_cast<const double2*>(src) + (size_t)site * 12;
#pragma unroll
        for (int k = 0; k < 12; k++)
          if ((k >= 6 && s == 0) || (k < 6 && s == g.Ls - 1)) a[l].c[k] = cmake(b[k].x, b[k].y);
      }
    }
    Store64::store_pair(half, m, NP, a[0], a[1]);
  }
}

// z_1 = P_- psi_1 + P_+ psi_Ls, one thread per component of a site
__global__ void extract_z1_kernel(const Geom g, double* prop, const void* p0, const void* p1) {
  const size_t total = (size_t)g.Vh * 24;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total;
       i += (size_t)gridDim.x * blockDim.x) {
    const int site = (int)(i / 12), k = (int)(i - (size_t)site * 12), h = site >> 1;
    const void* half = (row_parity(g, h) ^ (site & 1)) ? p1 : p0;
    const double* q = Store64::at(half, k, site5(h, k < 6 ? g.Ls - 1 : 0, g.Ls), g.N5);
    reinterpret_cast<double2*>(prop)[i] = make_double2(__ldg(q), __ldg(q + 2));
  }
}

// ---- BLAS-1 -------------------------------------------------------------------
// One thread per slice pair m (two 5D sites), vector loads of the pair layout.

// *num / *den, divided by one warp of the CTA (see sum_in); every thread calls it.
__device__ __forceinline__ double quotient(const double* num, const double* den) {
  __shared__ double q;
  if (threadIdx.x < 32) {
    const double v = *num / *den;
    if (threadIdx.x == 0) q = v;
  }
  __syncthreads();
  return q;
}

template <class SPX, class SP>
__global__ void __launch_bounds__(kBlasThreads) xr_update_kernel(
    const Geom g, void* x, void* r, const void* p, const void* w, const double* num,
    const double* den, int sstride, size_t stride_x, size_t stride, Reduce red, const int* active) {
  using T = typename SP::T;
  using TX = typename SPX::T;
  const int rhs = blockIdx.y;
  if (active && !active[rhs]) return;
  const size_t off = rhs * stride, offx = rhs * stride_x;
  const double ad = quotient(num + (size_t)rhs * sstride, den + (size_t)rhs * sstride);
  const T a = (T)ad;
  const TX ax = (TX)ad;
  const int NP = g.N5 >> 1;
  double acc = 0.0;
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < NP; m += gridDim.x * blockDim.x) {
    Spinor<TX> xv[2];
    Spinor<T> rv[2], pv[2], wv[2];
    SPX::load_pair(reinterpret_cast<const char*>(x) + offx, m, NP, xv[0], xv[1]);
    SP::load_pair(reinterpret_cast<const char*>(r) + off, m, NP, rv[0], rv[1]);
    SP::load_pair(reinterpret_cast<const char*>(p) + off, m, NP, pv[0], pv[1]);
    SP::load_pair(reinterpret_cast<const char*>(w) + off, m, NP, wv[0], wv[1]);
#pragma unroll
    for (int l = 0; l < 2; l++)
#pragma unroll
      for (int k = 0; k < 12; k++) {
        xv[l].c[k] = cmake(fma(ax, (TX)pv[l].c[k].re, xv[l].c[k].re), fma(ax, (TX)pv[l].c[k].im, xv[l].c[k].im));
        rv[l].c[k] = cmake(fma(-a, wv[l].c[k].re, rv[l].c[k].re), fma(-a, wv[l].c[k].im, rv[l].c[k].im));
      }
    SPX::store_pair(reinterpret_cast<char*>(x) + offx, m, NP, xv[0], xv[1]);
    SP::store_pair(reinterpret_cast<char*>(r) + off, m, NP, rv[0], rv[1]);
    acc += sqd(rv[0]) + sqd(rv[1]);
  }
  block_sum_to(acc, red, rhs, gridDim.x, blockIdx.x);
}

template <class SP>
__global__ void __launch_bounds__(kBlasThreads) p_update_kernel(
    const Geom g, void* p, const void* z, const double* num, const double* den, int sstride,
    size_t stride, const int* active) {
  using T = typename SP::T;
  const int rhs = blockIdx.y;
  if (active && !active[rhs]) return;
  const size_t off = rhs * stride;
  const T beta = (T)quotient(num + (size_t)rhs * sstride, den + (size_t)rhs * sstride);
  const int NP = g.N5 >> 1;
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < NP; m += gridDim.x * blockDim.x) {
    Spinor<T> pv[2], zv[2];
    SP::load_pair(reinterpret_cast<const char*>(p) + off, m, NP, pv[0], pv[1]);
    SP::load_pair(reinterpret_cast<const char*>(z) + off, m, NP, zv[0], zv[1]);
#pragma unroll
    for (int l = 0; l < 2; l++)
#pragma unroll
      for (int k = 0; k < 12; k++)
        pv[l].c[k] = cmake(fma(beta, pv[l].c[k].re, zv[l].c[k].re), fma(beta, pv[l].c[k].im, zv[l].c[k].im));
    SP::store_pair(reinterpret_cast<char*>(p) + off, m, NP, pv[0], pv[1]);
  }
}


template <class SPX, class SP>
__global__ void __launch_bounds__(kBlasThreads) px_update_kernel(
    const Geom g, void* x, void* p, const void* z, const double* a_ptr, const double* num,
    const double* den, int sstride, size_t stride_x, size_t stride, const int* active, int do_p) {
  using T = typename SP::T;
  using TX = typename SPX::T;
  const int rhs = blockIdx.y;
  if (active && !active[rhs]) return;
  const size_t off = rhs * stride, offx = rhs * stride_x;
  const TX a = (TX)a_ptr[(size_t)rhs * sstride];
  const T beta = do_p ? (T)quotient(num + (size_t)rhs * sstride, den + (size_t)rhs * sstride) : (T)0;
  const int NP = g.N5 >> 1;
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < NP; m += gridDim.x * blockDim.x) {
    Spinor<T> pv[2];
    Spinor<TX> xv[2];
    SP::load_pair(reinterpret_cast<const char*>(p) + off, m, NP, pv[0], pv[1]);
    SPX::load_pair(reinterpret_cast<const char*>(x) + offx, m, NP, xv[0], xv[1]);
#pragma unroll
    for (int l = 0; l < 2; l++)
#pragma unroll
      for (int k = 0; k < 12; k++)
        xv[l].c[k] = cmake(fma(a, (TX)pv[l].c[k].re, xv[l].c[k].re), fma(a, (TX)pv[l].c[k].im, xv[l].c[k].im));
    SPX::store_pair(reinterpret_cast<char*>(x) + offx, m, NP, xv[0], xv[1]);
    if (do_p) {
      Spinor<T> zv[2];
      SP::load_pair(reinterpret_cast<const char*>(z) + off, m, NP, zv[0], zv[1]);
#pragma unroll
      for (int l = 0; l < 2; l++)
#pragma unroll
        for (int k = 0; k < 12; k++)
          pv[l].c[k] = cmake(fma(beta, pv[l].c[k].re, zv[l].c[k].re), fma(beta, pv[l].c[k].im, zv[l].c[k].im));
      SP::store_pair(reinterpret_cast<char*>(p) + off, m, NP, pv[0], pv[1]);
    }
  }
}

// p_new = z + beta p_old (and, with do_x, the deferred x += a_prev p_old) for one
// slice pair m of site h, t = m mod (Ls/2), plus bp = B p_new: B is cyclic
// bidiagonal per chirality (Eq. mobius1 with D_w -> 1),
//   (B v)+(s) = d+(s) v+(s) + o+(s) v+(s-1),  (B v)-(s) = d-(s) v-(s) + o-(s) v-(s+1),
// so v+ of slice 2t-1 (pair below) and v- of slice 2t+2 (pair above) enter as well: they are
// in the registers of the neighbouring lanes (a warp takes the pairs of 32 / (Ls/2) whole
// sites).  Used by the CG on the tuned path, whose D_bb pass A then hops B p directly.
// HBM bound: 6 half-field passes.  Forming the neighbours' slices again from loads of
// their own (48 words a thread) kept 16^3x32, Ls = 16, FP32 at 99 us, against 90 (cold, under ncu).
template <class SPX, class SP>
__global__ void __launch_bounds__(kBlasThreads, 2) pxb_update_kernel(
    const Geom g, void* x, const void* p, void* pnew, void* bp, const void* z, const double* a_ptr,
    const SumIn num, const double* den, int sstride, size_t stride_x, size_t stride,
    const typename SP::T* bdiag, const typename SP::T* boff, size_t cstride, const int* active,
    int do_x) {
  using T = typename SP::T;
  using TX = typename SPX::T;
  const int rhs = blockIdx.y;
  ahead_trigger();
  if (active && !active[rhs]) return;
  const size_t off = rhs * stride, offx = rhs * stride_x;
  ahead_wait();
  __shared__ T beta_sh;
  bool have_beta = false;
  T beta = 0;
  const int NP = g.N5 >> 1, half = g.Ls >> 1;
  const int per = 32 / half * half;  // pairs of a warp
  const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const T* bd = bdiag + (size_t)rhs * cstride;
  const T* bo = boff + (size_t)rhs * cstride;
  const char* pb = reinterpret_cast<const char*>(p) + off;
  const char* zb = reinterpret_cast<const char*>(z) + off;
  // whole blocks go round the loop, for the barrier and the shuffles
  for (int m0 = blockIdx.x * warps * per; m0 < NP; m0 += gridDim.x * warps * per) {
    const int mt = m0 + (threadIdx.x >> 5) * per + lane;
    const bool mine = lane < per && mt < NP;
    const int m = mine ? mt : NP - 1;
    const int t = m % half;
    const int below = t == 0 ? lane + half - 1 : lane - 1, above = t + 1 == half ? lane - t : lane + 1;
    Spinor<T> pv[2], q[2];
    SP::load_pair(pb, m, NP, pv[0], pv[1]);
    SP::load_pair(zb, m, NP, q[0], q[1]);
    if (!have_beta) {  // by one warp, while the loads are on their way
      if (threadIdx.x < 32) {
        const double b = sum_in(num, rhs, blockIdx.x == 0) / den[(size_t)rhs * sstride];
        if (threadIdx.x == 0) beta_sh = (T)b;
      }
      __syncthreads();
      beta = beta_sh;
      have_beta = true;
    }
#pragma unroll
    for (int l = 0; l < 2; l++)
#pragma unroll
      for (int k = 0; k < 12; k++)
        q[l].c[k] = cmake(fma(beta, pv[l].c[k].re, q[l].c[k].re), fma(beta, pv[l].c[k].im, q[l].c[k].im));
    if (do_x && mine) {
      const TX a = (TX)a_ptr[(size_t)rhs * sstride];
      Spinor<TX> xv[2];
      SPX::load_pair(reinterpret_cast<const char*>(x) + offx, m, NP, xv[0], xv[1]);
#pragma unroll
      for (int l = 0; l < 2; l++)
#pragma unroll
        for (int k = 0; k < 12; k++)
          xv[l].c[k] = cmake(fma(a, (TX)pv[l].c[k].re, xv[l].c[k].re), fma(a, (TX)pv[l].c[k].im, xv[l].c[k].im));
      SPX::store_pair(reinterpret_cast<char*>(x) + offx, m, NP, xv[0], xv[1]);
    }
    if (mine) SP::store_pair(reinterpret_cast<char*>(pnew) + off, m, NP, q[0], q[1]);
    if constexpr (SP::kScaled) {
      // 16-bit storage: B acts on the stored (rounded) p_new, as pass B's local term sees it
      SP::quantize(q[0]);
      SP::quantize(q[1]);
    }
    const int s0 = 2 * t;
    const T dp0 = bd[s0], dp1 = bd[s0 + 1], op0 = bo[s0], op1 = bo[s0 + 1];
    const T dm0 = bd[g.Ls + s0], dm1 = bd[g.Ls + s0 + 1], om0 = bo[g.Ls + s0], om1 = bo[g.Ls + s0 + 1];
    Spinor<T> b[2];
#pragma unroll
    for (int k = 0; k < 6; k++) {
      const cplx<T> lo = cmake(__shfl_sync(0xffffffffu, q[1].c[k].re, below),
                               __shfl_sync(0xffffffffu, q[1].c[k].im, below));
      const cplx<T> up = cmake(__shfl_sync(0xffffffffu, q[0].c[6 + k].re, above),
                               __shfl_sync(0xffffffffu, q[0].c[6 + k].im, above));
      b[0].c[k] = cmake(fma(op0, lo.re, dp0 * q[0].c[k].re), fma(op0, lo.im, dp0 * q[0].c[k].im));
      b[1].c[k] = cmake(fma(op1, q[0].c[k].re, dp1 * q[1].c[k].re), fma(op1, q[0].c[k].im, dp1 * q[1].c[k].im));
      b[0].c[6 + k] = cmake(fma(om0, q[1].c[6 + k].re, dm0 * q[0].c[6 + k].re),
                            fma(om0, q[1].c[6 + k].im, dm0 * q[0].c[6 + k].im));
      b[1].c[6 + k] = cmake(fma(om1, up.re, dm1 * q[1].c[6 + k].re), fma(om1, up.im, dm1 * q[1].c[6 + k].im));
    }
    if (mine) SP::store_pair(reinterpret_cast<char*>(bp) + off, m, NP, b[0], b[1]);
  }
}

// dst <- src converted; the norm (optional) is that of the stored dst values.
template <class SPD, class SPS>
__global__ void __launch_bounds__(kBlasThreads) convert_kernel(
    const Geom g, void* dst, const void* src, size_t sd, size_t ss, Reduce red, int do_norm,
    const int* active) {
  using TD = typename SPD::T;
  using TS = typename SPS::T;
  const int rhs = blockIdx.y;
  if (active && !active[rhs]) return;
  const int NP = g.N5 >> 1;
  double acc = 0.0;
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < NP; m += gridDim.x * blockDim.x) {
    Spinor<TS> a[2];
    SPS::load_pair(reinterpret_cast<const char*>(src) + rhs * ss, m, NP, a[0], a[1]);
    Spinor<TD> b[2];
    cvt(b[0], a[0]);
    cvt(b[1], a[1]);
    SPD::store_pair(reinterpret_cast<char*>(dst) + rhs * sd, m, NP, b[0], b[1]);
    if (do_norm) {
      if constexpr (SPD::kScaled) {
        SPD::quantize(b[0]);
        SPD::quantize(b[1]);
      }
      acc += sqd(b[0]) + sqd(b[1]);
    }
  }
  if (do_norm) block_sum_to(acc, red, rhs, gridDim.x, blockIdx.x);
}

template <class SPS>
__global__ void __launch_bounds__(kBlasThreads) accumulate64_kernel(
    const Geom g, void* x64, void* src, int zero_src, size_t sd, size_t ss, const int* active) {
  using TS = typename SPS::T;
  const int rhs = blockIdx.y;
  if (active && !active[rhs]) return;
  const int NP = g.N5 >> 1;
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < NP; m += gridDim.x * blockDim.x) {
    Spinor<TS> a[2];
    SPS::load_pair(reinterpret_cast<const char*>(src) + rhs * ss, m, NP, a[0], a[1]);
    Spinor<double> x[2];
    Store64::load_pair(reinterpret_cast<const char*>(x64) + rhs * sd, m, NP, x[0], x[1]);
#pragma unroll
    for (int l = 0; l < 2; l++)
#pragma unroll
      for (int k = 0; k < 12; k++)
        x[l].c[k] = cmake(x[l].c[k].re + (double)a[l].c[k].re, x[l].c[k].im + (double)a[l].c[k].im);
    Store64::store_pair(reinterpret_cast<char*>(x64) + rhs * sd, m, NP, x[0], x[1]);
    if (zero_src) {
      Spinor<TS> zz;
#pragma unroll
      for (int k = 0; k < 12; k++) zz.c[k] = cmake<TS>(0, 0);
      SPS::store_pair(reinterpret_cast<char*>(src) + rhs * ss, m, NP, zz, zz);
    }
  }
}

__global__ void __launch_bounds__(kBlasThreads) sub64_norm_kernel(
    const Geom g, void* out, const void* a, const void* b, size_t stride, Reduce red,
    const int* active) {
  const int rhs = blockIdx.y;
  if (active && !active[rhs]) return;
  const size_t off = rhs * stride;
  const int NP = g.N5 >> 1;
  double acc = 0.0;
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < NP; m += gridDim.x * blockDim.x) {
    Spinor<double> x[2], y[2];
    Store64::load_pair(reinterpret_cast<const char*>(a) + off, m, NP, x[0], x[1]);
    Store64::load_pair(reinterpret_cast<const char*>(b) + off, m, NP, y[0], y[1]);
#pragma unroll
    for (int l = 0; l < 2; l++)
#pragma unroll
      for (int k = 0; k < 12; k++) x[l].c[k] = x[l].c[k] - y[l].c[k];
    Store64::store_pair(reinterpret_cast<char*>(out) + off, m, NP, x[0], x[1]);
    acc += sqd(x[0]) + sqd(x[1]);
  }
  block_sum_to(acc, red, rhs, gridDim.x, blockIdx.x);
}

// dst <- a - b with a FP64 and b FP32 (the difference in FP64), stored in the
// precision of SPD; |dst|^2 of the stored values.
template <class SPD>
__global__ void __launch_bounds__(kBlasThreads) sub_to_kernel(
    const Geom g, void* dst, const void* a, const void* b, size_t sd, size_t sa, size_t sb,
    Reduce red, const int* active) {
  using TD = typename SPD::T;
  const int rhs = blockIdx.y;
  if (active && !active[rhs]) return;
  const int NP = g.N5 >> 1;
  double acc = 0.0;
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < NP; m += gridDim.x * blockDim.x) {
    Spinor<double> x[2];
    Spinor<float> y[2];
    Store64::load_pair(reinterpret_cast<const char*>(a) + rhs * sa, m, NP, x[0], x[1]);
    Store32::load_pair(reinterpret_cast<const char*>(b) + rhs * sb, m, NP, y[0], y[1]);
    Spinor<TD> d[2];
#pragma unroll
    for (int l = 0; l < 2; l++)
#pragma unroll
      for (int k = 0; k < 12; k++)
        d[l].c[k] = cmake<TD>((TD)(x[l].c[k].re - (double)y[l].c[k].re),
                              (TD)(x[l].c[k].im - (double)y[l].c[k].im));
    SPD::store_pair(reinterpret_cast<char*>(dst) + rhs * sd, m, NP, d[0], d[1]);
    if constexpr (SPD::kScaled) {
      SPD::quantize(d[0]);
      SPD::quantize(d[1]);
    }
    acc += sqd(d[0]) + sqd(d[1]);
  }
  block_sum_to(acc, red, rhs, gridDim.x, blockIdx.x);
}

template <class SP>
__global__ void __launch_bounds__(kBlasThreads) norm_kernel(const Geom g, const void* x,
                                                             size_t stride, Reduce red) {
  using T = typename SP::T;
  const int rhs = blockIdx.y;
  const int NP = g.N5 >> 1;
  double acc = 0.0;
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < NP; m += gridDim.x * blockDim.x) {
    Spinor<T> a[2];
    SP::load_pair(reinterpret_cast<const char*>(x) + rhs * stride, m, NP, a[0], a[1]);
    acc += sqd(a[0]) + sqd(a[1]);
  }
  block_sum_to(acc, red, rhs, gridDim.x, blockIdx.x);
}

// Re <a, b> of two FP64 half-fields (one right-hand side per blockIdx.y).
__global__ void __launch_bounds__(kBlasThreads) dot_re64_kernel(const Geom g, const void* a,
                                                                 const void* b, size_t stride,
                                                                 Reduce red) {
  const int rhs = blockIdx.y;
  const int NP = g.N5 >> 1;
  double acc = 0.0;
  for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < NP; m += gridDim.x * blockDim.x) {
    Spinor<double> x[2], y[2];
    Store64::load_pair(reinterpret_cast<const char*>(a) + rhs * stride, m, NP, x[0], x[1]);
    Store64::load_pair(reinterpret_cast<const char*>(b) + rhs * stride, m, NP, y[0], y[1]);
#pragma unroll
    for (int l = 0; l < 2; l++)
#pragma unroll
      for (int k = 0; k < 12; k++)
        acc = fma(x[l].c[k].re, y[l].c[k].re, fma(x[l].c[k].im, y[l].c[k].im, acc));
  }
  block_sum_to(acc, red, rhs, gridDim.x, blockIdx.x);
}

__global__ void finish_sum_kernel(const SumIn in, const int* active) {
  const int rhs = blockIdx.x;
  if (active && !active[rhs]) return;
  sum_in(in, rhs, true);
}

// Launch shape of n elements, one per thread up to 16 CTAs of kBlasThreads per SM.  Below
// two CTAs of 256 per SM the CTAs are of 64 threads, so that a small lattice still
// spreads over all SMs.
struct Shape {
  int blocks, threads;
};
Shape elementwise(size_t n) {
  const int threads = n < (size_t)152 * 2 * kBlasThreads ? 64 : kBlasThreads;
  const size_t b = (n + threads - 1) / threads;
  return Shape{(int)std::min<size_t>(std::max<size_t>(b, 1), 152 * 16), threads};
}

}  // namespace

int blas_grid_blocks(const Geom& g) { return elementwise((size_t)g.N5 / 2).blocks; }

size_t field_bytes(const Geom& g, int prec) {
  size_t b = 0;
  switch (prec) {
    case P64: b = (size_t)g.N5 * 192; break;
    case P32: b = (size_t)g.N5 * 96; break;
    case P16:
    case PB16: b = (size_t)g.N5 * 52; break;
    default: return 0;
  }
  return (b + 255) / 256 * 256;
}

size_t gauge_bytes(const Geom& g, int prec) {
  const size_t links = (size_t)g.Vh * 2 * 4;
  switch (prec) {
    case P64: return links * 144;
    case P32: return links * 80;
    default: return links * 48;
  }
}

#define DWF_PREC_SWITCH(prec, SP, ...)                 \
  switch (prec) {                                      \
    case P64: { using SP = Store64; __VA_ARGS__; } break;        \
    case P32: { using SP = Store32; __VA_ARGS__; } break;        \
    case P16: { using SP = Store16<false>; __VA_ARGS__; } break; \
    case PB16: { using SP = Store16<true>; __VA_ARGS__; } break; \
    default: return cudaErrorInvalidValue;             \
  }

template <class SP, bool PACK>
void run_half(const Geom& g, void* field, double* canon, int nrhs, size_t stride, cudaStream_t s) {
  const size_t ts = sizeof(typename SP::T);
  const int sites = tile_sites(g.Ls, ts, 1);
  const int tiles = (g.Vh + sites - 1) / sites;
  auto k = (reinterpret_cast<uintptr_t>(field) & 15) == 0 ? half_kernel<SP, PACK, true> : half_kernel<SP, PACK, false>;
  k<<<(unsigned)tiles * nrhs, kBlasThreads, tile_bytes(g.Ls, sites, ts, 1), s>>>(g, field, canon, stride, sites, tiles);
}

cudaError_t launch_pack_half(const Geom& g, int prec, void* dst, const double* src, int nrhs,
                             cudaStream_t s) {
  DWF_PREC_SWITCH(prec, SP, run_half<SP, true>(g, dst, const_cast<double*>(src), nrhs, field_bytes(g, prec), s));
  return cudaGetLastError();
}

cudaError_t launch_unpack_half(const Geom& g, int prec, double* dst, const void* src, int nrhs,
                               cudaStream_t s) {
  DWF_PREC_SWITCH(prec, SP, run_half<SP, false>(g, const_cast<void*>(src), dst, nrhs, field_bytes(g, prec), s));
  return cudaGetLastError();
}

template <bool SPLIT>
cudaError_t run_full(const Geom& g, void* p0, void* p1, double* full, cudaStream_t s) {
  const int sites = tile_sites(g.Ls, 8, 2);
  full_kernel<SPLIT><<<(g.Vh + sites - 1) / sites, kBlasThreads, tile_bytes(g.Ls, sites, 8, 2), s>>>(g, p0, p1, full, sites);
  return cudaGetLastError();
}

cudaError_t launch_split_full(const Geom& g, void* p0, void* p1, const double* full, cudaStream_t s) {
  return run_full<true>(g, p0, p1, const_cast<double*>(full), s);
}

cudaError_t launch_merge_full(const Geom& g, double* full, const void* p0, const void* p1,
                              cudaStream_t s) {
  return run_full<false>(g, const_cast<void*>(p0), const_cast<void*>(p1), full, s);
}

cudaError_t launch_gauge_convert(const Geom& g, const double* U, void* g64, void* g32, void* g16,
                                 cudaStream_t s) {
  const int per = kGaugeSites / 2;
  gauge_convert_kernel<<<(g.Vh + per - 1) / per, kBlasThreads, 0, s>>>(
      g, U, reinterpret_cast<double2*>(g64), reinterpret_cast<float4*>(g32),
      reinterpret_cast<uint4*>(g16));
  return cudaGetLastError();
}

cudaError_t launch_source_pb(const Geom& g, void* p0, void* p1, const double* src, cudaStream_t s) {
  const Shape sh = elementwise((size_t)g.N5 / 2);
  source_pb_kernel<<<dim3(sh.blocks, 2), sh.threads, 0, s>>>(g, p0, p1, src);
  return cudaGetLastError();
}

cudaError_t launch_extract_z1(const Geom& g, double* prop, const void* p0, const void* p1,
                              cudaStream_t s) {
  const Shape sh = elementwise((size_t)g.Vh * 24);
  extract_z1_kernel<<<sh.blocks, sh.threads, 0, s>>>(g, prop, p0, p1);
  return cudaGetLastError();
}

cudaError_t launch_xr_update(const Geom& g, int prec, int xprec, void* x, void* r, const void* p,
                             const void* w, const double* num, const double* den, int sstride,
                             int nrhs, size_t stride_x, size_t stride, const Reduce* red,
                             cudaStream_t s, const int* active) {
  const Shape sh = elementwise((size_t)g.N5 / 2);
  const dim3 grid(sh.blocks, nrhs);
  if (xprec == prec) {
    DWF_PREC_SWITCH(prec, SP, xr_update_kernel<SP, SP><<<grid, sh.threads, 0, s>>>(g, x, r, p, w, num, den, sstride, stride_x, stride, *red, active));
  } else if (xprec == P32) {
    DWF_PREC_SWITCH(prec, SP, xr_update_kernel<Store32, SP><<<grid, sh.threads, 0, s>>>(g, x, r, p, w, num, den, sstride, stride_x, stride, *red, active));
  } else {
    return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_p_update(const Geom& g, int prec, void* p, const void* z, const double* num,
                            const double* den, int sstride, int nrhs, size_t stride,
                            cudaStream_t s, const int* active) {
  const Shape sh = elementwise((size_t)g.N5 / 2);
  const dim3 grid(sh.blocks, nrhs);
  DWF_PREC_SWITCH(prec, SP, p_update_kernel<SP><<<grid, sh.threads, 0, s>>>(g, p, z, num, den, sstride, stride, active));
  return cudaGetLastError();
}

template <class SPD>
cudaError_t convert_from(const Geom& g, void* dst, int prec_s, const void* src, int nrhs, size_t sd,
                         size_t ss, const Reduce* red, cudaStream_t s, const int* active) {
  const Shape sh = elementwise((size_t)g.N5 / 2);
  const dim3 grid(sh.blocks, nrhs);
  Reduce r{};
  if (red) r = *red;
  const int dn = red != nullptr;
  DWF_PREC_SWITCH(prec_s, SPS, convert_kernel<SPD, SPS><<<grid, sh.threads, 0, s>>>(g, dst, src, sd, ss, r, dn, active));
  return cudaGetLastError();
}

cudaError_t launch_convert(const Geom& g, int prec_d, void* dst, int prec_s, const void* src,
                           int nrhs, size_t sd, size_t ss, const Reduce* red, cudaStream_t s,
                           const int* active) {
  switch (prec_d) {
    case P64: return convert_from<Store64>(g, dst, prec_s, src, nrhs, sd, ss, red, s, active);
    case P32: return convert_from<Store32>(g, dst, prec_s, src, nrhs, sd, ss, red, s, active);
    case P16: return convert_from<Store16<false>>(g, dst, prec_s, src, nrhs, sd, ss, red, s, active);
    case PB16: return convert_from<Store16<true>>(g, dst, prec_s, src, nrhs, sd, ss, red, s, active);
  }
  return cudaErrorInvalidValue;
}


template <class SPX>
cudaError_t px_from(const Geom& g, int prec, void* x, void* p, const void* z, const double* a_ptr,
                    const double* num, const double* den, int sstride, int nrhs, size_t sx,
                    size_t sp, cudaStream_t s, const int* active, int do_p) {
  const Shape sh = elementwise((size_t)g.N5 / 2);
  const dim3 grid(sh.blocks, nrhs);
  DWF_PREC_SWITCH(prec, SP, px_update_kernel<SPX, SP><<<grid, sh.threads, 0, s>>>(g, x, p, z, a_ptr, num, den, sstride, sx, sp, active, do_p));
  return cudaGetLastError();
}

cudaError_t launch_px_update(const Geom& g, int prec, int xprec, void* x, void* p, const void* z,
                             const double* a_ptr, const double* num, const double* den,
                             int sstride, int nrhs, size_t sx, size_t sp, cudaStream_t s,
                             const int* active) {
  if (xprec == P64) return px_from<Store64>(g, prec, x, p, z, a_ptr, num, den, sstride, nrhs, sx, sp, s, active, 1);
  return px_from<Store32>(g, prec, x, p, z, a_ptr, num, den, sstride, nrhs, sx, sp, s, active, 1);
}

cudaError_t launch_x_update(const Geom& g, int prec, int xprec, void* x, const void* p,
                            const double* a_ptr, int sstride, int nrhs, size_t sx, size_t sp,
                            cudaStream_t s, const int* active) {
  void* pp = const_cast<void*>(p);
  if (xprec == P64) return px_from<Store64>(g, prec, x, pp, nullptr, a_ptr, a_ptr, a_ptr, sstride, nrhs, sx, sp, s, active, 0);
  return px_from<Store32>(g, prec, x, pp, nullptr, a_ptr, a_ptr, a_ptr, sstride, nrhs, sx, sp, s, active, 0);
}

cudaError_t launch_pxb_update(const Geom& g, int prec, int xprec, void* x, const void* p,
                              void* pnew, void* bp, const void* z, const double* a_ptr, const SumIn& num,
                              const double* den, int sstride, int nrhs, size_t sx, size_t sp,
                              const void* bdiag, const void* boff, size_t cstride, cudaStream_t s,
                              const int* active, int do_x, bool ahead) {
  // threads for whole sites per warp
  const int half = g.Ls / 2, per = 32 / half * half;
  if (half > 16) return cudaErrorInvalidValue;
  const Shape sh = elementwise(((size_t)g.N5 / 2 + per - 1) / per * 32);
  const dim3 grid(sh.blocks, nrhs);
  if (prec == P32 && xprec == P32) {
    return launch_ahead(ahead, pxb_update_kernel<Store32, Store32>, grid, sh.threads, 0, s, g, x, p, pnew, bp, z, a_ptr, num,
                        den, sstride, sx, sp, reinterpret_cast<const float*>(bdiag),
                        reinterpret_cast<const float*>(boff), cstride, active, do_x);
  }
  if (prec == P32 && xprec == P64) {
    return launch_ahead(ahead, pxb_update_kernel<Store64, Store32>, grid, sh.threads, 0, s, g, x, p, pnew, bp, z, a_ptr, num,
                        den, sstride, sx, sp, reinterpret_cast<const float*>(bdiag),
                        reinterpret_cast<const float*>(boff), cstride, active, do_x);
  }
  if (prec == P64 && xprec == P64) {
    return launch_ahead(ahead, pxb_update_kernel<Store64, Store64>, grid, sh.threads, 0, s, g, x, p, pnew, bp, z, a_ptr, num,
                        den, sstride, sx, sp, reinterpret_cast<const double*>(bdiag),
                        reinterpret_cast<const double*>(boff), cstride, active, do_x);
  }
  if (prec == P16 && xprec == P32) {
    return launch_ahead(ahead, pxb_update_kernel<Store32, Store16<false>>, grid, sh.threads, 0, s, g, x, p, pnew, bp, z, a_ptr, num,
                        den, sstride, sx, sp, reinterpret_cast<const float*>(bdiag),
                        reinterpret_cast<const float*>(boff), cstride, active, do_x);
  }
  if (prec == PB16 && xprec == P32) {
    return launch_ahead(ahead, pxb_update_kernel<Store32, Store16<true>>, grid, sh.threads, 0, s, g, x, p, pnew, bp, z, a_ptr, num,
                        den, sstride, sx, sp, reinterpret_cast<const float*>(bdiag),
                        reinterpret_cast<const float*>(boff), cstride, active, do_x);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_finish_sum(const SumIn& in, int nrhs, cudaStream_t s, const int* active) {
  finish_sum_kernel<<<nrhs, 32, 0, s>>>(in, active);
  return cudaGetLastError();
}

cudaError_t launch_accumulate64(const Geom& g, void* x64, int prec_s, void* src, int zero_src,
                                int nrhs, size_t sd, size_t ss, cudaStream_t s, const int* active) {
  const Shape sh = elementwise((size_t)g.N5 / 2);
  const dim3 grid(sh.blocks, nrhs);
  DWF_PREC_SWITCH(prec_s, SPS, accumulate64_kernel<SPS><<<grid, sh.threads, 0, s>>>(g, x64, src, zero_src, sd, ss, active));
  return cudaGetLastError();
}

cudaError_t launch_sub64_norm(const Geom& g, void* out, const void* a, const void* b, int nrhs,
                              size_t stride, const Reduce* red, cudaStream_t s, const int* active) {
  const Shape sh = elementwise((size_t)g.N5 / 2);
  const dim3 grid(sh.blocks, nrhs);
  sub64_norm_kernel<<<grid, sh.threads, 0, s>>>(g, out, a, b, stride, *red, active);
  return cudaGetLastError();
}

cudaError_t launch_sub_to(const Geom& g, int prec_d, void* dst, const void* a64, const void* b32,
                          int nrhs, size_t sd, size_t sa, size_t sb, const Reduce* red,
                          cudaStream_t s, const int* active) {
  const Shape sh = elementwise((size_t)g.N5 / 2);
  const dim3 grid(sh.blocks, nrhs);
  switch (prec_d) {
    case P32:
      sub_to_kernel<Store32><<<grid, sh.threads, 0, s>>>(g, dst, a64, b32, sd, sa, sb, *red, active);
      break;
    case P16:
      sub_to_kernel<Store16<false>><<<grid, sh.threads, 0, s>>>(g, dst, a64, b32, sd, sa, sb, *red,
                                                                  active);
      break;
    case PB16:
      sub_to_kernel<Store16<true>><<<grid, sh.threads, 0, s>>>(g, dst, a64, b32, sd, sa, sb, *red,
                                                                 active);
      break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_norm(const Geom& g, int prec, const void* x, int nrhs, size_t stride,
                        const Reduce* red, cudaStream_t s) {
  const Shape sh = elementwise((size_t)g.N5 / 2);
  const dim3 grid(sh.blocks, nrhs);
  DWF_PREC_SWITCH(prec, SP, norm_kernel<SP><<<grid, sh.threads, 0, s>>>(g, x, stride, *red));
  return cudaGetLastError();
}

cudaError_t launch_dot_re64(const Geom& g, const void* a, const void* b, int nrhs, size_t stride,
                            const Reduce* red, cudaStream_t s) {
  const Shape sh = elementwise((size_t)g.N5 / 2);
  const dim3 grid(sh.blocks, nrhs);
  dot_re64_kernel<<<grid, sh.threads, 0, s>>>(g, a, b, stride, *red);
  return cudaGetLastError();
}

}  // namespace dwf
