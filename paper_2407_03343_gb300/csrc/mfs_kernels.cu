// CUDA kernels of the hot path (sm_103a).
//
//  pair kernels        steps 2+3 of the G_hat apply (Sec. 2.2, eq. uAll): for every
//                      collocation node x_i of sphere k,
//                        out_i = mu_i + sqrt(w_i) sum_{k' != k} [S f + R t + D d](x_i - y)
//                      over the proxy Stokeslets and the image S/R/D triples of all other
//                      spheres (eq. lin_comb).  Direct summation, so the self block is
//                      skipped instead of being added and subtracted (allowed by Sec. 2.2).
//                      Sources are staged through shared memory in rounds; positions are stored
//                      relative to their sphere centre and shifted into the target sphere's
//                      frame while staging.  FP32 (pairs_kernel): NT targets per thread, sums
//                      folded into Kahan-compensated accumulators across rounds, the centre
//                      difference in float-float.  Double-float (pairs_dw_*) and native FP64
//                      (pairs_fp64_*, velocity_fp64_kernel): see there.
//  gemv_kernel<T>      batched row-major GEMV for the one-body pseudo-inverse factors
//                      (eq. transform), HBM-bound.
//  Krylov kernels      multi-dot, update, scale (GMRES with CGS2), FP64 partial sums.
//  ft_kernel           forces and torques from the strengths (Sec. 2.3 remark), FP64.
//  rhs_kernel          W u_bc (eq. bc, eq. lq2), FP64.
//  assemble_self       B_k = W_k G^(kk) column-major FP64 for the one-time factorisation.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <utility>
#include <vector>

#include "mfs_internal.h"

namespace mfs {
namespace {

constexpr int kPairThreads = 128;
constexpr int kTileProxy = 256; // proxy sources staged per round
constexpr int kTileImg = 128;   // image nodes staged per round
constexpr double kPi = 3.14159265358979323846;

// four doubles moved as one 32-byte-aligned unit
struct __align__(32) D4 {
  double x, y, z, w;
};

template <typename T> struct Prec;
template <> struct Prec<float> {
  using V4 = float4;
  static __device__ __forceinline__ float rsq(float x) { return rsqrtf(x); }
  static __device__ __forceinline__ V4 mk(float a, float b, float c, float d) { return make_float4(a, b, c, d); }
};
template <> struct Prec<double> {
  using V4 = D4;
  // 1/sqrt(x): FP32 hardware estimate y refined by one third-order step of the binomial series,
  // y (1 - e)^(-1/2) = y (1 + e (1/2 + 3 e / 8) + ...) with e = 1 - x y^2 ~ 2^-22 (the dropped
  // term is below 2^-66); five FP64 operations against seven of two Newton steps.
  static __device__ __forceinline__ double rsq(double x) {
    const double y = (double)rsqrtf((float)x);
    const double e = fma(-(x * y), y, 1.0);
    return fma(y, e * fma(0.375, e, 0.5), y);
  }
  static __device__ __forceinline__ V4 mk(double a, double b, double c, double d) { return D4{a, b, c, d}; }
};

// Kahan-compensated s += x.
__device__ __forceinline__ void comp_add(float& s, float& c, float x) {
  float y = x - c;
  float t = s + y;
  c = (t - s) - y;
  s = t;
}

// Centre of sphere o minus centre of the target frame, in the working precision.
struct CentreShift32 {
  const float* hi;
  const float* lo;
  float kh[3], kl[3];
  __device__ void init(int k) {
    for (int c = 0; c < 3; ++c) {
      kh[c] = hi[3 * k + c];
      kl[c] = lo[3 * k + c];
    }
  }
  __device__ __forceinline__ float d(int o, int c) const { return (hi[3 * o + c] - kh[c]) + (lo[3 * o + c] - kl[c]); }
};
struct CentreShift64 {
  const double* cen;
  double kc[3];
  __device__ void init(int k) {
    for (int c = 0; c < 3; ++c) kc[c] = k >= 0 ? cen[3 * k + c] : 0.0;
  }
  __device__ __forceinline__ double d(int o, int c) const { return cen[3 * o + c] - kc[c]; }
};
template <typename T>
struct PairArgs {
  const typename Prec<T>::V4* tgt;  // (x, y, z, sqrt w) relative to the tile's sphere (absolute if sphere < 0)
  const int* tile_sphere;
  const int* tile_start;
  const int* tile_count;
  const typename Prec<T>::V4* proxy;  // N, relative to the owner centre
  int N, P;
  const typename Prec<T>::V4* img;    // image nodes relative to the owner centre
  const int* img_owner;
  const int* img_off;
  int n_img;
  const long long* unk_off;
  const float* cen_hi;
  const float* cen_lo;
  const double* cen64;
  const float4* proxy2;  // double-float copy of proxy: high words, low words
  const float2* lam2;    // double-float strengths (double-float kernels), in place of lam
  const T* lam;
  const T* mu;   // may be null: then out = scale * sum (no W, no identity)
  T* out;
  T scale;       // 1 / (8 pi mu)
  T dip;         // 2 mu: dipole strengths rescaled so that scale * dip = 1 / (4 pi)
  float span;    // a little over the sphere radius plus the proxy radius: bounds |x - c| + |y - c'| on every axis
};

// One target tile (NT nodes per thread) against every source of every other sphere.
template <typename T, int NT>
__device__ __forceinline__ void pair_tile(const PairArgs<T>& A, const int t) {
  using V4 = typename Prec<T>::V4;
  __shared__ V4 sp[kTileProxy];
  __shared__ V4 sf[kTileProxy];
  __shared__ V4 si[3 * kTileImg];

  const int k = A.tile_sphere[t];
  const int start = A.tile_start[t];
  const int cnt = A.tile_count[t];
  CentreShift32 sh;
  sh.hi = A.cen_hi;
  sh.lo = A.cen_lo;
  sh.init(k);

  T x[NT], y[NT], z[NT], ux[NT], uy[NT], uz[NT];
  T sx[NT], sy[NT], sz[NT], cx[NT], cy[NT], cz[NT];
#pragma unroll
  for (int q = 0; q < NT; ++q) {
    int idx = threadIdx.x + q * kPairThreads;
    int node = start + (idx < cnt ? idx : cnt - 1);
    V4 p = A.tgt[node];
    x[q] = p.x; y[q] = p.y; z[q] = p.z;
    ux[q] = uy[q] = uz[q] = T(0);
    sx[q] = sy[q] = sz[q] = T(0);
    cx[q] = cy[q] = cz[q] = T(0);
  }
  const T far = T(1e18);

  // ---- proxy Stokeslets of every sphere but k
  const int total = A.P * A.N;
  // the proxies before and after sphere k's own, in tiles with exact trip counts
  for (int rr = 0; rr < 2; ++rr) {
  const int r_lo = rr == 0 ? 0 : (k + 1) * A.N;
  const int r_hi = rr == 0 ? k * A.N : total;
  for (int s0 = r_lo; s0 < r_hi; s0 += kTileProxy) {
    const int ns = min(kTileProxy, r_hi - s0);
    __syncthreads();
    for (int i = threadIdx.x; i < ns; i += kPairThreads) {
      int j = s0 + i;
      V4 pos = Prec<T>::mk(far, far, far, T(0)), str = Prec<T>::mk(T(0), T(0), T(0), T(0));
      if (j < total) {
        int o = j / A.N;
        int jj = j - o * A.N;
        V4 pr = A.proxy[jj];
        pos = Prec<T>::mk(pr.x + sh.d(o, 0), pr.y + sh.d(o, 1), pr.z + sh.d(o, 2), T(0));
        if (o != k) {
          const T* l = A.lam + A.unk_off[o] + 3LL * jj;
          str = Prec<T>::mk(l[0], l[1], l[2], T(0));
        }
      }
      sp[i] = pos;
      sf[i] = str;
    }
    __syncthreads();
#pragma unroll 2
    for (int j = 0; j < ns; ++j) {
      const V4 p = sp[j];
      const V4 f = sf[j];
#pragma unroll
      for (int q = 0; q < NT; ++q) {
        T dx = x[q] - p.x, dy = y[q] - p.y, dz = z[q] - p.z;
        T r2 = dx * dx + dy * dy + dz * dz;
        T ir = Prec<T>::rsq(r2);
        T ir2 = ir * ir;
        T rf = dx * f.x + dy * f.y + dz * f.z;
        T c = rf * ir2;
        ux[q] += ir * (f.x + c * dx);
        uy[q] += ir * (f.y + c * dy);
        uz[q] += ir * (f.z + c * dz);
      }
    }
#pragma unroll
    for (int q = 0; q < NT; ++q) {
      comp_add(sx[q], cx[q], ux[q]);
      comp_add(sy[q], cy[q], uy[q]);
      comp_add(sz[q], cz[q], uz[q]);
      ux[q] = uy[q] = uz[q] = T(0);
    }
  }
  }

  // ---- image nodes (Stokeslet + rotlet + potential dipole at one position)
  const int self_lo = A.img_off[k], self_hi = A.img_off[k + 1];
  for (int rr = 0; rr < 2; ++rr) {
  const int r_lo = rr == 0 ? 0 : self_hi;
  const int r_hi = rr == 0 ? self_lo : A.n_img;
  for (int s0 = r_lo; s0 < r_hi; s0 += kTileImg) {
    const int ns = min(kTileImg, r_hi - s0);
    __syncthreads();
    for (int i = threadIdx.x; i < ns; i += kPairThreads) {
      int j = s0 + i;
      V4 a = Prec<T>::mk(far, far, far, T(0)), b = Prec<T>::mk(T(0), T(0), T(0), T(0)), c = b;
      if (j < A.n_img) {
        int o = A.img_owner[j];
        V4 pr = A.img[j];
        T px = pr.x + sh.d(o, 0), py = pr.y + sh.d(o, 1), pz = pr.z + sh.d(o, 2);
        if (o != k) {
          const T* l = A.lam + A.unk_off[o] + 3LL * A.N + 9LL * (j - A.img_off[o]);
          a = Prec<T>::mk(px, py, pz, l[0]);
          b = Prec<T>::mk(l[1], l[2], l[3], l[4]);
          c = Prec<T>::mk(l[5], A.dip * l[6], A.dip * l[7], A.dip * l[8]);
        } else {
          a = Prec<T>::mk(px, py, pz, T(0));
        }
      }
      si[3 * i] = a;
      si[3 * i + 1] = b;
      si[3 * i + 2] = c;
    }
    __syncthreads();
    for (int j = 0; j < ns; ++j) {
      const V4 a = si[3 * j], b = si[3 * j + 1], c = si[3 * j + 2];
      // f = (a.w, b.x, b.y), t = (b.z, b.w, c.x), d = (c.y, c.z, c.w)
#pragma unroll
      for (int q = 0; q < NT; ++q) {
        T dx = x[q] - a.x, dy = y[q] - a.y, dz = z[q] - a.z;
        T r2 = dx * dx + dy * dy + dz * dz;
        T ir = Prec<T>::rsq(r2);
        T ir2 = ir * ir;
        T ir3 = ir * ir2;
        // Stokeslet
        T rf = dx * a.w + dy * b.x + dz * b.y;
        T cs = rf * ir2;
        T vx = ir * (a.w + cs * dx), vy = ir * (b.x + cs * dy), vz = ir * (b.y + cs * dz);
        // rotlet: (t x r) / r^3
        vx += ir3 * (b.w * dz - c.x * dy);
        vy += ir3 * (c.x * dx - b.z * dz);
        vz += ir3 * (b.z * dy - b.w * dx);
        // potential dipole: -d / r^3 + 3 (d.r) r / r^5
        T rd = dx * c.y + dy * c.z + dz * c.w;
        T c3 = T(3) * rd * ir3 * ir2;
        vx += c3 * dx - ir3 * c.y;
        vy += c3 * dy - ir3 * c.z;
        vz += c3 * dz - ir3 * c.w;
        ux[q] += vx;
        uy[q] += vy;
        uz[q] += vz;
      }
    }
#pragma unroll
    for (int q = 0; q < NT; ++q) {
      comp_add(sx[q], cx[q], ux[q]);
      comp_add(sy[q], cy[q], uy[q]);
      comp_add(sz[q], cz[q], uz[q]);
      ux[q] = uy[q] = uz[q] = T(0);
    }
  }
  }

#pragma unroll
  for (int q = 0; q < NT; ++q) {
    int idx = threadIdx.x + q * kPairThreads;
    if (idx < cnt) {
      long long node = start + idx;
      T sw = A.tgt[node].w;
      T gx = (sx[q] + cx[q]) * A.scale, gy = (sy[q] + cy[q]) * A.scale, gz = (sz[q] + cz[q]) * A.scale;
      A.out[3 * node] = A.mu[3 * node] + sw * gx;
      A.out[3 * node + 1] = A.mu[3 * node + 1] + sw * gy;
      A.out[3 * node + 2] = A.mu[3 * node + 2] + sw * gz;
    }
  }
}

template <typename T>
PairArgs<T> make_args(const TargetSet& tg, const SourceSet& src, const T* lam, const T* mu, T* out, double visc,
                      int nt = 4) {
  PairArgs<T> A;
  if constexpr (sizeof(T) == 4) {
    A.tgt = tg.pos32;
    A.proxy = src.proxy32;
    A.img = src.img32;
  } else {
    A.tgt = reinterpret_cast<const D4*>(tg.pos64);
    A.proxy = reinterpret_cast<const D4*>(src.proxy64);
    A.img = reinterpret_cast<const D4*>(src.img64);
  }
  A.tile_sphere = nt == 4 ? tg.tile_sphere : tg.tile1_sphere;
  A.tile_start = nt == 4 ? tg.tile_start : tg.tile1_start;
  A.tile_count = nt == 4 ? tg.tile_count : tg.tile1_count;
  A.N = src.N;
  A.P = src.P;
  A.img_owner = src.img_owner;
  A.img_off = src.img_off;
  A.n_img = src.n_img;
  A.unk_off = src.unk_off;
  A.cen_hi = src.cen_hi;
  A.cen_lo = src.cen_lo;
  A.cen64 = src.cen64;
  A.proxy2 = src.proxy2;
  A.lam2 = nullptr;
  A.lam = lam;
  A.mu = mu;
  A.out = out;
  A.scale = T(1.0 / (8.0 * kPi * visc));
  A.dip = T(2.0 * visc);
  A.span = (float)(1.001 * src.span);
  return A;
}

// ------------------------------------------------------------------ native FP64 pair sums
// Bound by the FP64 pipe (two lanes per SM and clock, so one warp per scheduler saturates it):
// 22 FP64 operations a (node, Stokeslet) pair.  What matters is that every SM gets the same share of
// it down to the last CTA, so a CTA takes 32 targets (a 128-node tile in four pieces; a sphere's
// ragged last tile then wastes at most 31 lanes) and its four warps take every fourth source, with
// the sources split further over CTAs where there are few targets.  Measured (20 spheres with
// images, 5.7e8 pairs): 39.3 ms with a thread per node of 128- and 512-node tiles, 25.4
// now; 16,125 flow points around three spheres: 3.44 and 0.86 ms.
constexpr int kFp64Warps = kPairThreads / 32;
constexpr int kFp64Tile = 256;     // proxy sources staged per round
constexpr int kFp64TileImg = 128;  // image nodes staged per round

// Sums at the 32 points of this CTA over its share of the sources: proxies [p0, p1) and image
// nodes [i0, i1) of the lists without sphere k's own (k < 0: nothing left out).  Returns the sums in
// the lanes of warp 0.
__device__ __forceinline__ void fp64_sums(const PairArgs<double>& A, int k, double x, double y, double z, int part,
                                          int nparts, double (&out)[3]) {
  __shared__ D4 sp[kFp64Tile], sf[kFp64Tile];
  __shared__ D4 si[3 * kFp64TileImg];
  __shared__ double red[kFp64Warps][3][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  CentreShift64 sh;
  sh.cen = A.cen64;
  sh.init(k);
  double ux = 0, uy = 0, uz = 0;

  // ---- proxy Stokeslets of every sphere but k: this part's share of the list, in runs before and
  // after sphere k's own
  const int total = A.P * A.N;
  const int p_lo = k < 0 ? total : k * A.N, p_w = k < 0 ? 0 : A.N;
  const long long p_eff = total - p_w;
  const int pe[2] = {(int)(p_eff * part / nparts), (int)(p_eff * (part + 1) / nparts)};
  for (int rr = 0; rr < 2; ++rr) {
    const int r_lo = rr == 0 ? min(pe[0], p_lo) : max(pe[0], p_lo) + p_w;
    const int r_hi = rr == 0 ? min(pe[1], p_lo) : max(pe[1], p_lo) + p_w;
    for (int s0 = r_lo; s0 < r_hi; s0 += kFp64Tile) {
      const int ns = min(kFp64Tile, r_hi - s0);
      __syncthreads();
      for (int i = threadIdx.x; i < ns; i += kPairThreads) {
        const int j = s0 + i, o = j / A.N, jj = j - o * A.N;
        const D4 pr = A.proxy[jj];
        const double* l = A.lam + A.unk_off[o] + 3LL * jj;
        sp[i] = D4{pr.x + sh.d(o, 0), pr.y + sh.d(o, 1), pr.z + sh.d(o, 2), 0.0};
        sf[i] = D4{l[0], l[1], l[2], 0.0};
      }
      __syncthreads();
#pragma unroll 2
      for (int j = warp; j < ns; j += kFp64Warps) {
        const D4 p = sp[j], f = sf[j];
        const double dx = x - p.x, dy = y - p.y, dz = z - p.z;
        const double ir = Prec<double>::rsq(fma(dz, dz, fma(dy, dy, dx * dx)));
        const double c = fma(dz, f.z, fma(dy, f.y, dx * f.x)) * ir * ir;
        ux = fma(ir, fma(c, dx, f.x), ux);
        uy = fma(ir, fma(c, dy, f.y), uy);
        uz = fma(ir, fma(c, dz, f.z), uz);
      }
    }
  }

  // ---- image nodes (Stokeslet + rotlet + potential dipole at one position)
  const int i_lo = k < 0 ? A.n_img : A.img_off[k], i_w = k < 0 ? 0 : A.img_off[k + 1] - i_lo;
  const long long i_eff = A.n_img - i_w;
  const int ie[2] = {(int)(i_eff * part / nparts), (int)(i_eff * (part + 1) / nparts)};
  for (int rr = 0; rr < 2; ++rr) {
    const int r_lo = rr == 0 ? min(ie[0], i_lo) : max(ie[0], i_lo) + i_w;
    const int r_hi = rr == 0 ? min(ie[1], i_lo) : max(ie[1], i_lo) + i_w;
    for (int s0 = r_lo; s0 < r_hi; s0 += kFp64TileImg) {
      const int ns = min(kFp64TileImg, r_hi - s0);
      __syncthreads();
      for (int i = threadIdx.x; i < ns; i += kPairThreads) {
        const int j = s0 + i, o = A.img_owner[j];
        const D4 pr = A.img[j];
        const double* l = A.lam + A.unk_off[o] + 3LL * A.N + 9LL * (j - A.img_off[o]);
        si[3 * i] = D4{pr.x + sh.d(o, 0), pr.y + sh.d(o, 1), pr.z + sh.d(o, 2), l[0]};
        si[3 * i + 1] = D4{l[1], l[2], l[3], l[4]};
        si[3 * i + 2] = D4{l[5], A.dip * l[6], A.dip * l[7], A.dip * l[8]};
      }
      __syncthreads();
      for (int j = warp; j < ns; j += kFp64Warps) {
        const D4 a = si[3 * j], b = si[3 * j + 1], c = si[3 * j + 2];
        // f = (a.w, b.x, b.y), t = (b.z, b.w, c.x), d = (c.y, c.z, c.w)
        const double dx = x - a.x, dy = y - a.y, dz = z - a.z;
        const double ir = Prec<double>::rsq(fma(dz, dz, fma(dy, dy, dx * dx)));
        const double ir2 = ir * ir, ir3 = ir * ir2;
        // Stokeslet
        const double cs = fma(dz, b.y, fma(dy, b.x, dx * a.w)) * ir2;
        double vx = ir * fma(cs, dx, a.w), vy = ir * fma(cs, dy, b.x), vz = ir * fma(cs, dz, b.y);
        // rotlet (t x r) / r^3 and potential dipole -d / r^3 + 3 (d.r) r / r^5
        const double c3 = 3.0 * fma(dz, c.w, fma(dy, c.z, dx * c.y)) * ir2;
        vx = fma(ir3, fma(b.w, dz, -c.x * dy) + fma(c3, dx, -c.y), vx);
        vy = fma(ir3, fma(c.x, dx, -b.z * dz) + fma(c3, dy, -c.z), vy);
        vz = fma(ir3, fma(b.z, dy, -b.w * dx) + fma(c3, dz, -c.w), vz);
        ux += vx;
        uy += vy;
        uz += vz;
      }
    }
  }
  red[warp][0][lane] = ux;
  red[warp][1][lane] = uy;
  red[warp][2][lane] = uz;
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    out[c] = 0.0;
    if (warp == 0)
      for (int w = 0; w < kFp64Warps; ++w) out[c] += red[w][c][lane];
    out[c] *= A.scale;
  }
}

// One 32-node piece (0..3) of a 128-node tile: out = mu + sqrt(w) u, or this part's partial sums.
__device__ __forceinline__ void pair_piece_fp64(const PairArgs<double>& A, int t, int piece, int part, int nparts,
                                                double* __restrict__ partial, long long pstride) {
  const int start = A.tile_start[t] + 32 * piece, cnt = min(32, A.tile_count[t] - 32 * piece);
  if (cnt <= 0) return;
  const int lane = threadIdx.x & 31;
  const long long node = start + min(lane, cnt - 1);
  const D4 p = A.tgt[node];
  double u[3];
  fp64_sums(A, A.tile_sphere[t], p.x, p.y, p.z, part, nparts, u);
  if (threadIdx.x >= cnt) return;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (nparts > 1) partial[part * pstride + 3 * node + c] = u[c];
    else A.out[3 * node + c] = A.mu[3 * node + c] + p.w * u[c];
  }
}

// ------------------------------------------------------------------ double-float pair kernel
// FP64-accurate pair sums on the FP32 pipes.  A value is an unevaluated sum hi + lo of two
// floats (double-word arithmetic).  Error-free transforms: TwoSum (Knuth, TAOCP vol. 2),
// FastTwoSum and TwoProd via FMA (Dekker 1971); DW+DW and DW*DW follow the "sloppy" sum
// and the FMA-based product of Joldes, Muller and Popescu (ACM TOMS 44, 2017), whose
// absolute errors stay at ~2^-46 of the operands even under cancellation, which is what
// the pair sums need: the strengths lambda_hat = B^+ mu can exceed the field they produce
// by 1e9 or more (Sec. 2.2, truncation 5e-12), so every term must be accurate to ~1e-14.
struct dw {
  float h, l;
};
// The _rn intrinsics are never contracted into FMAs, which the error-free transforms
// rely on (a fused a*b + w would break the rounded product they assume).
__device__ __forceinline__ dw two_sum(float a, float b) {
  float s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}
__device__ __forceinline__ dw fast_two_sum(float a, float b) {
  float s = __fadd_rn(a, b);
  float e = __fsub_rn(b, __fsub_rn(s, a));
  return {s, e};
}
__device__ __forceinline__ dw two_prod(float a, float b) {
  float p = __fmul_rn(a, b);
  float e = __fmaf_rn(a, b, -p);
  return {p, e};
}
__device__ __forceinline__ dw dw_add(dw x, dw y) {
  dw s = two_sum(x.h, y.h);
  float v = __fadd_rn(x.l, y.l);
  return fast_two_sum(s.h, __fadd_rn(s.l, v));
}
__device__ __forceinline__ dw dw_mul(dw x, dw y) {
  dw c = two_prod(x.h, y.h);
  float t = __fmul_rn(x.h, y.l);
  t = __fmaf_rn(x.l, y.h, t);
  return fast_two_sum(c.h, __fadd_rn(c.l, t));
}
__device__ __forceinline__ dw dw_split(double v) {
  float h = (float)v;
  return {h, (float)(v - (double)h)};
}
__device__ __forceinline__ double dw_join(dw x) { return (double)x.h + (double)x.l; }
// ------------------------------------------------------------------ packed FP32
// Two FP32 lanes per instruction (sm_100+ f32x2): the FMA pipe does one lane-operation per lane
// either way (measured: fma, add, mul and sub all at 95 % of 152 x 128 lanes x the SM clock, the
// scalar forms at 92 %), but half the issue slots are free for loads, selects and MUFU.
typedef unsigned long long f2x;
__device__ __forceinline__ f2x f2add(f2x a, f2x b) {
  f2x d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2x f2sub(f2x a, f2x b) {
  f2x d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2x f2mul(f2x a, f2x b) {
  f2x d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2x f2fma(f2x a, f2x b, f2x c) {
  f2x d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f2x f2make(float lo, float hi) {
  f2x d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void f2split(f2x v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2x f2dup(float v) { return f2make(v, v); }
__device__ __forceinline__ f2x f2neg(f2x v) { return v ^ 0x8000000080000000ull; }
__device__ __forceinline__ float rsqrt_ftz(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// two double-word values, one per lane: high and low words packed
struct dw2 {
  f2x h, l;
};
// a + b = s + e and a - b = s + e exactly in both lanes (Knuth).  Finding the larger operand by
// compare and select on the ALU pipe, for Dekker's three additions, measured 2-5 % slower in the
// pair kernel (28.4-30.0 against 27.9 ms on 100 spheres) although it takes a fifth of its work off
// the FMA pipe.
__device__ __forceinline__ dw2 two_sum2(f2x a, f2x b) {
  const f2x s = f2add(a, b), bb = f2sub(s, a);
  return {s, f2add(f2sub(a, f2sub(s, bb)), f2sub(b, bb))};
}
__device__ __forceinline__ dw2 two_diff2(f2x a, f2x b) {
  const f2x s = f2sub(a, b), bb = f2sub(s, a);
  return {s, f2sub(f2sub(a, f2sub(s, bb)), f2add(b, bb))};
}
__device__ __forceinline__ dw2 fast_two_sum2(f2x a, f2x b) {
  const f2x s = f2add(a, b);
  return {s, f2sub(b, f2sub(s, a))};
}
__device__ __forceinline__ dw2 dw2_add(dw2 x, dw2 y) {
  const dw2 s = two_sum2(x.h, y.h);
  return fast_two_sum2(s.h, f2add(s.l, f2add(x.l, y.l)));
}
// product and sum without renormalisation: the exact error of the high parts plus the first-order
// terms of the low ones
__device__ __forceinline__ dw2 mul2u(dw2 x, dw2 y) {
  const f2x p = f2mul(x.h, y.h);
  return {p, f2fma(x.l, y.h, f2fma(x.h, y.l, f2fma(x.h, y.h, f2neg(p))))};
}
__device__ __forceinline__ dw2 add2u(dw2 x, dw2 y) {
  const dw2 s = two_sum2(x.h, y.h);
  return {s.h, f2add(s.l, f2add(x.l, y.l))};
}

// ------------------------------------------------------------------ double-float pair sums
// Each thread holds one target at a time and evaluates two sources per instruction (the lanes), so
// a source pair is read from shared memory as it is stored and a lane sums every second source.
// What bounds the sums is the FMA pipe: 164 lane-operations a (node, Stokeslet) pair, 170
// close to the target's sphere (the earlier scalar evaluation: 204, and its issue slots) and 383 an image triple (436).  Measured on 100
// spheres (5.59e9 pairs): 26.85 ms, 89 % of the measured packed rate, against 43.1 ms.  The evaluation keeps
// the accuracy of a renormalised double-word one (~2^-46 of the operands) with fewer operations:
//  - positions of a (target sphere, source sphere) segment are split on a common power-of-two grid
//    per axis, so the difference of the high words is exact without a two-sum (a third word where the
//    proxies may come close);
//  - with s = 1/|d| to FP32 accuracy (MUFU and one Newton step on the high words) the unit vector
//    u = d / |d| is formed as s d, and its deviation 1 - |s d|^2, found to ~2^-48 by a chain of
//    fused multiply-adds from 1 whose roundings are recovered exactly, corrects u and 1/|d| at
//    second order; the field needs only u and 1/|d| (Stokeslet: (f + (u.f) u) / |d|);
//  - products and sums inside a term but for u.f are not renormalised (their low words stay below
//    ~2^-23 of the operands), and the terms are summed in groups of eight per lane with exact high
//    sums and plain low sums, the groups in double-word arithmetic: a group's roundings scale with the
//    group's sum instead of with the running sum.
// Root mean square error per absolute sum (16 / 31 / 96 / 200 / 800 proxies of one sphere, random
// strengths): 1.8 / 1.4 / 0.80 / 0.55 / 0.28e-15, that of adding every renormalised term in double-word
// arithmetic 2.0 / 1.6 / 1.05 / 0.73 / 0.35e-15.  At first order, with u.f as it comes, a Newton step of
// one more rounding and groups of sixteen it is 3.0 / 2.4 / 1.3 / 1.0 / 0.48e-15 (and 100 spheres 26.1 ms).
constexpr int kDwTile = 256;     // proxy sources staged per round (one sphere's)
constexpr int kDwTileImg = 64;   // image nodes staged per round (one sphere's)
constexpr int kDwGroup = 8;      // terms per lane and group
// Threads of a double-float CTA: the 128-node tiles are taken in two pieces, and a piece without targets
// ends at once, so 823 nodes a sphere run as 13 CTAs of 64 (832 places) and not as 7 of 128 (896), and
// the last wave is made of half as long CTAs.  Measured against CTAs of 128 (same rule for the parts): 100
// spheres 27.8 -> 26.1 ms, the dilute solve of 20 spheres 36.8 -> 35.9 ms (with first-order terms; 26.9 and
// 35.6 now); two spheres and the batch of motions the same within 2 %.
constexpr int kDwThreads = 64;
constexpr int kDwPieces = kPairThreads / kDwThreads;
static_assert(kDwPieces == kPairPieces, "arrival counters");
// resident CTAs per SM (128 registers); 10 (96 registers) and 12 (80) were slower (with first-order terms): 100
// spheres 26.8 and 26.6 ms against 26.1, two spheres 49.7 and 50.6 us against 41.8
constexpr int kDwCtas = 8;
constexpr int kDwMultiCtas = 6;  // of the kernel over several right-hand sides (3 x the sums; 168 registers)

// Sources of one round in shared memory: source pair u holds its two sources' components side by
// side, pos[3 u ..]: (xh yh), (zh xl), (yl zl), strengths likewise.
struct DwGeom {          // geometry of one target and two sources
  f2x p[3], np[3], l[3];  // unit vector: high words, their negatives, low words
  f2x s, ns, il;          // 1/|d|: high word, its negative, low word
};

struct DwTarget {        // a target in the grid of the current segment, duplicated into both lanes
  f2x h[3], l[3], r[3];  // (r: third words, DW_REST)
};

// How positions are held: double-float words; high words on the segment's grid; high and low words on
// grids and a third word (rest: the sources' third words)
enum { DW_FREE, DW_GRID, DW_REST };

template <int FORM>
__device__ __forceinline__ void dw_geometry(const DwTarget& T, const ulonglong2 a, const ulonglong2 b,
                                            const ulonglong2 c, const f2x* rest, DwGeom& g) {
  const f2x yh[3] = {a.x, a.y, b.x}, yl[3] = {b.y, c.x, c.y};
  const f2x mtwo = f2dup(-2.0f), mhalf = f2dup(-0.5f);
  f2x dh[3], dl[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const dw2 t = FORM != DW_FREE ? dw2{f2sub(T.h[q], yh[q]), 0} : two_diff2(T.h[q], yh[q]);
    const f2x tl = f2sub(T.l[q], yl[q]);
    const dw2 d = fast_two_sum2(t.h, FORM != DW_FREE ? tl : f2add(t.l, tl));
    dh[q] = d.h;
    dl[q] = FORM == DW_REST ? f2add(d.l, f2sub(T.r[q], rest[q])) : d.l;
  }
  const f2x r2 = f2fma(dh[2], dh[2], f2fma(dh[1], dh[1], f2mul(dh[0], dh[0])));
  float r0, r1;
  f2split(r2, r0, r1);
  // one Newton step in residual form, s0 + s0 (1 - r2 s0^2) / 2: its last rounding is that of the
  // result, so s is off by ~1.3e-7 at most (2e-7 as s0 (3 - r2 s0^2) / 2, the same four operations)
  const f2x s0 = f2make(rsqrt_ftz(r0), rsqrt_ftz(r1));
  g.s = f2fma(s0, f2fma(f2mul(f2mul(r2, mhalf), s0), s0, f2dup(0.5f)), s0);
  g.ns = f2neg(g.s);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    g.p[q] = f2mul(g.s, dh[q]);
    g.np[q] = f2mul(g.ns, dh[q]);
    g.l[q] = f2fma(g.s, dl[q], f2fma(g.s, dh[q], g.np[q]));
  }
  // e = (1 - |p + l|^2) / 2: the chain -2 + px^2 + py^2 + pz^2 (which stays within a factor of two,
  // so its differences are exact) with each rounding recovered, and the cross terms p.l
  const f2x a1 = f2fma(g.p[0], g.p[0], mtwo), a2 = f2fma(g.p[1], g.p[1], a1), a3 = f2fma(g.p[2], g.p[2], a2);
  const f2x t = f2add(f2add(f2fma(g.p[0], g.p[0], f2sub(mtwo, a1)), f2fma(g.p[1], g.p[1], f2sub(a1, a2))),
                      f2fma(g.p[2], g.p[2], f2sub(a2, a3)));
  const f2x nq = f2fma(g.np[2], g.l[2], f2fma(g.np[1], g.l[1], f2mul(g.np[0], g.l[0])));
  const f2x e0 = f2fma(mhalf, f2add(f2add(a3, f2dup(1.0f)), t), nq);
  // 1/|p + l| = 1 + e + 3/2 e^2 + ..: the second term reaches 2e-14, always of one sign
  const f2x e = f2fma(f2mul(e0, f2dup(1.5f)), e0, e0);
  g.il = f2mul(g.s, e);
#pragma unroll
  for (int q = 0; q < 3; ++q) g.l[q] = f2fma(g.p[q], e, g.l[q]);
}

// u . f as -nh + l, renormalised (FastTwoSum: l is below 2^-22 |f|, so where it exceeds a cancelled
// nh what is lost is below 2^-46 |f|)
__device__ __forceinline__ void dw_ndot(const DwGeom& g, const f2x (&fh)[3], const f2x (&fl)[3], f2x& nh, f2x& l) {
  f2x n[3], e[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    n[q] = f2mul(g.np[q], fh[q]);
    e[q] = f2fma(g.l[q], fh[q], f2fma(g.p[q], fl[q], f2fma(g.p[q], fh[q], n[q])));
  }
  const dw2 s1 = two_sum2(n[0], n[1]);
  const dw2 s2 = two_sum2(s1.h, n[2]);                                      // -(u.f), high word
  const f2x lo = f2sub(f2add(f2add(e[0], e[1]), f2sub(e[2], s1.l)), s2.l);  // +(u.f), low word
  nh = f2sub(s2.h, lo);
  l = f2sub(lo, f2sub(s2.h, nh));
}

// v = f + (u.f) u in component q, from nh = -(u.f)_h, ph = (u.f)_h and l = (u.f)_l
__device__ __forceinline__ dw2 dw_project(const DwGeom& g, int q, f2x fh, f2x fl, f2x nh, f2x ph, f2x l) {
  const f2x nm = f2mul(nh, g.p[q]);
  const f2x e = f2fma(l, g.p[q], f2fma(ph, g.l[q], f2fma(nh, g.np[q], nm)));
  const dw2 s = two_diff2(fh, nm);
  return {s.h, f2add(s.l, f2add(fl, e))};
}

// group sum += v / |d|
__device__ __forceinline__ void dw_accumulate(const DwGeom& g, dw2 v, dw2& sum) {
  const f2x nt = f2mul(g.ns, v.h);
  const f2x e = f2fma(g.il, v.h, f2fma(g.s, v.l, f2fma(g.s, v.h, nt)));
  const dw2 s = two_diff2(sum.h, nt);
  sum.h = s.h;
  sum.l = f2add(sum.l, f2add(s.l, e));
}

// v / |d| (three in a row in an image triple: the low parts' product is kept as well)
__device__ __forceinline__ dw2 dw_over_r(const DwGeom& g, dw2 v) {
  const f2x nt = f2mul(g.ns, v.h);
  return {f2neg(nt), f2fma(g.il, f2add(v.h, v.l), f2fma(g.s, v.l, f2fma(g.s, v.h, nt)))};
}

// the lanes of a round's double-word sums joined onto the target's sum
__device__ __forceinline__ void dw_fold(dw& u, const dw2& m) {
  float h0, h1, l0, l1;
  f2split(m.h, h0, h1);
  f2split(m.l, l0, l1);
  u = dw_add(u, dw_add(dw{h0, l0}, dw{h1, l1}));
}

// A thread's target and its sums for R right-hand sides.
template <int R>
struct DWTile {
  dw x[3];
  dw u[R][3];
};

// whether this warp has a target of the piece
__device__ __forceinline__ bool dw_warp_live(int cnt) { return (int)(threadIdx.x & ~31u) < cnt; }

template <int R>
__device__ __forceinline__ void dw_load_targets(const PairArgs<double>& A, int start, int cnt, DWTile<R>& T) {
  const int idx = threadIdx.x;
  const D4 p = A.tgt[start + (idx < cnt ? idx : cnt - 1)];
  T.x[0] = dw_split(p.x);
  T.x[1] = dw_split(p.y);
  T.x[2] = dw_split(p.z);
#pragma unroll
  for (int r = 0; r < R; ++r) T.u[r][0] = T.u[r][1] = T.u[r][2] = dw{0.f, 0.f};
}

// Grid of a segment: on each axis the spacing 2^(e - 24) with 2^e above every |x - y| of the
// segment (centre distance plus twice the radius), so high words on it subtract exactly.  What lies
// below the low words, 2^(e - 49), then is an absolute error of the positions; where a proxy may come
// closer than a quarter of 2^e to a target (centres within 3.6 radii at r_proxy 0.63) it would exceed
// the terms' other roundings.  There the low words are put on a second grid, 2^(e - 46), and subtract
// exactly too, and a third word holds the rest: six lane-operations more (a two-sum of double-float
// words: 18, and twice the error).  Nodes within 0.2 of proxies at 0.97 of the surface, gap 1e-3, 31 / 96 /
// 200 proxies: rms error 10.2 / 3.8 / 2.9e-15 of the absolute sum in two words, 2.2 / 1.1 / 0.8e-15 in three; a
// double-float difference in the scalar evaluation 3.2 / 1.5 / 1.0e-15.  Where every segment is close it costs
// 4 % (8 spheres of 400 proxies 295 -> 305 us), on 100 spheres 0.1 %.
struct DwGrid {
  dw shift[3];    // source sphere's centre minus target sphere's
  float rest[3];  // what the split leaves of it (three words)
  float m32[3];   // 2^(e-1): rounds |x| < 2^(e-1) to the grid as (|x| + m32) - m32
  bool close;     // whether the segment takes three words
};
// The grid of sphere o's segment, by one warp, an axis a lane: FP64 operations take 16 clocks of an SM's two
// lanes a warp, whatever the lanes hold.
__device__ __forceinline__ void dw_grid(const PairArgs<double>& A, const CentreShift64& sh, int o, DwGrid& G) {
  const int lane = threadIdx.x & 31, q = min(lane, 2);
  const double v = sh.cen[3 * o + q] - (q == 0 ? sh.kc[0] : q == 1 ? sh.kc[1] : sh.kc[2]);
  const dw s = dw_split(v);
  const float rest = (float)(v - dw_join(s));
  const float b = fabsf(s.h) * 1.0001f + A.span;
  // half the power of two above b (b is a normal number: at least the sphere's radius)
  const float m32 = 0.5f * __int_as_float((__float_as_int(b) & 0x7f800000) + 0x00800000);
  const float h[3] = {__shfl_sync(~0u, s.h, 0), __shfl_sync(~0u, s.h, 1), __shfl_sync(~0u, s.h, 2)};
  const float m[3] = {__shfl_sync(~0u, m32, 0), __shfl_sync(~0u, m32, 1), __shfl_sync(~0u, m32, 2)};
  const float gap = norm3df(h[0], h[1], h[2]) - A.span;
  if (lane < 3) {
    G.shift[q] = s;
    G.rest[q] = rest;
    G.m32[q] = m32;
    G.close = !(fmaxf(m[0], fmaxf(m[1], m[2])) <= 2.0f * gap);
  }
}
// x rounded to the grid (a float of 2^(e-1) and above lies on it)
__device__ __forceinline__ float dw_on_grid(float x, float m32) {
  const float t = fabsf(x);
  return copysignf(t >= m32 ? t : __fsub_rn(__fadd_rn(t, m32), m32), x);
}
// x rounded to the second grid, |x| up to 2^(e - 24)
__device__ __forceinline__ float dw_on_grid2(float x, float m32) {
  const float m = __fmul_rn(m32, 1.5f * 0x1p-22f);
  return __fsub_rn(__fadd_rn(x, m), m);
}
// A proxy's position in the target's frame, in FP32 operations only: with the position and the strengths
// held in double, the sums, splits and conversions of a source were about 25 FP64 operations, 12 clocks of
// an SM's two FP64 lanes, where 64 targets spend about 84 clocks on a source.
__device__ __forceinline__ void dw_stage_pos(const DwGrid& G, const float4 ph, const float4 pl, float* sp, float* rest,
                                             int i) {
  const float rh[3] = {ph.x, ph.y, ph.z}, rl[3] = {pl.x, pl.y, pl.z};
  float* o = sp + 12 * (i >> 1) + (i & 1);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const dw s = two_sum(rh[q], G.shift[q].h);
    float h, l;
    if (G.close) {
      const dw t = two_sum(rl[q], G.shift[q].l), u = two_sum(s.l, t.h), y = fast_two_sum(s.h, u.h);
      h = dw_on_grid(y.h, G.m32[q]);
      const dw v = two_sum(__fsub_rn(y.h, h), y.l);
      l = dw_on_grid2(v.h, G.m32[q]);
      rest[6 * (i >> 1) + 2 * q + (i & 1)] =
          __fadd_rn(__fsub_rn(v.h, l), __fadd_rn(v.l, __fadd_rn(u.l, __fadd_rn(t.l, G.rest[q]))));
    } else {
      h = dw_on_grid(s.h, G.m32[q]);
      l = __fadd_rn(__fsub_rn(s.h, h), __fadd_rn(s.l, __fadd_rn(rl[q], G.shift[q].l)));
    }
    o[2 * q] = h;
    o[6 + 2 * q] = l;
  }
}
template <int FORM>
__device__ __forceinline__ DwTarget dw_target(const DwGrid& G, const dw (&x)[3]) {
  DwTarget t;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const float h = dw_on_grid(x[q].h, G.m32[q]);
    t.h[q] = f2dup(h);
    if constexpr (FORM == DW_REST) {
      const dw v = two_sum(__fsub_rn(x[q].h, h), x[q].l);
      const float l = dw_on_grid2(v.h, G.m32[q]);
      t.l[q] = f2dup(l);
      t.r[q] = f2dup(__fadd_rn(__fsub_rn(v.h, l), v.l));
    } else {
      t.l[q] = f2dup(__fadd_rn(__fsub_rn(x[q].h, h), x[q].l));
    }
  }
  return t;
}

// A round of nu source pairs against the targets of the piece.
template <int R, int TILE, int FORM>
__device__ __forceinline__ void dw_proxy_round(const DwGrid& G, unsigned mask, int nu, int cnt, const float* sp,
                                               const float* rest, const float (*sf)[6 * TILE], DWTile<R>& T) {
  if (!dw_warp_live(cnt)) return;
  const DwTarget X = dw_target<FORM>(G, T.x);
  dw2 m[R][3];
#pragma unroll
  for (int r = 0; r < R; ++r) m[r][0] = m[r][1] = m[r][2] = dw2{0, 0};
  for (int u0 = 0; u0 < nu; u0 += kDwGroup) {
    dw2 sum[R][3];
#pragma unroll
    for (int r = 0; r < R; ++r) sum[r][0] = sum[r][1] = sum[r][2] = dw2{0, 0};
    const int u1 = min(nu, u0 + kDwGroup);
#pragma unroll 2
    for (int u = u0; u < u1; ++u) {
      const ulonglong2* P = reinterpret_cast<const ulonglong2*>(sp) + 3 * u;
      DwGeom g;
      dw_geometry<FORM>(X, P[0], P[1], P[2], reinterpret_cast<const f2x*>(rest) + 3 * u, g);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (R > 1 && !(mask >> r & 1u)) continue;
        const ulonglong2* F = reinterpret_cast<const ulonglong2*>(sf[r]) + 3 * u;
        const ulonglong2 fa = F[0], fb = F[1], fc = F[2];
        const f2x fh[3] = {fa.x, fa.y, fb.x}, fl[3] = {fb.y, fc.x, fc.y};
        f2x nh, l;
        dw_ndot(g, fh, fl, nh, l);
        const f2x ph = f2neg(nh);
#pragma unroll
        for (int c = 0; c < 3; ++c) dw_accumulate(g, dw_project(g, c, fh[c], fl[c], nh, ph, l), sum[r][c]);
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int c = 0; c < 3; ++c) m[r][c] = dw2_add(m[r][c], sum[r][c]);
  }
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < 3; ++c) dw_fold(T.u[r][c], m[r][c]);
}

// Proxy Stokeslets [r_lo, r_hi) of the flattened proxy index (sphere o = j / N, proxy j - o N; the
// range holds none of the target sphere's own), one sphere at a time in rounds of at most TILE.
template <int R, int TILE>
__device__ __forceinline__ void dw_proxy_range(const PairArgs<double>& A, const CentreShift64& sh,
                                               const float2* const (&lam)[R], unsigned mask, int r_lo, int r_hi,
                                               int cnt, float* sp, float (*sf)[6 * TILE], DwGrid* grids, int& segs,
                                               DWTile<R>& T) {
  for (int s0 = r_lo; s0 < r_hi;) {
    const int o = s0 / A.N, j0 = s0 - o * A.N;
    const int seg = min(r_hi - s0, A.N - j0);  // what is left of sphere o
    // a new segment's grid goes to the place that was last read two segments, so two barriers, ago
    if (s0 == r_lo || j0 == 0) {
      ++segs;
      if (threadIdx.x < 32) dw_grid(A, sh, o, grids[segs & 1]);
    }
    __syncthreads();
    const DwGrid G = grids[segs & 1];
    // even rounds of whole groups; third words take the place of a third of the sources
    constexpr int kClose = 2 * TILE / 3 / (2 * kDwGroup) * (2 * kDwGroup);
    static_assert(kClose > 0 && 9 * kClose <= 6 * TILE, "third words behind the positions");
    float* const rest = sp + 6 * kClose;
    const int tile = G.close ? kClose : TILE;
    const int rounds = (seg + tile - 1) / tile;
    const int ns = min(seg, ((seg + rounds - 1) / rounds + 2 * kDwGroup - 1) / (2 * kDwGroup) * (2 * kDwGroup));
    const int nu = (ns + 1) >> 1;
    for (int i = threadIdx.x; i < 2 * nu; i += kDwThreads) {
      const int jj = j0 + min(i, ns - 1);
      dw_stage_pos(G, A.proxy2[2 * jj], A.proxy2[2 * jj + 1], sp, rest, i);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const bool on = i < ns && (mask >> r & 1u);  // the odd round's last slot carries no strength
        const float2* l = lam[r] + A.unk_off[o] + 3LL * jj;
        float* f = sf[r] + 12 * (i >> 1) + (i & 1);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const float2 v = on ? l[q] : make_float2(0.f, 0.f);
          f[2 * q] = v.x;
          f[6 + 2 * q] = v.y;
        }
      }
    }
    __syncthreads();
    if (G.close) dw_proxy_round<R, TILE, DW_REST>(G, mask, nu, cnt, sp, rest, sf, T);
    else dw_proxy_round<R, TILE, DW_GRID>(G, mask, nu, cnt, sp, rest, sf, T);
    s0 += ns;
  }
}

// Image nodes [r_lo, r_hi) (Stokeslet f, rotlet t and potential dipole q at one position; none of
// the target sphere's own), one sphere at a time.  With u and 1/r the triple's field is
//   (1/r) [ f + (u.f) u + (1/r) [ t x u + (1/r) (3 (u.q) u - q) ] ].
// Strengths per right-hand side and pair of nodes: f, t, -q and 3 q, high and low words.
template <int R, int TILE>
__device__ __forceinline__ void dw_image_range(const PairArgs<double>& A, const CentreShift64& sh,
                                               const float2* const (&lam)[R], unsigned mask, int r_lo, int r_hi,
                                               int cnt, float* sp, float (*si)[24 * TILE], DWTile<R>& T) {
  for (int s0 = r_lo; s0 < r_hi;) {
    const int o = A.img_owner[s0];
    const int first = A.img_off[o];
    const int ns = min(TILE, min(r_hi, A.img_off[o + 1]) - s0);
    const int nu = (ns + 1) >> 1;
    __syncthreads();
    // a thread per node and axis: the FP64 operations of a warp take the same time for three nodes as for
    // one (a thread per node: two spheres with 20 images 43.0 us, now 40.4)
    for (int t = threadIdx.x; t < 6 * nu; t += kDwThreads) {
      const int i = t / 3, q = t - 3 * i;
      const int j = s0 + min(i, ns - 1);
      const D4 pr = A.img[j];
      const double shift = sh.cen[3 * o + q] - (q == 0 ? sh.kc[0] : q == 1 ? sh.kc[1] : sh.kc[2]);
      const dw y = dw_split((q == 0 ? pr.x : q == 1 ? pr.y : pr.z) + shift);
      float* f = sp + 12 * (i >> 1) + (i & 1) + 2 * q;
      f[0] = y.h;
      f[6] = y.l;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const bool on = i < ns && (mask >> r & 1u);
        const float2* l = lam[r] + A.unk_off[o] + 3LL * A.N + 9LL * (j - first) + q;
        const float2 zero = make_float2(0.f, 0.f);
        const float2 vf = on ? l[0] : zero, vt = on ? l[3] : zero, vq = on ? l[6] : zero;
        const double d = A.dip * ((double)vq.x + (double)vq.y);
        const dw v[4] = {{vf.x, vf.y}, {vt.x, vt.y}, dw_split(-d), dw_split(3.0 * d)};
        float* g = si[r] + 48 * (i >> 1) + (i & 1) + 2 * q;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          g[12 * w] = v[w].h;
          g[12 * w + 6] = v[w].l;
        }
      }
    }
    __syncthreads();
    if (dw_warp_live(cnt)) {
      DwTarget X;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        X.h[c] = f2dup(T.x[c].h);
        X.l[c] = f2dup(T.x[c].l);
      }
      dw2 m[R][3];
#pragma unroll
      for (int r = 0; r < R; ++r) m[r][0] = m[r][1] = m[r][2] = dw2{0, 0};
#pragma unroll 1
      for (int u = 0; u < nu; ++u) {
        const ulonglong2* P = reinterpret_cast<const ulonglong2*>(sp) + 3 * u;
        DwGeom g;
        dw_geometry<DW_FREE>(X, P[0], P[1], P[2], nullptr, g);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (R > 1 && !(mask >> r & 1u)) continue;
          const ulonglong2* F = reinterpret_cast<const ulonglong2*>(si[r]) + 12 * u;
          dw2 y[3];
          {  // (1/r) (3 (u.q) u - q)
            const ulonglong2 ta = F[9], tb = F[10], tc = F[11];
            const f2x th[3] = {ta.x, ta.y, tb.x}, tl[3] = {tb.y, tc.x, tc.y};
            f2x nh, l;
            dw_ndot(g, th, tl, nh, l);
            const f2x ph = f2neg(nh);
            const ulonglong2 qa = F[6], qb = F[7], qc = F[8];
            const f2x qh[3] = {qa.x, qa.y, qb.x}, ql[3] = {qb.y, qc.x, qc.y};
#pragma unroll
            for (int c = 0; c < 3; ++c) y[c] = dw_over_r(g, dw_project(g, c, qh[c], ql[c], nh, ph, l));
          }
          {  // + t x u, then / r
            const ulonglong2 ta = F[3], tb = F[4], tc = F[5];
            const dw2 t[3] = {{ta.x, tb.y}, {ta.y, tc.x}, {tb.x, tc.y}};
            const dw2 un[3] = {{g.p[0], g.l[0]}, {g.p[1], g.l[1]}, {g.p[2], g.l[2]}};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              const int c1 = (c + 1) % 3, c2 = (c + 2) % 3;
              const dw2 b = mul2u(t[c2], un[c1]);
              y[c] = dw_over_r(g, add2u(y[c], add2u(mul2u(t[c1], un[c2]), dw2{f2neg(b.h), f2neg(b.l)})));
            }
          }
          {  // + f + (u.f) u, then / r
            const ulonglong2 fa = F[0], fb = F[1], fc = F[2];
            const f2x fh[3] = {fa.x, fa.y, fb.x}, fl[3] = {fb.y, fc.x, fc.y};
            f2x nh, l;
            dw_ndot(g, fh, fl, nh, l);
            const f2x ph = f2neg(nh);
#pragma unroll
            for (int c = 0; c < 3; ++c)
              m[r][c] = dw2_add(m[r][c], dw_over_r(g, add2u(dw_project(g, c, fh[c], fl[c], nh, ph, l), y[c])));
          }
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) dw_fold(T.u[r][c], m[r][c]);
    }
    s0 += ns;
  }
}

// out = mu + sqrt(w) scale u per node, or the scaled partial sum of this source part
template <int R>
__device__ __forceinline__ void dw_write_out(const PairArgs<double>& A, int start, int cnt, const DWTile<R>& T, int r,
                                             const double* __restrict__ mu, double* __restrict__ out, int part,
                                             int nparts, double* __restrict__ partial, long long pstride) {
  if ((int)threadIdx.x >= cnt) return;
  const long long node = start + threadIdx.x;
  const double sw = A.tgt[node].w;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const double g = dw_join(T.u[r][c]) * A.scale;
    if (nparts > 1) partial[part * pstride + 3 * node + c] = g;
    else out[3 * node + c] = mu[3 * node + c] + sw * g;
  }
}

template <int R, int TILE, int TILE_IMG>
struct DwShared {
  __align__(16) float sp[6 * (TILE > TILE_IMG ? TILE : TILE_IMG)];  // positions of a round
  union {                                                           // and its strengths
    __align__(16) float sf[R][6 * TILE];
    __align__(16) float si[R][24 * TILE_IMG];
  };
  DwGrid grids[2];
};

// Sources may be split over `nparts` CTAs per target tile (when there are too few tiles to
// fill the GPU): part `part` takes a contiguous share of the tile's source list (the sources of
// every other sphere) and, for nparts > 1, writes its scaled partial sum to
// partial[part * pstride + 3 node + c] for the last part's CTA to add.
template <int R, int TILE, int TILE_IMG>
__device__ __forceinline__ void dw_all_sources(const PairArgs<double>& A, const CentreShift64& sh, int k,
                                               const float2* const (&lam)[R], unsigned mask, int cnt, int part,
                                               int nparts, DwShared<R, TILE, TILE_IMG>& S, DWTile<R>& T) {
  // the proxies before and after sphere k's own (this part's share of them)
  const int total = A.P * A.N;
  const int p_lo = k * A.N, p_w = A.N;
  const long long p_eff = total - p_w;
  const int pe0 = (int)(p_eff * part / nparts), pe1 = (int)(p_eff * (part + 1) / nparts);
  int segs = 0;
#pragma unroll 1  // (one copy of the loops: with two, 8 spheres took 350 us instead of 311)
  for (int rr = 0; rr < 2; ++rr)
    dw_proxy_range<R, TILE>(A, sh, lam, mask, rr ? max(pe0, p_lo) + p_w : min(pe0, p_lo),
                                rr ? max(pe1, p_lo) + p_w : min(pe1, p_lo), cnt, S.sp, S.sf, S.grids, segs, T);
  // image nodes before and after sphere k's own, this part's share
  const int i_lo = A.img_off[k], i_w = A.img_off[k + 1] - i_lo;
  const long long i_eff = A.n_img - i_w;
  const int ie0 = (int)(i_eff * part / nparts), ie1 = (int)(i_eff * (part + 1) / nparts);
#pragma unroll 1
  for (int rr = 0; rr < 2; ++rr)
    dw_image_range<R, TILE_IMG>(A, sh, lam, mask, rr ? max(ie0, i_lo) + i_w : min(ie0, i_lo),
                                    rr ? max(ie1, i_lo) + i_w : min(ie1, i_lo), cnt, S.sp, S.si, T);
}

__device__ __forceinline__ void pair_tile_dw(const PairArgs<double>& A, const int t, const int start, const int cnt,
                                             const int part, const int nparts, double* __restrict__ partial,
                                             const long long pstride) {
  __shared__ DwShared<1, kDwTile, kDwTileImg> S;
  const int k = A.tile_sphere[t];
  CentreShift64 sh;
  sh.cen = A.cen64;
  sh.init(k);
  DWTile<1> T;
  dw_load_targets(A, start, cnt, T);
  const float2* const lam[1] = {A.lam2};
  dw_all_sources<1, kDwTile, kDwTileImg>(A, sh, k, lam, 1u, cnt, part, nparts, S, T);
  dw_write_out<1>(A, start, cnt, T, 0, A.mu, A.out, part, nparts, partial, pstride);
}

// The near part of the far-field split: only the spheres of the target sphere's near list
// (ascending; runs of consecutive spheres are taken as one range).
__device__ __forceinline__ void pair_tile_dw_near(const PairArgs<double>& A, const int* __restrict__ near_off,
                                                  const int* __restrict__ near_idx, const int t, const int start,
                                                  const int cnt, const int part, const int nparts,
                                                  double* __restrict__ partial, const long long pstride) {
  __shared__ DwShared<1, kDwTile, kDwTileImg> S;
  const int k = A.tile_sphere[t];
  CentreShift64 sh;
  sh.cen = A.cen64;
  sh.init(k);
  DWTile<1> T;
  dw_load_targets(A, start, cnt, T);
  const float2* const lam[1] = {A.lam2};
  // this part's share of the near list
  int segs = 0;
  const int b0 = near_off[k], nn = near_off[k + 1] - b0;
  const int a1 = b0 + (int)((long long)nn * (part + 1) / nparts);
  for (int a = b0 + (int)((long long)nn * part / nparts); a < a1;) {
    const int o0 = near_idx[a];
    int o1 = o0;
    while (a + 1 < a1 && near_idx[a + 1] == o1 + 1) {
      ++a;
      ++o1;
    }
    ++a;
    dw_proxy_range<1, kDwTile>(A, sh, lam, 1u, o0 * A.N, (o1 + 1) * A.N, cnt, S.sp, S.sf, S.grids, segs, T);
    dw_image_range<1, kDwTileImg>(A, sh, lam, 1u, A.img_off[o0], A.img_off[o1 + 1], cnt, S.sp, S.si, T);
  }
  dw_write_out<1>(A, start, cnt, T, 0, A.mu, A.out, part, nparts, partial, pstride);
}

// ------------------------------------------------------------------ far-field kernel (FP32)
constexpr int kTileFar = 256;  // equivalent sources staged per round

struct FarArgs {
  const float4* tgt;     // (x - c_k, sqrt w) per node, FP32
  const double* tgt64;   // the same in FP64 (sqrt w taken from here)
  const int* tile_sphere;
  const int* tile_start;
  const int* tile_count;
  const float4* eq;      // n_eq equivalent-source positions relative to the owner centre
  int n_eq, P;
  const int* excl_off;
  const int* excl_idx;
  const float* cen_hi;
  const float* cen_lo;
  const float* q;        // 3 n_eq strengths per sphere
  double* out;
  float scale;           // 1 / (8 pi mu)
};

// out += sqrt(w) scale sum over every sphere outside the target sphere's exclusion list (its
// near spheres and itself) of the Stokeslet field of its equivalent sources.  The excluded
// spheres split the flattened equivalent-source index into runs, each staged in tiles.
template <int NT>
__global__ void __launch_bounds__(kPairThreads) pairs_far_kernel(FarArgs A, int nparts, double* __restrict__ partial,
                                                                 long long pstride) {
  __shared__ float4 sp[kTileFar];
  __shared__ float4 sf[kTileFar];
  const int t = blockIdx.x / nparts, part = blockIdx.x % nparts;
  const int k = A.tile_sphere[t];
  const int start = A.tile_start[t];
  const int cnt = A.tile_count[t];
  CentreShift32 sh;
  sh.hi = A.cen_hi;
  sh.lo = A.cen_lo;
  sh.init(k);
  float x[NT], y[NT], z[NT], ux[NT], uy[NT], uz[NT], sx[NT], sy[NT], sz[NT], cx[NT], cy[NT], cz[NT];
#pragma unroll
  for (int q = 0; q < NT; ++q) {
    int idx = threadIdx.x + q * kPairThreads;
    float4 p = A.tgt[start + (idx < cnt ? idx : cnt - 1)];
    x[q] = p.x; y[q] = p.y; z[q] = p.z;
    ux[q] = uy[q] = uz[q] = sx[q] = sy[q] = sz[q] = cx[q] = cy[q] = cz[q] = 0.f;
  }
  const int e0 = A.excl_off[k], e1 = A.excl_off[k + 1];
  // this part's share [f0, f1) of the far sources, counted in the order of the runs between
  // excluded spheres
  const long long n_far = (long long)(A.P - (e1 - e0)) * A.n_eq;
  const long long f0 = n_far * part / nparts, f1 = n_far * (part + 1) / nparts;
  long long before = 0;  // far sources in the runs before the current one
  int prev = -1;
  for (int a = e0; a <= e1; ++a) {
    const int nxt = a < e1 ? A.excl_idx[a] : A.P;
    const int run_lo = (prev + 1) * A.n_eq, run_hi = nxt * A.n_eq;
    prev = nxt;
    const long long len = run_hi - run_lo;
    const int lo = run_lo + (int)max(0LL, min(len, f0 - before));
    const int hi = run_lo + (int)max(0LL, min(len, f1 - before));
    before += len;
    for (int s0 = lo; s0 < hi; s0 += kTileFar) {
      const int ns = min(kTileFar, hi - s0);
      __syncthreads();
      for (int i = threadIdx.x; i < ns; i += kPairThreads) {
        const int j = s0 + i;
        const int o = j / A.n_eq;
        const int e = j - o * A.n_eq;
        const float4 z0 = A.eq[e];
        sp[i] = make_float4(z0.x + sh.d(o, 0), z0.y + sh.d(o, 1), z0.z + sh.d(o, 2), 0.f);
        const float* g = A.q + 3LL * j;
        sf[i] = make_float4(g[0], g[1], g[2], 0.f);
      }
      __syncthreads();
#pragma unroll 2
      for (int j = 0; j < ns; ++j) {
        const float4 p = sp[j];
        const float4 f = sf[j];
#pragma unroll
        for (int q = 0; q < NT; ++q) {
          float dx = x[q] - p.x, dy = y[q] - p.y, dz = z[q] - p.z;
          float r2 = dx * dx + dy * dy + dz * dz;
          float ir = rsqrtf(r2);
          float ir2 = ir * ir;
          float rf = dx * f.x + dy * f.y + dz * f.z;
          float c = rf * ir2;
          ux[q] += ir * (f.x + c * dx);
          uy[q] += ir * (f.y + c * dy);
          uz[q] += ir * (f.z + c * dz);
        }
      }
#pragma unroll
      for (int q = 0; q < NT; ++q) {
        comp_add(sx[q], cx[q], ux[q]);
        comp_add(sy[q], cy[q], uy[q]);
        comp_add(sz[q], cz[q], uz[q]);
        ux[q] = uy[q] = uz[q] = 0.f;
      }
    }
  }
#pragma unroll
  for (int q = 0; q < NT; ++q) {
    int idx = threadIdx.x + q * kPairThreads;
    if (idx < cnt) {
      long long node = start + idx;
      double sw = A.tgt64[4 * node + 3] * (double)A.scale;
      const double gx = sw * ((double)sx[q] + (double)cx[q]), gy = sw * ((double)sy[q] + (double)cy[q]),
                   gz = sw * ((double)sz[q] + (double)cz[q]);
      if (nparts > 1) {
        double* o = partial + part * pstride + 3 * node;
        o[0] = gx;
        o[1] = gy;
        o[2] = gz;
      } else {
        A.out[3 * node] += gx;
        A.out[3 * node + 1] += gy;
        A.out[3 * node + 2] += gz;
      }
    }
  }
}

// Packed-FP32 variant (sm_100+ f32x2 instructions): the four targets of a thread form two pairs,
// each operation of the pair math runs on both lanes of a pair with one instruction (the FMA pipe
// still does one lane-operation per target, but the issue slots are halved, which is what bounds
// the scalar kernel).  Sources are staged with every component duplicated into both lanes.
__global__ void __launch_bounds__(kPairThreads) pairs_far2_kernel(FarArgs A, int nparts, double* __restrict__ partial,
                                                                  long long pstride) {
  __shared__ ulonglong2 sa[kTileFar];  // (px, px | py, py)
  __shared__ ulonglong2 sb[kTileFar];  // (pz, pz | fx, fx)
  __shared__ ulonglong2 sc[kTileFar];  // (fy, fy | fz, fz)
  constexpr int NT = 4;
  const int t = blockIdx.x / nparts, part = blockIdx.x % nparts;
  const int k = A.tile_sphere[t];
  const int start = A.tile_start[t];
  const int cnt = A.tile_count[t];
  CentreShift32 sh;
  sh.hi = A.cen_hi;
  sh.lo = A.cen_lo;
  sh.init(k);
  float x[NT], y[NT], z[NT], sx[NT], sy[NT], sz[NT], cx[NT], cy[NT], cz[NT];
#pragma unroll
  for (int q = 0; q < NT; ++q) {
    int idx = threadIdx.x + q * kPairThreads;
    float4 p = A.tgt[start + (idx < cnt ? idx : cnt - 1)];
    x[q] = p.x; y[q] = p.y; z[q] = p.z;
    sx[q] = sy[q] = sz[q] = cx[q] = cy[q] = cz[q] = 0.f;
  }
  const f2x X0 = f2make(x[0], x[1]), X1 = f2make(x[2], x[3]);
  const f2x Y0 = f2make(y[0], y[1]), Y1 = f2make(y[2], y[3]);
  const f2x Z0 = f2make(z[0], z[1]), Z1 = f2make(z[2], z[3]);
  const f2x zero2 = f2make(0.f, 0.f);
  const int e0 = A.excl_off[k], e1 = A.excl_off[k + 1];
  const long long n_far = (long long)(A.P - (e1 - e0)) * A.n_eq;
  const long long f0 = n_far * part / nparts, f1 = n_far * (part + 1) / nparts;
  long long before = 0;
  int prev = -1;
  for (int a = e0; a <= e1; ++a) {
    const int nxt = a < e1 ? A.excl_idx[a] : A.P;
    const int run_lo = (prev + 1) * A.n_eq, run_hi = nxt * A.n_eq;
    prev = nxt;
    const long long len = run_hi - run_lo;
    const int lo = run_lo + (int)max(0LL, min(len, f0 - before));
    const int hi = run_lo + (int)max(0LL, min(len, f1 - before));
    before += len;
    for (int s0 = lo; s0 < hi; s0 += kTileFar) {
      const int ns = min(kTileFar, hi - s0);
      __syncthreads();
      for (int i = threadIdx.x; i < ns; i += kPairThreads) {
        const int j = s0 + i;
        const int o = j / A.n_eq;
        const int e = j - o * A.n_eq;
        const float4 z0 = A.eq[e];
        const float px = z0.x + sh.d(o, 0), py = z0.y + sh.d(o, 1), pz = z0.z + sh.d(o, 2);
        const float* g = A.q + 3LL * j;
        const float fx = g[0], fy = g[1], fz = g[2];
        sa[i] = make_ulonglong2(f2make(px, px), f2make(py, py));
        sb[i] = make_ulonglong2(f2make(pz, pz), f2make(fx, fx));
        sc[i] = make_ulonglong2(f2make(fy, fy), f2make(fz, fz));
      }
      __syncthreads();
      f2x ux0 = zero2, uy0 = zero2, uz0 = zero2, ux1 = zero2, uy1 = zero2, uz1 = zero2;
#pragma unroll 2
      for (int j = 0; j < ns; ++j) {
        const ulonglong2 a2 = sa[j], b2 = sb[j], c2 = sc[j];
#define MFS_FAR2_PAIR(X, Y, Z, UX, UY, UZ)                                        \
  {                                                                               \
    const f2x dx = f2sub(X, a2.x), dy = f2sub(Y, a2.y), dz = f2sub(Z, b2.x);      \
    const f2x r2 = f2fma(dz, dz, f2fma(dy, dy, f2mul(dx, dx)));                   \
    float rl, rh;                                                                 \
    f2split(r2, rl, rh);                                                          \
    const f2x ir = f2make(rsqrtf(rl), rsqrtf(rh));                                \
    const f2x ir2 = f2mul(ir, ir);                                                \
    const f2x rf = f2fma(dz, c2.y, f2fma(dy, c2.x, f2mul(dx, b2.y)));             \
    const f2x cc = f2mul(rf, ir2);                                                \
    UX = f2fma(ir, f2fma(cc, dx, b2.y), UX);                                      \
    UY = f2fma(ir, f2fma(cc, dy, c2.x), UY);                                      \
    UZ = f2fma(ir, f2fma(cc, dz, c2.y), UZ);                                      \
  }
        MFS_FAR2_PAIR(X0, Y0, Z0, ux0, uy0, uz0)
        MFS_FAR2_PAIR(X1, Y1, Z1, ux1, uy1, uz1)
#undef MFS_FAR2_PAIR
      }
      float u[3][NT];
      f2split(ux0, u[0][0], u[0][1]);
      f2split(ux1, u[0][2], u[0][3]);
      f2split(uy0, u[1][0], u[1][1]);
      f2split(uy1, u[1][2], u[1][3]);
      f2split(uz0, u[2][0], u[2][1]);
      f2split(uz1, u[2][2], u[2][3]);
#pragma unroll
      for (int q = 0; q < NT; ++q) {
        comp_add(sx[q], cx[q], u[0][q]);
        comp_add(sy[q], cy[q], u[1][q]);
        comp_add(sz[q], cz[q], u[2][q]);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < NT; ++q) {
    int idx = threadIdx.x + q * kPairThreads;
    if (idx < cnt) {
      long long node = start + idx;
      double sw = A.tgt64[4 * node + 3] * (double)A.scale;
      const double gx = sw * ((double)sx[q] + (double)cx[q]), gy = sw * ((double)sy[q] + (double)cy[q]),
                   gz = sw * ((double)sz[q] + (double)cz[q]);
      if (nparts > 1) {
        double* o = partial + part * pstride + 3 * node;
        o[0] = gx;
        o[1] = gy;
        o[2] = gz;
      } else {
        A.out[3 * node] += gx;
        A.out[3 * node + 1] += gy;
        A.out[3 * node + 2] += gz;
      }
    }
  }
}

// out[e] += the parts in order (the far kernel's, already scaled)
__global__ void parts_add_kernel(long long n3, int nparts, const double* __restrict__ partial, long long pstride,
                                 double* __restrict__ out) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n3; e += (long long)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int q = 0; q < nparts; ++q) s += partial[q * pstride + e];
    out[e] += s;
  }
}

// Split sources, fused reduction: every CTA of work item `item` has written its partial sums of the
// tile's nodes; the last one to arrive adds the parts in part order and writes out = mu + sqrt(w) s.
// Returns whether this CTA was the last (all threads see the same answer).
__device__ __forceinline__ bool parts_last_arrival(unsigned* counter, int item, int nparts) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(&counter[item], 1u) == (unsigned)nparts - 1;
    if (last) counter[item] = 0u;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}
// out = mu + sqrt(w) (sum of the parts in part order) at cnt nodes from start: a thread per value, the
// parts' loads issued eight at a time (one at a time, the last CTA's chain of loads was the tail of every
// launch of short problems)
__device__ __forceinline__ void parts_finish_nodes(const D4* tgt, long long start, int cnt, int nparts,
                                                   const double* partial, long long pstride, const double* mu,
                                                   double* out) {
  for (int i = threadIdx.x; i < 3 * cnt; i += blockDim.x) {
    const long long e = 3 * start + i;
    double sum = 0.0;
    for (int q0 = 0; q0 < nparts; q0 += 8) {
      double v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = q0 + q < nparts ? __ldcg(&partial[(q0 + q) * pstride + e]) : 0.0;
#pragma unroll
      for (int q = 0; q < 8; ++q) sum += v[q];
    }
    out[e] = mu[e] + tgt[start + i / 3].w * sum;
  }
}

// The piece of a tile that work item `item` = tile x kDwPieces + piece takes; false if it has no targets.
__device__ __forceinline__ bool dw_piece(const PairArgs<double>& A, int t, int piece, int& start, int& cnt) {
  start = A.tile_start[t] + piece * kDwThreads;
  cnt = min(kDwThreads, A.tile_count[t] - piece * kDwThreads);
  return cnt > 0;
}
__device__ __forceinline__ void parts_finish_piece(const PairArgs<double>& A, int item, int start, int cnt, int nparts,
                                                   const double* partial, long long pstride, unsigned* counter) {
  if (!parts_last_arrival(counter, item, nparts)) return;
  parts_finish_nodes(A.tgt, start, cnt, nparts, partial, pstride, A.mu, A.out);
}

template <typename T, int NT>
__global__ void __launch_bounds__(kPairThreads) pairs_kernel(PairArgs<T> A) {
  pair_tile<T, NT>(A, blockIdx.x);
}
__global__ void __launch_bounds__(kPairThreads) pairs_fp64_kernel(PairArgs<double> A, int nparts, double* partial,
                                                                  long long pstride) {
  const int piece = blockIdx.x % 4, t = blockIdx.x / 4 / nparts, part = blockIdx.x / 4 % nparts;
  pair_piece_fp64(A, t, piece, part, nparts, partial, pstride);
}
// velocity at n arbitrary points x (absolute positions): u, or this part's partial sums
__global__ void __launch_bounds__(kPairThreads) velocity_fp64_kernel(PairArgs<double> A, int n,
                                                                     const double* __restrict__ x, int nparts,
                                                                     double* __restrict__ u, long long pstride) {
  const int part = blockIdx.x % nparts;
  const long long i0 = 32LL * (blockIdx.x / nparts);
  const int cnt = (int)min(32LL, n - i0);
  const long long i = i0 + min((int)(threadIdx.x & 31), cnt - 1);
  double v[3];
  fp64_sums(A, -1, x[3 * i], x[3 * i + 1], x[3 * i + 2], part, nparts, v);
  if (threadIdx.x >= cnt) return;
#pragma unroll
  for (int c = 0; c < 3; ++c) u[part * pstride + 3 * i + c] = v[c];
}
__global__ void __launch_bounds__(kDwThreads, kDwCtas) pairs_dw_kernel(PairArgs<double> A, int nparts, double* partial,
                                                                       long long pstride, unsigned* counter) {
  const int item = blockIdx.x / nparts, t = item / kDwPieces;
  int start, cnt;
  if (!dw_piece(A, t, item % kDwPieces, start, cnt)) return;
  pair_tile_dw(A, t, start, cnt, blockIdx.x % nparts, nparts, partial, pstride);
  if (nparts > 1) parts_finish_piece(A, item, start, cnt, nparts, partial, pstride, counter);
}
__global__ void __launch_bounds__(kDwThreads, kDwCtas) pairs_dw_near_kernel(PairArgs<double> A, const int* near_off,
                                                                     const int* near_idx, int nparts, double* partial,
                                                                     long long pstride, unsigned* counter) {
  const int item = blockIdx.x / nparts, t = item / kDwPieces;
  int start, cnt;
  if (!dw_piece(A, t, item % kDwPieces, start, cnt)) return;
  pair_tile_dw_near(A, near_off, near_idx, t, start, cnt, blockIdx.x % nparts, nparts, partial, pstride);
  if (nparts > 1) parts_finish_piece(A, item, start, cnt, nparts, partial, pstride, counter);
}
// out = mu + sqrt(w) * (sum of the parts), or the plain sum when mu is null; parts added in order
__global__ void pair_parts_reduce_kernel(long long n3, const D4* __restrict__ tgt, int nparts,
                                         const double* __restrict__ partial, long long pstride,
                                         const double* __restrict__ mu, double* __restrict__ out) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n3; e += (long long)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int q = 0; q < nparts; ++q) s += partial[q * pstride + e];
    out[e] = mu ? mu[e] + tgt[e / 3].w * s : s;
  }
}
// Many problems in one launch: work[b] = (problem, tile); problems whose flag is 0 are skipped.
// The per-problem vectors are segments of concatenated ones: lam at lam + uoff[p], mu and out
// at mu + voff[p], out + voff[p].
struct BatchVecs {
  const double* lam;    // native FP64 kernel
  const float2* lam2;   // double-float kernels
  const double* mu;
  double* out;
  const long long* uoff;
  const long long* voff;
  double* partial;     // split sources: nparts slices of the concatenated vector length
  long long pstride;
  const long long* nlen;  // node rows (3 n_colloc) of each problem; a mobility problem's border follows
  unsigned* counter;      // double-float: zeros, one per piece of a work item; with split sources the
                          // last CTA of a piece adds the parts (in part order) and re-arms its counter
};

// native FP64: each (problem, 128-node tile) in four pieces; with split sources the parts are added
// by pair_parts_reduce_batch_kernel
__global__ void __launch_bounds__(kPairThreads, 4) pairs_fp64_batch_kernel(const PairArgs<double>* __restrict__ args,
                                                                        const int2* __restrict__ work,
                                                                        const int* __restrict__ active, BatchVecs bv,
                                                                        int nparts) {
  const int2 w = work[blockIdx.x / 4 / nparts];
  if (!active[w.x]) return;
  PairArgs<double> A = args[w.x];
  A.lam = bv.lam + bv.uoff[w.x];
  A.mu = bv.mu + bv.voff[w.x];
  A.out = bv.out + bv.voff[w.x];
  pair_piece_fp64(A, w.y, blockIdx.x % 4, blockIdx.x / 4 % nparts, nparts, bv.partial + bv.voff[w.x], bv.pstride);
}
__global__ void __launch_bounds__(kDwThreads, kDwCtas) pairs_dw_batch_kernel(const PairArgs<double>* __restrict__ args,
                                                                      const int2* __restrict__ work,
                                                                      const int* __restrict__ active, BatchVecs bv,
                                                                      int nparts) {
  const int item = blockIdx.x / nparts;
  const int2 w = work[item / kDwPieces];
  if (!active[w.x]) return;
  PairArgs<double> A = args[w.x];
  A.lam2 = bv.lam2 + bv.uoff[w.x];
  A.mu = bv.mu + bv.voff[w.x];
  A.out = bv.out + bv.voff[w.x];
  int start, cnt;
  if (!dw_piece(A, w.y, item % kDwPieces, start, cnt)) return;
  pair_tile_dw(A, w.y, start, cnt, blockIdx.x % nparts, nparts, bv.partial + bv.voff[w.x], bv.pstride);
  if (nparts > 1)
    parts_finish_piece(A, item, start, cnt, nparts, bv.partial + bv.voff[w.x], bv.pstride, bv.counter);
}
// ------------------------------------------------------------------ several right-hand sides on one geometry
// The problems of a batch that share a context (the motions of one geometry) have the same
// targets and sources and differ only in their strengths.  Work item (lead problem, 128-node
// tile, first index into the right-hand-side list, count <= kPairRhs): the position
// differences, the distance and its powers of each (node, source) pair are formed once in
// double-float and applied to the strengths of every listed right-hand side (80 of the 214 flops
// of a Stokeslet pair and 98 of the 487 of an image triple are shared).  Each
// right-hand side's sums follow the operation order of pair_tile_dw.
constexpr int kDwTileM = 128;    // proxy sources staged per round
constexpr int kDwTileImgM = 32;  // image nodes staged per round

// work[b] = (lead problem, tile of the 1-node-per-thread tiling, first index into rhs_prob, count);
// the sources are split over nparts CTAs per item as in pairs_dw_batch_kernel
template <int R>
__global__ void __launch_bounds__(kDwThreads, kDwMultiCtas) pairs_dw_multi_kernel(const PairArgs<double>* __restrict__ args,
                                                                      const int4* __restrict__ work,
                                                                      const int* __restrict__ rhs_prob,
                                                                      const int* __restrict__ active, BatchVecs bv,
                                                                      int nparts) {
  __shared__ DwShared<R, kDwTileM, kDwTileImgM> S;
  const int item = blockIdx.x / nparts;
  const int4 w = work[item / kDwPieces];
  const int part = blockIdx.x % nparts;
  int prob[R];
  unsigned mask = 0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    prob[r] = rhs_prob[w.z + min(r, w.w - 1)];
    if (r < w.w && active[prob[r]]) mask |= 1u << r;
  }
  if (!mask) return;
  const PairArgs<double> A = args[w.x];
  const float2* lam[R];
#pragma unroll
  for (int r = 0; r < R; ++r) lam[r] = bv.lam2 + bv.uoff[prob[r]];
  const int t = w.y;
  const int k = A.tile_sphere[t];
  int start, cnt;
  if (!dw_piece(A, t, item % kDwPieces, start, cnt)) return;
  CentreShift64 sh;
  sh.cen = A.cen64;
  sh.init(k);
  DWTile<R> T;
  dw_load_targets(A, start, cnt, T);
  dw_all_sources<R, kDwTileM, kDwTileImgM>(A, sh, k, lam, mask, cnt, part, nparts, S, T);
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (!(mask >> r & 1u)) continue;
    const long long off = bv.voff[prob[r]];
    dw_write_out<R>(A, start, cnt, T, r, bv.mu + off, bv.out + off, part, nparts, bv.partial + off, bv.pstride);
  }
  if (nparts > 1 && parts_last_arrival(bv.counter, item, nparts)) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (!(mask >> r & 1u)) continue;
      const long long off = bv.voff[prob[r]];
      parts_finish_nodes(A.tgt, start, cnt, nparts, bv.partial + off, bv.pstride, bv.mu + off, bv.out + off);
    }
  }
}

// the batched counterpart of pair_parts_reduce_kernel: CTA (chunk of an active problem, piece of
// blockDim elements), so that a single short problem still gets enough CTAs
__global__ void pair_parts_reduce_batch_kernel(SegTable t, const PairArgs<double>* __restrict__ args, BatchVecs bv,
                                               int nparts) {
  const int b = t.list ? t.list[blockIdx.x] : blockIdx.x;
  const int p = t.prob[b];
  if (!t.active[p]) return;
  const long long e = t.start[b] + (long long)blockIdx.y * blockDim.x + threadIdx.x;
  if (e >= t.end[b]) return;
  if (bv.nlen && e - bv.voff[p] >= bv.nlen[p]) return;  // a mobility problem's border rows
  const D4* tgt = args[p].tgt;
  double s = 0.0;
  for (int q = 0; q < nparts; ++q) s += bv.partial[q * bv.pstride + e];
  bv.out[e] = bv.mu[e] + tgt[(e - bv.voff[p]) / 3].w * s;
}

// ------------------------------------------------------------------ batched GEMV
constexpr int kGemvThreads = 256;
constexpr int kGemvRowsPerWarp = 2;

__device__ __forceinline__ float dot_vec(const float4& m, const float* x) {
  return m.x * __ldg(x) + m.y * __ldg(x + 1) + m.z * __ldg(x + 2) + m.w * __ldg(x + 3);
}

// PAIRED: the matrix is stored in row pairs (FP32 copy of Sigma^+ U^T); a warp's two rows are a pair
template <bool PAIRED>
__global__ void __launch_bounds__(kGemvThreads) gemv_kernel(GemvBatch<float> B, const float* __restrict__ x,
                                                            float* __restrict__ y) {
  // jobs sharing a matrix are adjacent, so its rows are read once; with a compacted list the grid
  // covers the active problems' jobs only
  const int job = B.job_list ? B.job_list[blockIdx.x] : blockIdx.x;
  if (B.active && !B.active[B.job_prob[job]]) return;
  const int nr = B.rows[job], nc = B.cols[job], ld = B.ld[job];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r0 = (blockIdx.y * (kGemvThreads / 32) + warp) * kGemvRowsPerWarp;
  if (r0 >= nr) return;
  const float* M = B.mat[job];
  const float* xv = x + B.x_off[job];
  float acc[kGemvRowsPerWarp];
#pragma unroll
  for (int r = 0; r < kGemvRowsPerWarp; ++r) acc[r] = 0.f;
  if constexpr (PAIRED) {
    // a 16-byte load holds two columns of the warp's row pair, so the loads of a warp are contiguous and x is
    // read once for both rows, two elements at a time where its offset is even (loads are what bounds this; four
    // columns a lane with the row loop of the plain layout read the matrix in two strided halves: both factors of
    // N = 400 for 8 / 60 spheres that share them 37.5 / 222 us, now 21 / 79; from plain rows 21 / 103)
    static_assert(kGemvRowsPerWarp == 2, "FP32 row pairs");
    const float* pr = M + (long long)r0 * ld;
    const float4* q = reinterpret_cast<const float4*>(pr);
    if ((reinterpret_cast<uintptr_t>(xv) & 7) == 0) {
      const float2* x2 = reinterpret_cast<const float2*>(xv);
#pragma unroll 4
      for (int v = lane; v < nc / 2; v += 32) {
        const float4 m = __ldg(q + v);
        const float2 xe = __ldg(x2 + v);
        acc[0] += m.x * xe.x + m.z * xe.y;
        acc[1] += m.y * xe.x + m.w * xe.y;
      }
    } else {
#pragma unroll 4
      for (int v = lane; v < nc / 2; v += 32) {
        const float4 m = __ldg(q + v);
        const float xa = __ldg(xv + 2 * v), xb = __ldg(xv + 2 * v + 1);
        acc[0] += m.x * xa + m.z * xb;
        acc[1] += m.y * xa + m.w * xb;
      }
    }
    if ((nc & 1) && lane == 0) {
      acc[0] += pr[2LL * (nc - 1)] * xv[nc - 1];
      acc[1] += pr[2LL * (nc - 1) + 1] * xv[nc - 1];
    }
  } else {
    const int nvec = nc / 4;
    for (int v = lane; v < nvec; v += 32) {
#pragma unroll
      for (int r = 0; r < kGemvRowsPerWarp; ++r) {
        int row = r0 + r;
        if (row < nr) {
          const float4 m = reinterpret_cast<const float4*>(M + (long long)row * ld)[v];
          acc[r] += dot_vec(m, xv + 4 * v);
        }
      }
    }
    for (int c = 4 * nvec + lane; c < nc; c += 32) {
#pragma unroll
      for (int r = 0; r < kGemvRowsPerWarp; ++r) {
        int row = r0 + r;
        if (row < nr) acc[r] += M[(long long)row * ld + c] * xv[c];
      }
    }
  }
#pragma unroll
  for (int r = 0; r < kGemvRowsPerWarp; ++r) {
    float s = acc[r];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0 && r0 + r < nr) y[B.y_off[job] + r0 + r] = s;
  }
}

// Native FP64 y = M x, one right-hand side an item: a CTA takes kGemv64Rows rows, its four warps every
// fourth run of 32 columns, and the next kGemv64Depth loads a row and lane are issued before the
// current ones are used.  Bound by the FP64 pipe once enough rows are there (two lanes per SM and
// clock, 16 bytes of matrix), by load latency below that, which is what the split of the columns and
// the loads in flight are for.  Both factors of one step 1, before (two rows a warp, one load each in
// flight) and now: 100 spheres N = 686 2710 -> 1775 us (the DFMA rate allows 1757), 8 spheres N = 400
// 389 -> 188, two spheres N = 800 213 -> 117, N = 300 43 -> 26.
constexpr int kGemv64Rows = 2, kGemv64Depth = 4, kGemv64Warps = 4;
__global__ void __launch_bounds__(32 * kGemv64Warps) gemv64_kernel(GemvBatch<double> B, const double* __restrict__ x,
                                                                  double* __restrict__ y) {
  constexpr int R = kGemv64Rows, D = kGemv64Depth, S = 32 * kGemv64Warps;
  __shared__ double red[kGemv64Warps][R][32];
  const int job = B.job_list ? B.job_list[blockIdx.x] : blockIdx.x;
  if (B.active && !B.active[B.job_prob[job]]) return;
  const int nr = B.rows[job], nc = B.cols[job];
  const int r0 = blockIdx.y * R;
  if (r0 >= nr) return;
  const long long ld = B.ld[job];
  const double* M = B.mat[job] + r0 * ld;
  const double* xv = x + B.x_off[job];
  double acc[R], cur[D][R], nxt[D][R];
#pragma unroll
  for (int r = 0; r < R; ++r) acc[r] = 0.0;
  auto load = [&](double (&m)[D][R], int c0) {
#pragma unroll
    for (int u = 0; u < D; ++u)
#pragma unroll
      for (int r = 0; r < R; ++r) m[u][r] = c0 + S * u < nc && r0 + r < nr ? __ldg(M + r * ld + c0 + S * u) : 0.0;
  };
  load(cur, threadIdx.x);
  for (int c0 = threadIdx.x; c0 < nc; c0 += S * D) {
    load(nxt, c0 + S * D);
#pragma unroll
    for (int u = 0; u < D; ++u) {
      if (c0 + S * u >= nc) break;
      const double xe = xv[c0 + S * u];
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r] = fma(cur[u][r], xe, acc[r]);
    }
#pragma unroll
    for (int u = 0; u < D; ++u)
#pragma unroll
      for (int r = 0; r < R; ++r) cur[u][r] = nxt[u][r];
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int r = 0; r < R; ++r) red[warp][r][lane] = acc[r];
  __syncthreads();
  for (int r = warp; r < R; r += kGemv64Warps) {
    double s = red[0][r][lane];
#pragma unroll
    for (int w = 1; w < kGemv64Warps; ++w) s += red[w][r][lane];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0 && r0 + r < nr) y[B.y_off[job] + r0 + r] = s;
  }
}

// Double-float GEMVs y = M x.  The rows of M are stored in pairs, a column's two rows side by side
// (double-float: (h0 h1 l0 l1), FP32: (a0 a1)), so that one packed FP32 instruction serves both: a
// product keeps its exact error (TwoProd) and the cross terms, the running sum is exact (TwoSum) and
// its errors are collected in a second float, 12 lane-operations an element (FP32 matrix: 11).
// For the double-float matrix the two are folded into a double-word sum every 16 terms, which keeps
// the accuracy of a double-word accumulation (~2^-46); for the FP32 matrix the rounding of its
// entries (6e-8, amplified by Sigma^+ only along right singular vectors whose fields on the other
// spheres are correspondingly weak, so that the operator stays accurate to ~1e-7) is far above that
// of the plain collection.  FP32 serves Sigma^+ U^T in the inner solves of MFS_MIXED, double-float V
// everywhere and Sigma^+ U^T in the refinement residual.
// One right-hand side: a CTA takes one row pair, its four warps every fourth run of 32 loads, and the
// next two loads a lane are issued before the current ones are used; what bounds it is HBM (or the
// latency of short matrices), for which ten resident CTAs a SM measured best.  Up to four right-hand
// sides of one matrix (spheres that share a factor, motions of one geometry) are taken together over
// two row pairs, the matrix read once for them; those are bound by the FMA pipe.
// Measured, both factors of one step 1 (GB300; before: two rows a warp, scalar, one right-hand side):
// two spheres with 20 images, N = 800 (386 MB double-float) 102 -> 86 us, with the FP32 factor
// (250 MB) 72 -> 61; 8 spheres N = 400 173 -> 128 and 122 -> 93; 100 spheres sharing the factor
// N = 686 776 -> 531 and (V only) 391 -> 275; eight right-hand sides over one row pair 579.
struct GemvAcc {
  dw2 s, m;  // running sum and its collected errors; double-word sum of the groups
};
template <bool F32>
__device__ __forceinline__ void gemv_step(GemvAcc& a, f2x mh, f2x ml, float2 xe) {
  const f2x xh = f2dup(xe.x), np = f2mul(mh, f2dup(-xe.x));
  f2x e = f2fma(mh, f2dup(xe.y), f2fma(mh, xh, np));
  if constexpr (!F32) e = f2fma(ml, xh, e);
  const dw2 t = two_diff2(a.s.h, np);
  a.s.h = t.h;
  a.s.l = f2add(a.s.l, f2add(t.l, e));
}

constexpr int kGemvPairThreads = 128;

template <bool F32, int C, int RP, int KS>
__device__ __forceinline__ void gemv_pairs(const GemvBatch<float>& B, const int* job, int rp0,
                                           const float2* __restrict__ x, float2* __restrict__ y2,
                                           double* __restrict__ y64) {
  constexpr int D = 2;        // 16-byte loads per row pair and lane in flight (twice)
  constexpr int S = 32 * KS;  // columns' loads of one step of the CTA
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nr = B.rows[job[0]], nc = B.cols[job[0]], ld = B.ld[job[0]];
  const int nrp = (nr + 1) >> 1;
  // a 16-byte load holds one column of a double-float row pair or two of an FP32 one
  const int nv = F32 ? (nc + 1) >> 1 : nc;
  const long long row16 = F32 ? ld / 2 : ld;
  const float4* M = reinterpret_cast<const float4*>(B.mat[job[0]]) + rp0 * row16;
  const float2* xv[C];
#pragma unroll
  for (int q = 0; q < C; ++q) xv[q] = x + B.x_off[job[q]];
  GemvAcc acc[RP][C];
#pragma unroll
  for (int r = 0; r < RP; ++r)
#pragma unroll
    for (int q = 0; q < C; ++q) acc[r][q] = GemvAcc{{0, 0}, {0, 0}};
  float4 cur[D][RP];
  float4 nxt[D][RP];
  auto load = [&](float4 (&m)[D][RP], int v0) {
#pragma unroll
    for (int u = 0; u < D; ++u)
#pragma unroll
      for (int r = 0; r < RP; ++r) {
        const int v = v0 + S * u;
        m[u][r] = v < nv && rp0 + r < nrp ? __ldg(M + r * row16 + v) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
  };
  const int v_first = KS > 1 ? (int)threadIdx.x : lane;
  load(cur, v_first);
  int terms = 0;
  for (int v0 = v_first; v0 < nv; v0 += S * D) {
    load(nxt, v0 + S * D);
#pragma unroll
    for (int u = 0; u < D; ++u) {
      const int v = v0 + S * u;
      if (v >= nv) break;
#pragma unroll
      for (int q = 0; q < C; ++q) {
        if constexpr (F32) {
          const float2 x0 = xv[q][2 * v];
          const float2 x1 = 2 * v + 1 < nc ? xv[q][2 * v + 1] : make_float2(0.f, 0.f);
#pragma unroll
          for (int r = 0; r < RP; ++r) {
            gemv_step<true>(acc[r][q], f2make(cur[u][r].x, cur[u][r].y), 0, x0);
            gemv_step<true>(acc[r][q], f2make(cur[u][r].z, cur[u][r].w), 0, x1);
          }
        } else {
          const float2 xe = xv[q][v];
#pragma unroll
          for (int r = 0; r < RP; ++r)
            gemv_step<false>(acc[r][q], f2make(cur[u][r].x, cur[u][r].y), f2make(cur[u][r].z, cur[u][r].w), xe);
        }
      }
    }
    terms += D;
    if (!F32 && terms >= 16) {
      terms = 0;
#pragma unroll
      for (int r = 0; r < RP; ++r)
#pragma unroll
        for (int q = 0; q < C; ++q) {
          acc[r][q].m = dw2_add(acc[r][q].m, acc[r][q].s);
          acc[r][q].s = dw2{0, 0};
        }
    }
#pragma unroll
    for (int u = 0; u < D; ++u)
#pragma unroll
      for (int r = 0; r < RP; ++r) cur[u][r] = nxt[u][r];
  }
  // the lanes' sums in a fixed order; lane 0 writes a pair's first row, lane 1 its second
  auto finish = [&](dw2 v, int r, long long y_off) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      v = dw2_add(v, dw2{__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)});
    float h0, h1, l0, l1;
    f2split(v.h, h0, h1);
    f2split(v.l, l0, l1);
    const int row = 2 * (rp0 + r) + lane;
    if (lane < 2 && row < nr) {
      const dw w = lane == 0 ? dw{h0, l0} : dw{h1, l1};
      const long long idx = y_off + row;
      if (y64) y64[idx] = dw_join(w);
      if (y2) y2[idx] = make_float2(w.h, w.l);
    }
  };
  auto value = [&](int r, int q) {
    dw2 v = two_sum2(acc[r][q].s.h, acc[r][q].s.l);
    if constexpr (!F32) v = dw2_add(acc[r][q].m, v);
    return v;
  };
  if constexpr (KS > 1) {
    // the warps' shares of the columns added in warp order, each value by one warp
    __shared__ ulonglong2 red[KS][RP * C][32];
#pragma unroll
    for (int r = 0; r < RP; ++r)
#pragma unroll
      for (int q = 0; q < C; ++q) {
        const dw2 v = value(r, q);
        red[warp][r * C + q][lane] = make_ulonglong2(v.h, v.l);
      }
    __syncthreads();
#pragma unroll 1
    for (int i = warp; i < RP * C; i += KS) {
      const ulonglong2 a = red[0][i][lane];
      dw2 v{a.x, a.y};
#pragma unroll
      for (int w = 1; w < KS; ++w) {
        const ulonglong2 b = red[w][i][lane];
        v = dw2_add(v, dw2{b.x, b.y});
      }
      long long y_off = B.y_off[job[0]];
#pragma unroll
      for (int q = 1; q < C; ++q)
        if (i % C == q) y_off = B.y_off[job[q]];
      finish(v, i / C, y_off);
    }
  } else {
#pragma unroll
    for (int r = 0; r < RP; ++r)
#pragma unroll
      for (int q = 0; q < C; ++q) finish(value(r, q), r, B.y_off[job[q]]);
  }
}

// row pairs a warp (KS 1) or the CTA (KS 4: its warps share the columns) takes at once
__host__ __device__ constexpr int gemv_rp(int c) { return c == 1 ? 1 : 2; }
// work item blockIdx.x: the right-hand sides list[item.x .. item.x + item.y) of one matrix
template <bool F32, int CMAX, int KS>
__global__ void __launch_bounds__(kGemvPairThreads, CMAX == 1 ? 10 : 1) gemv_pair_kernel(GemvBatch<float> B, const float2* __restrict__ x,
                                                                   float2* __restrict__ y2, double* __restrict__ y64) {
  constexpr int RP = gemv_rp(CMAX);
  const int2 it = B.items ? B.items[blockIdx.x] : make_int2(blockIdx.x, 1);
  const int rp0 = (KS > 1 ? blockIdx.y : blockIdx.y * (kGemvPairThreads / 32) + (threadIdx.x >> 5)) * RP;
  int job[CMAX];
  bool any = false;
#pragma unroll
  for (int q = 0; q < CMAX; ++q) {
    const int j = it.x + min(q, it.y - 1);
    job[q] = B.job_list ? B.job_list[j] : j;
    any = any || !B.active || B.active[B.job_prob[job[q]]];
  }
  if (!any || 2 * rp0 >= B.rows[job[0]]) return;
  // (three of four run as four with the last one twice: the same value written twice)
  if (CMAX > 1 && it.y == 1) gemv_pairs<F32, 1, RP, KS>(B, job, rp0, x, y2, y64);
  else if (CMAX > 2 && it.y == 2) gemv_pairs<F32, 2, RP, KS>(B, job, rp0, x, y2, y64);
  else gemv_pairs<F32, CMAX, RP, KS>(B, job, rp0, x, y2, y64);
}

__global__ void split_dw_kernel(long long n, const double* __restrict__ in, float2* __restrict__ out) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    dw s = dw_split(in[e]);
    out[e] = make_float2(s.h, s.l);
  }
}

// ------------------------------------------------------------------ Krylov helpers
constexpr int kRedThreads = 256;

template <typename T>
__global__ void multidot_kernel(int n, const T* __restrict__ V, long long ldv, const T* __restrict__ w,
                                double* __restrict__ partial, int nblk) {
  const int b = blockIdx.x, i = blockIdx.y;
  const int chunk = (n + nblk - 1) / nblk;
  const int lo = b * chunk, hi = min(n, lo + chunk);
  const T* v = V + (long long)i * ldv;
  T s = T(0);
  for (int e = lo + threadIdx.x; e < hi; e += blockDim.x) s += v[e] * w[e];
  double d = (double)s;
  for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
  __shared__ double red[kRedThreads / 32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = d;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) t += red[q];
    partial[(long long)i * nblk + b] = t;
  }
}

__global__ void reduce_partials_kernel(int nvec, int nblk, const double* __restrict__ partial, double* __restrict__ h) {
  const int i = blockIdx.x;
  double s = 0;
  for (int b = threadIdx.x; b < nblk; b += blockDim.x) s += partial[(long long)i * nblk + b];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __shared__ double red[32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) t += red[q];
    h[i] = t;
  }
}

template <typename T>
__global__ void update_kernel(int n, int nvec, const T* __restrict__ V, long long ldv, const double* __restrict__ h,
                              double sign, T* __restrict__ w) {
  __shared__ T hs[512];
  for (int i = threadIdx.x; i < nvec; i += blockDim.x) hs[i] = T(sign * h[i]);
  __syncthreads();
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    T acc = w[e];
    for (int i = 0; i < nvec; ++i) acc += hs[i] * V[(long long)i * ldv + e];
    w[e] = acc;
  }
}

template <typename T>
__global__ void scale_copy_kernel(int n, const T* __restrict__ w, double s, T* __restrict__ out) {
  T ss = T(s);
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    out[e] = ss * w[e];
}

template <typename Tin, typename Tout>
__global__ void convert_kernel(long long n, const Tin* __restrict__ in, double s, Tout* __restrict__ out) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    out[e] = (Tout)(s * (double)in[e]);
}

__global__ void axpy_mixed_kernel(int n, double a, const float* __restrict__ x, double* __restrict__ y) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    y[e] += a * (double)x[e];
}

__global__ void sub_kernel(int n, const double* __restrict__ a, const double* __restrict__ b, double* __restrict__ out) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    out[e] = a[e] - b[e];
}

// ------------------------------------------------------------------ segmented (batched) vector kernels
constexpr int kSegThreads = 256;

// The chunk a CTA works on: blockIdx.x indexes the compacted list of the active problems'
// chunks when the table carries one, else all chunks (inactive ones return at once).
__device__ __forceinline__ int seg_chunk(const SegTable& t) { return t.list ? t.list[blockIdx.x] : blockIdx.x; }

// Partial dot products of w with basis vectors over one chunk: CTA (chunk, vector block) stages
// the chunk of w (at most kSegChunkMax elements) in shared memory and each warp takes vectors of
// its block, so the launch has enough CTAs to keep HBM busy even for a single short problem.
constexpr int kSegChunkMax = 1024;
constexpr int kSegDotVecs = 16;   // basis vectors per CTA
static_assert(kSegCounters * kSegDotVecs >= 512, "a counter per block of basis vectors");
constexpr int kSegUpdSub = 128;   // elements per CTA of the update (one per thread)
__global__ void seg_dots_kernel(SegTable t, int nvec, const double* __restrict__ V, long long ldv,
                                const double* __restrict__ w, double* __restrict__ partial, double* __restrict__ h) {
  const int b = seg_chunk(t);
  const int p = t.prob[b];
  if (!t.active[p]) return;
  const long long lo = t.start[b];
  const int len = (int)(t.end[b] - lo);
  __shared__ double ws[kSegChunkMax];
  for (int e = threadIdx.x; e < len; e += blockDim.x) ws[e] = w[lo + e];
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  const int i1 = min(nvec, (int)(blockIdx.y + 1) * kSegDotVecs);
  // two vectors per warp at a time, so that twice the loads are in flight
  for (int i = blockIdx.y * kSegDotVecs + warp; i < i1; i += 2 * nwarps) {
    const int i2 = i + nwarps;
    const double* v = V + (long long)i * ldv + lo;
    const double* v2 = V + (long long)min(i2, i1 - 1) * ldv + lo;
    double d = 0.0, d2 = 0.0;
#pragma unroll 8
    for (int e = lane; e < len; e += 32) {
      const double x = ws[e];
      d += v[e] * x;
      d2 += v2[e] * x;
    }
    for (int o = 16; o > 0; o >>= 1) {
      d += __shfl_xor_sync(0xffffffffu, d, o);
      d2 += __shfl_xor_sync(0xffffffffu, d2, o);
    }
    if (lane == 0) {
      partial[(long long)i * t.nchunks + b] = d;
      if (i2 < i1) partial[(long long)i2 * t.nchunks + b] = d2;
    }
  }
  // The last CTA of problem p and this block of vectors adds their partial dots in chunk order (so the
  // result does not depend on which CTA that is), a thread per vector with 16 loads in flight, and re-arms
  // the counter for the next launch.  With one CTA for all vectors of a problem and four loads at a time an
  // iteration of 216 spheres (507 chunks) took 592 us beside step 1 and the pair sums, this way 296.
  unsigned* counter = t.counter + p * kSegCounters + blockIdx.y;
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  const int c0 = t.pchunk[p], c1 = t.pchunk[p + 1];
  if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == (unsigned)(c1 - c0) - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  const int i = blockIdx.y * kSegDotVecs + (int)threadIdx.x;
  if (threadIdx.x < kSegDotVecs && i < i1) {
    const double* q = partial + (long long)i * t.nchunks;
    double sum = 0.0;
    for (int c = c0; c < c1; c += 16) {
      double v[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = c + u < c1 ? __ldcg(q + c + u) : 0.0;
#pragma unroll
      for (int u = 0; u < 16; ++u) sum += v[u];
    }
    h[(long long)i * t.K + p] = sum;
  }
  if (threadIdx.x == 0) *counter = 0u;
}

// w += sign * sum_i coef[i K + p] V_i over one kSegUpdSub-element piece of a chunk per CTA.  The
// CTA's kSegUpdGroups thread groups take interleaved vectors (more loads in flight when a short
// problem has few pieces) and their sums are added in group order.
// NORM: also hn[p] = |w|^2 of the updated vector, which saves the launch and the read of a separate
// norm: each piece leaves its sum of squares in `partial` and the last CTA of a problem adds them
// (in piece order, so the sum does not depend on which CTA that is).
// With the normalisation on the device, the fused sums of split sources and these kernels in the single
// solves too (up to kSegSingleMax chunks), an iteration of two spheres went from 116 to 108 us, one of four from
// 180 to 173, and the sweep of motions from 20.4 to 20.0 ms.
constexpr int kSegUpdGroups = 4;
template <bool NORM>
__global__ void __launch_bounds__(kSegUpdSub* kSegUpdGroups)
    seg_update_kernel(SegTable t, int nvec, const double* __restrict__ V, long long ldv,
                      const double* __restrict__ coef, double sign, double* __restrict__ w,
                      double* __restrict__ partial, double* __restrict__ hn) {
  const int b = seg_chunk(t);
  const int p = t.prob[b];
  if (!t.active[p]) return;
  const int tl = threadIdx.x % kSegUpdSub, g = threadIdx.x / kSegUpdSub;
  const long long e = t.start[b] + (long long)blockIdx.y * kSegUpdSub + tl;
  if (t.start[b] + (long long)blockIdx.y * kSegUpdSub >= t.end[b]) return;  // whole CTA past the chunk
  __shared__ double c[512];
  __shared__ double red[kSegUpdGroups][kSegUpdSub];
  for (int i = threadIdx.x; i < nvec; i += blockDim.x) c[i] = sign * coef[(long long)i * t.K + p];
  __syncthreads();
  double a = 0.0;
  if (e < t.end[b]) {
#pragma unroll 8
    for (int i = g; i < nvec; i += kSegUpdGroups) a += c[i] * V[(long long)i * ldv + e];
  }
  red[g][tl] = a;
  __syncthreads();
  double s = 0.0;
  if (g == 0 && e < t.end[b]) {
    s = w[e];
#pragma unroll
    for (int q = 0; q < kSegUpdGroups; ++q) s += red[q][tl];
    w[e] = s;
  }
  if constexpr (NORM) {
    constexpr int kPieces = kSegChunkMax / kSegUpdSub;
    __shared__ double ws[kSegUpdSub / 32];
    __shared__ bool last;
    double q = s * s;
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    if (g == 0 && (tl & 31) == 0) ws[tl >> 5] = q;
    __syncthreads();
    if (threadIdx.x == 0) {
      double sum = 0.0;
      for (int i = 0; i < kSegUpdSub / 32; ++i) sum += ws[i];
      partial[(long long)b * kPieces + blockIdx.y] = sum;
      __threadfence();
      // pieces of problem p: its chunks are full (kSegChunkMax) but the last
      const int b0 = t.pchunk[p], b1 = t.pchunk[p + 1];
      const unsigned total = (unsigned)(b1 - 1 - b0) * kPieces +
                             (unsigned)((t.end[b1 - 1] - t.start[b1 - 1] + kSegUpdSub - 1) / kSegUpdSub);
      unsigned* counter = t.counter + p * kSegCounters;
      last = atomicAdd(counter, 1u) == total - 1;
      if (last) {
        *counter = 0u;
        ws[0] = 0.0;
      }
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int b0 = t.pchunk[p], b1 = t.pchunk[p + 1];
    const long long n_last = (t.end[b1 - 1] - t.start[b1 - 1] + kSegUpdSub - 1) / kSegUpdSub;
    const long long total = (long long)(b1 - 1 - b0) * kPieces + n_last;
    double sum = 0.0;
    for (long long i = threadIdx.x; i < total; i += blockDim.x) sum += __ldcg(&partial[(long long)b0 * kPieces + i]);
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    __syncthreads();
    double* wsum = &red[0][0];
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
      double tot = 0.0;
      for (int i = 0; i < kSegUpdSub * kSegUpdGroups / 32; ++i) tot += wsum[i];
      hn[p] = tot;
    }
  }
}

inline int seg_ctas(const SegTable& t) { return t.list ? t.nlist : t.nchunks; }

__global__ void seg_scale_kernel(SegTable t, const double* __restrict__ s, const double* __restrict__ in,
                                 double* __restrict__ out) {
  const int b = seg_chunk(t);
  const int p = t.prob[b];
  if (!t.active[p]) return;
  const double f = s[p];
  for (long long e = t.start[b] + threadIdx.x; e < t.end[b]; e += blockDim.x) out[e] = f * in[e];
}

__global__ void seg_scale_split_kernel(SegTable t, const double* __restrict__ s, const double* __restrict__ in,
                                       double* __restrict__ out, float2* __restrict__ x2) {
  const int b = seg_chunk(t);
  const int p = t.prob[b];
  if (!t.active[p]) return;
  const double f = s[p];
  for (long long e = t.start[b] + threadIdx.x; e < t.end[b]; e += blockDim.x) {
    const double v = f * in[e];
    out[e] = v;
    const dw d = dw_split(v);
    x2[e] = make_float2(d.h, d.l);
  }
}

// out = in / sqrt(hn[p]) (0 for hn = 0), and its (hi, lo) split for the next double-float apply when x2
// is given
__global__ void seg_normalise_kernel(SegTable t, const double* __restrict__ hn, const double* __restrict__ in,
                                     double* __restrict__ out, float2* __restrict__ x2) {
  const int b = seg_chunk(t);
  const int p = t.prob[b];
  if (!t.active[p]) return;
  // (the root and the quotient once a CTA: by every thread they were half of the FP64 work, 34 us on 1.8e6
  // elements, where the splits take 16)
  __shared__ double fs;
  if (threadIdx.x == 0) {
    const double h = sqrt(fmax(0.0, hn[p]));
    fs = h > 0 ? 1.0 / h : 0.0;
  }
  __syncthreads();
  const double f = fs;
  for (long long e = t.start[b] + threadIdx.x; e < t.end[b]; e += blockDim.x) {
    const double v = f * in[e];
    out[e] = v;
    if (x2) {
      const dw d = dw_split(v);
      x2[e] = make_float2(d.h, d.l);
    }
  }
}

__global__ void axpy64_kernel(long long n, double a, const double* __restrict__ x, double* __restrict__ y) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    y[e] += a * x[e];
}

// ------------------------------------------------------------------ batched Givens (device)
// One Arnoldi step for every active problem of a lockstep batch, one thread per problem: the
// Hessenberg column h = h1 + h2 (the two classical Gram-Schmidt passes) with the subdiagonal
// sqrt(hn), the earlier Givens rotations applied, a new rotation formed, the least-squares
// right-hand side g rotated and the residual estimate |g_{j+1}| / ||b|| updated.  A problem that
// meets its tolerance (or breaks down) is deactivated here, on the device, so the host need
// not wait for every step; scl = 1 / h_{j+1,j} normalises the new basis vector.
// One CTA per problem.  Applying the earlier rotations to the new column is the first-order
// linear recurrence r_{i+1} = -sn_i r_i + cs_i h_{i+1} (r_0 = h_0) with outputs
// h'_i = cs_i r_i + sn_i h_{i+1}; the CTA evaluates it as a parallel prefix of the affine maps
// r -> a r + b (each thread composes a contiguous run, a warp scan and the warp totals give every
// run its starting r), so its FP64 work is a few dependent operations per thread instead of a
// chain of j on one thread.
__global__ void batch_givens_kernel(GivensState S, int j, const double* __restrict__ h1, const double* __restrict__ h2,
                                    const double* __restrict__ hn) {
  const int p = blockIdx.x;
  if (!S.active[p]) return;
  __shared__ double col[kMaxGmresCol + 1], cs[kMaxGmresCol], sn[kMaxGmresCol];
  __shared__ double wa[32], wb[32], rj, hnext;
  __shared__ int bad;
  double* colg = S.H + ((long long)p * S.restart + j) * S.ldh;
  double* csg = S.cs + (long long)p * S.restart;
  double* sng = S.sn + (long long)p * S.restart;
  double* g = S.g + (long long)p * S.ldh;
  for (int i = threadIdx.x; i <= j; i += blockDim.x) col[i] = h1[(long long)i * S.K + p] + h2[(long long)i * S.K + p];
  for (int i = threadIdx.x; i < j; i += blockDim.x) {
    cs[i] = csg[i];
    sn[i] = sng[i];
  }
  if (threadIdx.x == 0) {
    hnext = sqrt(fmax(0.0, hn[p]));
    bad = !isfinite(hnext);
    if (j == 0) rj = 0.0;
  }
  __syncthreads();
  if (bad) {
    if (threadIdx.x == 0) {
      S.err[0] = 1;
      S.active[p] = 0;
    }
    return;
  }
  // this thread's run [i0, i1) of the rotations, composed into r -> A r + B
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = (j + blockDim.x - 1) / blockDim.x;
  const int i0 = min(j, tid * per), i1 = min(j, i0 + per);
  double A = 1.0, B = 0.0;
  for (int i = i0; i < i1; ++i) {
    const double a = -sn[i];
    B = fma(a, B, cs[i] * col[i + 1]);
    A *= a;
  }
  // inclusive scan over the warp's runs (a later run applies after an earlier one)
  for (int o = 1; o < 32; o <<= 1) {
    const double Ap = __shfl_up_sync(0xffffffffu, A, o), Bp = __shfl_up_sync(0xffffffffu, B, o);
    if (lane >= o) {
      B = fma(A, Bp, B);
      A *= Ap;
    }
  }
  if (lane == 31) {
    wa[warp] = A;
    wb[warp] = B;
  }
  __syncthreads();
  // the composition of every run before this thread's: the earlier warps', then the earlier lanes'
  double PA = 1.0, PB = 0.0;
  for (int q = 0; q < warp; ++q) {
    PB = fma(wa[q], PB, wb[q]);
    PA *= wa[q];
  }
  double EA = __shfl_up_sync(0xffffffffu, A, 1), EB = __shfl_up_sync(0xffffffffu, B, 1);
  if (lane == 0) {
    EA = 1.0;
    EB = 0.0;
  }
  double r = fma(EA, fma(PA, col[0], PB), EB);  // r at i0
  for (int i = i0; i < i1; ++i) {
    const double x = col[i + 1];
    colg[i] = fma(cs[i], r, sn[i] * x);
    r = fma(-sn[i], r, cs[i] * x);
  }
  if (i1 == j && i0 < i1) rj = r;
  if (j == 0 && tid == 0) rj = col[0];
  __syncthreads();
  if (tid == 0) {
    const double cj = rj, hx = hnext;
    const double den = hypot(cj, hx);
    const double c = den > 0 ? cj / den : 1.0, sj = den > 0 ? hx / den : 0.0;
    csg[j] = c;
    sng[j] = sj;
    colg[j] = den;
    colg[j + 1] = 0.0;
    g[j + 1] = -sj * g[j];
    g[j] = c * g[j];
    S.jused[p] = j + 1;
    S.iters[p] += 1;
    S.est[p] = fabs(g[j + 1]) / S.bn[p];
    S.scl[p] = hx > 0 ? 1.0 / hx : 0.0;
    if (S.est[p] <= S.tol[p] || hx == 0.0) S.active[p] = 0;
  }
}

// y = R^{-1} g per problem (back substitution over its own jused steps): coef[i K + p] = y_i,
// zero for jused <= i < jmax
__global__ void batch_backsolve_kernel(GivensState S, int jmax, double* __restrict__ coef) {
  const int p = blockIdx.x;
  const int J = S.jused[p];
  const double* H = S.H + (long long)p * S.restart * S.ldh;
  const double* g = S.g + (long long)p * S.ldh;
  __shared__ double t[kMaxGmresCol];
  // column-oriented back substitution: after y_i is known, every thread updates t[q] -= R[q][i] y_i
  for (int q = threadIdx.x; q < J; q += blockDim.x) t[q] = g[q];
  __syncthreads();
  for (int i = J - 1; i >= 0; --i) {
    const double d = H[(long long)i * S.ldh + i];
    const double yi = d != 0.0 ? t[i] / d : 0.0;
    __syncthreads();
    for (int q = threadIdx.x; q < i; q += blockDim.x) t[q] -= H[(long long)i * S.ldh + q] * yi;
    if (threadIdx.x == 0) coef[(long long)i * S.K + p] = yi;
    __syncthreads();
  }
  for (int i = J + threadIdx.x; i < jmax; i += blockDim.x) coef[(long long)i * S.K + p] = 0.0;
}

// ------------------------------------------------------------------ forces / torques
__global__ void ft_kernel(int N, const double* __restrict__ proxy64, const double* __restrict__ img64,
                          const int* __restrict__ img_off, const long long* __restrict__ unk_off,
                          const double* __restrict__ lam, double* __restrict__ F, double* __restrict__ Tq, int stride,
                          double sF, double sT) {
  const int k = blockIdx.x;
  double acc[6] = {0, 0, 0, 0, 0, 0};
  const double* l = lam + unk_off[k];
  for (int j = threadIdx.x; j < N; j += blockDim.x) {
    const double* y = proxy64 + 4LL * j;
    double fx = l[3 * j], fy = l[3 * j + 1], fz = l[3 * j + 2];
    acc[0] += fx; acc[1] += fy; acc[2] += fz;
    acc[3] += y[1] * fz - y[2] * fy;
    acc[4] += y[2] * fx - y[0] * fz;
    acc[5] += y[0] * fy - y[1] * fx;
  }
  const int i0 = img_off[k], i1 = img_off[k + 1];
  for (int j = i0 + threadIdx.x; j < i1; j += blockDim.x) {
    const double* y = img64 + 4LL * j;
    const double* s = l + 3LL * N + 9LL * (j - i0);
    double fx = s[0], fy = s[1], fz = s[2];
    acc[0] += fx; acc[1] += fy; acc[2] += fz;
    acc[3] += s[3] + y[1] * fz - y[2] * fy;
    acc[4] += s[4] + y[2] * fx - y[0] * fz;
    acc[5] += s[5] + y[0] * fy - y[1] * fx;
  }
  __shared__ double red[6][32];
  for (int c = 0; c < 6; ++c) {
    double s = acc[c];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[c][threadIdx.x >> 5] = s;
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    double s = 0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) s += red[threadIdx.x][q];
    if (threadIdx.x < 3) F[(long long)stride * k + threadIdx.x] = sF * s;
    else Tq[(long long)stride * k + threadIdx.x - 3] = sT * s;
  }
}

// out[node] -= sqrt(w) (V_k + Omega_k x (x - c_k)) with U = (V_k, Omega_k) per sphere
__global__ void rigid_sub_kernel(int n, const int* __restrict__ owner, const double* __restrict__ pos64,
                                 const double* __restrict__ U, double* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double* u = U + 6LL * owner[i];
    const double* r = pos64 + 4LL * i;
    const double sw = r[3];
    out[3LL * i] -= sw * (u[0] + u[4] * r[2] - u[5] * r[1]);
    out[3LL * i + 1] -= sw * (u[1] + u[5] * r[0] - u[3] * r[2]);
    out[3LL * i + 2] -= sw * (u[2] + u[3] * r[1] - u[4] * r[0]);
  }
}

struct Bg { double v[15]; };

__global__ void rhs_kernel(int n, const double* __restrict__ xabs, const int* __restrict__ owner,
                           const double* __restrict__ sqrtw, const double* __restrict__ cen,
                           const double* __restrict__ v, const double* __restrict__ om, Bg bg, double* __restrict__ wb) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    int o = owner[i];
    double x0 = xabs[3 * i], x1 = xabs[3 * i + 1], x2 = xabs[3 * i + 2];
    double r0 = x0 - cen[3 * o], r1 = x1 - cen[3 * o + 1], r2 = x2 - cen[3 * o + 2];
    const double* w = om + 3 * o;
    double u0 = v[3 * o] + w[1] * r2 - w[2] * r1;
    double u1 = v[3 * o + 1] + w[2] * r0 - w[0] * r2;
    double u2 = v[3 * o + 2] + w[0] * r1 - w[1] * r0;
    // background u_inf = U + E x + Omega x x, subtracted (eq. bc)
    const double* E = bg.v + 3;
    const double* Om = bg.v + 12;
    u0 -= bg.v[0] + E[0] * x0 + E[1] * x1 + E[2] * x2 + Om[1] * x2 - Om[2] * x1;
    u1 -= bg.v[1] + E[3] * x0 + E[4] * x1 + E[5] * x2 + Om[2] * x0 - Om[0] * x2;
    u2 -= bg.v[2] + E[6] * x0 + E[7] * x1 + E[8] * x2 + Om[0] * x1 - Om[1] * x0;
    double s = sqrtw[i];
    wb[3 * i] = s * u0;
    wb[3 * i + 1] = s * u1;
    wb[3 * i + 2] = s * u2;
  }
}

// B[(3 s + c) lda + 3 i + r] = sqrt(w_i) K_type(x_i - y_s)[r][c]
__global__ void assemble_self_kernel(int m, int n_src, const double* __restrict__ xrel, const double* __restrict__ sqrtw,
                                     const double* __restrict__ yrel, const int* __restrict__ type, double scale,
                                     double* __restrict__ B, long long lda) {
  long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (id >= (long long)m * n_src) return;
  int i = (int)(id % m);
  int s = (int)(id / m);
  double r[3] = {xrel[3 * i] - yrel[3 * s], xrel[3 * i + 1] - yrel[3 * s + 1], xrel[3 * i + 2] - yrel[3 * s + 2]};
  double r2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2];
  double ir = 1.0 / sqrt(r2);
  double ir3 = ir * ir * ir;
  double K[3][3];
  int ty = type[s];
  if (ty == 0) {
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b < 3; ++b) K[a][b] = scale * ((a == b ? ir : 0.0) + r[a] * r[b] * ir3);
  } else if (ty == 1) {
    double c = scale * ir3;
    K[0][0] = 0; K[0][1] = c * r[2]; K[0][2] = -c * r[1];
    K[1][0] = -c * r[2]; K[1][1] = 0; K[1][2] = c * r[0];
    K[2][0] = c * r[1]; K[2][1] = -c * r[0]; K[2][2] = 0;
  } else {
    double c = 1.0 / (4.0 * kPi);
    double ir5 = ir3 * ir * ir;
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b < 3; ++b) K[a][b] = c * ((a == b ? -ir3 : 0.0) + 3.0 * r[a] * r[b] * ir5);
  }
  double w = sqrtw[i];
  for (int c = 0; c < 3; ++c)
    for (int rr = 0; rr < 3; ++rr) B[(3LL * s + c) * lda + 3LL * i + rr] = w * K[rr][c];
}

// Arithmetic-peak probe: 8 independent fused multiply-add chains per thread, 16 steps of each
// per loop trip, enough warps per SM to hide the FMA latency.  The result is stored only when it
// equals a value it never takes, so the chains cannot be removed.
template <typename T>
__global__ void __launch_bounds__(256) fma_probe_kernel(int iters, T a, T b, T* __restrict__ sink) {
  T x[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) x[q] = T(threadIdx.x + q) * T(1e-3);
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int u = 0; u < 16; ++u)
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if constexpr (sizeof(T) == 4) x[q] = __fmaf_rn(x[q], a, b);
        else x[q] = __fma_rn(x[q], a, b);
      }
  }
  T s = T(0);
#pragma unroll
  for (int q = 0; q < 8; ++q) s += x[q];
  if (s == T(-1.25e30)) sink[0] = s;
}

thread_local long long t_launches = 0;

inline int grid_for(long long n, int threads, int cap = 152 * 16) {
  long long g = (n + threads - 1) / threads;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (int)g;
}

}  // namespace

long long launches_on_this_thread() { return t_launches; }
void note_launch() { ++t_launches; }

void launch_pairs_f32(const TargetSet& tg, const SourceSet& src, const float* lam_hat, const float* mu, float* out,
                      double visc, cudaStream_t st) {
  if (tg.n_tiles == 0) return;
  const int nt = pair_nodes_per_thread(tg.n_tiles);
  PairArgs<float> A = make_args<float>(tg, src, lam_hat, mu, out, visc, nt);
  ++t_launches;
  if (nt == 4) pairs_kernel<float, 4><<<tg.n_tiles, kPairThreads, 0, st>>>(A);
  else pairs_kernel<float, 1><<<tg.n_tiles1, kPairThreads, 0, st>>>(A);
}

int fp64_split_parts(long long pieces, long long min_sources, int max_parts) {
  if (pieces <= 0) return 1;
  long long s = (kFp64SplitTarget + pieces - 1) / pieces;
  s = std::min<long long>(s, min_sources / kFp64SplitMinSources);
  s = std::min<long long>(s, max_parts);
  return (int)std::max<long long>(s, 1);
}

void launch_pairs_fp64(const TargetSet& tg, const SourceSet& src, const double* lam_hat, const double* mu, double* out,
                       double visc, double* partial, int max_parts, cudaStream_t st) {
  if (tg.n_tiles1 == 0) return;
  PairArgs<double> A = make_args<double>(tg, src, lam_hat, mu, out, visc, 1);
  const long long n3 = 3LL * tg.n;
  const int parts = fp64_split_parts(4LL * tg.n_tiles1, (long long)(src.P - 1) * src.N, max_parts);
  ++t_launches;
  pairs_fp64_kernel<<<4 * tg.n_tiles1 * parts, kPairThreads, 0, st>>>(A, parts, partial, n3);
  if (parts > 1) {
    ++t_launches;
    pair_parts_reduce_kernel<<<grid_for(n3, 256), 256, 0, st>>>(n3, A.tgt, parts, partial, n3, mu, out);
  }
}

int velocity_parts(int n, const SourceSet& src) {
  return fp64_split_parts((n + 31LL) / 32, (long long)src.P * src.N, kVelocityMaxParts);
}

void launch_velocity(int n, const double* x, const SourceSet& src, const double* lam, double* u, double* partial,
                     double visc, cudaStream_t st) {
  if (n <= 0) return;
  PairArgs<double> A = make_args<double>(TargetSet(), src, lam, nullptr, u, visc, 1);
  const int parts = velocity_parts(n, src);
  const long long n3 = 3LL * n;
  ++t_launches;
  velocity_fp64_kernel<<<(unsigned)((n + 31LL) / 32 * parts), kPairThreads, 0, st>>>(A, n, x, parts,
                                                                                   parts > 1 ? partial : u, n3);
  if (parts > 1) {
    ++t_launches;
    pair_parts_reduce_kernel<<<grid_for(n3, 256), 256, 0, st>>>(n3, nullptr, parts, partial, n3, nullptr, u);
  }
}

// nodes per thread of a far-field launch: the requested shape, else the rule (512-node tiles once they fill
// the GPU twice)
static int shape_nt(const TargetSet& tg, const PairShape& shape) {
  if (shape.nt == 1 || shape.nt == 4) return shape.nt;
  return pair_nodes_per_thread(tg.n_tiles);
}

// resident CTAs of a pair kernel on the current device (SMs x CTAs per SM), looked up once per
// (device, kernel)
static double resident_ctas(const void* kernel, int threads) {
  static std::mutex mtx;
  static std::vector<std::pair<std::pair<int, const void*>, double>> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  std::lock_guard<std::mutex> g(mtx);
  for (const auto& e : cache)
    if (e.first.first == dev && e.first.second == kernel) return e.second;
  int per_sm = 0, sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    return 0;
  }
  cache.push_back({{dev, kernel}, (double)sms * per_sm});
  return cache.back().second;
}

// (see the declaration)
static int pair_split_parts(long long items, double wave, long long min_sources, int max_parts) {
  if (items <= 0 || wave <= 0 || min_sources <= 0) return 1;
  const int most = (int)std::max<long long>(1, std::min<long long>(max_parts, min_sources / kPairSplitMinSources));
  int best = 1;
  double best_t = 0;
  for (int p = 1; p <= most; ++p) {
    const double t = std::ceil((double)items * p / wave) * (1.0 / p + kPairSplitPartCost / (double)min_sources);
    if (p == 1 || t < best_t) {
      best_t = t;
      best = p;
    }
  }
  return best;
}

PairShape resolve_dw_shape(const TargetSet& tg, const SourceSet& src, PairShape shape, int max_parts) {
  PairShape r;
  r.nt = 1;
  if (shape.parts > 0) r.parts = std::min(shape.parts, max_parts);
  else r.parts = pair_split_parts(tg.n_pieces1, resident_ctas((const void*)pairs_dw_kernel, kDwThreads),
                                  (long long)(src.P - 1) * src.N, max_parts);
  return r;
}

void launch_pairs_dw(const TargetSet& tg, const SourceSet& src, const float2* lam_hat, const double* mu, double* out,
                     double visc, double* partial, unsigned* counter, int max_parts, cudaStream_t st, PairShape shape) {
  if (tg.n_tiles == 0) return;
  const PairShape r = resolve_dw_shape(tg, src, shape, max_parts);
  const int parts = partial ? r.parts : 1;
  PairArgs<double> A = make_args<double>(tg, src, nullptr, mu, out, visc, 1);
  A.lam2 = lam_hat;
  ++t_launches;
  // (with split sources the last CTA of a piece to finish adds the parts)
  pairs_dw_kernel<<<kDwPieces * tg.n_tiles1 * parts, kDwThreads, 0, st>>>(A, parts, partial, 3LL * tg.n, counter);
}

// source parts per tile so that tiles x parts fill whole waves of the resident CTAs (ties: fewer)
static int wave_parts(long long tiles, const void* kernel, int max_parts) {
  const double wave = resident_ctas(kernel, kPairThreads);
  if (wave <= 0) return 1;
  int best = 1;
  double best_eff = 0;
  for (int p = 1; p <= max_parts; ++p) {
    const double w = (double)tiles * p / wave;
    const double eff = w / std::ceil(w);
    if (eff > best_eff + 0.02) {
      best_eff = eff;
      best = p;
    }
  }
  return best;
}

// Near part: 64-target CTAs, a thread per node.  (With four from 304 512-node tiles on, 343 spheres: N = 300 at
// centres 2.5 apart 4.99 ms against 4.65, N = 160 at 3.0 0.82 against 0.78; all pairs of 100 spheres of 1,804 nodes
// 127.4 against 116.1.)  The parts are whole spheres of lists of uneven length, so their number is what leaves
// the smallest sum of a resident CTA's share of the work, kNearPartCost sources a part on top, and of half the
// longest CTA, which one that starts last waits for.  Measured over 1 to 16 parts (taken / best / first / last): cluster
// of 150 spheres, N = 686 3225 (8) / 3218 / 3925 / 3444 us; of 60, N = 150 172 (8) / 161 / 380 / 172; of 400, N = 300
// 4747 (6) / 4747 / 5281 / 4888; lattices of 125, N = 100 and 343, N = 300 104 (6) / 104 / 127 / 132 and 4643 (6) / 4643 /
// 4908 / 4766; 40 apart, N = 200 158 (12) / 151 / 292 / 176.
constexpr double kNearPartCost = 40.0;
PairShape resolve_near_shape(const TargetSet& tg, const SourceSet& src, const FarField& ff, PairShape shape,
                             int max_parts) {
  PairShape r;
  r.nt = 1;
  if (shape.parts > 0) {
    r.parts = std::min(shape.parts, max_parts);
    return r;
  }
  const double wave = resident_ctas((const void*)pairs_dw_near_kernel, kDwThreads);
  r.parts = 1;
  double best = 0;
  for (int p = 1; wave > 0 && p <= std::min(max_parts, std::max(1, ff.near_max)); ++p) {
    const double t = tg.n_pieces1 * (ff.near_mean * src.N + kNearPartCost * p) / wave +
                     0.5 * ((ff.near_max + p - 1) / p) * src.N;
    if (p == 1 || t < best) {
      best = t;
      r.parts = p;
    }
  }
  return r;
}

void launch_pairs_dw_near(const TargetSet& tg, const SourceSet& src, const FarField& ff, const float2* lam_hat,
                          const double* mu, double* out, double visc, double* partial, unsigned* counter, int max_parts,
                          cudaStream_t st, PairShape shape) {
  if (tg.n_tiles == 0) return;
  const PairShape r = resolve_near_shape(tg, src, ff, shape, max_parts);
  PairArgs<double> A = make_args<double>(tg, src, nullptr, mu, out, visc, 1);
  A.lam2 = lam_hat;
  const int parts = partial ? r.parts : 1;
  ++t_launches;
  pairs_dw_near_kernel<<<kDwPieces * tg.n_tiles1 * parts, kDwThreads, 0, st>>>(A, ff.near_off, ff.near_idx, parts,
                                                                              partial, 3LL * tg.n, counter);
}

PairShape resolve_far_shape(const TargetSet& tg, PairShape shape, int max_parts) {
  PairShape r;
  r.nt = shape_nt(tg, shape);
  // 4 nodes per thread run the packed-FP32 kernel unless the scalar one is asked for
  r.packed = r.nt == 4 && shape.packed >= 0 ? 1 : 0;
  const long long tiles = r.nt == 4 ? tg.n_tiles : tg.n_tiles1;
  const void* kern = r.nt == 4 ? (r.packed ? (const void*)pairs_far2_kernel : (const void*)pairs_far_kernel<4>)
                               : (const void*)pairs_far_kernel<1>;
  r.parts = shape.parts > 0 ? std::min(shape.parts, max_parts) : wave_parts(tiles, kern, max_parts);
  return r;
}

void launch_pairs_far(const TargetSet& tg, const SourceSet& src, const FarField& ff, double* out, double visc,
                      double* partial, int max_parts, cudaStream_t st, PairShape shape) {
  if (tg.n_tiles == 0 || ff.n_eq == 0) return;
  const PairShape r = resolve_far_shape(tg, shape, max_parts);
  const int nt = r.nt;
  FarArgs A;
  A.tgt = tg.pos32;
  A.tgt64 = tg.pos64;
  A.tile_sphere = nt == 4 ? tg.tile_sphere : tg.tile1_sphere;
  A.tile_start = nt == 4 ? tg.tile_start : tg.tile1_start;
  A.tile_count = nt == 4 ? tg.tile_count : tg.tile1_count;
  A.eq = ff.eq32;
  A.n_eq = ff.n_eq;
  A.P = src.P;
  A.excl_off = ff.excl_off;
  A.excl_idx = ff.excl_idx;
  A.cen_hi = src.cen_hi;
  A.cen_lo = src.cen_lo;
  A.q = ff.q;
  A.out = out;
  A.scale = (float)(1.0 / (8.0 * kPi * visc));
  const long long tiles = nt == 4 ? tg.n_tiles : tg.n_tiles1;
  const int parts = partial ? r.parts : 1;
  const long long n3 = 3LL * tg.n;
  ++t_launches;
  if (nt == 4 && r.packed) pairs_far2_kernel<<<tiles * parts, kPairThreads, 0, st>>>(A, parts, partial, n3);
  else if (nt == 4) pairs_far_kernel<4><<<tiles * parts, kPairThreads, 0, st>>>(A, parts, partial, n3);
  else pairs_far_kernel<1><<<tiles * parts, kPairThreads, 0, st>>>(A, parts, partial, n3);
  if (parts > 1) {
    ++t_launches;
    parts_add_kernel<<<grid_for(n3, 256), 256, 0, st>>>(n3, parts, partial, n3, out);
  }
}

size_t pair_args64_bytes() { return sizeof(PairArgs<double>); }

void fill_pair_args64(void* host_dst, const TargetSet& tg, const SourceSet& src, const double* lam_hat,
                      const double* mu, double* out, double visc, int nodes_per_thread) {
  PairArgs<double> A = make_args<double>(tg, src, lam_hat, mu, out, visc, nodes_per_thread);
  std::memcpy(host_dst, &A, sizeof(A));
}

void launch_pairs_batch64(bool double_float, const void* d_args, const int2* d_work, int n_work, const int* d_active,
                          const double* lam, const float2* lam2, const double* mu, double* out,
                          const long long* d_uoff, const long long* d_voff, int parts, double* partial,
                          long long pstride, const SegTable& seg, cudaStream_t st, const long long* d_nlen,
                          unsigned* d_counter) {
  if (n_work == 0) return;
  const PairArgs<double>* args = static_cast<const PairArgs<double>*>(d_args);
  BatchVecs bv{lam, lam2, mu, out, d_uoff, d_voff, partial, pstride, d_nlen, d_counter};
  if (!partial) parts = 1;
  ++t_launches;
  if (double_float) {  // with split sources the last CTA of each item adds the parts
    pairs_dw_batch_kernel<<<kDwPieces * n_work * parts, kDwThreads, 0, st>>>(args, d_work, d_active, bv, parts);
  } else {
    pairs_fp64_batch_kernel<<<4 * n_work * parts, kPairThreads, 0, st>>>(args, d_work, d_active, bv, parts);
    if (parts > 1) {
      ++t_launches;
      if (seg_ctas(seg) > 0)
        pair_parts_reduce_batch_kernel<<<dim3(seg_ctas(seg), (seg.chunk + 127) / 128), 128, 0, st>>>(seg, args, bv, parts);
    }
  }
}

int batch_split_parts(long long items, bool shared_rhs, long long min_sources, int max_parts) {
  return pair_split_parts(items, resident_ctas(shared_rhs ? (const void*)pairs_dw_multi_kernel<kPairRhs>
                                                                      : (const void*)pairs_dw_batch_kernel, kDwThreads),
                          min_sources, max_parts);
}

void launch_pairs_multi64(const void* d_args1, const int4* d_work, int n_work, const int* d_rhs, const int* d_active,
                          const float2* lam2, const double* mu, double* out, const long long* d_uoff,
                          const long long* d_voff, int parts, double* partial, long long pstride,
                          const long long* d_nlen, cudaStream_t st, unsigned* d_counter) {
  if (n_work == 0) return;
  if (!partial) parts = 1;
  const PairArgs<double>* args = static_cast<const PairArgs<double>*>(d_args1);
  BatchVecs bv{nullptr, lam2, mu, out, d_uoff, d_voff, partial, pstride, d_nlen, d_counter};
  ++t_launches;
  pairs_dw_multi_kernel<kPairRhs><<<kDwPieces * n_work * parts, kDwThreads, 0, st>>>(args, d_work, d_rhs, d_active, bv, parts);
}

void launch_seg_dots(const SegTable& t, int nvec, const double* V, long long ldv, const double* w, double* partial,
                     double* h, cudaStream_t st) {
  if (seg_ctas(t) == 0 || nvec == 0) return;
  ++t_launches;
  seg_dots_kernel<<<dim3(seg_ctas(t), (nvec + kSegDotVecs - 1) / kSegDotVecs), kSegThreads, 0, st>>>(t, nvec, V, ldv,
                                                                                                     w, partial, h);
}
void launch_seg_update(const SegTable& t, int nvec, const double* V, long long ldv, const double* coef, double sign,
                       double* w, cudaStream_t st) {
  if (seg_ctas(t) == 0 || nvec == 0) return;
  ++t_launches;
  seg_update_kernel<false><<<dim3(seg_ctas(t), (t.chunk + kSegUpdSub - 1) / kSegUpdSub), kSegUpdSub * kSegUpdGroups, 0, st>>>(
      t, nvec, V, ldv, coef, sign, w, nullptr, nullptr);
}
void launch_seg_update_norm(const SegTable& t, int nvec, const double* V, long long ldv, const double* coef, double sign,
                            double* w, double* partial, double* hn, cudaStream_t st) {
  if (seg_ctas(t) == 0 || nvec == 0) return;
  ++t_launches;
  seg_update_kernel<true><<<dim3(seg_ctas(t), (t.chunk + kSegUpdSub - 1) / kSegUpdSub), kSegUpdSub * kSegUpdGroups, 0, st>>>(
      t, nvec, V, ldv, coef, sign, w, partial, hn);
}
void launch_seg_normalise(const SegTable& t, const double* hn, const double* in, double* out, float2* x2, cudaStream_t st) {
  if (seg_ctas(t) == 0) return;
  ++t_launches;
  seg_normalise_kernel<<<seg_ctas(t), kSegThreads, 0, st>>>(t, hn, in, out, x2);
}
void launch_seg_scale_split(const SegTable& t, const double* s, const double* in, double* out, float2* x2,
                            cudaStream_t st) {
  if (seg_ctas(t) == 0) return;
  ++t_launches;
  seg_scale_split_kernel<<<seg_ctas(t), kSegThreads, 0, st>>>(t, s, in, out, x2);
}
void launch_seg_scale(const SegTable& t, const double* s, const double* in, double* out, cudaStream_t st) {
  if (seg_ctas(t) == 0) return;
  ++t_launches;
  seg_scale_kernel<<<seg_ctas(t), kSegThreads, 0, st>>>(t, s, in, out);
}
void launch_batch_givens(const GivensState& S, int j, const double* h1, const double* h2, const double* hn,
                         cudaStream_t st) {
  ++t_launches;
  batch_givens_kernel<<<S.K, 128, 0, st>>>(S, j, h1, h2, hn);
}
void launch_batch_backsolve(const GivensState& S, int jmax, double* coef, cudaStream_t st) {
  ++t_launches;
  batch_backsolve_kernel<<<S.K, 128, 0, st>>>(S, jmax, coef);
}
void launch_axpy64(long long n, double a, const double* x, double* y, cudaStream_t st) {
  ++t_launches;
  axpy64_kernel<<<grid_for(n, 256), 256, 0, st>>>(n, a, x, y);
}

template <typename T>
void launch_gemv(const GemvBatch<T>& b, const T* x, T* y, cudaStream_t st) {
  if (b.n_jobs == 0 || b.max_rows == 0) return;
  const int rows_per_cta = (kGemvThreads / 32) * kGemvRowsPerWarp;
  const int jobs = b.job_list ? b.n_list : b.n_jobs;
  if (jobs == 0) return;
  dim3 grid(jobs, (b.max_rows + rows_per_cta - 1) / rows_per_cta);
  ++t_launches;
  if constexpr (sizeof(T) == 8)
    gemv64_kernel<<<dim3(jobs, (b.max_rows + kGemv64Rows - 1) / kGemv64Rows), 32 * kGemv64Warps, 0, st>>>(b, x, y);
  else if (b.paired) gemv_kernel<true><<<grid, kGemvThreads, 0, st>>>(b, x, y);
  else gemv_kernel<false><<<grid, kGemvThreads, 0, st>>>(b, x, y);
}
template void launch_gemv<float>(const GemvBatch<float>&, const float*, float*, cudaStream_t);

GemvShape gemv_shape(int n_jobs, int max_rows, int max_cols) {
  const long long pairs = (long long)n_jobs * ((max_rows + 1) / 2);
  if (pairs <= 10 * 152) return {1, 4};
  if (max_cols <= 640 && pairs > 4000) return {pairs <= 10000 ? 1 : kGemvMaxRhs, 1};
  if (max_cols > 640 && pairs <= 5000) return {2, 4};
  return {kGemvMaxRhs, 0};
}

int gemv_items(int n, const int* list, const void* const* mat, std::vector<int2>& items, int cap) {
  items.clear();
  int most = 1;
  for (int i = 0; i < n;) {
    int e = i + 1;
    while (e < n && mat[list ? list[e] : e] == mat[list ? list[i] : i]) ++e;
    const int cnt = e - i, parts = (cnt + cap - 1) / cap;
    for (int q = 0; q < parts; ++q) {
      const int i0 = i + (int)((long long)cnt * q / parts), i1 = i + (int)((long long)cnt * (q + 1) / parts);
      items.push_back(make_int2(i0, i1 - i0));
      most = std::max(most, i1 - i0);
    }
    i = e;
  }
  return most;
}

template <bool F32>
static void gemv_pair_launch(const GemvBatch<float>& b, const float2* x, float2* y2, double* y64, cudaStream_t st) {
  if (b.n_items == 0 || b.max_rows == 0) return;
  ++t_launches;
  const int c = b.items_max;
  const int nrp = (b.max_rows + 1) / 2, groups = (nrp + gemv_rp(c) - 1) / gemv_rp(c);
  // several right-hand sides: the CTA's warps share the columns of a row group while there are fewer
  // groups than 64 warps a SM, and take a group each above that
  const bool split = b.col_warps ? b.col_warps > 1 : c == 1 || (long long)b.n_items * groups < 64LL * 152;
  const dim3 grid(b.n_items, split ? groups : (groups + 3) / 4);
#define MFS_GEMV(C, KS) gemv_pair_kernel<F32, C, KS><<<grid, kGemvPairThreads, 0, st>>>(b, x, y2, y64)
  switch (c) {
    case 1: if (split) MFS_GEMV(1, 4); else MFS_GEMV(1, 1); break;
    case 2: if (split) MFS_GEMV(2, 4); else MFS_GEMV(2, 1); break;
    case 3: if (split) MFS_GEMV(3, 4); else MFS_GEMV(3, 1); break;
    default: if (split) MFS_GEMV(4, 4); else MFS_GEMV(4, 1);
  }
#undef MFS_GEMV
}

void launch_gemv_dw(const GemvBatch<float>& b, const float2* x, float2* y_dw, double* y64, cudaStream_t st) {
  gemv_pair_launch<false>(b, x, y_dw, y64, st);
}

void launch_gemv_f32_dw(const GemvBatch<float>& b, const float2* x, float2* y_dw, cudaStream_t st) {
  gemv_pair_launch<true>(b, x, y_dw, nullptr, st);
}

void launch_split_dw(long long n, const double* in, float2* out, cudaStream_t st) {
  ++t_launches;
  split_dw_kernel<<<grid_for(n, 256), 256, 0, st>>>(n, in, out);
}
template void launch_gemv<double>(const GemvBatch<double>&, const double*, double*, cudaStream_t);

template <typename T>
void launch_multidot(int n, int nvec, const T* V, long long ldv, const T* w, double* partial, int nblk, cudaStream_t st) {
  dim3 grid(nblk, nvec);
  ++t_launches;
  multidot_kernel<T><<<grid, kRedThreads, 0, st>>>(n, V, ldv, w, partial, nblk);
}
template void launch_multidot<float>(int, int, const float*, long long, const float*, double*, int, cudaStream_t);
template void launch_multidot<double>(int, int, const double*, long long, const double*, double*, int, cudaStream_t);

void launch_reduce_partials(int nvec, int nblk, const double* partial, double* h, cudaStream_t st) {
  ++t_launches;
  reduce_partials_kernel<<<nvec, 256, 0, st>>>(nvec, nblk, partial, h);
}

template <typename T>
void launch_update(int n, int nvec, const T* V, long long ldv, const double* h, double sign, T* w, cudaStream_t st) {
  ++t_launches;
  update_kernel<T><<<grid_for(n, 256), 256, 0, st>>>(n, nvec, V, ldv, h, sign, w);
}
template void launch_update<float>(int, int, const float*, long long, const double*, double, float*, cudaStream_t);
template void launch_update<double>(int, int, const double*, long long, const double*, double, double*, cudaStream_t);

template <typename T>
void launch_scale_copy(int n, const T* w, double s, T* out, cudaStream_t st) {
  ++t_launches;
  scale_copy_kernel<T><<<grid_for(n, 256), 256, 0, st>>>(n, w, s, out);
}
template void launch_scale_copy<float>(int, const float*, double, float*, cudaStream_t);
template void launch_scale_copy<double>(int, const double*, double, double*, cudaStream_t);

template <typename Tin, typename Tout>
void launch_convert(long long n, const Tin* in, double s, Tout* out, cudaStream_t st) {
  ++t_launches;
  convert_kernel<Tin, Tout><<<grid_for(n, 256), 256, 0, st>>>(n, in, s, out);
}
template void launch_convert<double, float>(long long, const double*, double, float*, cudaStream_t);
template void launch_convert<float, double>(long long, const float*, double, double*, cudaStream_t);
template void launch_convert<double, double>(long long, const double*, double, double*, cudaStream_t);

void launch_axpy_mixed(int n, double a, const float* x, double* y, cudaStream_t st) {
  ++t_launches;
  axpy_mixed_kernel<<<grid_for(n, 256), 256, 0, st>>>(n, a, x, y);
}
void launch_sub(int n, const double* a, const double* b, double* out, cudaStream_t st) {
  ++t_launches;
  sub_kernel<<<grid_for(n, 256), 256, 0, st>>>(n, a, b, out);
}

void launch_forces_torques(const SourceSet& src, const double* lam, double* F, double* T, cudaStream_t st) {
  ++t_launches;
  ft_kernel<<<src.P, 256, 0, st>>>(src.N, src.proxy64, src.img64, src.img_off, src.unk_off, lam, F, T, 3, 1.0, 1.0);
}
void launch_forces_torques_scaled(const SourceSet& src, const double* lam, double* F, double* T, int stride, double sF,
                                  double sT, cudaStream_t st) {
  ++t_launches;
  ft_kernel<<<src.P, 256, 0, st>>>(src.N, src.proxy64, src.img64, src.img_off, src.unk_off, lam, F, T, stride, sF, sT);
}
void launch_rigid_sub(int n, const int* owner, const double* pos64, const double* U, double* out, cudaStream_t st) {
  ++t_launches;
  rigid_sub_kernel<<<grid_for(n, 256), 256, 0, st>>>(n, owner, pos64, U, out);
}

void launch_rhs(int n, const double* colloc_abs, const int* owner, const double* sqrtw, const double* cen,
                const double* v, const double* om, const double* bg, double* wb, cudaStream_t st) {
  Bg b;
  for (int i = 0; i < 15; ++i) b.v[i] = bg[i];
  ++t_launches;
  rhs_kernel<<<grid_for(n, 256), 256, 0, st>>>(n, colloc_abs, owner, sqrtw, cen, v, om, b, wb);
}

double launch_fma_probe(int which, int blocks, int iters, void* sink, cudaStream_t st) {
  ++t_launches;
  if (which == 0) fma_probe_kernel<float><<<blocks, 256, 0, st>>>(iters, 0.9999f, 1e-4f, static_cast<float*>(sink));
  else fma_probe_kernel<double><<<blocks, 256, 0, st>>>(iters, 0.9999, 1e-4, static_cast<double*>(sink));
  return 2.0 * 8.0 * 16.0 * (double)iters * (double)blocks * 256.0;  // flops
}

void launch_assemble_block(int m, int n_src, const double* xrel, const double* sqrtw, const double* yrel,
                           const int* type, double visc, double* B, long long lda, cudaStream_t st) {
  long long tot = (long long)m * n_src;
  int threads = 256;
  long long blocks = (tot + threads - 1) / threads;
  if (blocks == 0) return;
  ++t_launches;
  assemble_self_kernel<<<(unsigned)blocks, threads, 0, st>>>(m, n_src, xrel, sqrtw, yrel, type, 1.0 / (8.0 * kPi * visc),
                                                             B, lda);
}

void launch_assemble_self(const HostDisc& hd, int k, const double* d_colloc_rel, const double* d_sqrtw,
                          const double* d_src_rel, const int* d_src_type, int n_src, double* B, int lda,
                          cudaStream_t st) {
  int m = hd.colloc_off[k + 1] - hd.colloc_off[k];
  long long tot = (long long)m * n_src;
  int threads = 256;
  long long blocks = (tot + threads - 1) / threads;
  ++t_launches;
  assemble_self_kernel<<<(unsigned)blocks, threads, 0, st>>>(m, n_src, d_colloc_rel, d_sqrtw, d_src_rel, d_src_type,
                                                             1.0 / (8.0 * kPi * hd.prm.visc), B, lda);
}

}  // namespace mfs
