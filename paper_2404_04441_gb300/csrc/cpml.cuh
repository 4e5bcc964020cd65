// CPML absorbing layer for the second-order equation (the paper's CPML-like
// boundary, Sec. 2, after Komatitsch and Martin 2007; it prints no equations).
//
// From complex-frequency-shifted stretching of each axis,
//     u_tt = v^2 sum_a ( d_aa u + d_a psi_a + zeta_a ),
//     psi_a^n  = b_a psi_a^{n-1}  + a_a D1_a u^n,
//     zeta_a^n = b_a zeta_a^{n-1} + a_a ( D2_a u^n + D1_a psi_a^n ),
// b = exp(-(d + alpha) dt), a = d / (d + alpha) (b - 1), D2_a the axis part of
// Eq. 1 and D1_a the 8th-order central first derivative. psi_a and zeta_a are
// non-zero only in the two slabs of npml cells at the faces normal to a and
// are stored there.
//
// The leapfrog update with the layer is the plain update plus
//     C * sum_a ( D1_a psi_a^n + zeta_a^n ),
// and the axis-a term is non-zero only within w = npml + 4 cells of the two
// faces normal to a. So the sweep runs unchanged over the whole grid, and
// afterwards every line along each axis is walked through its two end segments
// of w cells (one segment of the whole line when the two would overlap), which
// updates psi_a and zeta_a from u^n (which the sweep does not overwrite) and
// adds the axis term to u^{n+1}. Corner points are updated by each axis in turn
// with no race. Where every axis holds two disjoint segments of a width they are
// unrolled for, one launch takes boxes that own their lines whole
// (cpml_lines_kernel), or one launch per axis where that is faster (kCpmlByAxis,
// kCpmlByAxisBeside); otherwise axis passes run one after another. Receivers
// within w of a face are then re-recorded.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>

#include "common.cuh"
#include "sweep.cuh"

namespace gbw {

struct CpmlGeom {
  int nx, ny, nz;
  int px;   // row pitch of v^2 dt^2 (floats)
  int pxu;  // row pitch of the wavefields (elements; px for FP32 storage)
  int npml, w;         // layer cells; correction width npml + 4
  float *psi[3], *zeta[3];           // slab storage per axis
  const float *bprof[3], *aprof[3];  // per-axis b, a (length n_a)
  float c2[3][5];  // D2 weights / h_a^2 (index 0: centre)
  float c1[3][5];  // D1 weights / h_a (index 1..4)
};

// The layer's profile along one axis of n cells (npml layer cells at each
// end), computed in FP64 and stored FP32: b = exp(-(d + alpha) dt) and
// a = d / (d + alpha) (b - 1), with d = d0 xi^2, d0 = 3 vmax ln(1/R) /
// (2 npml h), alpha = pi f_cps (1 - xi) and xi in (0, 1] the depth into the
// layer (1 at the face); b = 1 and a = 0 outside the layer.
inline void cpml_profile(int n, int npml, double R, double f_cps, double vmax, double h,
                         double dt, float *b, float *a) {
  const double pi = 3.14159265358979323846;
  const double d0 = 3.0 * vmax * std::log(1.0 / R) / (2.0 * npml * h);
  for (int i = 0; i < n; ++i) {
    double xi = 0.0;
    if (i < npml) xi = (double)(npml - i) / npml;
    if (i >= n - npml) xi = std::max(xi, (double)(i - (n - npml - 1)) / npml);
    if (xi <= 0.0) {
      b[i] = 1.f;
      a[i] = 0.f;
      continue;
    }
    const double dd = d0 * xi * xi, al = pi * f_cps * (1.0 - xi);
    const double bb = std::exp(-(dd + al) * dt);
    b[i] = (float)bb;
    a[i] = (float)(dd + al > 0.0 ? dd / (dd + al) * (bb - 1.0) : 0.0);
  }
}

// The layer's D2 (Eq. 1's axis part) and D1 weights along axis ax of
// spacing h.
inline void cpml_axis_coefs(CpmlGeom &g, int ax, double h) {
  g.c2[ax][0] = (float)(kW[0] / (h * h));
  g.c1[ax][0] = 0.f;
  for (int m = 1; m <= 4; ++m) {
    g.c2[ax][m] = (float)(kW[m] / (h * h));
    g.c1[ax][m] = (float)(kW1[m] / h);
  }
}

// Widest layer of the unrolled line ends, and the widths they are built for;
// other layers take the line walks. Each width adds 6 unrolled segments to every
// kernel of the layer, so the set is small: the widths of the bench and the tests
// (8, 16) and two common ones beside them (10, 20). Whole steps in us as boxes
// and as line walks, FP32 and FP16 fields: 150 x 141 x 133 with 8 cells 24 and
// 44, 25 and 66; with 20 39 and 68, 43 and 106 (12, walks only: 53, 80); 320 x
// 256 x 192 with 8 68 and 100, 65 and 130; with 20 108 and 143, 102 and 208 (12:
// 114, 156).
constexpr int kCpmlMaxCap = 20;
constexpr int kCpmlVariants = 4;

inline int cpml_variant(int npml) {
  return npml == 8 ? 0 : npml == 10 ? 1 : npml == 16 ? 2 : npml == 20 ? 3 : -1;
}

// Whether an axis of n cells takes the unrolled line ends: a layer width they
// are built for, two disjoint end segments (n >= 2 (npml + 4)), and 32-bit
// offsets along the line (fstep, sstep: the axis's field and slab steps);
// GBWAVE_CPML_GENERIC=1 keeps the line walks everywhere (the two forms give
// bitwise equal results).
inline bool cpml_seg_fits(int npml, int n, long long fstep, long long sstep) {
  const char *gen = std::getenv("GBWAVE_CPML_GENERIC");
  return cpml_variant(npml) >= 0 && n >= 2 * (npml + 4) &&
         (long long)(npml + 3) * fstep <= INT32_MAX &&
         (long long)(npml - 1) * sstep <= INT32_MAX && !(gen && std::atoi(gen) == 1);
}

// Slab storage, cell-major: cell in [0, 2 npml) counts the low slab's npml
// cells, then the high slab's; the x slabs hold ((cell nz + z) ny + y), the y
// slabs ((cell nz + z) nx + x), the z slabs ((cell ny + y) nx + x), so that
// adjacent lines (adjacent threads) are adjacent in memory.
__device__ __forceinline__ bool cpml_in_slab(int i, int n, int npml) {
  return i < npml || i >= n - npml;
}

__device__ __forceinline__ int cpml_cell(int i, int n, int npml) {
  return i < npml ? i : i - (n - 2 * npml);
}

constexpr int kCpmlChunk = 4;  // positions per batch of loads

// Wavefield elements in the layer kernels. FP32 fields are used as stored.
// 16-bit fields (BF16 / FP16 storage) hold value / 2^e, e the exponent of
// the time step the field holds (StepDesc::exps, chosen by the sweep that
// wrote it): a read converts exactly and multiplies by 2^e, a write
// multiplies by 2^-e (exact) and rounds once to the format, as the sweep's
// stores do. v^2 dt^2, psi and zeta stay FP32.
template <class T>
__device__ __forceinline__ float cpml_get(const T *p, float s) {
  if constexpr (std::is_same<T, float>::value) return *p;
  else return to_f32(*p) * s;
}

template <class T>
__device__ __forceinline__ void cpml_put(T *p, float v, float inv) {
  if constexpr (std::is_same<T, float>::value) *p = v;
  else if constexpr (std::is_same<T, __half>::value) *p = __float2half_rn(v * inv);
  else *p = __float2bfloat16_rn(v * inv);
}

// Four consecutive elements from p (16 bytes for FP32, 8 for 16-bit; p
// aligned to that).
template <class T>
__device__ __forceinline__ void cpml_get4(const T *p, float s, float *v) {
  if constexpr (std::is_same<T, float>::value) {
    const float4 t = *reinterpret_cast<const float4 *>(p);
    v[0] = t.x;
    v[1] = t.y;
    v[2] = t.z;
    v[3] = t.w;
  } else {
    const uint2 w = *reinterpret_cast<const uint2 *>(p);
    const T *e = reinterpret_cast<const T *>(&w);
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = to_f32(e[k]) * s;
  }
}

template <class T>
__device__ __forceinline__ void cpml_put4(T *p, const float *v, float inv) {
  if constexpr (std::is_same<T, float>::value) {
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
    uint2 w;
    T *e = reinterpret_cast<T *>(&w);
#pragma unroll
    for (int k = 0; k < 4; ++k) cpml_put(e + k, v[k], inv);
    *reinterpret_cast<uint2 *>(p) = w;
  }
}

// Scales of one step's fields (16-bit storage): 2^e of u^n and of u^{n+1},
// 2^-e of u^{n+1}, for absolute step step0 + n + koff; and the running
// maximum of |u^{n+1}| that the next step's scale is chosen from (the
// corrected shell values enter it). FP32: all ones, nothing read.
template <class T>
struct CpmlScale {
  float su = 1.f, so = 1.f, inv_so = 1.f;
  unsigned *maxbits = nullptr;
  __device__ __forceinline__ void init(const StepDesc *d, int koff) {
    if constexpr (!std::is_same<T, float>::value) {
      const long long ab = d->step0 + d->n + koff;
      su = exp2_int(d->exps[ab & 3]);
      const int eo = d->exps[(ab + 1) & 3];
      so = exp2_int(eo);
      inv_so = exp2_int(-eo);
      maxbits = const_cast<unsigned *>(&d->maxbits[(ab + 1) & 3]);
    }
  }
  // the largest |value| the warp's remaining lanes wrote (lanes past the
  // last line have returned), into the running maximum: non-negative floats
  // order as their bit patterns
  __device__ __forceinline__ void commit(float vmax) const {
    if constexpr (!std::is_same<T, float>::value) {
      const unsigned m = __activemask();
      const unsigned r = __reduce_max_sync(m, __float_as_uint(vmax));
      if ((threadIdx.x & 31) == __ffs(m) - 1 && r != 0u) atomicMax(maxbits, r);
    }
  }
};

// Four consecutive values of an x row from position p (p a multiple of 4,
// the row 16-byte aligned with its padding up to a multiple of 4 in
// bounds); positions outside [0, n) read as zero.
template <class T>
__device__ __forceinline__ void cpml_row4(const T *row, int p, int n, float *v, float s) {
  if (p < 0 || p >= n) {
    v[0] = v[1] = v[2] = v[3] = 0.f;
    return;
  }
  float t[4];
  cpml_get4(row + p, s, t);
  v[0] = t[0];
  v[1] = p + 1 < n ? t[1] : 0.f;
  v[2] = p + 2 < n ? t[2] : 0.f;
  v[3] = p + 3 < n ? t[3] : 0.f;
}

// One kernel per axis AX (0 = x, 1 = y, 2 = z): one thread per line along
// AX, adjacent lines (adjacent y for x, adjacent x for y and z) in adjacent
// threads. A thread walks its line's end segments, positions i0 .. i1-1
// ([0, w) and [n - w, n), or [0, n) when they would overlap), with register
// windows of u^n (positions i-4 .. i+F+7) and psi^n (i-4 .. i+F+3), F
// positions per batch: at position i it computes psi(k), k = i + 4, in the
// slab cells of the segment's own range i0 .. i1 + 3 (exactly the segment's
// slab cells, so each is updated once per step), then, for i0 <= i < i1,
// zeta^n(i) in the slab cells and u^{n+1}(i) += C (D1 psi^n + zeta^n). The
// walk starts at or before i0 - 4, where the psi used by the corrections is
// zero (before the grid, or between the slabs). The loads of the next batch
// are in flight while the current one is computed. x rows are walked in
// batches aligned to 4 positions and moved as float4 (a row is contiguous
// in one thread); y and z lines are coalesced across the threads.
// kStoreD (the gradient's recompute): the same correction C (D1 psi + zeta)
// is also added to dout, the step's forward increment D = u^{n+1} - 2u^n +
// u^{n-1} stored by the sweep (field layout).
// T: the wavefields' storage (float, or 16-bit with the step's scales read
// from d at absolute step step0 + n + koff). The walk of line t (index
// across the lines) in row q of lines (z for x and y lines, y for z lines).
template <int AX, class T, bool kStoreD>
__device__ __forceinline__ void cpml_line_walk(const CpmlGeom &g, int t, int q,
                                               const T *__restrict__ u, T *__restrict__ unext,
                                               const float *__restrict__ c,
                                               float *__restrict__ dout, const StepDesc *d,
                                               int koff) {
  static_assert(!kStoreD || std::is_same<T, float>::value, "D is stored for FP32 only");
  constexpr int F = kCpmlChunk;
  int n;
  // field offset and stride (pitch pxu), v^2 dt^2 offset and stride (px),
  // slab offset and stride
  long long ub, us, cb, cs, sb, ss;
  if (AX == 0) {
    if (t >= g.ny) return;
    n = g.nx;
    ub = ((long long)q * g.ny + t) * g.pxu;
    us = 1;
    cb = ((long long)q * g.ny + t) * g.px;
    cs = 1;
    sb = (long long)q * g.ny + t;
    ss = (long long)g.nz * g.ny;
  } else {
    if (t >= g.nx) return;
    n = AX == 1 ? g.ny : g.nz;
    ub = AX == 1 ? (long long)q * g.ny * g.pxu + t : (long long)q * g.pxu + t;
    us = AX == 1 ? (long long)g.pxu : (long long)g.ny * g.pxu;
    cb = AX == 1 ? (long long)q * g.ny * g.px + t : (long long)q * g.px + t;
    cs = AX == 1 ? (long long)g.px : (long long)g.ny * g.px;
    sb = (long long)q * g.nx + t;
    ss = AX == 1 ? (long long)g.nz * g.nx : (long long)g.ny * g.nx;
  }
  if constexpr (std::is_same<T, float>::value) {  // FP32 storage: pxu == px
    cb = ub;
    cs = us;
  }
  CpmlScale<T> sc;
  sc.init(d, koff);
  float vmax = 0.f;
  const T *__restrict__ ul = u + ub;
  const float *__restrict__ cl = c + cb;
  T *__restrict__ nl = unext + ub;
  float *__restrict__ dl = kStoreD ? dout + ub : nullptr;
  float *__restrict__ psi = g.psi[AX] + sb;
  float *__restrict__ zeta = g.zeta[AX] + sb;
  const float *bp = g.bprof[AX];
  const float *ap = g.aprof[AX];
  const int npml = g.npml, w = g.w;
  const bool two = n >= 2 * w;
  for (int sg = 0; sg < (two ? 2 : 1); ++sg) {
    const int i0 = (two && sg == 1) ? n - w : 0;
    const int i1 = two ? (sg == 0 ? w : n) : n;
    // Batch of positions i .. i+F-1: u(i+8+f), psi^{n-1}(i+4+f), zeta^{n-1},
    // C and u^{n+1} at i+f.
    float nw[F], npp[F], nzp[F], ncc[F], nun[F];
    auto load = [&](int i) {
      if (AX == 0) {
        cpml_row4(ul, i + 8, n, nw, sc.su);
        if (i + F > i0 && i < i1) {
          cpml_row4(cl, i, n, ncc, 1.f);
          cpml_row4(nl, i, n, nun, sc.so);
        } else {
#pragma unroll
          for (int f = 0; f < F; ++f) ncc[f] = nun[f] = 0.f;
        }
      }
#pragma unroll
      for (int f = 0; f < F; ++f) {
        const int k = i + 4 + f;
        npp[f] = (k >= 0 && k < n && k < i1 + 4 && cpml_in_slab(k, n, npml))
                     ? psi[cpml_cell(k, n, npml) * ss] : 0.f;
        const int p = i + f;
        const bool act = p >= i0 && p < i1;
        nzp[f] = (act && cpml_in_slab(p, n, npml)) ? zeta[cpml_cell(p, n, npml) * ss] : 0.f;
        if (AX != 0) {
          const int kw = i + 8 + f;
          nw[f] = (kw < n) ? cpml_get(ul + kw * us, sc.su) : 0.f;
          ncc[f] = act ? cl[p * cs] : 0.f;
          nun[f] = act ? cpml_get(nl + p * us, sc.so) : 0.f;
        }
      }
    };
    float W[12 + F];  // W[m] = u(i - 4 + m)
    float P[8 + F];   // P[m] = psi(i - 4 + m)
    int i = AX == 0 ? ((i0 - 4) & ~3) : i0 - 4;
    if (AX == 0) {
#pragma unroll
      for (int m = 0; m < 12; m += 4) cpml_row4(ul, i - 4 + m, n, W + m, sc.su);
    } else {
#pragma unroll
      for (int m = 0; m < 12; ++m) {
        const int k = i - 4 + m;
        W[m] = (k >= 0 && k < n) ? cpml_get(ul + k * us, sc.su) : 0.f;
      }
    }
#pragma unroll
    for (int m = 0; m < 8; ++m) P[m] = 0.f;
    load(i);
    for (; i < i1; i += F) {
      float pp[F], zp[F], cc[F], un[F];
#pragma unroll
      for (int f = 0; f < F; ++f) {
        W[12 + f] = nw[f];
        pp[f] = npp[f];
        zp[f] = nzp[f];
        cc[f] = ncc[f];
        un[f] = nun[f];
      }
      if (i + F < i1) load(i + F);
#pragma unroll
      for (int f = 0; f < F; ++f) {  // psi(i + 4 + f) from u(i + f .. i + f + 8)
        const int k = i + 4 + f;
        float v = 0.f;
        if (k >= 0 && k < n && k < i1 + 4 && cpml_in_slab(k, n, npml)) {
          float d1 = 0.f;
#pragma unroll
          for (int m = 1; m <= kR; ++m) d1 = fmaf(g.c1[AX][m], W[8 + f + m] - W[8 + f - m], d1);
          v = fmaf(__ldg(bp + k), pp[f], __ldg(ap + k) * d1);
          psi[cpml_cell(k, n, npml) * ss] = v;
        }
        P[8 + f] = v;
      }
      float out[F];
#pragma unroll
      for (int f = 0; f < F; ++f) {  // u^{n+1}(i + f) += C (D1 psi + zeta)
        const int p = i + f;
        out[f] = un[f];
        if (p < i0 || p >= i1) continue;
        float d1p = 0.f;
#pragma unroll
        for (int m = 1; m <= kR; ++m) d1p = fmaf(g.c1[AX][m], P[4 + f + m] - P[4 + f - m], d1p);
        float corr = d1p;
        if (cpml_in_slab(p, n, npml)) {
          float d2 = g.c2[AX][0] * W[4 + f];
#pragma unroll
          for (int m = 1; m <= kR; ++m) d2 = fmaf(g.c2[AX][m], W[4 + f + m] + W[4 + f - m], d2);
          const float zt = fmaf(__ldg(bp + p), zp[f], __ldg(ap + p) * (d2 + d1p));
          zeta[cpml_cell(p, n, npml) * ss] = zt;
          corr += zt;
        }
        out[f] = fmaf(cc[f], corr, un[f]);
        vmax = fmaxf(vmax, fabsf(out[f]));
        if (AX != 0) cpml_put(nl + p * us, out[f], sc.inv_so);
        if constexpr (kStoreD) dl[p * us] = fmaf(cc[f], corr, dl[p * us]);
      }
      // x: the whole aligned batch in one store (positions outside the
      // segment keep the value just read, which a 16-bit write reproduces
      // exactly; this thread owns the row)
      if (AX == 0 && i + F > i0 && i < i1) cpml_put4(nl + i, out, sc.inv_so);
#pragma unroll
      for (int m = 0; m < 12; ++m) W[m] = W[m + F];
#pragma unroll
      for (int m = 0; m < 8; ++m) P[m] = P[m + F];
    }
  }
  sc.commit(vmax);
}

template <int AX, class T, bool kStoreD = false>
__global__ void __launch_bounds__(128)
    cpml_line_kernel(CpmlGeom g, const T *__restrict__ u, T *__restrict__ unext,
                     const float *__restrict__ c, float *__restrict__ dout,
                     const StepDesc *d, int koff) {
  cpml_line_walk<AX, T, kStoreD>(g, blockIdx.x * blockDim.x + threadIdx.x, blockIdx.y, u,
                                 unext, c, dout, d, koff);
}


// Discrete adjoint of the layer (the gradient's backward steps), in the
// form the sweep runs it, p = C q. After the plain adjoint sweep has written
// p^k = 2p^{k+1} - p^{k+2} + C L p^{k+1} (+ injections), for each axis a:
//     nu_a^k = p^{k+1} + B_a nu_a^{k+1}              (slab cells)
//     mu_a^k = -D1_a (p^{k+1} + A_a nu_a^k) + B_a mu_a^{k+1}
//     p^k   += C ( D2_a (A_a nu_a^k) - D1_a (A_a mu_a^k) )
// (D2_a symmetric and D1_a antisymmetric with the zero halo). A nu and A mu
// vanish outside the slabs, so the correction reaches w = npml + 4 cells
// from each face, as in the forward. One thread per line, the same end
// segments; the walk starts 8 positions before a segment: at position i it
// forms nu (and g = p + A nu) at i + 8, mu at i + 4 (from g at i .. i + 8)
// and, inside the segment, the correction at i. Each slab cell is updated
// by the segment that owns it (the whole line when the segments overlap).
template <int AX>
__global__ void __launch_bounds__(128)
    cpml_adjoint_line_kernel(CpmlGeom g, const float *__restrict__ p1,
                             float *__restrict__ p0, const float *__restrict__ c,
                             float *__restrict__ nus, float *__restrict__ mus) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int q = blockIdx.y;
  int n;
  long long ub, us, sb, ss;
  if (AX == 0) {
    if (t >= g.ny) return;
    n = g.nx;
    ub = ((long long)q * g.ny + t) * g.px;
    us = 1;
    sb = (long long)q * g.ny + t;
    ss = (long long)g.nz * g.ny;
  } else {
    if (t >= g.nx) return;
    n = AX == 1 ? g.ny : g.nz;
    ub = AX == 1 ? (long long)q * g.ny * g.px + t : (long long)q * g.px + t;
    us = AX == 1 ? (long long)g.px : (long long)g.ny * g.px;
    sb = (long long)q * g.nx + t;
    ss = AX == 1 ? (long long)g.nz * g.nx : (long long)g.ny * g.nx;
  }
  const float *__restrict__ pl = p1 + ub;
  const float *__restrict__ cl = c + ub;
  float *__restrict__ ol = p0 + ub;
  float *__restrict__ nu = nus + sb;
  float *__restrict__ mu = mus + sb;
  const float *bp = g.bprof[AX];
  const float *ap = g.aprof[AX];
  const int npml = g.npml, w = g.w;
  const bool two = n >= 2 * w;
  for (int sg = 0; sg < (two ? 2 : 1); ++sg) {
    const int i0 = (two && sg == 1) ? n - w : 0;
    const int i1 = two ? (sg == 0 ? w : n) : n;
    // slab cells this segment updates
    auto owned = [&](int k) {
      if (k < 0 || k >= n || !cpml_in_slab(k, n, npml)) return false;
      return !two || (sg == 0 ? k < npml : k >= n - npml);
    };
    float G[9];    // g = p + A nu at positions i .. i+8
    float AN[13];  // A nu at i-4 .. i+8
    float AM[9];   // A mu at i-4 .. i+4
#pragma unroll
    for (int m = 0; m < 9; ++m) G[m] = AM[m] = 0.f;
#pragma unroll
    for (int m = 0; m < 13; ++m) AN[m] = 0.f;
    for (int i = i0 - 8; i < i1; ++i) {
      // nu and g at i + 8
      const int k8 = i + 8;
      float pv = 0.f, an = 0.f;
      if (k8 >= 0 && k8 < n) {
        pv = pl[k8 * us];
        if (cpml_in_slab(k8, n, npml)) {
          const long long cell = cpml_cell(k8, n, npml) * ss;
          const float nv = fmaf(__ldg(bp + k8), nu[cell], pv);
          if (owned(k8)) nu[cell] = nv;
          an = __fmul_rn(__ldg(ap + k8), nv);
        }
      }
      G[8] = __fadd_rn(pv, an);  // rounded as written (no contraction)
      AN[12] = an;
      // mu at i + 4 from g at i .. i + 8
      const int k4 = i + 4;
      float am = 0.f;
      if (k4 >= 0 && k4 < n && cpml_in_slab(k4, n, npml)) {
        float d1 = 0.f;
#pragma unroll
        for (int m = 1; m <= kR; ++m) d1 = fmaf(g.c1[AX][m], G[4 + m] - G[4 - m], d1);
        const long long cell = cpml_cell(k4, n, npml) * ss;
        const float mv = fmaf(__ldg(bp + k4), mu[cell], -d1);
        if (owned(k4)) mu[cell] = mv;
        am = __fmul_rn(__ldg(ap + k4), mv);
      }
      AM[8] = am;
      // correction at i
      if (i >= i0) {
        float d2 = g.c2[AX][0] * AN[4];
        float d1 = 0.f;
#pragma unroll
        for (int m = 1; m <= kR; ++m) {
          d2 = fmaf(g.c2[AX][m], AN[4 + m] + AN[4 - m], d2);
          d1 = fmaf(g.c1[AX][m], AM[4 + m] - AM[4 - m], d1);
        }
        const float corr = d2 - d1;
        if (corr != 0.f) ol[i * us] = fmaf(cl[i * us], corr, ol[i * us]);
      }
#pragma unroll
      for (int m = 0; m < 8; ++m) G[m] = G[m + 1];
#pragma unroll
      for (int m = 0; m < 12; ++m) AN[m] = AN[m + 1];
#pragma unroll
      for (int m = 0; m < 8; ++m) AM[m] = AM[m + 1];
    }
  }
}

// ---------------------------------------------------------------------------
// The layer in one launch.
//
// The three axis terms of a step meet only where shells cross: the axis-a
// term of a point needs u^n, psi_a and zeta_a along its own line, inside one
// end segment of w = npml + 4 cells, and nothing else. So the shell splits
// into boxes by whether each coordinate lies near a low face, between, or
// near a high one, and every box owns its lines whole:
//   * faces (one coordinate near a face): the lines normal to it;
//   * edges (two, tiled by T cells along the third axis): the lines of the
//     lower axis, then, after a barrier, those of the higher one, which add to
//     the points the first ones wrote;
//   * corners: x, then y, then z lines.
// Every point gets its x, y and z terms in that order, as three axis passes
// one after another would add them: the results are bitwise the same. A box's
// lines are shared by a cluster of kCpmlCluster CTAs, so that an edge tile is
// wide enough for whole sectors along x and still takes one line per thread
// and phase; the barrier is the cluster's.
//
// A line end is one thread: positions are counted from the face (j = 0 ..
// w-1, mirrored at the high face, where D1 changes sign: folded into the order
// of each difference, so every operation rounds as in the line walks above).
// The segment of a layer of NPML cells is unrolled with no per-position
// predicates: u^n is read only at the w positions the layer needs (psi reaches
// u up to npml + 3 cells from the face), the profile values travel in the
// kernel's parameters (constant operands), offsets along the line are 32-bit.
//
// What bounds it: on small grids the launches and two memory latencies a
// line (u^n, psi and zeta; then C and u^{n+1}), on large ones the traffic of
// lines that every array is read along. Against one launch per axis (line
// walks at 10 cells, unrolled at 16), with the sweep of that time, a whole step
// took 31 us instead of 56 at 150 x 141 x 133 with 10 cells (25 now), 102 instead
// of 103 at 320 x 256 x 192 in FP16 (82 now) and 296 instead of 297 at 512 x 512 x
// 256 with 16 (288 now); the gradient through autograd at 160 x 144 x 128 x 100
// steps 18.2 ms instead of 20.0 (15.6 now). CTAs of 256
// threads without clusters took 7 % longer at 320 x 256 x 192, 4 CTAs an SM
// (128 registers) 2 %, a second launch for the corners' z lines instead of the
// third phase 4 %, L2 prefetches of C and u^{n+1} 10 %.
constexpr int kCpmlThreads = 128;
constexpr int kCpmlCluster = 4;
constexpr int kCpmlLines = kCpmlThreads * kCpmlCluster;  // lines of a cluster

// CTAs per SM the line kernels are compiled for (168 registers a thread up to 16
// cells, 255 beyond; the server's 16-cell forms for 16-bit fields spill 208 bytes).
constexpr int cpml_ctas(int npml) { return npml > 16 ? 2 : 3; }

// Profile values by axis, face and depth from the face.
template <int NPML>
struct CpmlProf {
  float b[3][2][NPML], a[3][2][NPML];
};

template <int NPML>
inline void cpml_fill_prof(CpmlProf<NPML> &pf, int ax, const float *b, const float *a, int n,
                           int npml) {
  for (int j = 0; j < NPML && j < npml; ++j)
    for (int sd = 0; sd < 2; ++sd) {
      const int i = sd ? n - 1 - j : j;
      pf.b[ax][sd][j] = b[i];
      pf.a[ax][sd][j] = a[i];
    }
}

// Clusters of one launch: the corners, the edges of each pair of axes, then
// the faces of each axis. all: every axis at once; otherwise the lines of one
// axis alone, over the whole grid (a layer with an axis too short for two
// disjoint segments takes its axes one by one).
struct CpmlTiles {
  int w, T;
  int near[3];   // cells near a face: w, along x rounded up to 8 (whole
                 // sectors for the y and z faces) where the grid allows
  int all;
  int start[8];  // corners; xy, xz, yz edges; x, y, z faces; total
  struct {
    int half;               // clusters of one side
    int p0, np, q0, total;  // cross coordinates and lines of a side
  } face[3];
};

inline CpmlTiles cpml_tiles(int nx, int ny, int nz, int w, int only) {
  CpmlTiles t{};
  t.w = w;
  t.all = only < 0;
  const int n[3] = {nx, ny, nz};
  long long nb[7] = {};
  if (t.all) {
    const int r8 = (w + 7) & ~7;
    t.near[0] = 2 * r8 <= nx ? r8 : w;
    t.near[1] = t.near[2] = w;
    t.T = std::max(4, (kCpmlLines / t.near[0]) & ~3);
    nb[0] = 8;
    for (int e = 0; e < 3; ++e)
      nb[1 + e] = 4ll * ((n[2 - e] - 2 * t.near[2 - e] + t.T - 1) / t.T);
  }
  for (int ax = 0; ax < 3; ++ax) {
    if (!t.all && ax != only) continue;
    const int b = ax == 0 ? 1 : 0, c = ax == 2 ? 1 : 2;
    const long long p = n[b] - 2 * t.near[b], q = n[c] - 2 * t.near[c];
    t.face[ax].half = (int)((p * q + kCpmlLines - 1) / kCpmlLines);
    t.face[ax].p0 = t.near[b];
    t.face[ax].np = (int)p;
    t.face[ax].q0 = t.near[c];
    t.face[ax].total = (int)(p * q);
    nb[4 + ax] = 2ll * t.face[ax].half;
  }
  for (int k = 0; k < 7; ++k) t.start[k + 1] = t.start[k] + (int)nb[k];
  return t;
}

__host__ __device__ __forceinline__ int cpml_dim(const CpmlGeom &g, int ax) {
  return ax == 0 ? g.nx : ax == 1 ? g.ny : g.nz;
}

// A rectangle of lines: axis ax, face side, cross coordinates p in [p0, p0 +
// np) and q in [q0, q0 + nq), p along the lower of the two other axes (adjacent
// lines in adjacent threads).
struct CpmlRect {
  int ax, side, p0, np, q0, nq;
};

// A range of cells along one axis.
struct CpmlRange {
  int lo, n;
};

// The lines of cluster blk, in its phases. ctid: thread within the cluster;
// line(ax, side, p, q) takes a line, sync() is the cluster's barrier.
#pragma nv_exec_check_disable
template <class F, class S>
__host__ __device__ __forceinline__ void cpml_block(const CpmlGeom &g, const CpmlTiles &t,
                                                    int blk, int ctid, const F &line,
                                                    const S &sync) {
  CpmlRange r[3];
  unsigned sides, axes;
  int phases, ax = -1;
  CpmlRange p, q;
  int total, first = ctid, step = kCpmlLines;
  const bool face = blk >= t.start[4];
  if (face) {  // most blocks: one line a thread
    ax = blk >= t.start[6] ? 2 : blk >= t.start[5] ? 1 : 0;
    const auto &f = ax == 2 ? t.face[2] : ax == 1 ? t.face[1] : t.face[0];
    const int local = blk - (ax == 2 ? t.start[6] : ax == 1 ? t.start[5] : t.start[4]);
    const int side = local >= f.half;
    first += (local - (side ? f.half : 0)) * kCpmlLines;
    total = f.total;
    step = 1 << 30;
    p = CpmlRange{f.p0, f.np};
    q = CpmlRange{f.q0, 0};
    sides = side ? 7u : 0u;
    axes = 0;
    phases = 1;
  } else {
    auto near_range = [&](int k, int side) {
      return CpmlRange{side ? cpml_dim(g, k) - t.near[k] : 0, t.near[k]};
    };
    if (blk < 8) {  // corners
      axes = 7;
      sides = (unsigned)blk;
      phases = 3;
    } else {  // a tile of an edge along m
      const int cls = blk >= t.start[3] ? 3 : blk >= t.start[2] ? 2 : 1;
      const int local = blk - (cls == 3 ? t.start[3] : cls == 2 ? t.start[2] : t.start[1]);
      const int m = 3 - cls, a = cls == 3 ? 1 : 0, b = cls == 1 ? 1 : 2;
      const int nr = m == 0 ? t.near[0] : t.w, len = cpml_dim(g, m) - 2 * nr;
      const int per = (len + t.T - 1) / t.T, ci = local / per, m0 = (local - ci * per) * t.T;
      axes = (1u << a) | (1u << b);
      sides = ((ci & 1u) << a) | ((unsigned)(ci >> 1) << b);
      phases = 2;
      r[0] = r[1] = r[2] = CpmlRange{nr + m0, len - m0 < t.T ? len - m0 : t.T};
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if ((axes >> k) & 1) r[k] = near_range(k, (sides >> k) & 1);
  }
#pragma unroll 1
  for (int ph = 0; ph < phases; ++ph) {
    if (!face) {
      if (ph) sync();
      do ++ax;
      while (!((axes >> ax) & 1));
      p = ax == 0 ? r[1] : r[0];
      q = ax == 2 ? r[1] : r[2];
      total = p.n * q.n;
    }
#pragma unroll 1
    for (int i = first; i < total; i += step) {
      const int iq = (int)((unsigned)i / (unsigned)p.n);
      line(ax, (int)((sides >> ax) & 1), p.lo + (i - iq * p.n), q.lo + iq);
      if (face) break;
    }
  }
}

// Offsets of a line end: field (pitch pxu), v^2 dt^2 (pitch px) and slab of
// position j = 0, and the steps per position. The high face's slab cell of
// position j is 2 npml - 1 - j.
struct CpmlLine {
  long long u0, c0, s0;
  int ustep, cstep, sstep, n;
};

template <int AX, int SIDE>
__device__ __forceinline__ CpmlLine cpml_line_at(const CpmlGeom &g, int p, int q) {
  CpmlLine l;
  l.n = AX == 0 ? g.nx : AX == 1 ? g.ny : g.nz;
  const int x = AX == 0 ? 0 : p, y = AX == 0 ? p : AX == 1 ? 0 : q, z = AX == 2 ? 0 : q;
  const int us = AX == 0 ? 1 : AX == 1 ? g.pxu : g.ny * g.pxu;
  const int cs = AX == 0 ? 1 : AX == 1 ? g.px : g.ny * g.px;
  // slabs: ((cell nz + z) ny + y), ((cell nz + z) nx + x), ((cell ny + y) nx + x)
  const int ss = AX == 0 ? g.nz * g.ny : AX == 1 ? g.nz * g.nx : g.ny * g.nx;
  const long long row = (long long)z * g.ny + y;
  l.u0 = row * g.pxu + x;
  l.c0 = row * g.px + x;
  l.s0 = AX == 0 ? row : AX == 1 ? (long long)z * g.nx + x : (long long)y * g.nx + x;
  if (SIDE) {
    l.u0 += (long long)(l.n - 1) * us;
    l.c0 += (long long)(l.n - 1) * cs;
    l.s0 += (long long)(2 * g.npml - 1) * ss;
  }
  l.ustep = SIDE ? -us : us;
  l.cstep = SIDE ? -cs : cs;
  l.sstep = SIDE ? -ss : ss;
  return l;
}

// v[j] = f(position j) times s for the W positions (r: position
// 0). x lines are rows: read as 4-element vectors when the segment starts on
// a vector boundary (the low face always; the high face when n is a multiple
// of 4).
template <int AX, int SIDE, int W, class T>
__device__ __forceinline__ void cpml_line_load(const T *r, int step, int n, float s,
                                               float *v) {
  if (AX == 0 && (SIDE == 0 || (n & 3) == 0)) {
#pragma unroll
    for (int k = 0; k < W; k += 4) {
      float e[4];
      cpml_get4(SIDE == 0 ? r + k : r - (k + 3), s, e);
#pragma unroll
      for (int m = 0; m < 4; ++m)
        if (k + m < W) v[k + m] = SIDE == 0 ? e[m] : e[3 - m];
    }
  } else {
#pragma unroll
    for (int j = 0; j < W; ++j)
      v[j] = cpml_get(r + j * step, s);
  }
}

// A group of 4 that reaches past the segment is stored one by one: the points
// behind it may belong to another cluster.
template <int AX, int SIDE, int W, class T>
__device__ __forceinline__ void cpml_line_store(T *r, int step, int n, float inv,
                                                const float *v) {
  const bool vec = AX == 0 && (SIDE == 0 || (n & 3) == 0);
#pragma unroll
  for (int k = 0; k < W; k += 4) {
    if (vec && k + 4 <= W) {
      float e[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) e[m] = k + 4 <= W ? v[SIDE == 0 ? k + m : k + 3 - m] : 0.f;
      cpml_put4(SIDE == 0 ? r + k : r - (k + 3), e, inv);
    } else {
#pragma unroll
      for (int m = 0; m < 4; ++m)
        if (k + m < W) cpml_put(r + (k + m) * step, v[k + m], inv);
    }
  }
}

// Window value v[k], zero outside [0, N) (k is a compile-time constant
// after unrolling, so the test costs nothing).
template <int N>
__device__ __forceinline__ float cpml_seg_at(const float *v, int k) {
  return (k >= 0 && k < N) ? v[k] : 0.f;
}

// D1 at position j of a window v (zero outside [0, N)), as the line walks
// round it: sum over m of c1_m (f(i+m) - f(i-m)), i the grid position, which
// at the high face is v(j-m) - v(j+m).
template <int SIDE, int N>
__device__ __forceinline__ float cpml_seg_d1(const float *v, int j, const float *c1) {
  float d = 0.f;
#pragma unroll
  for (int m = 1; m <= kR; ++m) {
    const float hi = cpml_seg_at<N>(v, j + m);
    const float lo = cpml_seg_at<N>(v, j - m);
    d = fmaf(c1[m], SIDE == 0 ? hi - lo : lo - hi, d);
  }
  return d;
}

template <int N>
__device__ __forceinline__ float cpml_seg_d2(const float *v, int j, const float *c2) {
  float d = c2[0] * cpml_seg_at<N>(v, j);
#pragma unroll
  for (int m = 1; m <= kR; ++m)
    d = fmaf(c2[m], cpml_seg_at<N>(v, j + m) + cpml_seg_at<N>(v, j - m), d);
  return d;
}

// One line end of the forward step. Two phases, each issuing all of its loads
// before its first store (the slabs and the fields are not known to be
// distinct, so a load after a store waits for it): u^n, psi and zeta -> the
// new psi, zeta and the corrections; then C, u^{n+1} (and D) -> u^{n+1} (and
// D) updated. The live set stays about half of what one phase would hold.
// T: the wavefields' storage (float, or 16-bit with the step's scales); D is
// stored for FP32 only.
template <int AX, int SIDE, int NPML, class T, bool kStoreD, class P>
__device__ __forceinline__ void cpml_line_forward(const CpmlGeom &g, const P &pf, int p, int q,
                                                  const T *u, T *unext, const float *c,
                                                  float *dout, const CpmlScale<T> &sc) {
  constexpr int W = NPML + 4;
  const CpmlLine l = cpml_line_at<AX, SIDE>(g, p, q);
  float *psi = g.psi[AX] + l.s0;
  float *zeta = g.zeta[AX] + l.s0;
  float U[W], PS[NPML], ZT[NPML], CORR[W];
  cpml_line_load<AX, SIDE, W>(u + l.u0, l.ustep, l.n, sc.su, U);
#pragma unroll
  for (int j = 0; j < NPML; ++j) {
    PS[j] = psi[j * l.sstep];
    ZT[j] = zeta[j * l.sstep];
  }
#pragma unroll
  for (int j = 0; j < NPML; ++j) {
    const float d1 = cpml_seg_d1<SIDE, W>(U, j, g.c1[AX]);
    PS[j] = fmaf(pf.b[AX][SIDE][j], PS[j], pf.a[AX][SIDE][j] * d1);
  }
#pragma unroll
  for (int j = 0; j < W; ++j) {
    const float d1p = cpml_seg_d1<SIDE, NPML>(PS, j, g.c1[AX]);
    CORR[j] = d1p;
    if (j < NPML) {
      const float d2 = cpml_seg_d2<W>(U, j, g.c2[AX]);
      ZT[j] = fmaf(pf.b[AX][SIDE][j], ZT[j], pf.a[AX][SIDE][j] * (d2 + d1p));
      CORR[j] += ZT[j];
    }
  }
#pragma unroll
  for (int j = 0; j < NPML; ++j) {
    psi[j * l.sstep] = PS[j];
    zeta[j * l.sstep] = ZT[j];
  }
  float CC[W], UN[W], DO[kStoreD ? W : 1];
  if constexpr (std::is_same<T, float>::value)  // FP32 storage: pxu == px
    cpml_line_load<AX, SIDE, W>(c + l.u0, l.ustep, l.n, 1.f, CC);
  else
    cpml_line_load<AX, SIDE, W>(c + l.c0, l.cstep, l.n, 1.f, CC);
  cpml_line_load<AX, SIDE, W>((const T *)unext + l.u0, l.ustep, l.n, sc.so, UN);
  if constexpr (kStoreD)
    cpml_line_load<AX, SIDE, W>((const float *)dout + l.u0, l.ustep, l.n, 1.f, DO);
  float vmax = 0.f;
#pragma unroll
  for (int j = 0; j < W; ++j) {
    UN[j] = fmaf(CC[j], CORR[j], UN[j]);
    vmax = fmaxf(vmax, fabsf(UN[j]));
    if constexpr (kStoreD) DO[j] = fmaf(CC[j], CORR[j], DO[j]);
  }
  cpml_line_store<AX, SIDE, W>(unext + l.u0, l.ustep, l.n, sc.inv_so, UN);
  if constexpr (kStoreD)
    cpml_line_store<AX, SIDE, W>(dout + l.u0, l.ustep, l.n, 1.f, DO);
  sc.commit(vmax);
}

// One line end of the adjoint step (cpml_adjoint_line_kernel, unrolled): nu
// and g = p^{k+1} + A nu at the w positions, mu at the slab cells, then p^k +=
// C (D2 (A nu) - D1 (A mu)) over the segment; two phases as in the forward.
template <int AX, int SIDE, int NPML, class P>
__device__ __forceinline__ void cpml_line_adjoint(const CpmlGeom &g, const P &pf, int p, int q,
                                                  const float *p1, float *p0, const float *c,
                                                  float *nus, float *mus) {
  constexpr int W = NPML + 4;
  const CpmlLine l = cpml_line_at<AX, SIDE>(g, p, q);
  float *nu = nus + l.s0, *mu = mus + l.s0;
  float G[W], NU[NPML], MU[NPML], AN[NPML], AM[NPML], CORR[W];
  cpml_line_load<AX, SIDE, W>(p1 + l.u0, l.ustep, l.n, 1.f, G);
#pragma unroll
  for (int j = 0; j < NPML; ++j) {
    NU[j] = nu[j * l.sstep];
    MU[j] = mu[j * l.sstep];
  }
#pragma unroll
  for (int j = 0; j < NPML; ++j) {
    NU[j] = fmaf(pf.b[AX][SIDE][j], NU[j], G[j]);
    AN[j] = __fmul_rn(pf.a[AX][SIDE][j], NU[j]);
    G[j] = __fadd_rn(G[j], AN[j]);  // as the line walk: no contraction
  }
#pragma unroll
  for (int j = 0; j < NPML; ++j) {
    MU[j] = fmaf(pf.b[AX][SIDE][j], MU[j], -cpml_seg_d1<SIDE, W>(G, j, g.c1[AX]));
    AM[j] = __fmul_rn(pf.a[AX][SIDE][j], MU[j]);
  }
#pragma unroll
  for (int j = 0; j < W; ++j) {  // A nu and A mu are zero past the slab
    const float d2 = cpml_seg_d2<NPML>(AN, j, g.c2[AX]);
    const float d1 = cpml_seg_d1<SIDE, NPML>(AM, j, g.c1[AX]);
    CORR[j] = d2 - d1;
  }
#pragma unroll
  for (int j = 0; j < NPML; ++j) {
    nu[j * l.sstep] = NU[j];
    mu[j * l.sstep] = MU[j];
  }
  float CC[W], PO[W];
  cpml_line_load<AX, SIDE, W>(c + l.u0, l.ustep, l.n, 1.f, CC);  // FP32: pxu == px
  cpml_line_load<AX, SIDE, W>((const float *)p0 + l.u0, l.ustep, l.n, 1.f, PO);
#pragma unroll
  for (int j = 0; j < W; ++j)
    PO[j] = fmaf(CC[j], CORR[j], PO[j]);
  cpml_line_store<AX, SIDE, W>(p0 + l.u0, l.ustep, l.n, 1.f, PO);
}

// Fields of one layer pass. Forward: u^n, u^{n+1}, C, D (the gradient's
// recompute), the descriptor and offset of the step (the 16-bit fields'
// scales), and the shell receivers {x, y, z, id}, *nsrec of them. Adjoint:
// p^{k+1}, p^k, C and the nu, mu slabs.
struct CpmlPass {
  const void *u;
  void *unext;
  const float *c;
  float *dout;
  const StepDesc *d;
  int koff;
  const int4 *srec;
  const int *nsrec;
  float *nus[3], *mus[3];
};

// The shell receivers' row of the step before this pass's: u^n is that step's
// field with the layer's terms, and nothing writes it during this step, so the
// row rides in blocks beside the lines instead of in a launch of its own after
// them (2 us a step; the last step's row is recorded at the call's end).
constexpr int kCpmlRecClusters = 8;

template <class T>
__device__ __forceinline__ void cpml_record_previous(const CpmlGeom &g, const CpmlPass &a,
                                                     int first, int step) {
  const long long n = a.d->n + a.koff;
  const int nr = *a.nsrec;
  if (n == 0 || nr == 0) return;
  CpmlScale<T> sc;
  sc.init(a.d, a.koff);
  const T *u = static_cast<const T *>(a.u);
  float *row = a.d->traces + (size_t)(n - 1) * a.d->nrec;
  for (int r = first; r < nr; r += step) {
    const int4 e = a.srec[r];
    row[e.w] = cpml_get(u + ((size_t)e.z * g.ny + e.y) * g.pxu + e.x, sc.su);
  }
}

// Release and acquire over the cluster: global writes before it are visible
// to the cluster's reads after it.
__device__ __forceinline__ void cpml_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// A layer pass: the layer's width, the fields' storage T, and
// whether D is updated too.
template <int NPML_, class T, bool kStoreD>
struct CpmlForward {
  static constexpr int NPML = NPML_;
  static constexpr bool kRecords = !kStoreD;
  __device__ static __forceinline__ void record_previous(const CpmlGeom &g, const CpmlPass &a,
                                                         int first, int step) {
    cpml_record_previous<T>(g, a, first, step);
  }
  template <int AX, int SIDE, class P>
  __device__ static __forceinline__ void line(const CpmlGeom &g, const P &pf, const CpmlPass &a,
                                              int p, int q, const CpmlScale<T> &sc) {
    cpml_line_forward<AX, SIDE, NPML, T, kStoreD>(g, pf, p, q,
                                                         static_cast<const T *>(a.u),
                                                         static_cast<T *>(a.unext), a.c, a.dout,
                                                         sc);
  }
  __device__ static __forceinline__ CpmlScale<T> scale(const CpmlPass &a) {
    CpmlScale<T> sc;
    sc.init(a.d, a.koff);
    return sc;
  }
};

template <int NPML_>
struct CpmlAdjoint {
  static constexpr int NPML = NPML_;
  static constexpr bool kRecords = false;
  __device__ static __forceinline__ void record_previous(const CpmlGeom &, const CpmlPass &, int,
                                                         int) {}
  template <int AX, int SIDE, class P>
  __device__ static __forceinline__ void line(const CpmlGeom &g, const P &pf, const CpmlPass &a,
                                              int p, int q, const CpmlScale<float> &) {
    cpml_line_adjoint<AX, SIDE, NPML>(g, pf, p, q, static_cast<const float *>(a.u),
                                             static_cast<float *>(a.unext), a.c, a.nus[AX],
                                             a.mus[AX]);
  }
  __device__ static __forceinline__ CpmlScale<float> scale(const CpmlPass &) { return {}; }
};

// The lines of this CTA of cluster blk.
template <class OP, class P>
__device__ __forceinline__ void cpml_lines(const CpmlGeom &g, const CpmlTiles &t, const P &pf,
                                           const CpmlPass &a, int blk) {
  const auto sc = OP::scale(a);
  cpml_block(
      g, t, blk, (int)(blockIdx.x % kCpmlCluster) * kCpmlThreads + threadIdx.x,
      [&](int ax, int side, int p, int q) {
        if (side == 0) {
          if (ax == 0) OP::template line<0, 0>(g, pf, a, p, q, sc);
          else if (ax == 1) OP::template line<1, 0>(g, pf, a, p, q, sc);
          else OP::template line<2, 0>(g, pf, a, p, q, sc);
        } else {
          if (ax == 0) OP::template line<0, 1>(g, pf, a, p, q, sc);
          else if (ax == 1) OP::template line<1, 1>(g, pf, a, p, q, sc);
          else OP::template line<2, 1>(g, pf, a, p, q, sc);
        }
      },
      [] { cpml_cluster_sync(); });
}

template <class OP>
__global__ void __launch_bounds__(kCpmlThreads, cpml_ctas(OP::NPML))
    cpml_lines_kernel(const __grid_constant__ CpmlGeom g, const __grid_constant__ CpmlTiles t,
                      const __grid_constant__ CpmlProf<OP::NPML> pf,
                      const __grid_constant__ CpmlPass a) {
  const int blk = blockIdx.x / kCpmlCluster;
  if (OP::kRecords && blk >= t.start[7])
    OP::record_previous(g, a, (blockIdx.x - t.start[7] * kCpmlCluster) * kCpmlThreads + threadIdx.x,
                        kCpmlRecClusters * kCpmlLines);
  else
    cpml_lines<OP>(g, t, pf, a, blk);
}

// Receivers within w of a face: {x, y, z, receiver id}, recorded from the
// field after the step's layer terms (16-bit: the stored value times its
// scale).
template <class T>
__global__ void cpml_record_kernel(CpmlGeom g, const T *__restrict__ unext,
                                   const StepDesc *d, const int4 *srec,
                                   const int *nsrec, int koff) {
  const int nr = *nsrec;
  if (nr == 0) return;
  const long long n = d->n + koff;
  CpmlScale<T> sc;
  sc.init(d, koff);
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nr;
       t += gridDim.x * blockDim.x) {
    const int4 e = srec[t];
    d->traces[(size_t)n * d->nrec + e.w] =
        cpml_get(unext + ((size_t)e.z * g.ny + e.y) * g.pxu + e.x, sc.so);
  }
}

// What the host keeps of a layer to launch its passes.
struct CpmlPlan {
  CpmlGeom g;
  int axes;     // bit a: axis a takes the unrolled line ends
  int variant;  // which width (cpml_variant)
  // All three unrolled, but one launch per axis (kCpmlByAxis line ends or more).
  bool by_axis;
  CpmlProf<kCpmlMaxCap> prof;
  CpmlTiles all, one[3];  // every axis at once; single axes
};

// Line ends from which the axes take a launch each, without clusters: the
// launches' ends no longer count, and the cluster launch fills the chip a
// little less evenly. 16 cells, us a step in one launch and by axis: FP32 1024 x
// 1024 x 512 (4.2 M) 1736 and 1709, FP16 1319 and 1292, 512^3 (1.6 M) 514 and
// 508, 512 x 512 x 256 (1.0 M) 288 and 292; BF16 513 x 511 x 300 (1.1 M) 308 and
// 313.
constexpr long long kCpmlByAxis = 1500000;

inline long long cpml_line_ends(const CpmlGeom &g) {
  return 2 * ((long long)g.ny * g.nz + (long long)g.nx * g.nz + (long long)g.nx * g.ny);
}

// Points of line ends (w each) from which the axes take a launch each while
// another chain of launches runs beside this one (the gradient's recompute and
// adjoint): clusters of 4 CTAs that fill an SM's registers wait for places
// together. wave_gradient, checkpoint every 20 steps, us a step in one launch and
// by axis: 16 cells 144^3 (2.5 M) 113 and 118, 170^3 (3.5 M) 194 and 184; 8 cells
// 185^3 (2.5 M) 170 and 173, 200^3 (2.9 M) 199 and 193; 10 cells 128 x 128 x 400
// (3.3 M) 165 and 167, 200^3 (3.4 M) 211 and 205; 16 cells 256^3 (7.9 M),
// checkpoint every 40, 408 and 365, 512 x 512 x 256 (21 M) 1428 and 1315.
constexpr long long kCpmlByAxisBeside = 2800000;

inline void cpml_beside(CpmlPlan &p) {
  p.by_axis |= p.axes == 7 && p.g.w * cpml_line_ends(p.g) >= kCpmlByAxisBeside;
}

// Takes the plan's form on each axis from the grid and the layer's width
// (g.npml set), and its tiles.
inline void cpml_plan_forms(CpmlPlan &p) {
  const CpmlGeom &g = p.g;
  const int n[3] = {g.nx, g.ny, g.nz};
  const long long fstep[3] = {1, g.pxu, (long long)g.ny * g.pxu};
  const long long sstep[3] = {(long long)g.nz * g.ny, (long long)g.nz * g.nx,
                              (long long)g.ny * g.nx};
  p.axes = 0;
  for (int ax = 0; ax < 3; ++ax)
    if (cpml_seg_fits(g.npml, n[ax], fstep[ax], sstep[ax])) p.axes |= 1 << ax;
  p.variant = cpml_variant(g.npml);
  p.by_axis = p.axes == 7 && cpml_line_ends(g) >= kCpmlByAxis;
  p.all = cpml_tiles(g.nx, g.ny, g.nz, g.w, -1);
  for (int ax = 0; ax < 3; ++ax) p.one[ax] = cpml_tiles(g.nx, g.ny, g.nz, g.w, ax);
}

// Launches, enqueued on st (layer.cu): one forward step's layer terms and
// shell receivers (store_d: also into D, no receivers), one adjoint step's.
// a.koff and the descriptor give the step. Where every axis is unrolled a
// step records the receivers of the step before (cpml_record_previous), and
// cpml_record_last those of the last step once the descriptor is past it.
void cpml_forward(int storage, bool store_d, const CpmlPlan &p, const CpmlPass &a, int sms,
                  cudaStream_t st);
void cpml_record_last(int storage, const CpmlPlan &p, const CpmlPass &a, int sms,
                      cudaStream_t st);
void cpml_adjoint(const CpmlPlan &p, const CpmlPass &a, cudaStream_t st);

// The unrolled line ends on tiles t of the plan (layer_lines.cuh, compiled
// once per storage type, and for the gradient); record: with the shell
// receivers of the step before.
template <class T, bool kStoreD>
void cpml_launch_lines(const CpmlPlan &p, const CpmlTiles &t, const CpmlPass &a, bool record,
                       cudaStream_t st);
void cpml_launch_adjoint_lines(const CpmlPlan &p, const CpmlTiles &t, const CpmlPass &a,
                               cudaStream_t st);

// One served shot's layer in the shot server's batched layer launches: its
// plan, fields and receivers, step bookkeeping (batch step b0 is the shot's
// step 0, as in the batched sweep), and its first block in each launch of its
// group (a 1D grid that concatenates the shots' blocks): 0-2 the unrolled
// lines of every axis at once (0) or of one, 3-5 the line walks of one.
struct CpmlBatchShot {
  CpmlPlan plan;
  void *buf[2];  // buf[0] holds the shot's step 0
  const float *c;
  const StepDesc *desc;
  const int4 *srec;  // receivers within w of a face: {x, y, z, id}
  int nsrec;
  long long b0;
  int nsteps;
  int blk_begin[6];
};

// Launch groups: every axis unrolled (by width), some axes (by width), none.
constexpr int kCpmlGroups = 2 * kCpmlVariants + 1;
inline int cpml_batch_group(const CpmlPlan &p) {
  return p.axes == 7 ? p.variant : p.axes ? kCpmlVariants + p.variant : 2 * kCpmlVariants;
}
// Blocks of a shot in launch `which` (0..5) of its group. by_axis: a launch for
// each axis although every one is unrolled (as some_axes_group).
int cpml_batch_blocks(const CpmlBatchShot &s, int which, bool by_axis);
inline int some_axes_group(int all_axes_group) { return all_axes_group + kCpmlVariants; }
// Launches of a group's step, one after another: its line passes and the shell
// receivers.
inline int cpml_batch_launches(const int blocks[6]) {
  int n = 1;
  for (int i = 0; i < 6; ++i) n += blocks[i] > 0;
  return n;
}
// One batch step's launches over a group's n shots (layer.cu); blocks: their
// totals per launch; rec_blocks: blocks per shot for its receivers.
void cpml_batch_step(int storage, int group, const CpmlBatchShot *shots, int n,
                     const int blocks[6], int rec_blocks, long long k, cudaStream_t st);
// The unrolled lines of a group of one width, every axis (ax < 0) or one.
template <class T>
void cpml_launch_batched_lines(int variant, int ax, const CpmlBatchShot *shots, int n, int blocks,
                               long long k, cudaStream_t st);

}  // namespace gbw
