// FP64 interaction coefficients and their FP32 Fourier spectra.
//
// Coefficient of a box (cell or subcell) of edges hb for observer offset r from
// its centre (Eq. 9b times the box volume, Eq. 2 / Eq. 10):
//   g(r) = (V / dl) * sigma^AB(r),  dl = chord of the box through its centre along t,
// with sigma^AB the stress of the straight segment A = -dl/2 t, B = +dl/2 t
// (Eq. 6, Eq. 7a, Eq. 7b, prefactor mu / pi, evaluated at B minus at A).
// Near offsets (|r0 - r_i| < n_near * max h, Sec. 2.3) use
//   G = (1/M) sum_{u in target subcells} sum_{v in source subcells} g_sub(Delta + u - v)
// which is evaluated grouped by the subcell difference d = u - v (multiplicity
// prod_a (m_a - |d_a|)).  The self pair (observer on the segment midpoint) is 0.
//
// The table of G over all offsets is wrapped into the zero-padded periodic grid
// (offset D -> index D mod P), transformed by an FP64 R2C FFT, and because the
// table is odd (G(-D) = -G(D)) its spectrum is purely imaginary: only Im / (Px Py Pz)
// is kept, in FP32, laid out per tile of the fused z pass.  Oddness, and the mirrors a
// field has, also halve the table and each transform (see below).
#include <math.h>

#include <algorithm>
#include <utility>
#include <vector>

#include <cuda_fp16.h>

#include "dds_fft.cuh"
#include "dds_internal.h"

namespace dds {

namespace {

struct V3 {
  double x, y, z;
};
__host__ __device__ __forceinline__ V3 v3(double x, double y, double z) { return V3{x, y, z}; }
__host__ __device__ __forceinline__ V3 operator+(V3 a, V3 b) { return v3(a.x + b.x, a.y + b.y, a.z + b.z); }
__host__ __device__ __forceinline__ V3 operator*(double s, V3 a) { return v3(s * a.x, s * a.y, s * a.z); }
__host__ __device__ __forceinline__ double dot(V3 a, V3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__host__ __device__ __forceinline__ V3 cross(V3 a, V3 b) {
  return v3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ double comp(V3 a, int i) { return i == 0 ? a.x : (i == 1 ? a.y : a.z); }

// A box (cell or subcell) as a source: half its chord along t, and mu / pi times its
// volume over the chord.
struct Box {
  double hl, f;
};

// NF fields of one line direction: what their coefficients share.  TZ: t = (0, 0, 1) exactly
// (the vertical dislocations of the paper's layers); the terms that vanish are then left
// out: 64x64x8 with 15 replica shells, two fields, table 15.4 -> 11 ms.
template <int NF, bool TZ> struct Fields {
  V3 t;
  V3 b[NF], w[NF];          // Burgers vectors, b x t
  double k1;                // 1 / (1 - nu)
  Box cell, sub;
};

// Adds weight * (box coefficient) of every field at observer offset r (from the box
// centre) to acc[f][xx, yy, zz, xy, xz, yz].
//
// Eq. 6 at the ends A, B = -+hl t, with R from the observer to the end, splits into the
// part of R across the line, which both ends share, and the one along it:
//   R = rho + L t,  R_t = R + |R| t = rho + q t,  q = L + |R|,  R_t^2 = 2 |R| q,
// so the bracket of Eq. 6 is a sum of tensors in (rho, t, b) common to both ends, each
// times a scalar of the end.  With g = 1 / (2 |R|), i = g / q = 1 / R_t^2, l = L / |R|:
//   S = i (V - k1 X) + g (1 - k1) W
//       - k1 beta [ i (1 + t t) / 2 + i^2 (2 + l) rho rho + 2 g^3 (rho t + t rho) + l g^2 t t ],
// V = sym(b x rho, t), W = sym(w, t), X = sym(w, rho), w = b x t, beta = (b x rho) . t;
// only the differences of the five scalars between B and A remain per field.  Two
// reciprocal square roots and one division serve all fields of the direction: FP64
// units are scarce (1/64 of the FP32 rate), and this is about a tenth of the operations
// of evaluating Eq. 6 per end and field (GaN layer, five fields: tables 234 -> 12.4 ms
// with the offsets the symmetries leave; 15 replica shells on 64x64x8, two fields: 374 ->
// 15.4 ms).  The observer at the centre gives 0.
template <int NF, bool TZ>
__device__ __forceinline__ void box_add(const Fields<NF, TZ> &F, V3 r, const Box &box, double weight, double (&acc)[NF][6]) {
  if (r.x == 0.0 && r.y == 0.0 && r.z == 0.0) return;
  const double rt = TZ ? r.z : dot(r, F.t);
  V3 rho = TZ ? v3(-r.x, -r.y, 0.0) : v3(rt * F.t.x - r.x, rt * F.t.y - r.y, rt * F.t.z - r.z);
  const double rho2 = TZ ? r.x * r.x + r.y * r.y : dot(rho, rho);
  double LA = -box.hl - rt, LB = box.hl - rt;
  const double RA2 = LA * LA + rho2, RB2 = LB * LB + rho2;
  const double rsA = rsqrt(RA2), rsB = rsqrt(RB2);
  double lA = LA * rsA, lB = LB * rsB;
  if (lA + lB < 0.0) {     // observer ahead of the segment: R from the end to the observer
    LA = -LA;
    LB = -LB;
    lA = -lA;
    lB = -lB;
    rho = v3(-rho.x, -rho.y, TZ ? 0.0 : -rho.z);
  }
  // q = L + |R|; beside the segment (L < 0) the same as rho^2 / (|R| - L)
  double qA = fabs(LA) + RA2 * rsA, qB = fabs(LB) + RB2 * rsB;
  if (LA < 0.0) qA = rho2 / qA;
  if (LB < 0.0) qB = rho2 / qB;
  const double iq = 1.0 / (qA * qB);
  const double gA = 0.5 * rsA, gB = 0.5 * rsB;
  const double iA = gA * (iq * qB), iB = gB * (iq * qA);
  const double ga2 = gA * gA, gb2 = gB * gB;
  const double s = weight * box.f;
  const double d0 = s * (iB - iA), d1 = s * (gB - gA);
  const double d2 = s * (iB * iB * (2.0 + lB) - iA * iA * (2.0 + lA));
  const double d3 = 2.0 * s * (gb2 * gB - ga2 * gA);
  const double d4 = s * (lB * gb2 - lA * ga2);
  const double h0 = 0.5 * d0, dt = h0 + d4;
  constexpr int IA[6] = {0, 1, 2, 0, 0, 1}, IC[6] = {0, 1, 2, 1, 2, 2};
  double T[6];             // the tensor of the beta term, shared by the fields
  if constexpr (TZ) {
    const double px = d2 * rho.x, py = d2 * rho.y;
    T[0] = fma(rho.x, px, h0);
    T[1] = fma(rho.y, py, h0);
    T[2] = h0 + dt;
    T[3] = rho.x * py;
    T[4] = rho.x * d3;
    T[5] = rho.y * d3;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const V3 b = F.b[f], w = F.w[f];                     // w = (b_y, -b_x, 0)
      const double kb = F.k1 * (w.x * rho.x + w.y * rho.y);
      const double cw = 0.5 * d1 * (1.0 - F.k1), hz = h0 * b.z;
      const double yx = -h0 * F.k1 * rho.x, yy = -h0 * F.k1 * rho.y;
      acc[f][0] += kb * T[0] + 2.0 * (w.x * yx);
      acc[f][1] += kb * T[1] + 2.0 * (w.y * yy);
      acc[f][2] += kb * T[2] + 2.0 * (h0 * (b.x * rho.y - b.y * rho.x));
      acc[f][3] += kb * T[3] + (w.x * yy + w.y * yx);
      acc[f][4] += kb * T[4] + (cw * w.x - hz * rho.y);
      acc[f][5] += kb * T[5] + (cw * w.y + hz * rho.x);
    }
    return;
  }
  const V3 p = d2 * rho + d3 * F.t, z = d3 * rho + dt * F.t;     // rho (d2 rho + d3 t) + t (d3 rho + dt t)
#pragma unroll
  for (int c = 0; c < 6; ++c)
    T[c] = (IA[c] == IC[c] ? h0 : 0.0) + comp(rho, IA[c]) * comp(p, IC[c]) + comp(F.t, IA[c]) * comp(z, IC[c]);
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    const V3 w = F.w[f];
    const double kb = F.k1 * dot(w, rho);                // -k1 beta
    // d0 (V - k1 X) + d1 (1 - k1) W = sym(t, d0 v + d1 (1 - k1) w) - sym(w, d0 k1 rho), halves folded in
    const V3 x = h0 * cross(F.b[f], rho) + (0.5 * d1 * (1.0 - F.k1)) * w;
    const V3 y = (-h0 * F.k1) * rho;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const int a = IA[c], e = IC[c];
      double v;
      if (a == e) v = 2.0 * (comp(F.t, a) * comp(x, a) + comp(w, a) * comp(y, a));
      else v = comp(F.t, a) * comp(x, e) + comp(F.t, e) * comp(x, a) + comp(w, a) * comp(y, e) + comp(w, e) * comp(y, a);
      acc[f][c] += kb * T[c] + v;
    }
  }
}

__device__ __forceinline__ V3 offset_pos(const CoefGeom &g, int i, int j, int k) {
  return v3((double)i * g.h[0], (double)j * g.h[1], (double)k * g.h[2]);
}

__device__ __forceinline__ int near_terms(const CoefGeom &g) {
  return (2 * g.m[0] - 1) * (2 * g.m[1] - 1) * (2 * g.m[2] - 1);
}

// Near-field coefficient: adds the term of subcell difference index q of the (2m-1)^3
// lattice, times its multiplicity over the number of subcells.
template <int NF, bool TZ>
__device__ __forceinline__ void near_add(const CoefGeom &g, const Fields<NF, TZ> &F, V3 base, int q, double weight,
                                         double (&acc)[NF][6]) {
  const int Dx = 2 * g.m[0] - 1, Dy = 2 * g.m[1] - 1;
  const int dx = q % Dx - (g.m[0] - 1);
  const int dy = (q / Dx) % Dy - (g.m[1] - 1);
  const int dz = q / (Dx * Dy) - (g.m[2] - 1);
  const double mult = (double)((g.m[0] - abs(dx)) * (g.m[1] - abs(dy)) * (g.m[2] - abs(dz)));
  const V3 r = base + v3(dx * g.hs[0], dy * g.hs[1], dz * g.hs[2]);
  box_add(F, r, F.sub, weight * mult / (double)(g.m[0] * g.m[1] * g.m[2]), acc);
}

// Near field: |(i dx, j dy, k dz)|^2 < rn2, as ((x*x + y*y) + z*z) in round-to-nearest
// double without contraction (the same decision as the plain IEEE expression).
// Cells beyond near_lim along an axis are far without the FP64 test.
__device__ __forceinline__ bool near_dev(const CoefGeom &g, int i, int j, int k) {
  if (abs(i) > g.near_lim[0] || abs(j) > g.near_lim[1] || abs(k) > g.near_lim[2]) return false;
  const double x = __dmul_rn((double)i, g.h[0]), y = __dmul_rn((double)j, g.h[1]), z = __dmul_rn((double)k, g.h[2]);
  return __dadd_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)), __dmul_rn(z, z)) < g.rn2;
}

// Minimal image of offset i for period n, in (-n/2, n/2]; at the tie n/2 (n even) also
// -n/2, each with weight 1/2.  Returns the number of images (1 or 2).
__device__ __forceinline__ int min_images(int i, int n, int r[2], double w[2]) {
  int m = i % n;
  if (m < 0) m += n;
  w[0] = 1.0;
  if (2 * m < n) { r[0] = m; return 1; }
  if (2 * m > n) { r[0] = m - n; return 1; }
  r[0] = m;
  r[1] = -m;
  w[0] = w[1] = 0.5;
  return 2;
}

// Share `lane` of S of the coefficient at cell offset (i, j, k): one segment, or near the
// target the mean over target subcells of the sum over source subcells; with periodic
// boundary conditions (Sec. 4, Eq. 13) the sum over the replicas of the source cell,
// r_i + (k Lx, l Ly, 0), |k|, |l| <= n_shells, around the in-system offset or its minimal
// images (ties averaged: odd and periodic).  The lanes take the images in turn, and the
// subcell differences of every near image together (one near image is up to a few
// hundred terms), so they finish at about the same time.  Every lane of a warp calls
// this with the same number of images; `lanes`: the warp's mask of this offset's lanes.
template <int S, int NF, bool TZ>
__device__ __forceinline__ void coef_share(const CoefGeom &g, const Fields<NF, TZ> &F, int i, int j, int k, int lane,
                                           unsigned lanes, double (&acc)[NF][6]) {
  const int n = g.n_shells, side = 2 * n + 1, images = side * side;
  int rx[2] = {i, 0}, ry[2] = {j, 0};
  double wx[2] = {1.0, 0.0}, wy[2] = {1.0, 0.0};
  int nxr = 1, nyr = 1;
  if (n > 0 && g.periodic) {
    nxr = min_images(i, g.nx, rx, wx);
    nyr = min_images(j, g.ny, ry, wy);
  }
  const int terms = near_terms(g);
  for (int a = 0; a < nxr; ++a)
    for (int b = 0; b < nyr; ++b) {
      const double wt = wx[a] * wy[b];
      for (int m0 = 0; m0 < images; m0 += S) {
        const int m = m0 + lane;
        const int ii = rx[a] + (m / side - n) * g.nx, jj = ry[b] + (m % side - n) * g.ny;
        const bool near = m < images && near_dev(g, ii, jj, k);
        if (m < images && !near) box_add(F, offset_pos(g, ii, jj, k), F.cell, wt, acc);
        unsigned mask = S > 1 ? __ballot_sync(lanes, near) & lanes : (near ? 1u : 0u);
        while (mask) {                        // this offset's near images, all its lanes on each
          const int bit = __ffs(mask) - 1;
          mask &= mask - 1;
          const int q = m0 + (S > 1 ? bit % S : 0);
          const V3 base = offset_pos(g, rx[a] + (q / side - n) * g.nx, ry[b] + (q % side - n) * g.ny, k);
          for (int d = lane; d < terms; d += S) near_add(g, F, base, d, wt, acc);
        }
      }
    }
}

// ---- coefficients at listed offsets (parity queries) ------------------------
template <bool TZ>
__global__ void k_table_at(CoefGeom g, Fields<1, TZ> F, long n, const int *ijk, double *out) {
  const long q = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (q >= n) return;
  double acc[1][6] = {{0, 0, 0, 0, 0, 0}};
  coef_share<1>(g, F, ijk[3 * q], ijk[3 * q + 1], ijk[3 * q + 2], 0, 0u, acc);
#pragma unroll
  for (int c = 0; c < 6; ++c) out[6 * q + c] = acc[0][c];
}

// ---- coefficient table of the fields of one line direction --------------------
// Only offsets no symmetry gives: k >= 0 (the table is odd, G(-D) = -G(D)); i >= 0 when
// every field has the x mirror, j >= 0 when every field has the y mirror.  Row r of an
// axis with n cells holds offset r, or r - (2n - 1) from r = n on.
struct Tab {
  int nx, ny, nz;           // grid
  int mx, my;               // mirrors used
  int rx, ry;               // rows stored along x and y
};
__host__ __device__ __forceinline__ long tab_size(const Tab &T) { return (long)T.nz * T.ry * T.rx; }

// One segment per offset (near offsets are overwritten by k_table_near).
template <int NF, bool TZ>
__global__ void __launch_bounds__(256) k_table_far(CoefGeom g, Fields<NF, TZ> F, Tab T, double *tab) {
  const long N = tab_size(T), idx = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (idx >= N) return;
  const int ir = (int)(idx % T.rx), jr = (int)((idx / T.rx) % T.ry), k = (int)(idx / ((long)T.rx * T.ry));
  const int i = ir < T.nx ? ir : ir - (2 * T.nx - 1), j = jr < T.ny ? jr : jr - (2 * T.ny - 1);
  double acc[NF][6] = {};
  box_add(F, offset_pos(g, i, j, k), F.cell, 1.0, acc);
#pragma unroll
  for (int f = 0; f < NF; ++f)
#pragma unroll
    for (int c = 0; c < 6; ++c) tab[(f * 6 + c) * N + idx] = acc[f][c];
}

// Replica sums: S lanes per offset.
template <int NF, bool TZ, int S>
__global__ void __launch_bounds__(256) k_table_pbc(CoefGeom g, Fields<NF, TZ> F, Tab T, double *tab) {
  const long N = tab_size(T), idx = (blockIdx.x * (long)blockDim.x + threadIdx.x) / S;
  if (idx >= N) return;                       // all lanes of an offset together
  const int lane = threadIdx.x % S;
  const unsigned lanes = S == 32 ? 0xffffffffu : ((1u << S) - 1u) << ((threadIdx.x & 31) / S * S);
  const int ir = (int)(idx % T.rx), jr = (int)((idx / T.rx) % T.ry), k = (int)(idx / ((long)T.rx * T.ry));
  const int i = ir < T.nx ? ir : ir - (2 * T.nx - 1), j = jr < T.ny ? jr : jr - (2 * T.ny - 1);
  double acc[NF][6] = {};
  coef_share<S>(g, F, i, j, k, lane, lanes, acc);
#pragma unroll
  for (int f = 0; f < NF; ++f)
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      double v = acc[f][c];
      for (int o = S / 2; o > 0; o >>= 1) v += __shfl_xor_sync(lanes, v, o);
      if (lane == 0) tab[(f * 6 + c) * N + idx] = v;
    }
}

// One block per near offset (rows of the table): reduce the subcell-difference lattice.
template <int NF, bool TZ>
__global__ void __launch_bounds__(128) k_table_near(CoefGeom g, Fields<NF, TZ> F, Tab T, const int *ijk, double *tab) {
  const int q = blockIdx.x;
  const int i = ijk[3 * q], j = ijk[3 * q + 1], k = ijk[3 * q + 2];
  const V3 base = offset_pos(g, i, j, k);
  double acc[NF][6] = {};
  const int terms = near_terms(g);
  for (int d = threadIdx.x; d < terms; d += blockDim.x) near_add(g, F, base, d, 1.0, acc);
  __shared__ double red[4][NF * 6];
#pragma unroll
  for (int f = 0; f < NF; ++f)
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      double v = acc[f][c];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
      if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][f * 6 + c] = v;
    }
  __syncthreads();
  if (threadIdx.x < NF * 6) {
    double v = 0.0;
    for (int w = 0; w < 4; ++w) v += red[w][threadIdx.x];
    const int ir = i >= 0 ? i : i + 2 * T.nx - 1, jr = j >= 0 ? j : j + 2 * T.ny - 1;
    tab[threadIdx.x * tab_size(T) + ((long)k * T.ry + jr) * T.rx + ir] = v;
  }
}

// ---- FP64 FFT of the table ---------------------------------------------------
// The table of (component, field) wrapped into the padded grid is real and odd, so its
// transform is imaginary, and only half of each transform is work:
//   x: real-to-complex lines of 2M points, layers k >= 0 only;
//   y: layers k >= 0 only.  With the x mirror the x spectra are real or imaginary (one
//      number per bin): two columns form one complex column, rows ky <= py/2 remain, and
//      an x-even and an x-odd component share one real line (their sum: its spectrum's
//      real part belongs to the even one, the imaginary part to the odd one);
//   z: h(-z) = -conj h(z) gives the layers k < 0; two columns h1 + i h2 are transformed
//      as one, whose spectrum is i S1 - S2.
// FP64 arithmetic bounds every pass.  Full transforms of every padded value took 7.3 ms
// per component of the GaN layer (256x256x128, padded 512x512x256: 2.3 x, 3.4 y, 1.6 z);
// with the symmetries 2.0 ms (0.65 x, 0.93 y, 0.46 z).

// Components of one launch: line set s transforms component ce[s], plus the x-odd one
// co[s] when >= 0, into the spectra of slots se[s] and so[s]; sx, sy: mirror parities.
struct Comps {
  int sets, slots;
  int ce[6], co[6], se[6], so[6];
  int sx[6], sy[6];         // by component
  int comp_of[6];           // by slot
  int off;                  // first component of the field in the table (6 f)
};

// x: W lines (rows of the table) per block.  Without the x mirror: out[slot][k][jr][M + 1]
// complex; with it one number per bin: the real part (x-even component), or the imaginary
// part (x-odd).
template <int M>
__global__ void __launch_bounds__(128) k_x_lines_d(Tab T, Comps C, const double *tab, double *out, const double2 *tw) {
  constexpr int W = 4, LD = W + 1, NT = 128;
  extern __shared__ double2 sm_d[];
  double2 *buf = sm_d;
  const long lines = (long)T.nz * T.ry, l0 = (long)blockIdx.x * W;
  const int tid = threadIdx.x, set = blockIdx.y;
  const int ce = C.ce[set], co = C.co[set];
  const long N = tab_size(T);
  const double *te = tab + (C.off + ce) * N, *to = co >= 0 ? tab + (C.off + co) * N : nullptr;
  const double pe = C.sx[ce], po = co >= 0 ? C.sx[co] : 0.0;
  auto value = [&](long line, int n) {        // sample n of the wrapped line
    const int i = n < T.nx ? n : n - 2 * M;
    if (i <= -T.nx) return 0.0;
    const long row = line * T.rx;
    if (!T.mx) return __ldg(te + row + (i >= 0 ? i : i + 2 * T.nx - 1));
    const int a = abs(i);
    double v = __ldg(te + row + a);
    if (i < 0) v *= pe;
    if (to != nullptr) {
      const double u = __ldg(to + row + a);
      v += i < 0 ? po * u : u;
    }
    return v;
  };
  for (int e = tid; e < W * M; e += NT) {
    const int w = e / M, n = e % M;
    double2 z = make_double2(0.0, 0.0);
    if (l0 + w < lines) z = make_double2(value(l0 + w, 2 * n), value(l0 + w, 2 * n + 1));
    buf[n * LD + w] = z;
  }
  __syncthreads();
  fft_tile<M, W, LD, NT>(buf, tw + tw_offset(M), tid);
  const double2 *tw2 = tw + tw_offset(2 * M);
  for (int e = tid; e < W * (M + 1); e += NT) {
    const int w = e / (M + 1), k = e % (M + 1);
    if (l0 + w >= lines) continue;
    const double2 a = buf[(k % M) * LD + w];
    const double2 c = buf[((M - k) % M) * LD + w];
    // 2 E = Z[k] + conj Z[M-k],  2 O = (Z[k] - conj Z[M-k]) / i,  X = E + W^k O
    const double2 E = make_double2(a.x + c.x, a.y - c.y);
    const double2 O = make_double2(a.y + c.y, c.x - a.x);
    const double2 wk = (k < M) ? tw2[k] : make_double2(-1.0, 0.0);
    const long o = (l0 + w) * (M + 1) + k, S = lines * (M + 1);
    if (!T.mx) {
      reinterpret_cast<double2 *>(out)[C.se[set] * S + o] =
          make_double2(0.5 * (E.x + wk.x * O.x - wk.y * O.y), 0.5 * (E.y + wk.x * O.y + wk.y * O.x));
    } else {
      if (pe > 0.0 || to != nullptr) out[C.se[set] * S + o] = 0.5 * (E.x + wk.x * O.x - wk.y * O.y);
      else out[C.se[set] * S + o] = 0.5 * (E.y + wk.x * O.y + wk.y * O.x);
      if (to != nullptr) out[C.so[set] * S + o] = 0.5 * (E.y + wk.x * O.y + wk.y * O.x);
    }
  }
}

// y: padded row iy of layer k is table row j = iy, or iy - py (zero in the gap).  Without
// the x mirror W complex columns per tile, out[slot][k][ky < py][M + 1]; with it (PAIR) W
// pairs of columns, out[slot][k][ky <= py/2][M + 1], multiplied by i for x-odd components.
template <int P, int W, bool PAIR>
__global__ void __launch_bounds__(256) k_y_cols_d(Tab T, Comps C, int M, const double *in, double2 *out, const double2 *tw) {
  constexpr int NT = 256;
  extern __shared__ double2 sm_d[];
  double2 *buf = sm_d;
  const int cols = M + 1, tiles = PAIR ? (cols + 2 * W - 1) / (2 * W) : (cols + W - 1) / W;
  const int k = blockIdx.x / tiles, c0 = (blockIdx.x % tiles) * (PAIR ? 2 * W : W), slot = blockIdx.y;
  const int comp = C.comp_of[slot];
  const int tid = threadIdx.x;
  const long base = ((long)slot * T.nz + k) * T.ry;
  for (int e = tid; e < P * W; e += NT) {
    const int n = e / W, w = e % W;
    const int j = n < T.ny ? n : n - P;
    double2 v = make_double2(0.0, 0.0);
    if (j > -T.ny) {
      const int jr = j >= 0 ? j : (T.my ? -j : j + 2 * T.ny - 1);
      const double sg = j < 0 && T.my ? (double)C.sy[comp] : 1.0;
      const long row = (base + jr) * cols;
      if (PAIR) {
        const int c = c0 + 2 * w;
        if (c < cols) v.x = sg * __ldg(in + row + c);
        if (c + 1 < cols) v.y = sg * __ldg(in + row + c + 1);
      } else if (c0 + w < cols) {
        v = __ldg(reinterpret_cast<const double2 *>(in) + row + c0 + w);
        v.x *= sg;
        v.y *= sg;
      }
    }
    buf[n * W + w] = v;
  }
  __syncthreads();
  fft_tile<P, W, W, NT>(buf, tw + tw_offset(P), tid);
  if (!PAIR) {
    double2 *dst = out + ((long)slot * T.nz + k) * P * cols;
    for (int e = tid; e < P * W; e += NT) {
      const int n = e / W, w = e % W;
      if (c0 + w < cols) dst[(long)n * cols + c0 + w] = buf[n * W + w];
    }
  } else {
    const bool odd = C.sx[comp] < 0;
    double2 *dst = out + ((long)slot * T.nz + k) * (P / 2 + 1) * cols;
    for (int e = tid; e < (P / 2 + 1) * 2 * W; e += NT) {
      const int n = e / (2 * W), q = e % (2 * W), w = q / 2;
      if (c0 + q >= cols) continue;
      const double2 a = buf[n * W + w], b = buf[((P - n) % P) * W + w];
      // columns f1 + i f2, both real: F1 = (C[k] + conj C[-k]) / 2, F2 = (C[k] - conj C[-k]) / 2i
      double2 v = (q & 1) ? make_double2(0.5 * (a.y + b.y), 0.5 * (b.x - a.x))
                          : make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
      if (odd) v = make_double2(-v.y, v.x);
      dst[(long)n * cols + c0 + q] = v;
    }
  }
}

// z: pairs of adjacent columns of in[slot][k < nz][cols]; out[slot][kz < P][cols], the
// imaginary part of the transform.
template <int P, int W>
__global__ void __launch_bounds__(256) k_z_cols_d(int nz, long cols, const double2 *in, double *out, const double2 *tw) {
  constexpr int NT = 256;
  extern __shared__ double2 sm_d[];
  double2 *buf = sm_d;
  const long c0 = (long)blockIdx.x * 2 * W;
  const int slot = blockIdx.y, tid = threadIdx.x;
  in += (long)slot * nz * cols;
  out += (long)slot * P * cols;
  for (int e = tid; e < (P / 2 + 1) * W; e += NT) {
    const int n = e / W, w = e % W;
    const long c = c0 + 2 * w;
    double2 a = make_double2(0.0, 0.0), b = a;
    if (n < nz && c < cols) a = __ldg(in + n * cols + c);
    if (n < nz && c + 1 < cols) b = __ldg(in + n * cols + c + 1);
    buf[n * W + w] = make_double2(a.x - b.y, a.y + b.x);                       // h1 + i h2
    if (n > 0 && n < P / 2) buf[(P - n) * W + w] = make_double2(-a.x - b.y, a.y - b.x);   // -conj h1 - i conj h2
  }
  __syncthreads();
  fft_tile<P, W, W, NT>(buf, tw + tw_offset(P), tid);
  for (int e = tid; e < P * 2 * W; e += NT) {
    const int n = e / (2 * W), q = e % (2 * W);
    if (c0 + q >= cols) continue;
    const double2 v = buf[n * W + q / 2];
    out[n * cols + c0 + q] = (q & 1) ? -v.x : v.y;
  }
}

// The imaginary part at (kx, ky, kz) of out[kz][ky][kx]; fold != 0: only ky <= py/2 are
// held, and g(kx, -ky, -kz) = fold * g(kx, ky, kz) gives the others.
__device__ __forceinline__ double spec_at(const double *spec, int M, int py, int pz, int fold, int kx, int ky, int kz) {
  double s = 1.0;
  int rows = py;
  if (fold != 0) {
    rows = py / 2 + 1;
    if (ky > py / 2) {
      ky = py - ky;
      kz = kz == 0 ? 0 : pz - kz;
      s = fold;
    }
  }
  return s * spec[((long)kz * rows + ky) * (M + 1) + kx];
}

// Imaginary part of the spectrum of component c of field e, scaled, into the layout
// the fused z pass reads:
//   shared-memory variant (zg = 0): kspec[tile][6][fe][pz][wz], tiles of wz columns;
//   register variant (zg = G > 0):  kspec[warp tile][6][fe][lane][E], E = pz / G, warp
//     tiles of 32/G columns, lane g * (32/G) + w holding kz = k1 + E bitrev_G(g), k1 < E;
//   three-stage variant (k_extract_four): see there.
// Main tiles cover (ky, kx < M) row by row; the Nyquist tiles (kx = M) follow.
__device__ __forceinline__ void store_val(float *p, double v) { *p = (float)v; }
__device__ __forceinline__ void store_val(__half *p, double v) { *p = __float2half_rn((float)v); }

// Largest |Im| of one spectrum (for the FP16 scale); bit patterns of non-negative
// doubles order like unsigned integers.
__global__ void k_absmax_imag(const double *spec, long n, unsigned long long *out) {
  double m = 0.0;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
    m = fmax(m, fabs(spec[i]));
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

// FP16 scale of (component c, field e): the largest |value| after the FFT scaling.
__global__ void k_store_scale(const unsigned long long *amax, double scale, float *kscale, int idx) {
  const double m = __longlong_as_double((long long)*amax) * scale;
  kscale[idx] = m > 0.0 ? (float)m : 1.0f;
}

template <typename OT>
__global__ void k_extract(const double *spec, int fold, int M, int py, int pz, int wz, int zg, int fe, int e, int c,
                          double scale, const unsigned long long *amax, OT *kspec) {
  const int cw = zg > 0 ? 32 / zg : wz;                  // columns per tile
  const int E = zg > 0 ? pz / zg : 0;                     // registers per lane
  const long per_tile = zg > 0 ? 32L * E : (long)pz * wz;
  const long tiles_main = (long)py * (M / cw);
  const long tiles = tiles_main + py / cw;
  const long idx = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (idx >= tiles * per_tile) return;
  const long tau = idx / per_tile;
  const int r = (int)(idx % per_tile);
  int kz, w;
  const long dst = ((tau * 6 + c) * fe + e) * per_tile + r;
  if (zg > 0) {
    const int lane = r / E, k1 = r % E, g = lane / cw;
    const int gb = zg == 4 ? (((g & 1) << 1) | (g >> 1))
                 : zg == 8 ? (((g & 1) << 2) | (g & 2) | (g >> 2)) : g;
    w = lane % cw;
    kz = k1 + E * gb;
  } else {
    kz = r / wz;
    w = r % wz;
  }
  int kx, ky;
  if (tau < tiles_main) {
    ky = (int)(tau / (M / cw));
    kx = (int)(tau % (M / cw)) * cw + w;
  } else {
    ky = (int)(tau - tiles_main) * cw + w;
    kx = M;
  }
  double v = spec_at(spec, M, py, pz, fold, kx, ky, kz) * scale;
  if (amax != nullptr) {                 // FP16 storage: values relative to the largest
    const double m = __longlong_as_double((long long)*amax) * scale;
    if (m > 0.0) v /= m;
  }
  store_val(&kspec[dst], v);
}

// Imaginary part of the spectrum of component c of field e, scaled, into the layout
// the three-stage z pass reads (pz = R1 R2, tiles of W = wz columns): per stored tile s
// and component c, 16-byte chunks [j][thread t = k1 W + w], the value of
// (e, kz = k1 + R1 k2) at position (R2 e + k2) % V of chunk j = (R2 e + k2) / V, V values
// per chunk.  Stored tiles: the main tiles (ky, kx tile) row by row -- all of them, or
// those with ky <= py/2 when every field has the x-mirror parity (ZSym::xall) -- then
// the Nyquist tiles (kx = M).
template <typename OT>
__global__ void k_extract_four(const double *spec, int fold, Shape sh, int e, int c, double scale,
                               const unsigned long long *amax, OT *kspec) {
  constexpr int V = 16 / (int)sizeof(OT);
  const int W = sh.wz, R2 = zfour_r2(sh.pz), R1 = sh.pz / R2, M = sh.M, py = sh.py, fe = sh.fe;
  // 32-bit indices: at most 1024 x 513 x 512 values
  const unsigned per_tile = sh.pz * W, idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (unsigned)zf_stored_tiles(sh) * per_tile) return;
  const int s = idx / per_tile, r = idx - s * per_tile, t = r / R2, k2 = r % R2, k1 = t / W, w = t % W, q = R2 * e + k2;
  const int ktiles = M / W;
  const int main_tiles = (sh.zs.xall ? py / 2 + 1 : py) * ktiles;
  int kx, ky;
  if (s < main_tiles) {
    ky = s / ktiles;
    kx = (s - ky * ktiles) * W + w;
  } else {
    ky = (s - main_tiles) * W + w;
    kx = M;
  }
  double v = spec_at(spec, M, py, sh.pz, fold, kx, ky, k1 + R1 * k2) * scale;
  if (amax != nullptr) {                 // FP16 storage: values relative to the largest
    const double m = __longlong_as_double((long long)*amax) * scale;
    if (m > 0.0) v /= m;
  }
  const size_t dst = ((size_t)s * 6 + c) * fe * per_tile + ((size_t)(q / V) * (R1 * W) + t) * V + q % V;
  store_val(&kspec[dst], v);
}

template <typename K>
cudaError_t big_smem(K kernel, size_t smem) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

template <int M>
cudaError_t x_lines(const Tab &T, const Comps &C, const double *tab, double *out, const double2 *tw, cudaStream_t s) {
  const size_t smem = sizeof(double2) * M * 5;
  cudaError_t err = big_smem(k_x_lines_d<M>, smem);
  if (err != cudaSuccess) return err;
  const dim3 grid((unsigned)(((long)T.nz * T.ry + 3) / 4), C.sets);
  k_x_lines_d<M><<<grid, 128, smem, s>>>(T, C, tab, out, tw);
  return cudaGetLastError();
}

template <int P>
cudaError_t y_cols(const Tab &T, const Comps &C, int M, const double *in, double2 *out, const double2 *tw, cudaStream_t s) {
  constexpr int W = P >= 512 ? 4 : 8;
  const size_t smem = sizeof(double2) * P * W;
  cudaError_t err = T.mx ? big_smem(k_y_cols_d<P, W, true>, smem) : big_smem(k_y_cols_d<P, W, false>, smem);
  if (err != cudaSuccess) return err;
  const int per = T.mx ? 2 * W : W;
  const dim3 grid((unsigned)((long)T.nz * ((M + per) / per)), C.slots);      // ceil((M + 1) / per) tiles per layer
  if (T.mx) k_y_cols_d<P, W, true><<<grid, 256, smem, s>>>(T, C, M, in, out, tw);
  else k_y_cols_d<P, W, false><<<grid, 256, smem, s>>>(T, C, M, in, out, tw);
  return cudaGetLastError();
}

template <int P>
cudaError_t z_cols(int nz, long cols, int slots, const double2 *in, double *out, const double2 *tw, cudaStream_t s) {
  constexpr int W = P >= 512 ? 4 : 8;
  const size_t smem = sizeof(double2) * P * W;
  cudaError_t err = big_smem(k_z_cols_d<P, W>, smem);
  if (err != cudaSuccess) return err;
  const dim3 grid((unsigned)((cols + 2 * W - 1) / (2 * W)), slots);
  k_z_cols_d<P, W><<<grid, 256, smem, s>>>(nz, cols, in, out, tw);
  return cudaGetLastError();
}

cudaError_t x_dispatch(int M, const Tab &T, const Comps &C, const double *tab, double *out, const double2 *tw,
                       cudaStream_t s) {
  switch (M) {
    case 16: return x_lines<16>(T, C, tab, out, tw, s);
    case 32: return x_lines<32>(T, C, tab, out, tw, s);
    case 64: return x_lines<64>(T, C, tab, out, tw, s);
    case 128: return x_lines<128>(T, C, tab, out, tw, s);
    case 256: return x_lines<256>(T, C, tab, out, tw, s);
    case 512: return x_lines<512>(T, C, tab, out, tw, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t y_dispatch(int P, const Tab &T, const Comps &C, int M, const double *in, double2 *out, const double2 *tw,
                       cudaStream_t s) {
  switch (P) {
    case 32: return y_cols<32>(T, C, M, in, out, tw, s);
    case 64: return y_cols<64>(T, C, M, in, out, tw, s);
    case 128: return y_cols<128>(T, C, M, in, out, tw, s);
    case 256: return y_cols<256>(T, C, M, in, out, tw, s);
    case 512: return y_cols<512>(T, C, M, in, out, tw, s);
    case 1024: return y_cols<1024>(T, C, M, in, out, tw, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t z_dispatch(int P, int nz, long cols, int slots, const double2 *in, double *out, const double2 *tw,
                       cudaStream_t s) {
  switch (P) {
    case 16: return z_cols<16>(nz, cols, slots, in, out, tw, s);
    case 32: return z_cols<32>(nz, cols, slots, in, out, tw, s);
    case 64: return z_cols<64>(nz, cols, slots, in, out, tw, s);
    case 128: return z_cols<128>(nz, cols, slots, in, out, tw, s);
    case 256: return z_cols<256>(nz, cols, slots, in, out, tw, s);
    case 512: return z_cols<512>(nz, cols, slots, in, out, tw, s);
    default: return cudaErrorInvalidValue;
  }
}

CoefGeom coef_geom(const dds_ctx *ctx) {
  CoefGeom g;
  for (int a = 0; a < 3; ++a) g.h[a] = ctx->h[a];
  subcell_counts(ctx->h, g.m);
  for (int a = 0; a < 3; ++a) g.hs[a] = ctx->h[a] / (double)g.m[a];
  g.mu = ctx->mu;
  g.nu = ctx->nu;
  const double hmax = fmax(ctx->h[0], fmax(ctx->h[1], ctx->h[2]));
  const double rn = ctx->n_near * hmax;
  g.rn2 = rn * rn;
  // |i| h < rn in exact arithmetic, with a cell to spare for rounding
  for (int a = 0; a < 3; ++a) g.near_lim[a] = (int)fmin(1e9, ceil(rn / ctx->h[a]) + 1.0);
  g.nx = ctx->nx;
  g.ny = ctx->ny;
  g.n_shells = ctx->n_shells;
  g.periodic = ctx->pbc_periodic ? 1 : 0;
  return g;
}

}  // namespace


namespace {

Box make_box(const double hb[3], const double t[3], double mu) {
  const double dl = chord_length(hb, t);
  return Box{0.5 * dl, mu * 0.31830988618379067154 * (hb[0] * hb[1] * hb[2]) / dl};
}

// Fields of one line direction (nf <= NF of them; the rest repeat the last).
template <int NF, bool TZ>
Fields<NF, TZ> make_fields(const CoefGeom &g, const double t[3], const double *b) {
  Fields<NF, TZ> F;
  F.t = v3(t[0], t[1], t[2]);
  for (int f = 0; f < NF; ++f) {
    const double *q = b + 3 * f;
    F.b[f] = v3(q[0], q[1], q[2]);
    F.w[f] = cross(F.b[f], F.t);
  }
  F.k1 = 1.0 / (1.0 - g.nu);
  F.cell = make_box(g.h, t, g.mu);
  F.sub = make_box(g.hs, t, g.mu);
  return F;
}

// Table of NF fields (near: the stored near offsets, open boundary only).
template <int NF, bool TZ>
cudaError_t fill_table_dir(const CoefGeom &g, const double t[3], const double *b, const Tab &T, int n_near,
                       const int *d_near, double *tab, cudaStream_t s) {
  const Fields<NF, TZ> F = make_fields<NF, TZ>(g, t, b);
  const long N = tab_size(T);
  if (g.n_shells > 2)                         // 49 images and more: a warp per offset
    k_table_pbc<NF, TZ, 32><<<(unsigned)((N * 32 + 255) / 256), 256, 0, s>>>(g, F, T, tab);
  else if (g.n_shells > 0)                    // 9 or 25 images
    k_table_pbc<NF, TZ, 8><<<(unsigned)((N * 8 + 255) / 256), 256, 0, s>>>(g, F, T, tab);
  else
    k_table_far<NF, TZ><<<(unsigned)((N + 255) / 256), 256, 0, s>>>(g, F, T, tab);
  cudaError_t err = cudaGetLastError();
  if (err == cudaSuccess && n_near > 0) {
    k_table_near<NF, TZ><<<n_near, 128, 0, s>>>(g, F, T, d_near, tab);
    err = cudaGetLastError();
  }
  return err;
}

bool vertical(const double t[3]) { return t[0] == 0.0 && t[1] == 0.0 && t[2] == 1.0; }

template <int NF>
cudaError_t fill_table(const CoefGeom &g, const double t[3], const double *b, const Tab &T, int n_near,
                       const int *d_near, double *tab, cudaStream_t s) {
  return vertical(t) ? fill_table_dir<NF, true>(g, t, b, T, n_near, d_near, tab, s)
                     : fill_table_dir<NF, false>(g, t, b, T, n_near, d_near, tab, s);
}

// Consecutive effective fields whose tables are made together; components per launch.
struct Batch {
  int e0, n, mx, my, slots;
};

}  // namespace

// -------------------------------------------------------------------------------
cudaError_t launch_table_at(const CoefGeom &g, const double t[3], const double b[3], long n,
                            const int *d_ijk, double *d_out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int nt = 128;
  const unsigned blocks = (unsigned)((n + nt - 1) / nt);
  if (vertical(t)) k_table_at<true><<<blocks, nt, 0, s>>>(g, make_fields<1, true>(g, t, b), n, d_ijk, d_out);
  else k_table_at<false><<<blocks, nt, 0, s>>>(g, make_fields<1, false>(g, t, b), n, d_ijk, d_out);
  return cudaGetLastError();
}

CoefGeom make_coef_geom(const dds_ctx *ctx) { return coef_geom(ctx); }

int build_spectra(dds_ctx *ctx, cudaStream_t s) {
  const Shape &sh = ctx->shape;
  const int px = 2 * sh.M, py = sh.py, pz = sh.pz, M = sh.M;
  const size_t P = (size_t)px * py * pz;
  const CoefGeom g = coef_geom(ctx);
  const double *ft = ctx->field_t.data(), *fb = ctx->field_b.data();

  auto tab_of = [&](int mx, int my) {
    Tab T;
    T.nx = sh.nx;
    T.ny = sh.ny;
    T.nz = sh.nz;
    T.mx = mx;
    T.my = my;
    T.rx = mx ? sh.nx : 2 * sh.nx - 1;
    T.ry = (my || py == sh.ny) ? sh.ny : 2 * sh.ny - 1;      // periodic in y: rows 0 .. ny - 1
    return T;
  };
  // Runs of up to three fields of one direction and mirrors share tables, and up to six
  // components share a launch.  The three buffers are each sized for the run that needs most
  // of it; their sum is kept within what a full padded FP64 table of one field and one complex
  // spectrum take (sized run by run without that rule, 18 families on 256x256x128 took 4.03 GB
  // against 3.76, a mirrored and an unmirrored direction together 4.83).  Components per launch
  // are reduced first, where they take most, then fields per table.  The fewest of both always
  // fit: half of that table, and half of that spectrum in each buffer.
  struct Run {
    int e0, fields, mx, my;
    int n, slots;               // fields per table, components per launch
    size_t tab, x, y;           // bytes per field of a table, per component of either buffer
    int least() const { return mx ? 2 : 1; }
  };
  std::vector<Run> runs;
  for (int e = 0; e < ctx->fe;) {
    auto flag = [&](int q, int a) { return mirror_ok(ft + 3 * q, fb + 3 * q, a) ? 1 : 0; };
    Run r{e, 1, flag(e, 0), flag(e, 1), 0, 6, 0, 0, 0};
    while (r.fields < 3 && e + r.fields < ctx->fe && flag(e + r.fields, 0) == r.mx && flag(e + r.fields, 1) == r.my &&
           ft[3 * e] == ft[3 * (e + r.fields)] && ft[3 * e + 1] == ft[3 * (e + r.fields) + 1] &&
           ft[3 * e + 2] == ft[3 * (e + r.fields) + 2])
      ++r.fields;
    const Tab T = tab_of(r.mx, r.my);
    const size_t ky = T.mx ? py / 2 + 1 : py, c = M + 1;
    r.n = r.fields;
    r.tab = 48 * (size_t)tab_size(T);
    r.x = std::max((size_t)T.nz * T.ry * c * (T.mx ? 8 : 16), (size_t)pz * ky * c * 8);
    r.y = (size_t)T.nz * ky * c * 16;
    runs.push_back(r);
    e += r.fields;
  }
  size_t tab_max = 0, buf1_max = 0, buf2_max = 0;
  const size_t limit = 48 * P + 16 * (size_t)(M + 1) * py * pz;
  for (;;) {
    tab_max = buf1_max = buf2_max = 0;
    Run *wide = nullptr, *deep = nullptr;     // most in the buffers and reducible; largest table
    for (Run &r : runs) {
      tab_max = std::max(tab_max, r.n * r.tab);
      buf1_max = std::max(buf1_max, r.slots * r.x);
      buf2_max = std::max(buf2_max, r.slots * r.y);
      if (r.slots > r.least() && (!wide || r.slots * (r.x + r.y) > wide->slots * (wide->x + wide->y))) wide = &r;
      if (r.n > 1 && (!deep || r.n * r.tab > deep->n * deep->tab)) deep = &r;
    }
    if (tab_max + buf1_max + buf2_max <= limit) break;
    if (wide) wide->slots = wide->slots > 2 ? wide->slots - 2 : wide->least();
    else if (deep) --deep->n;
    else break;
  }
  std::vector<Batch> batches;
  for (const Run &r : runs)
    for (int f = 0; f < r.fields; f += r.n) batches.push_back({r.e0 + f, std::min(r.n, r.fields - f), r.mx, r.my, r.slots});

  // near offsets the tables hold (decided on the host, same expression as the
  // definition): all of them, then those with i >= 0, j >= 0 and both, by (mx, my)
  std::vector<int> near;                 // with replica shells the table kernel handles them
  int near_at[2][2] = {{0, 0}, {0, 0}}, near_n[2][2] = {{0, 0}, {0, 0}};
  if (ctx->n_near > 0.0 && ctx->n_shells == 0) {
    double hmax = fmax(ctx->h[0], fmax(ctx->h[1], ctx->h[2]));
    int lim[3] = {ctx->nx - 1, ctx->ny - 1, ctx->nz - 1};
    for (int a = 0; a < 3; ++a) {
      const double c = ceil(ctx->n_near * hmax / ctx->h[a]) + 1.0;
      if (c < lim[a]) lim[a] = (int)c;
    }
    for (int mx = 0; mx < 2; ++mx)
      for (int my = 0; my < 2; ++my) {
        bool used = false;
        for (const Batch &b : batches) used = used || (b.mx == mx && b.my == my);
        if (!used) continue;
        near_at[mx][my] = (int)near.size();
        for (int k = 0; k <= lim[2]; ++k)
          for (int j = my ? 0 : -lim[1]; j <= lim[1]; ++j)
            for (int i = mx ? 0 : -lim[0]; i <= lim[0]; ++i)
              if (is_near(ctx->h, ctx->n_near, i, j, k)) {
                near.push_back(i);
                near.push_back(j);
                near.push_back(k);
              }
        near_n[mx][my] = ((int)near.size() - near_at[mx][my]) / 3;
      }
  }

  double *tab = nullptr, *buf1 = nullptr;
  double2 *buf2 = nullptr;
  int *d_near = nullptr;
  unsigned long long *d_amax = nullptr;
  cudaError_t err = cudaMallocAsync(&tab, tab_max, s);
  if (err == cudaSuccess) err = cudaMallocAsync(&d_amax, sizeof(unsigned long long), s);
  if (err == cudaSuccess) err = cudaMallocAsync(&buf1, buf1_max, s);
  if (err == cudaSuccess) err = cudaMallocAsync(&buf2, buf2_max, s);
  if (err == cudaSuccess && !near.empty()) err = cudaMallocAsync(&d_near, sizeof(int) * near.size(), s);
  if (err != cudaSuccess) {
    cudaFreeAsync(tab, s);
    cudaFreeAsync(buf1, s);
    cudaFreeAsync(buf2, s);
    cudaFreeAsync(d_near, s);
    cudaFreeAsync(d_amax, s);
    cudaGetLastError();
    return fail(ctx, DDS_ERR_OOM, "build_kernels: cannot allocate %.2f GB of FP64 table workspace: %s",
                (double)(tab_max + buf1_max + buf2_max) / 1e9, cudaGetErrorString(err));
  }
  if (!near.empty())
    err = cudaMemcpyAsync(d_near, near.data(), sizeof(int) * near.size(), cudaMemcpyHostToDevice, s);

  const double scale = 1.0 / ((double)px * (double)py * (double)pz);
  for (size_t ib = 0; ib < batches.size() && err == cudaSuccess; ++ib) {
    const Batch &b = batches[ib];
    const Tab T = tab_of(b.mx, b.my);
    const double *t = ft + 3 * b.e0, *bv = fb + 3 * b.e0;
    const int nn = near_n[b.mx][b.my];
    const int *dn = d_near + near_at[b.mx][b.my];
    if (b.n == 1) err = fill_table<1>(g, t, bv, T, nn, dn, tab, s);
    else if (b.n == 2) err = fill_table<2>(g, t, bv, T, nn, dn, tab, s);
    else err = fill_table<3>(g, t, bv, T, nn, dn, tab, s);
    for (int f = 0; f < b.n && err == cudaSuccess; ++f) {
      const int e = b.e0 + f;
      Comps all{};
      all.off = 6 * f;
      for (int c = 0; c < 6; ++c) {
        all.sx[c] = b.mx ? mirror_parity(fb + 3 * e, 0, c) : 1;
        all.sy[c] = b.my ? mirror_parity(fb + 3 * e, 1, c) : 1;
      }
      // line sets: with the x mirror each x-odd component shares the line of an x-even one
      std::vector<std::pair<int, int>> sets;
      std::vector<int> even, odd;
      for (int c = 0; c < 6; ++c) (b.mx && all.sx[c] < 0 ? odd : even).push_back(c);
      for (size_t q = 0; q < std::max(even.size(), odd.size()); ++q) {
        if (q >= even.size()) sets.push_back({odd[q], -1});
        else sets.push_back({even[q], q < odd.size() ? odd[q] : -1});
      }
      const size_t cols = (size_t)(b.mx ? py / 2 + 1 : py) * (M + 1);
      for (size_t q = 0; q < sets.size() && err == cudaSuccess;) {
        Comps C = all;
        for (; q < sets.size(); ++q) {
          const int add = sets[q].second >= 0 ? 2 : 1;
          if (C.slots + add > b.slots) break;
          C.ce[C.sets] = sets[q].first;
          C.co[C.sets] = sets[q].second;
          C.se[C.sets] = C.slots;
          C.comp_of[C.slots++] = sets[q].first;
          C.so[C.sets] = 0;
          if (add == 2) {
            C.so[C.sets] = C.slots;
            C.comp_of[C.slots++] = sets[q].second;
          }
          ++C.sets;
        }
        err = x_dispatch(M, T, C, tab, buf1, ctx->tw.f64, s);
        if (err == cudaSuccess) err = y_dispatch(py, T, C, M, buf1, buf2, ctx->tw.f64, s);
        if (err == cudaSuccess) err = z_dispatch(pz, T.nz, (long)cols, C.slots, buf2, buf1, ctx->tw.f64, s);
        for (int slot = 0; slot < C.slots && err == cudaSuccess; ++slot) {
          const int c = C.comp_of[slot];
          const double *spec = buf1 + (size_t)slot * pz * cols;
          const int fold = b.mx ? -C.sx[c] : 0;
          const long n = sh.zfour ? zf_stored_tiles(sh) * pz * sh.wz : (long)py * (M + 1) * pz;
          const unsigned blocks = (unsigned)((n + 255) / 256);
          if (ctx->spectra_fp16) {
            err = cudaMemsetAsync(d_amax, 0, sizeof(unsigned long long), s);
            if (err == cudaSuccess) {
              k_absmax_imag<<<1024, 256, 0, s>>>(spec, (long)(pz * cols), d_amax);
              k_store_scale<<<1, 1, 0, s>>>(d_amax, scale, ctx->kscale, c * sh.fe + e);
              __half *out = static_cast<__half *>(ctx->kspec);
              if (sh.zfour) k_extract_four<__half><<<blocks, 256, 0, s>>>(spec, fold, sh, e, c, scale, d_amax, out);
              else k_extract<__half><<<blocks, 256, 0, s>>>(spec, fold, M, py, pz, sh.wz, sh.zreg_g, sh.fe, e, c,
                                                            scale, d_amax, out);
              err = cudaGetLastError();
            }
          } else {
            float *out = static_cast<float *>(ctx->kspec);
            if (sh.zfour) k_extract_four<float><<<blocks, 256, 0, s>>>(spec, fold, sh, e, c, scale, nullptr, out);
            else k_extract<float><<<blocks, 256, 0, s>>>(spec, fold, M, py, pz, sh.wz, sh.zreg_g, sh.fe, e, c, scale,
                                                         nullptr, out);
            err = cudaGetLastError();
          }
        }
      }
    }
  }
  cudaFreeAsync(tab, s);
  cudaFreeAsync(buf1, s);
  cudaFreeAsync(buf2, s);
  cudaFreeAsync(d_near, s);
  cudaFreeAsync(d_amax, s);
  if (err == cudaSuccess) err = cudaStreamSynchronize(s);
  if (err != cudaSuccess) return fail(ctx, DDS_ERR_CUDA, "build_kernels: %s", cudaGetErrorString(err));
  return DDS_OK;
}

}  // namespace dds
