// Relaxation of the dislocation stress to free top and bottom surfaces
// (Sec. 5, Eqs. 14-18), FP32.
//
// The displacement u (three components, [c][z][y][x], metres) relaxes by
// explicit Euler steps of Eq. 17,
//     u <- u + dt (A grad div u - B rot rot u + f),   f_a = sum_b d sigma^dis_ab / db (Eq. 15),
// with u periodic in x and y (Eq. 16a) and the traction-free surface conditions
// of Eq. 16c imposed through one ghost layer below the first and above the last
// film layer (Eq. 18b and its counterparts).  Ghost values are functions of the
// film values of the same step, so the step kernel evaluates them where it needs
// them instead of storing them.  Differences: second differences, 4-point mixed
// derivatives, central first derivatives; d sigma^dis / dz one-sided (second
// order) on the surface layers.  dt = min(h)^2 / (5A - 3B).
//
// The coefficients are folded with dt on the host (double, then rounded once),
// so every quantity the kernels touch is in units of u.  One step reads u and
// dt f and writes u: 36 bytes per cell from HBM.
#include <algorithm>
#include <type_traits>

#include "dds_internal.h"
#include "stress_common.cuh"

namespace dds {
namespace {

struct RelaxCoef {
  int nx, ny, nz;
  // dt-scaled operator: u_a += sum_b lap2[a][b] (u_a[+b] - 2 u_a + u_a[-b])
  //                          + sum_{b != a} mix2[a][b] (4-point cross of u_b in a, b),
  // each value twice, for packed pairs of cells
  float2 lap2[3][3], mix2[3][3];
  // ghost layers: first derivatives 1/(2 h) and the factors of Eq. 18b
  float inv2h[3];
  float two_dz;      // 2 dz
  float zfac;        // 2 dz / (1 - nu)
  float nu;
  // Hooke's law for sigma(u): lambda, mu
  float lam, mu;
  // phi of Eq. 16c from sigma^dis: -(1 + nu) / E and -(1 + nu)(1 - 2 nu) / E
  float phi_shear, phi_normal;
  // dt for f
  float dt;
};

__device__ __forceinline__ int wrap(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

__device__ __forceinline__ long cidx(const RelaxCoef &r, int c, int k, int j, int i) {
  return (((long)c * r.nz + k) * r.ny + j) * r.nx + i;
}

// dt f (Eq. 15) at every film cell and phi (Eq. 16c) on the two surface layers.
__global__ void k_relax_prep(RelaxCoef r, const float *__restrict__ sig, float *__restrict__ gf,
                             float *__restrict__ phi) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y, k = blockIdx.z;
  if (i >= r.nx || j >= r.ny) return;
  // component index of the pair (a, b): xx yy zz xy xz yz
  constexpr int PAIR[3][3] = {{0, 3, 4}, {3, 1, 5}, {4, 5, 2}};
  const int ip = wrap(i + 1, r.nx), im = wrap(i - 1, r.nx), jp = wrap(j + 1, r.ny), jm = wrap(j - 1, r.ny);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int cx = PAIR[a][0], cy = PAIR[a][1], cz = PAIR[a][2];
    float d = (__ldg(sig + cidx(r, cx, k, j, ip)) - __ldg(sig + cidx(r, cx, k, j, im))) * r.inv2h[0] +
              (__ldg(sig + cidx(r, cy, k, jp, i)) - __ldg(sig + cidx(r, cy, k, jm, i))) * r.inv2h[1];
    float dz;
    if (r.nz >= 3) {
      if (k == 0)
        dz = (-3.f * __ldg(sig + cidx(r, cz, 0, j, i)) + 4.f * __ldg(sig + cidx(r, cz, 1, j, i)) - __ldg(sig + cidx(r, cz, 2, j, i))) * r.inv2h[2];
      else if (k == r.nz - 1)
        dz = (3.f * __ldg(sig + cidx(r, cz, k, j, i)) - 4.f * __ldg(sig + cidx(r, cz, k - 1, j, i)) + __ldg(sig + cidx(r, cz, k - 2, j, i))) * r.inv2h[2];
      else
        dz = (__ldg(sig + cidx(r, cz, k + 1, j, i)) - __ldg(sig + cidx(r, cz, k - 1, j, i))) * r.inv2h[2];
    } else {
      dz = (__ldg(sig + cidx(r, cz, 1, j, i)) - __ldg(sig + cidx(r, cz, 0, j, i))) * (2.f * r.inv2h[2]);
    }
    gf[cidx(r, a, k, j, i)] = r.dt * (d + dz);
  }
  if (k == 0 || k == r.nz - 1) {
    const long plane = (long)r.ny * r.nx;
    float *ph = phi + (long)(k == 0 ? 0 : 3) * plane + (long)j * r.nx + i;
    ph[0] = r.phi_shear * __ldg(sig + cidx(r, 4, k, j, i));
    ph[plane] = r.phi_shear * __ldg(sig + cidx(r, 5, k, j, i));
    ph[2 * plane] = r.phi_normal * __ldg(sig + cidx(r, 2, k, j, i));
  }
}

// The march over the film, shared by the step and the stress kernels.  256 threads take a
// tile of 64 x 8 (or 32 x 16) columns, two x-adjacent cells per thread, up a chunk of layers.  Planes of
// u (three components, one-cell halo) arrive in a ring of shared-memory slots by
// cp.async, up to three layers ahead of the layer that uses them; ghost planes are evaluated
// into their slot.  A plane is read from shared memory once, when it is the one above the
// current layer: every term of the operator is a combination of in-plane terms of the
// layer's own plane and of differences between the planes above and below, so a thread
// carries the centre values, four in-plane differences and the in-plane part of the
// operator in registers.  That is 12 shared-memory loads per cell against 45 with three
// resident planes, and one barrier per layer against two.  The march is unrolled by three:
// the carried terms then stay in fixed registers.  The two
// cells' arithmetic is packed (add/fma on pairs of FP32).  FULL: rows are whole tiles and everything is aligned, so no
// access is predicated.  What bounds it: shared-memory wavefronts (about half the time) and
// the latency of a layer's chain at two CTAs per SM (their registers), with DRAM at half its
// rate; deeper rings and one cell per thread measured the same or slower.  Step, GaN grid
// 256x256x128: 94 -> 77 us, 512x512x16: 61 -> 49 us; total stress: 442 -> 105 us and 226 ->
// 63 us (it evaluated ghost layers and offsets per value before).
constexpr int NTM = 256, RING = 4, X0 = 4;         // column x of the tile at X0 + x: 16-byte aligned rows
template <int PX> struct March {                   // PX threads along x
  static constexpr int TX = 2 * PX, TY = NTM / PX, HY = TY + 2, LD = TX + 8, CS = HY * LD, PLANE = 3 * CS;
  // a slot: one plane, and the threads' own inputs (NC fields) of the layer below it
  template <int NC> static constexpr int slot_floats() { return PLANE + NC * 2 * NTM; }
};

__device__ __forceinline__ float ld_cg1(const float *p) {
  float v;
  asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}

__device__ __forceinline__ int mod(int i, int n) { return ((i % n) + n) % n; }

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

__device__ __forceinline__ void cp_async4(float *dst, const float *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async8f(float *dst, const float *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async16f(float *dst, const float *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// The part of every plane one thread stages: two groups of four columns and, for the first
// threads, one halo column, as offsets of the film element in layer 0 and of the slot
// element (fixed for the whole march; source -1: none).
struct Stage {
  int src[3], dst[3];
  int col;                 // first column of the groups
};
template <int PX>
__device__ __forceinline__ Stage make_stage(const RelaxCoef &r, int i0, int j0) {
  constexpr int TX = March<PX>::TX, HY = March<PX>::HY, LD = March<PX>::LD;
  constexpr int G = TX / 4, ROWS = 3 * HY, PASS = NTM / G;
  static_assert(ROWS <= 2 * PASS && 2 * ROWS <= NTM, "two passes over the rows, one over the halo columns");
  auto film = [&](int row, int i) { return (int)cidx(r, row / HY, 0, mod(j0 + row % HY - 1, r.ny), i); };
  Stage st;
  const int x = 4 * (threadIdx.x % G);
  st.col = i0 + x;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int row = threadIdx.x / G + PASS * e;
    st.src[e] = row < ROWS && st.col <= r.nx ? film(row, st.col) : -1;   // column nx is the last that is read
    st.dst[e] = row * LD + X0 + x;
  }
  const int row = threadIdx.x >> 1, hx = threadIdx.x & 1 ? TX : -1;
  st.src[2] = row < ROWS && i0 + hx <= r.nx ? film(row, mod(i0 + hx, r.nx)) : -1;
  st.dst[2] = row * LD + X0 + hx;
  return st;
}

// Ghost plane k = -1 or nz of a tile and its halo (Eq. 18b and its counterparts) into slot
// pl: the inner neighbour of the surface layer plus or minus 2 dz times
//   u_x: 2 phi_xz - du_z/dx,  u_y: 2 phi_yz - du_z/dy,
//   u_z: (phi_zz - nu (du_x/dx + du_y/dy)) / (1 - nu).  A thread evaluates
// all components at its three positions with every load in flight: one position and
// component at a time, the surface chunks waited 8 times a memory latency for it.
template <int PX>
__device__ __forceinline__ void ghost_plane(const RelaxCoef &r, const float *u, const float *phi, int i0, int j0, int k,
                                            float *pl) {
  constexpr int TX = March<PX>::TX, HY = March<PX>::HY, LD = March<PX>::LD, CS = March<PX>::CS;
  constexpr int W = TX + 2, NP = (HY * W + NTM - 1) / NTM;
  const bool top = k >= r.nz;
  const int plane = r.ny * r.nx, cs = r.nz * plane;
  const float *us = u + (top ? r.nz - 1 : 0) * plane, *un = u + (top ? r.nz - 2 : 1) * plane;
  const float *ph = phi + (top ? 3 : 0) * plane;
  const float sgn = top ? 1.f : -1.f;
  float in[NP][3], f[NP][3], zx[NP][2], zy[NP][2], xx[NP][2], yy[NP][2];
#pragma unroll
  for (int e = 0; e < NP; ++e) {
    const int p = threadIdx.x + NTM * e, hy = p / W, x = i0 + p - hy * W - 1;
    const bool used = p < HY * W && x <= r.nx;     // column nx is the last that is read
    const int i = used ? wrap(x, r.nx) : 0, j = used ? mod(j0 + hy - 1, r.ny) : 0;
    const int o = j * r.nx + i, oe = j * r.nx + wrap(i + 1, r.nx), ow = j * r.nx + wrap(i - 1, r.nx);
    const int on = wrap(j + 1, r.ny) * r.nx + i, os = wrap(j - 1, r.ny) * r.nx + i;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      in[e][c] = ld_cg1(un + c * cs + o);
      f[e][c] = ld_cg1(ph + c * plane + o);
    }
    zx[e][0] = ld_cg1(us + 2 * cs + oe);
    zx[e][1] = ld_cg1(us + 2 * cs + ow);
    zy[e][0] = ld_cg1(us + 2 * cs + on);
    zy[e][1] = ld_cg1(us + 2 * cs + os);
    xx[e][0] = ld_cg1(us + oe);
    xx[e][1] = ld_cg1(us + ow);
    yy[e][0] = ld_cg1(us + cs + on);
    yy[e][1] = ld_cg1(us + cs + os);
  }
#pragma unroll
  for (int e = 0; e < NP; ++e) {
    const int p = threadIdx.x + NTM * e, hy = p / W, x = p - hy * W - 1;
    if (p >= HY * W || i0 + x > r.nx) continue;
    float *d = pl + hy * LD + X0 + x;
    d[0] = in[e][0] + sgn * r.two_dz * (2.f * f[e][0] - (zx[e][0] - zx[e][1]) * r.inv2h[0]);
    d[CS] = in[e][1] + sgn * r.two_dz * (2.f * f[e][1] - (zy[e][0] - zy[e][1]) * r.inv2h[1]);
    d[2 * CS] = in[e][2] + sgn * r.zfac * (f[e][2] - r.nu * ((xx[e][0] - xx[e][1]) * r.inv2h[0] + (yy[e][0] - yy[e][1]) * r.inv2h[1]));
  }
}

// Starts plane k (a layer, or a ghost layer at -1 and nz) into slot pl, in the current copy group.
// vec: rows of u are 16-byte aligned (whole groups of four).
template <int PX, bool FULL>
__device__ __forceinline__ void start_plane(const RelaxCoef &r, const float *u, const float *phi, const Stage &st, int i0,
                                            int j0, int k, bool vec, float *pl) {
  if (k >= 0 && k < r.nz) {
    const float *layer = u + (long)k * (r.ny * r.nx);
    if constexpr (FULL) {
      cp_async16f(pl + st.dst[0], layer + st.src[0]);
      if (st.src[1] >= 0) cp_async16f(pl + st.dst[1], layer + st.src[1]);
    } else {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        if (st.src[e] < 0) continue;
        const float *src = layer + st.src[e];
        float *dst = pl + st.dst[e];
        if (vec && st.col < r.nx) {
          cp_async16f(dst, src);
          if (st.col + 4 == r.nx) cp_async4(dst + 4, src + 4 - r.nx);    // a row that ends inside the tile: its halo
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q) {            // past the last column: the first again
            const int i = st.col + q;
            if (i <= r.nx) cp_async4(dst + q, src + q - (i == r.nx ? r.nx : 0));
          }
        }
      }
    }
    if (st.src[2] >= 0) cp_async4(pl + st.dst[2], layer + st.src[2]);
  } else {
    ghost_plane<PX>(r, u, phi, i0, j0, k, pl);
  }
}

// What a thread keeps of a plane for its two cells: centre values; u_x(x+1) - u_x(x-1) and
// the same of u_z; u_y(y+1) - u_y(y-1) and the same of u_z.  STEP: in[a] = the in-plane
// part of the operator; otherwise in[0], in[1] = the x difference of u_y and the y
// difference of u_x.
struct PlaneTerms {
  float2 c[3], ax, az, by, bz, in[3];
};

// The values at x (the two cells), x - 1 and x + 1 of one row.
struct Row {
  float2 m, w, e;
};
template <bool SIDES>
__device__ __forceinline__ Row load_row(const float *p) {
  Row v;
  v.m = *reinterpret_cast<const float2 *>(p);
  if (SIDES) {
    v.w = make_float2(p[-1], v.m.x);
    v.e = make_float2(v.m.y, p[2]);
  }
  return v;
}

template <int PX, bool STEP>
__device__ __forceinline__ void read_plane(const RelaxCoef &r, const float *p, PlaneTerms &t) {
  constexpr int CS = March<PX>::CS, LD = March<PX>::LD;
  float2 xs[3], ys[3], cross[2];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const Row m = load_row<true>(p + c * CS);
    const Row d = c < 2 ? load_row<STEP>(p + c * CS - LD) : load_row<false>(p + c * CS - LD);
    const Row n = c < 2 ? load_row<STEP>(p + c * CS + LD) : load_row<false>(p + c * CS + LD);
    t.c[c] = m.m;
    if (STEP) {
      xs[c] = add2(sub2(m.e, m.m), sub2(m.w, m.m));
      ys[c] = add2(sub2(n.m, m.m), sub2(d.m, m.m));
      if (c < 2) cross[c] = sub2(add2(n.e, d.w), add2(d.e, n.w));
    }
    if (c == 0) {
      t.ax = sub2(m.e, m.w);
      if (!STEP) t.in[1] = sub2(n.m, d.m);
    } else if (c == 1) {
      t.by = sub2(n.m, d.m);
      if (!STEP) t.in[0] = sub2(m.e, m.w);
    } else {
      t.az = sub2(m.e, m.w);
      t.bz = sub2(n.m, d.m);
    }
  }
  if (STEP) {                                      // d2u_y/dxdy into x, d2u_x/dxdy into y
    t.in[0] = fma2(r.lap2[0][0], xs[0], fma2(r.lap2[0][1], ys[0], __fmul2_rn(r.mix2[0][1], cross[1])));
    t.in[1] = fma2(r.lap2[1][0], xs[1], fma2(r.lap2[1][1], ys[1], __fmul2_rn(r.mix2[1][0], cross[0])));
    t.in[2] = fma2(r.lap2[2][0], xs[2], __fmul2_rn(r.lap2[2][1], ys[2]));
  }
}

// STEP: one explicit step, out[3] = u + dt (navier(u) + f), gin[3] = dt f.  Otherwise the
// total stress, out[6] = gin[6] + lambda div u delta + mu (du_a/db + du_b/da).
template <int PX, bool STEP, bool FULL>
__global__ void __launch_bounds__(NTM, 2)
k_relax_march(RelaxCoef r, const float *u, const float *gin, const float *phi, float *out, int kz, int vec) {
  using C = March<PX>;
  constexpr int TX = C::TX, TY = C::TY, LD = C::LD, PLANE = C::PLANE, NC = STEP ? 3 : 6;
  constexpr int SLOT = C::template slot_floats<NC>();
  extern __shared__ __align__(16) float ring[];
  const int tx = threadIdx.x % PX, ty = threadIdx.x / PX;
  const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY, i = i0 + 2 * tx;
  const int kb = blockIdx.z * kz, ke = min(kb + kz, r.nz);
  const bool live = FULL || (i < r.nx && j0 + ty < r.ny), second = FULL || i + 1 < r.nx;
  const int plane = r.ny * r.nx, cstride = r.nz * plane, own = (j0 + ty) * r.nx + i;
  pdl_trigger();
  const Stage st = make_stage<PX>(r, i0, j0);
  pdl_wait();                                      // u of the step before
  const int mine = (ty + 1) * LD + X0 + 2 * tx, own_in = PLANE + 2 * threadIdx.x;
  // one copy group, into slot q: plane k and the cells' inputs of layer k - 1 (nothing past
  // the plane above the chunk)
  auto start = [&](int k, int q) {
    if (k <= ke) {
      start_plane<PX, FULL>(r, u, phi, st, i0, j0, k, vec, ring + q * SLOT);
      if (live && k > kb) {
        float *dst = ring + q * SLOT + own_in;
        const int o = own + (k - 1) * plane;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const float *src = gin + (o + c * cstride);
          if constexpr (FULL) {
            cp_async8f(dst + 2 * NTM * c, src);
          } else {
            cp_async4(dst + 2 * NTM * c, src);
            if (second) cp_async4(dst + 2 * NTM * c + 1, src + 1);
          }
        }
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  PlaneTerms t[3];
  int sq = 2;                                      // slot of plane k + 1
  // layer k with the terms of the planes k - 1, k, k + 1 in t[P], t[P + 1], t[P + 2] (mod 3)
  auto layer = [&](int k, auto P) {
    constexpr int A = decltype(P)::value, B = (A + 1) % 3, D = (A + 2) % 3;
    asm volatile("cp.async.wait_group %0;\n" ::"n"(RING - 2) : "memory");      // plane k + 1 has landed
    __syncthreads();                               // ... for every thread; planes up to k are read
    start(k + RING, sq == 0 ? RING - 1 : sq - 1);
    const float *slot = ring + sq * SLOT;
    sq = sq == RING - 1 ? 0 : sq + 1;
    read_plane<PX, STEP>(r, slot + mine, t[D]);
    float2 g[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) g[c] = *reinterpret_cast<const float2 *>(slot + own_in + 2 * NTM * c);
    const PlaneTerms &lo = t[A], &mi = t[B], &up = t[D];
    float2 v[NC];
    if (STEP) {
      const float2 mz[3] = {fma2(r.mix2[0][2], sub2(up.az, lo.az), mi.in[0]), fma2(r.mix2[1][2], sub2(up.bz, lo.bz), mi.in[1]),
                            fma2(r.mix2[2][0], sub2(up.ax, lo.ax), fma2(r.mix2[2][1], sub2(up.by, lo.by), mi.in[2]))};
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float2 c0 = mi.c[a];
        const float2 w = fma2(r.lap2[a][2], add2(sub2(up.c[a], c0), sub2(lo.c[a], c0)), g[a]);
        v[a] = add2(c0, add2(w, mz[a]));
      }
    } else {
      const float2 hx = make_float2(r.inv2h[0], r.inv2h[0]), hy = make_float2(r.inv2h[1], r.inv2h[1]);
      const float2 hz = make_float2(r.inv2h[2], r.inv2h[2]), mu = make_float2(r.mu, r.mu), mu2 = make_float2(2.f * r.mu, 2.f * r.mu);
      const float2 xx = __fmul2_rn(mi.ax, hx), yy = __fmul2_rn(mi.by, hy), zz = __fmul2_rn(sub2(up.c[2], lo.c[2]), hz);
      const float2 xy = fma2(mi.in[1], hy, __fmul2_rn(mi.in[0], hx));
      const float2 xz = fma2(sub2(up.c[0], lo.c[0]), hz, __fmul2_rn(mi.az, hx));
      const float2 yz = fma2(sub2(up.c[1], lo.c[1]), hz, __fmul2_rn(mi.bz, hy));
      const float2 ld = __fmul2_rn(make_float2(r.lam, r.lam), add2(add2(xx, yy), zz));
      const float2 e[6] = {fma2(mu2, xx, ld), fma2(mu2, yy, ld), fma2(mu2, zz, ld), __fmul2_rn(mu, xy), __fmul2_rn(mu, xz), __fmul2_rn(mu, yz)};
#pragma unroll
      for (int c = 0; c < NC; ++c) v[c] = add2(g[c], e[c]);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      float *p = out + (own + k * plane + c * cstride);
      if constexpr (FULL) {
        *reinterpret_cast<float2 *>(p) = v[c];
      } else if (live) {
        p[0] = v[c].x;
        if (second) p[1] = v[c].y;
      }
    }
  };
#pragma unroll
  for (int q = 0; q < RING; ++q) start(kb - 1 + q, q);
  asm volatile("cp.async.wait_group %0;\n" ::"n"(RING - 2) : "memory");
  __syncthreads();
  read_plane<PX, STEP>(r, ring + mine, t[0]);
  read_plane<PX, STEP>(r, ring + SLOT + mine, t[1]);
  __syncthreads();                                 // slot 0 is read
  start(kb - 1 + RING, 0);
  using I0 = std::integral_constant<int, 0>;
  using I1 = std::integral_constant<int, 1>;
  using I2 = std::integral_constant<int, 2>;
  for (int k = kb; k < ke; k += 3) {
    layer(k, I0{});
    if (k + 1 < ke) layer(k + 1, I1{});
    if (k + 2 < ke) layer(k + 2, I2{});
  }
}

RelaxCoef relax_coef(const dds_ctx *ctx, double *dt_out) {
  RelaxCoef r{};
  r.nx = ctx->nx;
  r.ny = ctx->ny;
  r.nz = ctx->nz;
  const double mu = ctx->mu, nu = ctx->nu;
  const double E = 2.0 * mu * (1.0 + nu);
  const double A = E * (1.0 - nu) / ((1.0 + nu) * (1.0 - 2.0 * nu));
  const double B = E / (2.0 * (1.0 + nu));
  const double *h = ctx->h;
  const double hmin = std::min(h[0], std::min(h[1], h[2]));
  const double dt = hmin * hmin / (5.0 * A - 3.0 * B);
  for (int a = 0; a < 3; ++a) {
    for (int b = 0; b < 3; ++b) {
      const float lap = (float)(dt * (a == b ? A : B) / (h[b] * h[b]));
      const float mix = a == b ? 0.f : (float)(dt * (A - B) / (4.0 * h[a] * h[b]));
      r.lap2[a][b] = make_float2(lap, lap);
      r.mix2[a][b] = make_float2(mix, mix);
    }
    r.inv2h[a] = (float)(1.0 / (2.0 * h[a]));
  }
  r.two_dz = (float)(2.0 * h[2]);
  r.zfac = (float)(2.0 * h[2] / (1.0 - nu));
  r.nu = (float)nu;
  r.lam = (float)(A - 2.0 * B);
  r.mu = (float)B;
  r.phi_shear = (float)(-(1.0 + nu) / E);
  r.phi_normal = (float)(-(1.0 + nu) * (1.0 - 2.0 * nu) / E);
  r.dt = (float)dt;
  if (dt_out) *dt_out = dt;
  return r;
}

template <int PX, bool STEP>
cudaError_t launch_march_px(const RelaxCoef &r, const float *u, const float *in, const float *phi, float *out, bool early,
                            cudaStream_t s) {
  using C = March<PX>;
  // Layers per chunk: 16 where that makes two full waves (two CTAs per SM each), 8 where that
  // makes one, else 4.  Longer chunks restart the march less often, but leave an emptier last
  // wave (step on 256x256x128: 8 / 16 / 32 / 64 layers 82 / 77 / 82 / 81 us; 512x512x16: 8 /
  // 16 layers 49 / 51 us; 100x90x40: 4 / 8 / 16 layers 9 / 12 / 20 us).  Shorter still while
  // all chunks are resident at once: a layer's chain and the two ghost planes are then all the
  // time (1 / 2 / 4 layers, ten steps and the total: 16x16x4 49 / 62 / 91 us, 64x64x8 47 / 54 /
  // 65, 64x64x64, 512 CTAs at one layer, 86 / 71 / 84; the total alone, 16x16x4 8.4 / 9.1 / 12.4)
  int dev = 0, sms = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err == cudaSuccess) err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (err != cudaSuccess) return err;
  const long tiles = (long)((r.nx + C::TX - 1) / C::TX) * ((r.ny + C::TY - 1) / C::TY);
  auto ctas = [&](int layers) { return tiles * ((r.nz + layers - 1) / layers); };
  int kz = ctas(16) >= 4 * sms ? 16 : (ctas(8) >= 2 * sms ? 8 : 4);
  while (kz > 1 && ctas(kz / 2) <= 2 * sms) kz /= 2;
  const dim3 grid((unsigned)((r.nx + C::TX - 1) / C::TX), (unsigned)((r.ny + C::TY - 1) / C::TY),
                  (unsigned)((r.nz + kz - 1) / kz));
  const int vec = r.nx % 4 == 0 && ((uintptr_t)u & 15) == 0;
  const bool full = vec && r.nx % C::TX == 0 && r.ny % C::TY == 0 && (((uintptr_t)in | (uintptr_t)out) & 7) == 0;
  const size_t smem = sizeof(float) * RING * C::template slot_floats<STEP ? 3 : 6>();
  if (full) return launch_pass<k_relax_march<PX, STEP, true>>(early, grid, NTM, smem, s, r, u, in, phi, out, kz, vec);
  return launch_pass<k_relax_march<PX, STEP, false>>(early, grid, NTM, smem, s, r, u, in, phi, out, kz, vec);
}

template <bool STEP>
cudaError_t launch_march(const RelaxCoef &r, const float *u, const float *in, const float *phi, float *out, bool early,
                         cudaStream_t s) {
  // tiles of 64 x 8 columns, or of 32 x 16 where those overhang the rows less (step on
  // 160x160x32 15.9 -> 11.9 us, 32x512x4 9.2 -> 6.1 us; on 256x256x128 they take 87 against
  // 76 us)
  const int w64 = (r.nx + 63) / 64 * 64, w32 = (r.nx + 31) / 32 * 32;
  return w32 < w64 ? launch_march_px<16, STEP>(r, u, in, phi, out, early, s)
                   : launch_march_px<32, STEP>(r, u, in, phi, out, early, s);
}

}  // namespace

int enqueue_relax(dds_ctx *ctx, const float *sig, float *u, int n_steps, float *sig_tot, cudaStream_t s) {
  const RelaxCoef r = relax_coef(ctx, nullptr);
  const size_t N = (size_t)r.nx * r.ny * r.nz;
  const size_t need = 3 * N + 3 * N + 6 * (size_t)r.nx * r.ny;     // dt f, u ping-pong, phi
  if (ctx->relax_n < need) {
    cudaFree(ctx->relax_buf);
    ctx->relax_buf = nullptr;
    ctx->relax_n = 0;
    if (cudaMalloc(&ctx->relax_buf, sizeof(float) * need) != cudaSuccess) {
      cudaGetLastError();
      return fail(ctx, DDS_ERR_OOM, "relax: cannot allocate %.2f GB of work space", sizeof(float) * need / 1e9);
    }
    ctx->relax_n = need;
  }
  // a captured chain keeps full dependencies (see the evaluation's passes)
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  cudaError_t err = cudaStreamIsCapturing(s, &capture);
  const bool early = err == cudaSuccess && capture == cudaStreamCaptureStatusNone;
  float *gf = ctx->relax_buf, *tmp = gf + 3 * N, *phi = tmp + 3 * N;
  const dim3 blk(32, 4, 1);
  const dim3 grid((unsigned)((r.nx + 31) / 32), (unsigned)((r.ny + 3) / 4), (unsigned)r.nz);
  k_relax_prep<<<grid, blk, 0, s>>>(r, sig, gf, phi);
  if (err == cudaSuccess) err = cudaGetLastError();
  // ping-pong so that the last step writes into u
  float *a = u, *b = tmp;
  if (n_steps % 2 == 1 && err == cudaSuccess) {
    err = cudaMemcpyAsync(tmp, u, sizeof(float) * 3 * N, cudaMemcpyDeviceToDevice, s);
    a = tmp;
    b = u;
  }
  for (int t = 0; t < n_steps && err == cudaSuccess; ++t) {
    err = launch_march<true>(r, a, gf, phi, b, early, s);
    std::swap(a, b);
  }
  if (err == cudaSuccess && sig_tot) err = launch_march<false>(r, u, sig, phi, sig_tot, early, s);
  if (err != cudaSuccess) return fail(ctx, DDS_ERR_CUDA, "relax: kernel launch failed: %s", cudaGetErrorString(err));
  return DDS_OK;
}

double relax_time_step(const dds_ctx *ctx) {
  double dt = 0.0;
  relax_coef(ctx, &dt);
  return dt;
}

}  // namespace dds
