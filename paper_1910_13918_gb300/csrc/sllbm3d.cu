// 3D extension of the SLLBM step (the paper's stated next step): D3Q125, the tensor product of
// D1Q5 three times (Sec. II.B), on a uniform grid of hexahedral Lagrange cells (Sec. II.E per
// axis), the fourth-order equilibrium of Sec. II.A with index tuples over {x, y, z}, g^eq =
// (2 C_v - 3) theta f^eq (Sec. II.D) and BGK (Eq. streaming_fg, Pr = 1).  A plain FP64 step on
// full populations, one thread per vertex: the first pass interpolates every velocity of f and g
// at its departure point (tensor product of the three 1D Lagrange bases, per-axis tables as in
// 2D) into the destination and sums the moments, the second relaxes each value in place.  The
// equilibrium is the factorised form: the tensor coefficients a_eq^(n) of an isotropic Maxwellian
// are products of per-axis Hermite moments A_k(u) (A_0 = 1, A_1 = u, A_2 = u^2 + q, A_3 = u^3 +
// 3uq, A_4 = u^4 + 6u^2 q + 3q^2, q = theta - 1), so
//   f_abc^eq = w_a w_b w_c rho sum_{k+l+m <= 4} A_k(u_x) he_k(a) A_l(u_y) he_l(b) A_m(u_z) he_m(c).
// This file has its own context and entry points (sllbm3d_* in include/sllbm.h); it shares the
// axis-table kernel and the device helpers with the 2D library.
#include <math.h>

#include <new>
#include <string>
#include <vector>

#include "../../include/sllbm.h"
#include "kernels.h"
#include "tma.cuh"

using namespace sllbm;

namespace {

constexpr int kQ3 = kQ1 * kQ1 * kQ1;   // D3Q125

struct Step3Args {
  const double* src;
  double* dst;
  int nx, ny, nz;
  long long nv;
  int px, py, pz;                        // periodic axes
  const int *offx, *offy, *offz;         // [5][n]: stencil start - vertex index
  const double *wx, *wy, *wz;            // [5][n][p+1]
  Consts cs;
  double omega, K, cv;
  int npop, iso;
  int* flag;                             // bit 0: unstable
};

// Layout of an FP32 pair state: plane i, vertex (x, y, z) at
// i * plane + origin + (z * rows + y) * pitch + x, with g ghost cells before the interior on
// every axis (g = 0: the dense [125][nz][ny][nx]; the sum-factorised step keeps g = 2, or 4 at orders 3
// and 4, and the periodic images in the ghost cells, so that its staged regions never wrap).
struct Pad3 {
  int g, pitch, rows;
  size_t plane, origin;
  __host__ __device__ size_t at(int i, int x, int y, int z) const {
    return (size_t)i * plane + origin + ((size_t)z * rows + y) * pitch + x;
  }
};

struct Field3Args {
  const double *rho, *u, *v, *w, *T;     // init inputs
  double *orho, *ou, *ov, *ow, *oT;      // moment outputs
  double* state;                         // FP64: full populations [npop][125][nv]
  float2* state32;                       // FP32: (f - w, g - K w) pairs in layout lay (else null)
  Pad3 lay;
  int nx, ny;
  long long nv;
  Consts cs;
  double K, cv;
  int npop;
  int* flag;
};

// FP32 step: deviations from the lattice weights, f and g of a (velocity, vertex) side by side.
struct Step3F32Args {
  const float2* src;
  float2* dst;
  int nx, ny, nz;
  long long nv;
  int px, py, pz;
  const int *offx, *offy, *offz;         // [5][n]
  const float *wx, *wy, *wz;             // [5][n][p+1]
  Consts cs;
  float omega, K, cv, inv2cv;
  int npop, iso;
  int* flag;
};

// Per-axis Hermite moments A_k(u), k = 0..4, of the Maxwellian with q = theta - 1.
__device__ __forceinline__ void hermite_moments(double u, double q, double (&A)[5]) {
  A[0] = 1.0;
  A[1] = u;
  A[2] = u * u + q;
  A[3] = u * (u * u + 3.0 * q);
  A[4] = u * u * (u * u + 6.0 * q) + 3.0 * q * q;
}

// f^eq of velocity (a, b, c), given the per-axis factors X[k] = A_k(u_x) he_k(a) etc.
__device__ __forceinline__ double eq3(const Consts& cs, double rho, const double (&Ax)[5],
                                      const double (&Ay)[5], const double (&Az)[5], int a, int b, int c) {
  double s = 0.0;
#pragma unroll
  for (int k = 0; k <= 4; ++k) {
    const double xk = Ax[k] * cs.he[k][a];
#pragma unroll
    for (int l = 0; l <= 4 - k; ++l) {
      const double yl = Ay[l] * cs.he[l][b];
      double zs = 0.0;
#pragma unroll
      for (int m = 0; m <= 4 - k - l; ++m) zs += Az[m] * cs.he[m][c];
      s += xk * yl * zs;
    }
  }
  return cs.w[a] * cs.w[b] * cs.w[c] * rho * s;
}

template <int P>
__global__ void __launch_bounds__(128) step3d_f64_kernel(const __grid_constant__ Step3Args a) {
  const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= a.nv) return;
  const int ix = (int)(v % a.nx);
  const long long t = v / a.nx;
  const int iy = (int)(t % a.ny), iz = (int)(t / a.ny);
  const size_t plane = (size_t)a.nv;
  const bool two = a.npop == 2;
  double rho = 0.0, jx = 0.0, jy = 0.0, jz = 0.0, e2 = 0.0;
#pragma unroll 1
  for (int i = 0; i < kQ3; ++i) {
    const int ia = i / 25, ib = (i / 5) % 5, ic = i % 5;
    const int sx = ix + a.offx[ia * a.nx + ix], sy = iy + a.offy[ib * a.ny + iy],
              sz = iz + a.offz[ic * a.nz + iz];
    const double* wx = a.wx + (size_t)(ia * a.nx + ix) * (P + 1);
    const double* wy = a.wy + (size_t)(ib * a.ny + iy) * (P + 1);
    const double* wz = a.wz + (size_t)(ic * a.nz + iz) * (P + 1);
    const double* pf = a.src + (size_t)i * plane;
    const double* pg = two ? a.src + (size_t)(kQ3 + i) * plane : pf;
    double accf = 0.0, accg = 0.0;
#pragma unroll
    for (int kc = 0; kc <= P; ++kc) {
      const size_t zoff = (size_t)wrap_index(sz + kc, a.nz, a.pz) * a.ny;
      double yf = 0.0, yg = 0.0;
#pragma unroll
      for (int kb = 0; kb <= P; ++kb) {
        const size_t row = (zoff + (size_t)wrap_index(sy + kb, a.ny, a.py)) * a.nx;
        double xf = 0.0, xg = 0.0;
#pragma unroll
        for (int ka = 0; ka <= P; ++ka) {
          const size_t o = row + (size_t)wrap_index(sx + ka, a.nx, a.px);
          xf += wx[ka] * __ldg(pf + o);
          if (two) xg += wx[ka] * __ldg(pg + o);
        }
        yf += wy[kb] * xf;
        yg += wy[kb] * xg;
      }
      accf += wz[kc] * yf;
      accg += wz[kc] * yg;
    }
    a.dst[(size_t)i * plane + v] = accf;
    if (two) a.dst[(size_t)(kQ3 + i) * plane + v] = accg;
    const double cx = a.cs.xi[ia], cy = a.cs.xi[ib], cz = a.cs.xi[ic];
    rho += accf;
    jx += accf * cx;
    jy += accf * cy;
    jz += accf * cz;
    e2 += accf * (cx * cx + cy * cy + cz * cz) + accg;
  }
  const double ux = jx / rho, uy = jy / rho, uz = jz / rho;
  const double theta = a.iso ? 1.0 : (e2 - rho * (ux * ux + uy * uy + uz * uz)) / (2.0 * a.cv * rho);
  const double q = theta - 1.0;
  double Ax[5], Ay[5], Az[5];
  hermite_moments(ux, q, Ax);
  hermite_moments(uy, q, Ay);
  hermite_moments(uz, q, Az);
#pragma unroll 1
  for (int i = 0; i < kQ3; ++i) {
    const double feq = eq3(a.cs, rho, Ax, Ay, Az, i / 25, (i / 5) % 5, i % 5);
    double* df = a.dst + (size_t)i * plane + v;
    *df -= a.omega * (*df - feq);
    if (two) {
      double* dg = a.dst + (size_t)(kQ3 + i) * plane + v;
      *dg -= a.omega * (*dg - a.K * theta * feq);
    }
  }
  if (!(rho > 0.0 && theta > 0.0 && isfinite(rho) && isfinite(theta))) atomicOr(a.flag, 1);
}

// Index j of an axis of n vertices, wrapped once on periodic axes: stencil nodes lie within one
// period of the vertex (the departure displacement is far below the domain length).
__device__ __forceinline__ int wrap1(int j, int n, int periodic) {
  if (!periodic) return j;
  return j < 0 ? j + n : (j >= n ? j - n : j);
}


// Fused FP32 step, one thread per vertex, one launch.  First sweep: every velocity's (f, g) pair
// is interpolated at its departure point (tensor product of the three 1D Lagrange bases, each in
// the difference form v_0 + sum_{k>=1} w_k (v_k - v_0), which keeps constant fields exact) and
// written to the destination, and its moments are summed.  Second sweep: the thread reads its
// own 125 pairs back (from L1/L2: no second pass over HBM), relaxes them toward the factorised
// equilibrium and sums the residual moments of (f^eq - f); the residuals (the FP32 rounding of
// the equilibrium) are then removed at the rest velocity and at (s, 0, 0), (0, s, 0), (0, 0, s)
// for mass and momentum, and on g at the rest velocity for the energy.
// Two forms. Grids of one wave (4 blocks an SM): the registers go to the (p+1)^3 gathers in flight, which
// such a grid waits for, and f^eq - w is summed by order (18 x 22 x 28 vertices, p = 2:
// 109 us a step, 130 in the other form; 20 x 36 x 80, p = 4: 458 and 595).  Larger grids (no bound): more warps
// share L1 and L2, and the nested sum, whose products hide the loads of the second sweep, is the
// faster one (96^3, p = 4, departures beyond the neighbouring cells: 6.10 ms, 6.33 with the sum by order and 7 blocks).
// Neither forms the leading 1 of the sum and takes it off afterwards: that left its rounding on every
// value (44^3, deviations of 1e-4 of the weights: 6e-3 of the largest deviation in one step, 3e-6 now).
template <int P, int BLOCKS>
__global__ void __launch_bounds__(128, BLOCKS) step3d_f32_kernel(const __grid_constant__ Step3F32Args a) {
  const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= a.nv) return;
  const int ix = (int)(v % a.nx);
  const long long t = v / a.nx;
  const int iy = (int)(t % a.ny), iz = (int)(t / a.ny);
  const size_t plane = (size_t)a.nv;
  float drho = 0.f, jx = 0.f, jy = 0.f, jz = 0.f, a2 = 0.f, G = 0.f;
#pragma unroll 1
  for (int i = 0; i < kQ3; ++i) {
    const int ia = i / 25, ib = (i / 5) % 5, ic = i % 5;
    const int sx = ix + a.offx[ia * a.nx + ix], sy = iy + a.offy[ib * a.ny + iy],
              sz = iz + a.offz[ic * a.nz + iz];
    const float* wx = a.wx + (size_t)(ia * a.nx + ix) * (P + 1);
    const float* wy = a.wy + (size_t)(ib * a.ny + iy) * (P + 1);
    const float* wz = a.wz + (size_t)(ic * a.nz + iz) * (P + 1);
    const float2* pl = a.src + (size_t)i * plane;
    int cx[P + 1], cy[P + 1], cz[P + 1];
#pragma unroll
    for (int k = 0; k <= P; ++k) {
      cx[k] = wrap1(sx + k, a.nx, a.px);
      cy[k] = wrap1(sy + k, a.ny, a.py);
      cz[k] = wrap1(sz + k, a.nz, a.pz);
    }
    float2 zs[P + 1];
#pragma unroll
    for (int kc = 0; kc <= P; ++kc) {
      const size_t zoff = (size_t)cz[kc] * a.ny;
      float2 ys[P + 1];
#pragma unroll
      for (int kb = 0; kb <= P; ++kb) {
        const float2* row = pl + (zoff + (size_t)cy[kb]) * a.nx;
        const float2 b0 = __ldg(row + cx[0]);
        float2 acc = b0;
#pragma unroll
        for (int ka = 1; ka <= P; ++ka) acc = fma2(bcast2(__ldg(wx + ka)), sub2(__ldg(row + cx[ka]), b0), acc);
        ys[kb] = acc;
      }
      float2 acc = ys[0];
#pragma unroll
      for (int kb = 1; kb <= P; ++kb) acc = fma2(bcast2(__ldg(wy + kb)), sub2(ys[kb], ys[0]), acc);
      zs[kc] = acc;
    }
    float2 acc = zs[0];
#pragma unroll
    for (int kc = 1; kc <= P; ++kc) acc = fma2(bcast2(__ldg(wz + kc)), sub2(zs[kc], zs[0]), acc);
    a.dst[(size_t)i * plane + v] = acc;
    const float ex = a.cs.xif[ia], ey = a.cs.xif[ib], ez = a.cs.xif[ic];
    drho += acc.x;
    jx += ex * acc.x;
    jy += ey * acc.x;
    jz += ez * acc.x;
    a2 += (ex * ex + ey * ey + ez * ez) * acc.x;
    G += acc.y;
  }
  if (a.npop != 2) G = 0.f;
  const float rho = 1.f + drho, inv_rho = __frcp_rn(rho);
  const float ux = jx * inv_rho, uy = jy * inv_rho, uz = jz * inv_rho;
  // theta - 1 = (A2 + G - rho |u|^2 - 2 C_v drho) / (2 C_v rho)   (sum w |xi|^2 + K = 2 C_v)
  const float qk = (a2 + G - rho * (ux * ux + uy * uy + uz * uz) - 2.f * a.cv * drho) * inv_rho * a.inv2cv;
  const float q = a.iso ? 0.f : qk;
  // per-axis factors X_k(a) = A_k(u_x) he_k(a), Y_l(b) likewise, and Zc_n(c) = sum_{1 <= m <= n}
  // A_m(u_z) he_m(c): S_abc = sum_{k + l + m <= 4} X_k(a) Y_l(b) Z_m(c) - 1 = sum_n C_n (1 + Zc_n(c)) - 1
  // with C_n = sum_{k + l = 4 - n} X_k(a) Y_l(b), C_4 = 1, without forming the leading 1; and
  // f^eq - w = w (drho + rho S)
  float Ax[5], Ay[5], Az[5];
  {
    const float u3[3] = {ux, uy, uz};
    float* A3[3] = {Ax, Ay, Az};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float u = u3[d];
      A3[d][0] = 1.f;
      A3[d][1] = u;
      A3[d][2] = u * u + q;
      A3[d][3] = u * (u * u + 3.f * q);
      A3[d][4] = u * u * (u * u + 6.f * q) + 3.f * q * q;
    }
  }
  // (nested: sum_k X_k sum_l Y_l (1 + Zc_{4-k-l}), the term k = l = 0 being Zc_4 alone)
  float Zc[5][5], Z4[5];   // [n][c] and Zc_4, compile-time indices only (nested: 1 + Zc_n)
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    float acc = 0.f, z = 0.f;
    if constexpr (BLOCKS == 4) Zc[0][c] = 0.f;
#pragma unroll
    for (int m = BLOCKS == 4 ? 1 : 0; m < 5; ++m) {
      acc += Az[m] * a.cs.hef[m][c];
      if (m > 0) z += Az[m] * a.cs.hef[m][c];
      Zc[m][c] = acc;
    }
    Z4[c] = z;
  }
  const float om = a.omega, Kq1 = a.K * (1.f + q), Kq = a.K * q;
  const float2 om2 = bcast2(om);
  float r0 = 0.f, r1 = 0.f, r2 = 0.f, r3 = 0.f, re = 0.f;
#pragma unroll 1
  for (int ia = 0; ia < kQ1; ++ia) {
    float Xa[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) Xa[k] = Ax[k] * a.cs.hef[k][ia];
    const float ex = a.cs.xif[ia], wa = a.cs.wf[ia];
#pragma unroll 1
    for (int ib = 0; ib < kQ1; ++ib) {
      float Yb[5];
#pragma unroll
      for (int l = 0; l < 5; ++l) Yb[l] = Ay[l] * a.cs.hef[l][ib];
      const float ey = a.cs.xif[ib], wab = wa * a.cs.wf[ib];
      const float C3 = Xa[1] + Yb[1], C2 = Xa[2] + Yb[2] + Xa[1] * Yb[1],
                  C1 = Xa[3] + Yb[3] + Xa[2] * Yb[1] + Xa[1] * Yb[2],
                  C0 = Xa[4] + Yb[4] + Xa[3] * Yb[1] + Xa[1] * Yb[3] + Xa[2] * Yb[2];
      const float Cs = C0 + C1 + C2 + C3;
#pragma unroll
      for (int ic = 0; ic < kQ1; ++ic) {
        const int i = 25 * ia + 5 * ib + ic;
        float em1;
        if constexpr (BLOCKS == 4) {
          em1 = fmaf(C1, Zc[1][ic], fmaf(C2, Zc[2][ic], fmaf(C3, Zc[3][ic], Cs + Z4[ic])));
        } else {
          em1 = 0.f;
#pragma unroll
          for (int k = 0; k <= 4; ++k) {
            float sl = k == 0 ? Z4[ic] : 0.f;
#pragma unroll
            for (int l = k == 0 ? 1 : 0; l <= 4 - k; ++l) sl += Yb[l] * Zc[4 - k - l][ic];
            em1 += Xa[k] * sl;
          }
        }
        const float w = wab * a.cs.wf[ic];
        const float ef = w * fmaf(rho, em1, drho);
        const float eg = Kq1 * ef + Kq * w;   // g^eq - K w = K ((1 + q)(f^eq - w) + q w)
        float2* o = a.dst + (size_t)i * plane + v;
        const float2 fg = *o;
        const float2 d = sub2(make_float2(ef, a.npop == 2 ? eg : 0.f), fg);
        const float ez = a.cs.xif[ic];
        r0 += d.x;
        r1 += ex * d.x;
        r2 += ey * d.x;
        r3 += ez * d.x;
        re += (ex * ex + ey * ey + ez * ez) * d.x + d.y;
        *o = fma2(om2, d, fg);
      }
    }
  }
  {   // remove the residuals (see above): i = 25 a + 5 b + c; s = xi of index 1
    const float inv_s = a.cs.inv_xi1f, s2 = a.cs.xi1sqf;
    const float d1 = r1 * inv_s, d2 = r2 * inv_s, d3 = r3 * inv_s;
    const float d0 = r0 - d1 - d2 - d3;
    const float de = re - s2 * (d1 + d2 + d3);
    float2* o = a.dst + v;
    o[0].x -= om * d0;
    o[25 * plane].x -= om * d1;
    o[5 * plane].x -= om * d2;
    o[1 * plane].x -= om * d3;
    if (a.npop == 2) {
      o[0].y -= om * de;
    } else if (!a.iso) {   // one population: energy along (+-s, 0, 0) and -2 at rest
      const float e = om * 0.5f * de * inv_s * inv_s;
      o[25 * plane].x -= e;
      o[75 * plane].x -= e;
      o[0].x += 2.f * e;
    }
  }
  if (!((rho > 0.f) && (qk > -1.f) && isfinite(rho) && isfinite(qk))) atomicOr(a.flag, 1);
}

// ---- sum-factorised FP32 step ----
//
// Two launches a step.  stream3d_kernel: a CTA takes a tile of 32 x 8 x TZ vertices and walks the
// 125 velocity planes; per plane one TMA tensor copy brings the source region (the tile and the
// stencil halo: XO = p rounded up to even columns on both sides in x, p in y and z) into a ring of
// NS stages.  The state keeps ghost cells on every axis, holding the periodic images on periodic
// axes (zero, and never read by an interior vertex, on zero-gradient ones), so a region never
// wraps.  The interpolation is sum-factorised: z pass over the region's (y, x) columns, y pass
// over the tile's z and the region's x, x pass into the destination, each in a centred tail-sum
// form
//   sum_d W_d v_{c+d} = v_c + sum_{j=1..p} T+_j (v_{c+j} - v_{c+j-1}) - sum_{j=1..p} T-_j (v_{c-j+1} - v_{c-j}),
//   T+_j = sum_{d >= j} W_d, T-_j = sum_{d <= -j} W_d  (d the offset from the vertex, W_d its weight),
// equal to the Lagrange sum because the weights sum to one and exact for constant fields in FP32.
// The passes are pipelined over the planes: phase i runs the z pass of plane i, the y pass of plane
// i - 1 and the x pass of plane i - 2, on double-buffered results, so a phase has one barrier and
// three independent pieces of work in place of three dependent ones with a barrier each.  In the x
// pass a thread takes two neighbouring vertices: their common window comes in 16-byte loads, and
// the two results leave in one 16-byte store.  The thread sums its vertices' moments over the 125
// planes.  collide3d_kernel then relaxes every vertex's 125 pairs in place and writes the periodic
// images of the vertices next to periodic faces.  On grids of few tiles five CTAs share a tile's planes
// (stream3d_parts).
//
// What bounds it: the latency of the phases and shared memory together (64^3: the LSU pipe at 65 %,
// issue at 39 %; 128^3: 1.187 ms, 1.38 ms with three barriers a plane and one vertex a task).  Deeper
// tiles (32 x 8 x 8, three stages, one CTA of 512 threads) take the same time; 24 warps an SM on
// tiles of 3 or 2 slices take 1.50 and 1.44 ms, as their regions grow.  250 values a vertex rule out a
// collision in registers, so the two kernels move 16 bytes an update.
constexpr int kT3X = 32, kT3Y = 8;

// Tile depth, threads and stages by order.
template <int P>
struct T3Config {
  static constexpr int TZ = 4, NT = P <= 2 ? 256 : 512, NS = 2, MINB = P <= 2 ? 2 : 1;
};

template <int P>
struct T3Shape {
  using C = T3Config<P>;
  static constexpr int TZ = C::TZ, NT = C::NT, NS = C::NS;
  static constexpr int XO = (P + 1) / 2 * 2;   // the region starts at x0 - XO: 16-byte aligned
  static constexpr int RX = kT3X + 2 * XO, RY = kT3Y + 2 * P, RZ = TZ + 2 * P;
  static constexpr int RE = RX * RY * RZ;   // region pairs
  static constexpr int NW = 2 * P;          // tail sums per (component, node): T+_1..p, -T-_1..p
  static constexpr int ZT = RY * RX;        // z-pass columns
  static constexpr int YT = TZ * RX;        // y-pass columns
  // slices of the z and y results, padded so that the columns of a warp that crosses from one slice
  // to the next go on over the shared-memory banks as in one row (16 pairs)
  static constexpr int ZS = RY * RX + ((RX - RY * RX) % 16 + 16) % 16, YS = kT3Y * RX + ((RX - kT3Y * RX) % 16 + 16) % 16;
  static constexpr int ZB = TZ * ZS, YB = TZ * YS;   // pairs of one z / y result
  static constexpr int NWT = kQ1 * (TZ + kT3Y + kT3X) * NW;   // the tile's tail sums
  static constexpr size_t kStage = sizeof(float2) * RE;
  static constexpr size_t kStride = (kStage + 127) / 128 * 128;
  static constexpr size_t kBytes = 128 + NS * kStride + sizeof(float2) * 2 * (size_t)(ZB + YB) +
                                   sizeof(float) * NWT + sizeof(uint64_t) * NS;
  static constexpr int XT = kT3X / 2 * kT3Y * TZ / NT;   // x-pass tasks (two vertices each) per thread
  static_assert(YT <= NT && XT * NT == kT3X / 2 * kT3Y * TZ, "one y column a thread at most, x tasks split evenly");
  static_assert((sizeof(float2) * (ZB + YB)) % 16 == 0 && NWT % 2 == 0, "16-byte rows, 8-byte barriers");
  static constexpr int G = XO;   // ghost cells of the state on every axis
};

struct Stream3Args {
  const float2* src;     // pairs in layout lay (deviations)
  float2* dst;
  Pad3 lay;
  float* sums;           // [parts][6][nv]: sum f, sum f xi_x, sum f xi_y, sum f xi_z, sum f |xi|^2, sum g
  int nx, ny, nz;
  long long nv;
  const float* tx;       // [5][nx][2p] tail sums per (component, node)
  const float* ty;
  const float* tz;
  Consts cs;
  int* flag;             // bit 2: a staging copy timed out
};

// centred tail-sum interpolation at window position c (see above); w = T+_1..p, -T-_1..p
template <int P, int N>
__device__ __forceinline__ float2 tail_interp(const float2 (&v)[N], const float2 (&d)[N - 1], int c, const float* w) {
  float2 acc = v[c];
#pragma unroll
  for (int j = 1; j <= P; ++j) {
    acc = fma2(bcast2(w[j - 1]), d[c + j - 1], acc);
    acc = fma2(bcast2(w[P + j - 1]), d[c - j], acc);
  }
  return acc;
}

// NPL: the planes of a CTA, 125 or those of the x component blockIdx.y (25).
template <int P, int NPL>
__global__ void __launch_bounds__(T3Config<P>::NT, T3Config<P>::MINB)
    stream3d_kernel(const __grid_constant__ Stream3Args a, const __grid_constant__ CUtensorMap smap) {
  using SH = T3Shape<P>;
  constexpr int TZ = SH::TZ, NT = SH::NT, NS = SH::NS, XO = SH::XO;
  constexpr int RX = SH::RX, RY = SH::RY, RZ = SH::RZ, NW = SH::NW, XT = SH::XT;
  extern __shared__ unsigned char s3_smem[];
  unsigned char* base = s3_smem + ((128 - (smem_u32(s3_smem) & 127)) & 127);
  float2* Zb = reinterpret_cast<float2*>(base + NS * SH::kStride);      // [2][TZ][RY][RX] (slices ZS apart), after the stages
  float2* Yb = Zb + 2 * SH::ZB;                                        // [2][TZ][TY][RX] (slices YS apart)
  float* Wz = reinterpret_cast<float*>(Yb + 2 * SH::YB);               // [5][TZ][NW]
  float* Wy = Wz + kQ1 * TZ * NW;                                      // [5][TY][NW]
  float* Wx = Wy + kQ1 * kT3Y * NW;                                    // [5][TX][NW]
  uint64_t* BAR = reinterpret_cast<uint64_t*>(Wx + kQ1 * kT3X * NW);   // [NS]
  const int tid = threadIdx.x;
  const int tiles_x = (a.nx + kT3X - 1) / kT3X, tiles_y = (a.ny + kT3Y - 1) / kT3Y;
  const int byz = (int)blockIdx.x / tiles_x, first = NPL * (int)blockIdx.y;   // this CTA's planes
  const int x0 = ((int)blockIdx.x - byz * tiles_x) * kT3X, y0 = (byz % tiles_y) * kT3Y,
            z0 = (byz / tiles_y) * TZ;
  // the tile's tail sums of all components (nodes past the grid clamped: those outputs are not
  // stored)
  for (int e = tid; e < SH::NWT; e += NT) {
    const int q = e % NW, r = e / NW;
    float t;
    if (r < kQ1 * TZ) {
      const int c = r / TZ, n = min(z0 + r - c * TZ, a.nz - 1);
      t = __ldg(a.tz + ((size_t)c * a.nz + n) * NW + q);
    } else if (r < kQ1 * (TZ + kT3Y)) {
      const int r2 = r - kQ1 * TZ, c = r2 / kT3Y, n = min(y0 + r2 - c * kT3Y, a.ny - 1);
      t = __ldg(a.ty + ((size_t)c * a.ny + n) * NW + q);
    } else {
      const int r2 = r - kQ1 * (TZ + kT3Y), c = r2 / kT3X, n = min(x0 + r2 - c * kT3X, a.nx - 1);
      t = __ldg(a.tx + ((size_t)c * a.nx + n) * NW + q);
    }
    Wz[e] = t;   // Wz, Wy and Wx are consecutive
  }
  if (tid == 0) {
    for (int k = 0; k < NS; ++k) mbar_init(&BAR[k], 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();
  // region origin in the ghost-padded layout (g = XO): x0 (x in floats: 2 x0, a multiple of 4, i.e.
  // 16 bytes), y0 - p + g, z0 - p + g
  const int cx = 2 * (x0 - XO + a.lay.g), cy = y0 - P + a.lay.g, cz = z0 - P + a.lay.g;
  auto issue = [&](int i, int st) {   // thread 0: this CTA's plane i into stage st
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    mbar_expect_tx(&BAR[st], (unsigned)SH::kStage);
    tma_load_4d(base + (size_t)st * SH::kStride, &smap, cx, cy, cz, first + i, &BAR[st]);
  };
  if (tid == 0)
    for (int k = 0; k < NS - 1; ++k) issue(k, k);
  // y pass: this thread's column (tz, rx); the last threads of the CTA, as the first ones have the
  // most z columns
  const int yt = tid - (NT - SH::YT);
  const int ytz = yt < 0 ? 0 : yt / RX, ycol = yt < 0 ? 0 : yt - ytz * RX;
  // x pass: task r = tid + k NT is the vertices x0 + 2 (r % 16) and the next one of tile row
  // r / 16 (z = row / TY, y = row % TY)
  const int xp = tid & 15;
  const int vx = x0 + 2 * xp;
  float2* out[XT];   // destination of the tasks, advancing plane by plane
  bool on[XT];
#pragma unroll
  for (int k = 0; k < XT; ++k) {
    const int row = (tid + k * NT) >> 4, vy = y0 + row % kT3Y, vz = z0 + row / kT3Y;
    on[k] = vx < a.nx && vy < a.ny && vz < a.nz;
    out[k] = a.dst + a.lay.at(first, vx, vy, vz);
  }
  const bool both = vx + 1 < a.nx;   // an odd x count ends with half a task
  // per vertex: (sum f, sum g), sum f xi_y, sum f xi_z, sum f (xi_y^2 + xi_z^2); over the planes of
  // one x component (f alone), and over all
  float2 fg[XT][2], part[XT][2];
  float my[XT][2], mz[XT][2], m2[XT][2], mx[XT][2];
#pragma unroll
  for (int k = 0; k < XT; ++k)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      fg[k][v] = part[k][v] = make_float2(0.f, 0.f);
      my[k][v] = mz[k][v] = m2[k][v] = mx[k][v] = 0.f;
    }
  float wx[2][NW];
  int st = 0, par = 0;          // stage of plane i and the parity of its phase
  int zc = 0, yb = 0, yc = 0;   // component of the z pass (plane i); of the y pass (plane i - 1)
  int xa = first / 25, xb = 0, xc = 0;   // components of the x pass (plane i - 2)
#pragma unroll 1
  for (int i = 0; i < NPL + 2; ++i) {
    const bool late = i < NPL && !mbar_wait(&BAR[st], (unsigned)par, a.flag);
    if (__syncthreads_or(late)) {
      // the copy of plane i did not land in time: stop, after it and the ones issued behind it
      for (int k = i, s2 = st, p2 = par; k < i + NS - 1 && k < NPL; ++k) {
        if (!mbar_wait(&BAR[s2], (unsigned)p2, a.flag)) break;
        if (++s2 == NS) {
          s2 = 0;
          p2 ^= 1;
        }
      }
      return;
    }
    if (tid == 0 && i + NS - 1 < NPL) issue(i + NS - 1, st == 0 ? NS - 1 : st - 1);   // every thread is past plane i - 1
    // z pass of plane i: column (ry, rx) of the region, the tile's z rows
    if (i < NPL) {
      constexpr int ZR = (SH::ZT + NT - 1) / NT;
      const float2* Sst = reinterpret_cast<const float2*>(base + (size_t)st * SH::kStride);
      float2* zout = Zb + (i & 1) * SH::ZB;
      float wz[TZ * NW];
#pragma unroll
      for (int q = 0; q < TZ * NW; ++q) wz[q] = Wz[zc * TZ * NW + q];
#pragma unroll
      for (int c = 0; c < ZR; ++c) {
        const int t = tid + c * NT;
        if (t < SH::ZT) {
          if (zc == 0) {   // at rest along z: the vertex's own slice
#pragma unroll
            for (int tz = 0; tz < TZ; ++tz) zout[tz * SH::ZS + t] = Sst[(tz + P) * RY * RX + t];
            continue;
          }
          float2 v[RZ], d[RZ - 1];
#pragma unroll
          for (int r = 0; r < RZ; ++r) v[r] = Sst[r * RY * RX + t];
#pragma unroll
          for (int r = 0; r + 1 < RZ; ++r) d[r] = sub2(v[r + 1], v[r]);
#pragma unroll
          for (int tz = 0; tz < TZ; ++tz) zout[tz * SH::ZS + t] = tail_interp<P>(v, d, tz + P, wz + tz * NW);
        }
      }
      if (++st == NS) {
        st = 0;
        par ^= 1;
      }
      if (++zc == kQ1) zc = 0;
    }
    // y pass of plane i - 1: column (tz, rx), the tile's y rows
    if (i >= 1 && i <= NPL) {
      if (yt >= 0) {
        const float* wy = Wy + yb * kT3Y * NW;
        const float2* zin = Zb + ((i - 1) & 1) * SH::ZB + ytz * SH::ZS + ycol;
        float2* yout = Yb + ((i - 1) & 1) * SH::YB + ytz * SH::YS + ycol;
        if (yb == 0) {   // at rest along y
#pragma unroll
          for (int ty = 0; ty < kT3Y; ++ty) yout[ty * RX] = zin[(ty + P) * RX];
        } else {
          float2 v[RY], d[RY - 1];
#pragma unroll
          for (int r = 0; r < RY; ++r) v[r] = zin[r * RX];
#pragma unroll
          for (int r = 0; r + 1 < RY; ++r) d[r] = sub2(v[r + 1], v[r]);
#pragma unroll
          for (int ty = 0; ty < kT3Y; ++ty) yout[ty * RX] = tail_interp<P>(v, d, ty + P, wy + ty * NW);
        }
      }
      if (++yc == kQ1) {
        yc = 0;
        if (++yb == kQ1) yb = 0;
      }
    }
    // x pass of plane i - 2: two neighbouring vertices a task, into the destination; their moments
    if (i >= 2) {
      if (xb == 0 && xc == 0) {   // a new x component: the tail sums of this thread's columns
#pragma unroll
        for (int q = 0; q < NW; ++q) {
          wx[0][q] = Wx[(xa * kT3X + 2 * xp) * NW + q];
          wx[1][q] = Wx[(xa * kT3X + 2 * xp + 1) * NW + q];
        }
      }
      const float ey = a.cs.xif[xb], ez = a.cs.xif[xc], e2 = ey * ey + ez * ez;
#pragma unroll
      for (int k = 0; k < XT; ++k) {
        const int row = (tid + k * NT) >> 4;
        const float4* in = reinterpret_cast<const float4*>(Yb + (i & 1) * SH::YB + (row / kT3Y) * SH::YS +
                                                           (row % kT3Y) * RX + 2 * xp);
        float2 r0, r1;
        if (xa == 0) {   // at rest along x
          const float4 q = in[XO / 2];
          r0 = make_float2(q.x, q.y);
          r1 = make_float2(q.z, q.w);
        } else {
          float2 v[2 * XO + 2], d[2 * XO + 1];
#pragma unroll
          for (int j = 0; j <= XO; ++j) {
            const float4 q = in[j];
            v[2 * j] = make_float2(q.x, q.y);
            v[2 * j + 1] = make_float2(q.z, q.w);
          }
#pragma unroll
          for (int j = 0; j < 2 * XO + 1; ++j) d[j] = sub2(v[j + 1], v[j]);
          r0 = tail_interp<P>(v, d, XO, wx[0]);
          r1 = tail_interp<P>(v, d, XO + 1, wx[1]);
        }
        if (on[k]) {
          if (both)
            *reinterpret_cast<float4*>(out[k]) = make_float4(r0.x, r0.y, r1.x, r1.y);
          else
            *out[k] = r0;
        }
        out[k] += a.lay.plane;
        const float2 r[2] = {r0, r1};
#pragma unroll
        for (int v2 = 0; v2 < 2; ++v2) {
          part[k][v2] = __fadd2_rn(part[k][v2], r[v2]);
          my[k][v2] = fmaf(ey, r[v2].x, my[k][v2]);
          mz[k][v2] = fmaf(ez, r[v2].x, mz[k][v2]);
          m2[k][v2] = fmaf(e2, r[v2].x, m2[k][v2]);
        }
      }
      if (++xc == kQ1) {
        xc = 0;
        if (++xb == kQ1) {   // the planes of one x component are done
          xb = 0;
          const float ex = a.cs.xif[xa];
#pragma unroll
          for (int k = 0; k < XT; ++k)
#pragma unroll
            for (int v2 = 0; v2 < 2; ++v2) {
              fg[k][v2] = __fadd2_rn(fg[k][v2], part[k][v2]);
              mx[k][v2] = fmaf(ex, part[k][v2].x, mx[k][v2]);
              m2[k][v2] = fmaf(ex * ex, part[k][v2].x, m2[k][v2]);
              part[k][v2] = make_float2(0.f, 0.f);
            }
          ++xa;
        }
      }
    }
  }
#pragma unroll
  for (int k = 0; k < XT; ++k) {
    const int row = (tid + k * NT) >> 4, vy = y0 + row % kT3Y, vz = z0 + row / kT3Y;
    if (!on[k]) continue;
    const size_t v = ((size_t)vz * a.ny + vy) * a.nx + vx;
#pragma unroll
    for (int v2 = 0; v2 < 2; ++v2) {
      if (v2 == 1 && !both) continue;
      const float m[6] = {fg[k][v2].x, mx[k][v2], my[k][v2], mz[k][v2], m2[k][v2], fg[k][v2].y};
#pragma unroll
      for (int q = 0; q < 6; ++q) a.sums[(size_t)(6 * blockIdx.y + q) * a.nv + v + v2] = m[q];
    }
  }
}

// Second sweep of the sum-factorised step: one thread per vertex relaxes its 125 pairs in place
// (read back from the destination), from the moment sums of the stream kernel, with the residual
// correction of step3d_f32_kernel, and writes them to the periodic images of the vertex in the
// ghost cells as well.  It moves 16 bytes an update, at 4.9 TB/s on 128^3 vertices (0.919 ms, with
// rows of 5 pairs asked for two rows ahead in five blocks an SM; one row ahead in six: 1.011 ms; the
// copying of the images was a launch of 0.18 ms of its own).  Per row (a, b) the products
// X_k(a) Y_l(b) are summed by order first, so that a velocity takes 5 multiply-adds.
struct Collide3Args {
  float2* dst;
  Pad3 lay;
  const float* sums;
  int parts;             // of the moment sums
  int nx, ny, nz, px, py, pz;
  long long nv;
  Consts cs;
  float omega, K, cv, inv2cv;
  int npop, iso;
  int* flag;
};

__global__ void __launch_bounds__(128, 5) collide3d_kernel(const __grid_constant__ Collide3Args a) {
  const unsigned v = blockIdx.x * 128u + threadIdx.x;   // at most 2^27 vertices
  if (v >= (unsigned)a.nv) return;
  const unsigned yz = v / (unsigned)a.nx;
  const int x = (int)(v - yz * (unsigned)a.nx), z = (int)(yz / (unsigned)a.ny), y = (int)(yz - (unsigned)z * (unsigned)a.ny);
  // value i of this vertex: the plane's address (the same for all threads) and the vertex's offset
  // in a plane
  char* const base = reinterpret_cast<char*>(a.dst);
  const size_t plane = a.lay.plane * sizeof(float2);
  const size_t off = a.lay.at(0, x, y, z) * sizeof(float2);
  auto at = [&](int i) { return reinterpret_cast<float2*>(base + (size_t)i * plane + off); };
  // the vertex's periodic images in the ghost cells (axes are at least two ghost widths long: one
  // image an axis).  The x image is one predicated store, since half the warps hold some; the others
  // are whole rows and slices, behind a branch that few warps take.
  const int g = a.lay.g;
  const int dx = !a.px ? 0 : x < g ? a.nx : x >= a.nx - g ? -a.nx : 0;
  const int dy = !a.py ? 0 : y < g ? a.ny : y >= a.ny - g ? -a.ny : 0;
  const int dz = !a.pz ? 0 : z < g ? a.nz : z >= a.nz - g ? -a.nz : 0;
  const int sy = a.lay.pitch * dy, sz = a.lay.pitch * a.lay.rows * dz;   // below a plane: < 2^31 pairs
  auto put = [&](int i, float2 val) {
    float2* o = at(i);
    *o = val;
    if (dx) o[dx] = val;
    if (dy | dz) {
      if (dy) {
        o[sy] = val;
        if (dx) o[sy + dx] = val;
      }
      if (dz) {
        o[sz] = val;
        if (dx) o[sz + dx] = val;
        if (dy) {
          o[sz + sy] = val;
          if (dx) o[sz + sy + dx] = val;
        }
      }
    }
  };
  float2 cur[kQ1], nxt[kQ1];
#pragma unroll
  for (int ic = 0; ic < kQ1; ++ic) cur[ic] = *at(ic);
#pragma unroll
  for (int ic = 0; ic < kQ1; ++ic) nxt[ic] = *at(kQ1 + ic);
  const size_t sp = (size_t)a.nv;
  float mom[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) mom[q] = a.sums[q * sp + v];
  for (int k = 1; k < a.parts; ++k)
#pragma unroll
    for (int q = 0; q < 6; ++q) mom[q] += a.sums[(6 * k + q) * sp + v];
  const float drho = mom[0], jx = mom[1], jy = mom[2], jz = mom[3], a2 = mom[4], G = a.npop == 2 ? mom[5] : 0.f;
  const float rho = 1.f + drho, inv_rho = __frcp_rn(rho);
  const float ux = jx * inv_rho, uy = jy * inv_rho, uz = jz * inv_rho;
  const float qk = (a2 + G - rho * (ux * ux + uy * uy + uz * uz) - 2.f * a.cv * drho) * inv_rho * a.inv2cv;
  const float q = a.iso ? 0.f : qk;
  float Ax[5], Ay[5], Az[5];
  {
    const float u3[3] = {ux, uy, uz};
    float* A3[3] = {Ax, Ay, Az};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float u = u3[d];
      A3[d][0] = 1.f;
      A3[d][1] = u;
      A3[d][2] = u * u + q;
      A3[d][3] = u * (u * u + 3.f * q);
      A3[d][4] = u * u * (u * u + 6.f * q) + 3.f * q * q;
    }
  }
  // Zc[n][c] = sum_{1 <= m <= n} A_m(u_z) he_m(c): the sums to order n without their leading 1
  float Zc[5][5];
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    float acc = 0.f;
    Zc[0][c] = 0.f;
#pragma unroll
    for (int m = 1; m < 5; ++m) {
      acc += Az[m] * a.cs.hef[m][c];
      Zc[m][c] = acc;
    }
  }
  const float om = a.omega, Kq1 = a.K * (1.f + q), Kq = a.K * q;
  const float2 om2 = bcast2(om);
  const bool two = a.npop == 2;
  float r0 = 0.f, r1 = 0.f, r2 = 0.f, r3 = 0.f, re = 0.f, rg = 0.f;
#pragma unroll 1
  for (int row = 0; row < kQ1 * kQ1; ++row) {
    const int ia = row / kQ1, ib = row - kQ1 * ia;
    float2 aft[kQ1];   // two rows ahead
    if (row + 2 < kQ1 * kQ1) {
#pragma unroll
      for (int ic = 0; ic < kQ1; ++ic) aft[ic] = *at(kQ1 * (row + 2) + ic);
    }
    // C[n] = sum_{k + l = 4 - n} X_k(a) Y_l(b): E - 1 = sum_n C[n] (1 + Zc[n][c]) - 1, C[4] = 1
    float X[5], Y[5], C[4];
#pragma unroll
    for (int k = 1; k < 5; ++k) {
      X[k] = Ax[k] * a.cs.hef[k][ia];
      Y[k] = Ay[k] * a.cs.hef[k][ib];
    }
    C[3] = X[1] + Y[1];
    C[2] = X[2] + Y[2] + X[1] * Y[1];
    C[1] = X[3] + Y[3] + X[2] * Y[1] + X[1] * Y[2];
    C[0] = X[4] + Y[4] + X[3] * Y[1] + X[1] * Y[3] + X[2] * Y[2];
    const float Cs = C[0] + C[1] + C[2] + C[3];
    const float ex = a.cs.xif[ia], ey = a.cs.xif[ib], wab = a.cs.wf[ia] * a.cs.wf[ib];
    float rs = 0.f, rz = 0.f, rzz = 0.f;
#pragma unroll
    for (int ic = 0; ic < kQ1; ++ic) {
      float em1 = Cs + Zc[4][ic];
#pragma unroll
      for (int n = 1; n < 4; ++n) em1 = fmaf(C[n], Zc[n][ic], em1);
      const float w = wab * a.cs.wf[ic];
      const float ef = w * fmaf(rho, em1, drho);
      const float eg = Kq1 * ef + Kq * w;   // g^eq - K w = K ((1 + q)(f^eq - w) + q w)
      const float2 d = sub2(make_float2(ef, two ? eg : 0.f), cur[ic]);
      const float ez = a.cs.xif[ic];
      rs += d.x;
      rz = fmaf(ez, d.x, rz);
      rzz = fmaf(ez * ez, d.x, rzz);
      rg += d.y;
      const float2 val = fma2(om2, d, cur[ic]);
      put(kQ1 * row + ic, val);
    }
    r0 += rs;
    r1 = fmaf(ex, rs, r1);
    r2 = fmaf(ey, rs, r2);
    r3 += rz;
    re += fmaf(fmaf(ex, ex, ey * ey), rs, rzz);
#pragma unroll
    for (int ic = 0; ic < kQ1; ++ic) {
      cur[ic] = nxt[ic];
      nxt[ic] = aft[ic];
    }
  }
  {
    const float inv_s = a.cs.inv_xi1f, s2 = a.cs.xi1sqf;
    const float d1 = r1 * inv_s, d2 = r2 * inv_s, d3 = r3 * inv_s;
    const float d0 = r0 - d1 - d2 - d3;
    const float de = re + rg - s2 * (d1 + d2 + d3);
    // (held in registers to the end instead, these cost the fifth block: 0.956 ms against 0.919 on 128^3)
    float2 v0 = *at(0), v1 = *at(1), v5 = *at(5), v25 = *at(25), v75 = *at(75);
    v0.x -= om * d0;
    v25.x -= om * d1;
    v5.x -= om * d2;
    v1.x -= om * d3;
    if (two) {
      v0.y -= om * de;
    } else if (!a.iso) {   // one population: energy along (+-s, 0, 0) and -2 at rest
      const float e = om * 0.5f * de * inv_s * inv_s;
      v25.x -= e;
      v75.x -= e;
      v0.x += 2.f * e;
    }
    put(0, v0);
    put(1, v1);
    put(5, v5);
    put(25, v25);
    put(75, v75);
  }
  if (!((rho > 0.f) && (qk > -1.f) && isfinite(rho) && isfinite(qk))) atomicOr(a.flag, 1);
}

// The periodic images of the ghost cells of a padded pair state (after init and set_state), one
// thread per (plane, ghost cell).  The ghost cells of a plane are enumerated as three disjoint
// sets: the 2g slices before and after the interior slices (whole rows), then in the interior
// slices the 2g ghost rows, then in the interior rows the columns outside the interior.  A cell
// past a zero-gradient face, or in the row padding past the ghost columns, is skipped.
__global__ void __launch_bounds__(256) ghost_refresh3d_kernel(float2* pairs, Pad3 lay, int nx, int ny, int nz,
                                                              int px, int py, int pz, unsigned per_plane) {
  const unsigned e = blockIdx.x * 256u + threadIdx.x;
  if (e >= per_plane) return;
  const int i = blockIdx.y;
  unsigned r = e;
  const unsigned g = lay.g, W = lay.pitch, R = lay.rows, S = W - nx;   // S: columns outside the interior
  const unsigned nzs = 2 * g * R * W, nys = (unsigned)nz * 2 * g * W;
  int X, Y, Z;   // interior coordinates of the ghost cell (outside [0, n) on some axis)
  if (r < nzs) {
    const int zz = (int)(r / (R * W));
    r -= (unsigned)zz * R * W;
    Z = zz < (int)g ? zz - (int)g : nz + zz - (int)g;
    Y = (int)(r / W) - (int)g;
    X = (int)(r % W) - (int)g;
  } else if ((r -= nzs) < nys) {
    Z = (int)(r / (2 * g * W));
    r -= (unsigned)Z * 2 * g * W;
    const int yy = (int)(r / W);
    Y = yy < (int)g ? yy - (int)g : ny + yy - (int)g;
    X = (int)(r % W) - (int)g;
  } else {
    r -= nys;
    Z = (int)(r / ((unsigned)ny * S));
    r -= (unsigned)Z * ny * S;
    Y = (int)(r / S);
    const int xx = (int)(r % S);
    X = xx < (int)g ? xx - (int)g : nx + xx - (int)g;
  }
  if (X >= nx + (int)g) return;   // row padding
  const bool ox = X < 0 || X >= nx, oy = Y < 0 || Y >= ny, oz = Z < 0 || Z >= nz;
  if ((ox && !px) || (oy && !py) || (oz && !pz)) return;
  const int x = ox ? (X < 0 ? X + nx : X - nx) : X, y = oy ? (Y < 0 ? Y + ny : Y - ny) : Y,
            z = oz ? (Z < 0 ? Z + nz : Z - nz) : Z;
  pairs[lay.at(i, X, Y, Z)] = pairs[lay.at(i, x, y, z)];
}

// Tail sums T+_j, -T-_j (j = 1..p) of every (component, node) of one axis, from the FP64 tables:
// the stencil of node n starts at n + off and has weights w_0..w_p, offsets d = off + k.
template <int P>
__global__ void __launch_bounds__(128) tail_table_kernel(const int* off, const double* w, int n, float* out) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= kQ1 * n) return;
  double W[2 * P + 1];
#pragma unroll
  for (int d = 0; d <= 2 * P; ++d) W[d] = 0.0;
  const int o = off[e];
#pragma unroll
  for (int k = 0; k <= P; ++k)   // o + k is in [-P, P] (tiled3d_usable)
    if (o + k >= -P && o + k <= P) W[o + k + P] += w[(size_t)e * (P + 1) + k];
#pragma unroll
  for (int j = 1; j <= P; ++j) {
    double tp = 0.0, tm = 0.0;
    for (int d = j; d <= P; ++d) tp += W[d + P];
    for (int d = -P; d <= -j; ++d) tm += W[d + P];
    out[(size_t)e * 2 * P + j - 1] = (float)tp;
    out[(size_t)e * 2 * P + P + j - 1] = (float)(-tm);
  }
}

// FP32 pairs (layout lay) <-> dense FP64 full populations [npop][125][nv]: plane i = blockIdx.y, whose
// lattice weights the block forms once.  (With four FP64 products a value and FP64 conversions the
// FP64 pipe bound it: 2.94 ms for the 2.1 M vertices of 128^3, now 1.27 ms in and 1.31 out, 0.95 ms of it HBM traffic.)
constexpr int kConvPer = 4;   // vertices a thread
__global__ void __launch_bounds__(256) convert3d_kernel(float2* pairs, Pad3 lay, double* dense, int nx, int ny,
                                                        unsigned nv, int npop, double K, const __grid_constant__ Consts cs,
                                                        int to_dense) {
  __shared__ double ws[2];
  const int i = blockIdx.y;
  if (threadIdx.x == 0) {
    ws[0] = cs.w[i / 25] * cs.w[(i / 5) % 5] * cs.w[i % 5];
    ws[1] = K * ws[0];
  }
  __syncthreads();
  const double w = ws[0], Kw = ws[1];
  double *df = dense + (size_t)i * nv, *dg = dense + (size_t)(kQ3 + i) * nv;
  unsigned v[kConvPer];
  size_t o[kConvPer];
#pragma unroll
  for (int k = 0; k < kConvPer; ++k) {
    v[k] = (blockIdx.x * kConvPer + k) * 256u + threadIdx.x;
    const unsigned vk = min(v[k], nv - 1), yz = vk / (unsigned)nx, z = yz / (unsigned)ny;
    o[k] = lay.at(i, (int)(vk - yz * (unsigned)nx), (int)(yz - z * (unsigned)ny), (int)z);
  }
  if (to_dense) {
    float2 p[kConvPer];
#pragma unroll
    for (int k = 0; k < kConvPer; ++k) p[k] = pairs[o[k]];   // past the end: the last vertex again
#pragma unroll
    for (int k = 0; k < kConvPer; ++k)
      if (v[k] < nv) {
        df[v[k]] = exact_double(p[k].x) + w;
        if (npop == 2) dg[v[k]] = exact_double(p[k].y) + Kw;
      }
  } else {
    double f[kConvPer], g[kConvPer];
#pragma unroll
    for (int k = 0; k < kConvPer; ++k) {
      f[k] = df[min(v[k], nv - 1)];
      g[k] = npop == 2 ? dg[min(v[k], nv - 1)] : Kw;
    }
#pragma unroll
    for (int k = 0; k < kConvPer; ++k)
      if (v[k] < nv) pairs[o[k]] = make_float2(nearest_float(f[k] - w), nearest_float(g[k] - Kw));
  }
}

__global__ void init3d_kernel(const __grid_constant__ Field3Args a) {
  const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= a.nv) return;
  const double rho = a.rho[v], theta = a.T[v], q = theta - 1.0;
  double Ax[5], Ay[5], Az[5];
  hermite_moments(a.u[v], q, Ax);
  hermite_moments(a.v[v], q, Ay);
  hermite_moments(a.w[v], q, Az);
  const size_t plane = (size_t)a.nv;
  const int x = (int)(v % a.nx), y = (int)((v / a.nx) % a.ny), z = (int)(v / ((long long)a.nx * a.ny));
  for (int i = 0; i < kQ3; ++i) {
    const double feq = eq3(a.cs, rho, Ax, Ay, Az, i / 25, (i / 5) % 5, i % 5);
    if (a.state32) {
      const double w = a.cs.w[i / 25] * a.cs.w[(i / 5) % 5] * a.cs.w[i % 5];
      a.state32[a.lay.at(i, x, y, z)] =
          make_float2((float)(feq - w), a.npop == 2 ? (float)(a.K * theta * feq - a.K * w) : 0.f);
    } else {
      a.state[(size_t)i * plane + v] = feq;
      if (a.npop == 2) a.state[(size_t)(kQ3 + i) * plane + v] = a.K * theta * feq;
    }
  }
}

__global__ void moments3d_kernel(const __grid_constant__ Field3Args a) {
  const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= a.nv) return;
  const size_t plane = (size_t)a.nv;
  const int x = (int)(v % a.nx), y = (int)((v / a.nx) % a.ny), z = (int)(v / ((long long)a.nx * a.ny));
  double rho = 0.0, jx = 0.0, jy = 0.0, jz = 0.0, e2 = 0.0;
  for (int i = 0; i < kQ3; ++i) {
    double f, g;
    if (a.state32) {
      const float2 p = a.state32[a.lay.at(i, x, y, z)];
      const double w = a.cs.w[i / 25] * a.cs.w[(i / 5) % 5] * a.cs.w[i % 5];
      f = (double)p.x + w;
      g = a.npop == 2 ? (double)p.y + a.K * w : 0.0;
    } else {
      f = a.state[(size_t)i * plane + v];
      g = a.npop == 2 ? a.state[(size_t)(kQ3 + i) * plane + v] : 0.0;
    }
    const double cx = a.cs.xi[i / 25], cy = a.cs.xi[(i / 5) % 5], cz = a.cs.xi[i % 5];
    rho += f;
    jx += f * cx;
    jy += f * cy;
    jz += f * cz;
    e2 += f * (cx * cx + cy * cy + cz * cz) + g;
  }
  const double ux = jx / rho, uy = jy / rho, uz = jz / rho;
  const double theta = (e2 - rho * (ux * ux + uy * uy + uz * uz)) / (2.0 * a.cv * rho);
  if (a.orho) a.orho[v] = rho;
  if (a.ou) a.ou[v] = ux;
  if (a.ov) a.ov[v] = uy;
  if (a.ow) a.ow[v] = uz;
  if (a.oT) a.oT[v] = theta;
  if (!(rho > 0.0 && theta > 0.0 && isfinite(rho) && isfinite(theta))) atomicOr(a.flag, 1);
}

__global__ void coords3d_kernel(AxisK ax, AxisK ay, AxisK az, double* x, double* y, double* z) {
  const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nv = (long long)ax.nv * ay.nv * az.nv;
  if (v >= nv) return;
  const int ix = (int)(v % ax.nv);
  const long long t = v / ax.nv;
  x[v] = vertex_ref_coord(ix, ax);
  y[v] = vertex_ref_coord((int)(t % ay.nv), ay);
  z[v] = vertex_ref_coord((int)(t / ay.nv), az);
}

// D1Q5 in Table I order and he[k][a] = He_k(xi_a) / k! (recurrence He_{k+1} = x He_k - k He_{k-1}).
void d1q5_consts(Consts& cs) {
  cs = Consts{};
  const double s10 = sqrt(10.0), sm = sqrt(5.0 - s10), lg = sqrt(5.0 + s10);
  const double xi[5] = {0.0, sm, lg, -sm, -lg};
  const double w[5] = {8.0 / 15.0, (7.0 + 2.0 * s10) / 60.0, (7.0 - 2.0 * s10) / 60.0,
                       (7.0 + 2.0 * s10) / 60.0, (7.0 - 2.0 * s10) / 60.0};
  cs.nq1 = kQ1;
  for (int a = 0; a < kQ1; ++a) {
    cs.xi[a] = xi[a];
    cs.w[a] = w[a];
    double hm1 = 0.0, h = 1.0, fact = 1.0;
    for (int k = 0; k < kQ1; ++k) {
      if (k > 0) fact *= k;
      cs.he[k][a] = h / fact;
      const double hn = xi[a] * h - k * hm1;
      hm1 = h;
      h = hn;
    }
    cs.xif[a] = (float)xi[a];
    cs.wf[a] = (float)w[a];
    for (int k = 0; k < kQ1; ++k) {
      cs.hef[k][a] = (float)cs.he[k][a];
      cs.whf[k][a] = (float)(cs.w[a] * cs.he[k][a]);
    }
  }
  cs.inv_xi1f = (float)(1.0 / xi[1]);
  cs.xi1sqf = (float)(xi[1] * xi[1]);
}

void axis3(AxisK& ax, int n_cells, int p, double lo, double hi, int periodic, int nodes) {
  ax = AxisK{};
  ax.n_cells = n_cells;
  ax.p = p;
  ax.periodic = periodic;
  ax.nv = periodic ? n_cells * p : n_cells * p + 1;
  ax.lo = lo;
  ax.hi = hi;
  ax.len = hi - lo;
  ax.hc = (hi - lo) / n_cells;
  const double pi = 3.141592653589793238462643383279502884;
  for (int k = 0; k <= p; ++k)   // Gauss-Lobatto-Chebyshev points (Sec. II.E) or equidistant
    ax.nodes[k] = nodes == SLLBM_NODES_GLC ? 0.5 * (1.0 - cos(k * pi / p)) : (double)k / p;
}

}  // namespace

struct sllbm3d_ctx {
  sllbm_grid3_desc g;
  sllbm_params p;
  cudaStream_t stream = nullptr;
  AxisK ax{}, ay{}, az{};
  Consts cs{};
  int npop = 2;
  bool f32 = false;                      // FP32 deviation pairs (else FP64 full populations)
  int n_sm = 0;                          // of the device
  long long nv = 0;
  double* state[2] = {nullptr, nullptr}; // FP32: reinterpreted as float2 [125][nv]
  int cur = 0;
  bool precomputed = false, initialized = false;
  int* off[3] = {nullptr, nullptr, nullptr};
  float* w32[3] = {nullptr, nullptr, nullptr};
  double* w64[3] = {nullptr, nullptr, nullptr};
  // sum-factorised FP32 step: tail sums per axis, moment sums
  bool tiled = false;
  Pad3 lay{};                            // layout of the FP32 pair state
  float* tail[3] = {nullptr, nullptr, nullptr};
  float* sums = nullptr;                 // [parts][6][nv]
  int parts = 1;                         // CTAs a tile in stream3d_kernel, an x component each, or one
  int* flag = nullptr;
  std::vector<void*> allocations;
  std::string err;
};

namespace {

sllbm_status fail3(sllbm3d_ctx* c, sllbm_status s, const std::string& msg) {
  if (c) c->err = msg;
  return s;
}

sllbm_status cuda3(sllbm3d_ctx* c, cudaError_t e, const char* where) {
  if (e == cudaSuccess) return SLLBM_OK;
  return fail3(c, SLLBM_ERR_CUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

template <typename T>
sllbm_status alloc3(sllbm3d_ctx* c, T** ptr, size_t count) {
  void* p = nullptr;
  const cudaError_t e = cudaMalloc(&p, (count ? count : 1) * sizeof(T));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail3(c, SLLBM_ERR_OOM, std::string("cudaMalloc failed: ") + cudaGetErrorString(e));
  }
  c->allocations.push_back(p);
  *ptr = static_cast<T*>(p);
  return SLLBM_OK;
}

unsigned blocks_for(long long n, int threads) { return (unsigned)((n + threads - 1) / threads); }

// storage of one state buffer in 8-byte units: FP64 populations or FP32 (f, g) pairs
size_t state_doubles(const sllbm3d_ctx* c) {
  return c->f32 ? (size_t)kQ3 * c->lay.plane : (size_t)c->npop * kQ3 * c->nv;
}
float2* pairs(const sllbm3d_ctx* c, int k) { return reinterpret_cast<float2*>(c->state[k]); }

template <int P>
long long tiles3d(int nx, int ny, int nz) {
  return (long long)((nx + kT3X - 1) / kT3X) * ((ny + kT3Y - 1) / kT3Y) * ((nz + T3Config<P>::TZ - 1) / T3Config<P>::TZ);
}

// The sum-factorised FP32 step: stream3d_kernel then collide3d_kernel.
template <int P, int NPL>
cudaError_t launch_stream3d_planes(const Stream3Args& a, cudaStream_t s) {
  using SH = T3Shape<P>;
  EncodeTiledFn enc = encode_fn();
  if (!enc) return cudaErrorNotSupported;
  if (a.lay.g != SH::G || a.lay.pitch % 2) return cudaErrorInvalidValue;
  // 4D map of the ghost-padded source pairs as floats: (2 x column, row, slice, velocity plane)
  CUtensorMap smap;
  const cuuint64_t dims[4] = {(cuuint64_t)2 * a.lay.pitch, (cuuint64_t)a.lay.rows,
                              (cuuint64_t)(a.lay.plane / ((size_t)a.lay.pitch * a.lay.rows)), (cuuint64_t)kQ3};
  const cuuint64_t strides[3] = {(cuuint64_t)a.lay.pitch * sizeof(float2),
                                 (cuuint64_t)a.lay.pitch * a.lay.rows * sizeof(float2),
                                 (cuuint64_t)a.lay.plane * sizeof(float2)};
  const cuuint32_t box[4] = {(cuuint32_t)(2 * SH::RX), (cuuint32_t)SH::RY, (cuuint32_t)SH::RZ, 1u};
  const cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
  if (enc(&smap, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float2*>(a.src), dims, strides, box, estr,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(stream3d_kernel<P, NPL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::kBytes);
  if (e != cudaSuccess) return e;
  stream3d_kernel<P, NPL><<<dim3((unsigned)tiles3d<P>(a.nx, a.ny, a.nz), kQ3 / NPL), SH::NT, SH::kBytes, s>>>(a, smap);
  return cudaGetLastError();
}

template <int P>
cudaError_t launch_stream3d(const Stream3Args& a, int parts, cudaStream_t s) {
  return parts == kQ1 ? launch_stream3d_planes<P, kQ3 / kQ1>(a, s) : launch_stream3d_planes<P, kQ3>(a, s);
}

// Whether a tile's 125 planes go to five CTAs, an x component each (with moment sums of their own), or to one.
// A CTA runs one phase a plane and two more, at about 1 us each whatever the load: 127 phases a wave of
// tiles, or 27 a wave of parts, which is what grids of a few tiles wait for (36 x 12 x 8, p = 1: 129 -> 50 us a step,
// and 83 by the gather step; 49^3, p = 2: 230 -> 175; 64 x 32 x 32, p = 4: 216 -> 157).  Not where the tiles
// fill the device as they are (64^3, p = 2, 256 tiles on 304 places: 298, 311 in parts) or beyond two
// waves (128^3: 2.12 and 2.23 ms).
int stream3d_parts(const sllbm3d_ctx* c) {
  const int nx = c->ax.nv, ny = c->ay.nv, nz = c->az.nv;
  long long tiles = 0, places = c->n_sm;
  switch (c->g.order) {
    case 1: tiles = tiles3d<1>(nx, ny, nz); places *= T3Config<1>::MINB; break;
    case 2: tiles = tiles3d<2>(nx, ny, nz); places *= T3Config<2>::MINB; break;
    case 3: tiles = tiles3d<3>(nx, ny, nz); places *= T3Config<3>::MINB; break;
    default: tiles = tiles3d<4>(nx, ny, nz); places *= T3Config<4>::MINB; break;
  }
  auto waves = [&](long long n) { return (n + places - 1) / places; };
  return places > 0 && tiles <= 2 * places && (kQ3 / kQ1 + 2) * waves(kQ1 * tiles) < (kQ3 + 2) * waves(tiles) ? kQ1 : 1;
}

// Whether the sum-factorised step takes the grid: FP32, axes at least as long as a staged region of
// order 2 (36 x 12 x 8 vertices; also two ghost widths), and every stencil within p vertices of its vertex: from
// an inner node the departures stay in the cell, from a cell face they reach no further than the
// neighbouring cells.  At the least sizes it takes, by order: 50, 54, 60 (36 x 12 x 9) and 62 us a step
// (36 x 12 x 12); the gather step 83, 106, 168 and 295.
bool tiled3d_usable(const sllbm3d_ctx* c, double dt) {
  if (!c->f32 || encode_fn() == nullptr) return false;
  const AxisK* axes[3] = {&c->ax, &c->ay, &c->az};
  const int least[3] = {36, 12, 8};
  for (int k = 0; k < 3; ++k) {
    const AxisK& ax = *axes[k];
    if (ax.nv < least[k] || (ax.periodic && ax.n_cells < 3)) return false;   // (two cells: each is both neighbours)
    for (int a = 0; a < kQ1; ++a) {
      const double d = dt * c->cs.xi[a] / ax.hc;   // in cells; 1e-9 keeps clear of rounding
      if (!(fabs(d) < 1.0 - 1e-9)) return false;
      for (int l = 1; l < ax.p; ++l)
        if (!(ax.nodes[l] - d > 1e-9 && ax.nodes[l] - d < 1.0 - 1e-9)) return false;
    }
  }
  return true;
}

// The layout of the state, its two buffers and, for the sum-factorised step, the moment sums.
sllbm_status alloc_state3d(sllbm3d_ctx* c) {
  Pad3& L = c->lay;
  L.g = c->tiled ? (c->g.order <= 2 ? T3Shape<2>::G : T3Shape<4>::G) : 0;
  L.pitch = c->tiled ? (c->ax.nv + 2 * L.g + 1) / 2 * 2 : c->ax.nv;
  L.rows = c->ay.nv + 2 * L.g;
  L.plane = (size_t)L.pitch * L.rows * (c->az.nv + 2 * L.g);
  L.origin = ((size_t)L.g * L.rows + L.g) * L.pitch + L.g;
  sllbm_status s = SLLBM_OK;
  for (int k = 0; k < 2 && s == SLLBM_OK; ++k) s = alloc3(c, &c->state[k], state_doubles(c));
  if (!c->tiled) return s;
  c->parts = stream3d_parts(c);
  if (s == SLLBM_OK) s = alloc3(c, &c->sums, (size_t)6 * c->parts * c->nv);
  for (int k = 0; k < 2 && s == SLLBM_OK; ++k)   // ghosts of zero-gradient faces stay 0
    s = cuda3(c, cudaMemsetAsync(c->state[k], 0, state_doubles(c) * sizeof(double), c->stream), "cudaMemsetAsync");
  return s;
}

// The periodic images of the current state's ghost cells (after init and set_state).
cudaError_t fill_ghosts3d(sllbm3d_ctx* c) {
  if (!c->tiled) return cudaSuccess;
  const unsigned per_plane = (unsigned)(c->lay.plane - (size_t)c->nv);   // cells outside the interior
  ghost_refresh3d_kernel<<<dim3((per_plane + 255) / 256, kQ3), 256, 0, c->stream>>>(
      pairs(c, c->cur), c->lay, c->ax.nv, c->ay.nv, c->az.nv, c->ax.periodic, c->ay.periodic, c->az.periodic, per_plane);
  return cudaGetLastError();
}

cudaError_t launch_tiled3d(sllbm3d_ctx* c, const float2* src, float2* dst) {
  Stream3Args a{};
  a.src = src;
  a.dst = dst;
  a.sums = c->sums;
  a.nx = c->ax.nv;
  a.ny = c->ay.nv;
  a.nz = c->az.nv;
  a.nv = c->nv;
  a.lay = c->lay;
  a.tx = c->tail[0];
  a.ty = c->tail[1];
  a.tz = c->tail[2];
  a.cs = c->cs;
  a.flag = c->flag;
  cudaError_t e = cudaErrorInvalidValue;
  switch (c->g.order) {
    case 1: e = launch_stream3d<1>(a, c->parts, c->stream); break;
    case 2: e = launch_stream3d<2>(a, c->parts, c->stream); break;
    case 3: e = launch_stream3d<3>(a, c->parts, c->stream); break;
    case 4: e = launch_stream3d<4>(a, c->parts, c->stream); break;
  }
  if (e != cudaSuccess) return e;
  Collide3Args b{};
  b.dst = dst;
  b.lay = c->lay;
  b.sums = c->sums;
  b.parts = c->parts;
  b.nx = c->ax.nv;
  b.ny = c->ay.nv;
  b.nz = c->az.nv;
  b.px = c->ax.periodic;
  b.py = c->ay.periodic;
  b.pz = c->az.periodic;
  b.nv = c->nv;
  b.cs = c->cs;
  b.omega = (float)(1.0 / c->p.tau);
  b.K = (float)(2.0 * c->p.cv - 3.0);
  b.cv = (float)c->p.cv;
  b.inv2cv = (float)(0.5 / c->p.cv);
  b.npop = c->npop;
  b.iso = c->p.isothermal;
  b.flag = c->flag;
  collide3d_kernel<<<blocks_for(c->nv, 128), 128, 0, c->stream>>>(b);
  return cudaGetLastError();
}

}  // namespace

extern "C" {

sllbm_status sllbm3d_create(const sllbm_grid3_desc* g, const sllbm_params* p, void* stream, sllbm3d_ctx** out) {
  if (!g || !p || !out) return SLLBM_ERR_ARG;
  *out = nullptr;
  if (g->order < 1 || g->order > 4) return SLLBM_ERR_UNSUPPORTED;
  if (p->velset != SLLBM_VEL_D3Q125 || (p->prec != SLLBM_PREC_F64_PLAIN && p->prec != SLLBM_PREC_F32))
    return SLLBM_ERR_UNSUPPORTED;
  if (p->pr != 0.0 && p->pr != 1.0) return SLLBM_ERR_UNSUPPORTED;
  if (g->nx_cells < 1 || g->ny_cells < 1 || g->nz_cells < 1 || !(g->x1 > g->x0) || !(g->y1 > g->y0) ||
      !(g->z1 > g->z0))
    return SLLBM_ERR_ARG;
  for (int bc : {g->bc_x, g->bc_y, g->bc_z})
    if (bc != SLLBM_BC_PERIODIC && bc != SLLBM_BC_ZERO_GRADIENT) return SLLBM_ERR_ARG;
  if (g->nodes != SLLBM_NODES_GLC && g->nodes != SLLBM_NODES_EQUIDISTANT) return SLLBM_ERR_ARG;
  if (!(p->dt > 0.0) || !(p->tau > 0.5) || !(p->cv >= 1.5) || p->T0 != 1.0) return SLLBM_ERR_ARG;
  if (p->isothermal != 0 && (p->isothermal != 1 || p->cv != 1.5)) return SLLBM_ERR_ARG;
  const long long nvx = (long long)g->nx_cells * g->order + 1, nvy = (long long)g->ny_cells * g->order + 1,
                  nvz = (long long)g->nz_cells * g->order + 1;
  if (nvx > (1 << 16) || nvy > (1 << 16) || nvz > (1 << 16) || nvx * nvy * nvz > (1LL << 27))
    return SLLBM_ERR_UNSUPPORTED;   // 125 x 2 doubles a vertex: keep the state within the device
  sllbm3d_ctx* c = new (std::nothrow) sllbm3d_ctx();
  if (!c) return SLLBM_ERR_OOM;
  c->g = *g;
  c->p = *p;
  c->stream = static_cast<cudaStream_t>(stream);
  d1q5_consts(c->cs);
  axis3(c->ax, g->nx_cells, g->order, g->x0, g->x1, g->bc_x == SLLBM_BC_PERIODIC, g->nodes);
  axis3(c->ay, g->ny_cells, g->order, g->y0, g->y1, g->bc_y == SLLBM_BC_PERIODIC, g->nodes);
  axis3(c->az, g->nz_cells, g->order, g->z0, g->z1, g->bc_z == SLLBM_BC_PERIODIC, g->nodes);
  c->nv = (long long)c->ax.nv * c->ay.nv * c->az.nv;
  c->npop = p->cv == 1.5 ? 1 : 2;
  c->f32 = p->prec == SLLBM_PREC_F32;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&c->n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();   // (no device: the allocations below fail)
    c->n_sm = 0;
  }
  // The sum-factorised step's state keeps ghost cells, in rows of whole 16-byte units (1.2 times the dense one
  // on 128^3 vertices, up to 4 times on thin grids of orders 3 and 4).  If the device has no room for it,
  // the gather step takes the grid on the dense layout.
  c->tiled = tiled3d_usable(c, p->dt);
  sllbm_status s = alloc_state3d(c);
  if (s == SLLBM_ERR_OOM && c->tiled) {
    for (void* q : c->allocations) cudaFree(q);
    c->allocations.clear();
    c->tiled = false;
    s = alloc_state3d(c);
  }
  if (s == SLLBM_OK) s = alloc3(c, &c->flag, 1);
  if (s == SLLBM_OK) s = cuda3(c, cudaMemsetAsync(c->flag, 0, sizeof(int), c->stream), "cudaMemsetAsync");
  if (s != SLLBM_OK) {
    sllbm3d_destroy(c);
    return s;
  }
  *out = c;
  return SLLBM_OK;
}

sllbm_status sllbm3d_destroy(sllbm3d_ctx* c) {
  if (!c) return SLLBM_ERR_ARG;
  if (c->stream || !c->allocations.empty()) cudaStreamSynchronize(c->stream);
  for (void* p : c->allocations) cudaFree(p);
  delete c;
  return SLLBM_OK;
}

sllbm_status sllbm3d_grid_info(const sllbm3d_ctx* c, int* nx, int* ny, int* nz, int* npop) {
  if (!c) return SLLBM_ERR_ARG;
  if (nx) *nx = c->ax.nv;
  if (ny) *ny = c->ay.nv;
  if (nz) *nz = c->az.nv;
  if (npop) *npop = c->npop;
  return SLLBM_OK;
}

sllbm_status sllbm3d_vertex_coords(sllbm3d_ctx* c, double* x, double* y, double* z) {
  if (!c || !x || !y || !z) return fail3(c, SLLBM_ERR_ARG, "null pointer");
  coords3d_kernel<<<blocks_for(c->nv, 128), 128, 0, c->stream>>>(c->ax, c->ay, c->az, x, y, z);
  return cuda3(c, cudaGetLastError(), "coords3d_kernel");
}

sllbm_status sllbm3d_precompute_departures(sllbm3d_ctx* c) {
  if (!c) return SLLBM_ERR_ARG;
  const AxisK* axes[3] = {&c->ax, &c->ay, &c->az};
  for (int k = 0; k < 3; ++k) {
    const size_t n = (size_t)kQ1 * axes[k]->nv;
    if (!c->off[k]) {
      sllbm_status s = alloc3(c, &c->off[k], n);
      if (s == SLLBM_OK) s = alloc3(c, &c->w32[k], n * (c->g.order + 1));
      if (s == SLLBM_OK) s = alloc3(c, &c->w64[k], n * (c->g.order + 1));
      if (s != SLLBM_OK) return s;
    }
    const sllbm_status s = cuda3(c, launch_axis_tables(*axes[k], c->cs, c->p.dt, c->off[k], c->w32[k], c->w64[k],
                                                       c->stream), "launch_axis_tables");
    if (s != SLLBM_OK) return s;
  }
  if (c->tiled) {
    const int P = c->g.order;
    for (int k = 0; k < 3; ++k) {
      const int n = axes[k]->nv;
      if (!c->tail[k]) {
        const sllbm_status s = alloc3(c, &c->tail[k], (size_t)kQ1 * n * 2 * P);
        if (s != SLLBM_OK) return s;
      }
      const unsigned nb = blocks_for((long long)kQ1 * n, 128);
      switch (P) {
        case 1: tail_table_kernel<1><<<nb, 128, 0, c->stream>>>(c->off[k], c->w64[k], n, c->tail[k]); break;
        case 2: tail_table_kernel<2><<<nb, 128, 0, c->stream>>>(c->off[k], c->w64[k], n, c->tail[k]); break;
        case 3: tail_table_kernel<3><<<nb, 128, 0, c->stream>>>(c->off[k], c->w64[k], n, c->tail[k]); break;
        default: tail_table_kernel<4><<<nb, 128, 0, c->stream>>>(c->off[k], c->w64[k], n, c->tail[k]); break;
      }
      const sllbm_status s = cuda3(c, cudaGetLastError(), "tail_table_kernel");
      if (s != SLLBM_OK) return s;
    }
  }
  c->precomputed = true;
  return SLLBM_OK;
}

sllbm_status sllbm3d_init_equilibrium(sllbm3d_ctx* c, const double* rho, const double* u, const double* v,
                                      const double* w, const double* T) {
  if (!c || !rho || !u || !v || !w || !T) return fail3(c, SLLBM_ERR_ARG, "null pointer");
  if (!c->precomputed) return fail3(c, SLLBM_ERR_STATE, "precompute_departures first");
  Field3Args a{};
  a.rho = rho;
  a.u = u;
  a.v = v;
  a.w = w;
  a.T = T;
  a.state = c->state[c->cur];
  a.state32 = c->f32 ? pairs(c, c->cur) : nullptr;
  a.lay = c->lay;
  a.nx = c->ax.nv;
  a.ny = c->ay.nv;
  a.nv = c->nv;
  a.cs = c->cs;
  a.K = 2.0 * c->p.cv - 3.0;
  a.cv = c->p.cv;
  a.npop = c->npop;
  init3d_kernel<<<blocks_for(c->nv, 128), 128, 0, c->stream>>>(a);
  sllbm_status s = cuda3(c, cudaGetLastError(), "init3d_kernel");
  if (s == SLLBM_OK) s = cuda3(c, fill_ghosts3d(c), "ghost3d_kernel");
  if (s == SLLBM_OK) c->initialized = true;
  return s;
}

sllbm_status sllbm3d_step(sllbm3d_ctx* c, int nsteps) {
  if (!c || nsteps < 0) return fail3(c, SLLBM_ERR_ARG, "bad arguments");
  if (!c->precomputed || !c->initialized) return fail3(c, SLLBM_ERR_STATE, "precompute and init first");
  Step3Args a{};
  a.nx = c->ax.nv;
  a.ny = c->ay.nv;
  a.nz = c->az.nv;
  a.nv = c->nv;
  a.px = c->ax.periodic;
  a.py = c->ay.periodic;
  a.pz = c->az.periodic;
  a.offx = c->off[0];
  a.offy = c->off[1];
  a.offz = c->off[2];
  a.wx = c->w64[0];
  a.wy = c->w64[1];
  a.wz = c->w64[2];
  a.cs = c->cs;
  a.omega = 1.0 / c->p.tau;
  a.K = 2.0 * c->p.cv - 3.0;
  a.cv = c->p.cv;
  a.npop = c->npop;
  a.iso = c->p.isothermal;
  a.flag = c->flag;
  const unsigned blocks = blocks_for(c->nv, 128);
  if (c->f32) {
    Step3F32Args b{};
    b.nx = a.nx;
    b.ny = a.ny;
    b.nz = a.nz;
    b.nv = a.nv;
    b.px = a.px;
    b.py = a.py;
    b.pz = a.pz;
    b.offx = a.offx;
    b.offy = a.offy;
    b.offz = a.offz;
    b.wx = c->w32[0];
    b.wy = c->w32[1];
    b.wz = c->w32[2];
    b.cs = c->cs;
    b.omega = (float)a.omega;
    b.K = (float)a.K;
    b.cv = (float)a.cv;
    b.inv2cv = (float)(0.5 / a.cv);
    b.npop = a.npop;
    b.iso = a.iso;
    b.flag = a.flag;
    for (int k = 0; k < nsteps; ++k) {
      if (c->tiled) {
        const sllbm_status s = cuda3(c, launch_tiled3d(c, pairs(c, c->cur), pairs(c, c->cur ^ 1)), "stream3d/collide3d");
        if (s != SLLBM_OK) return s;
        c->cur ^= 1;
        continue;
      }
      b.src = pairs(c, c->cur);
      b.dst = pairs(c, c->cur ^ 1);
      if (blocks <= 4u * (unsigned)c->n_sm) {   // one wave
        switch (c->g.order) {
          case 1: step3d_f32_kernel<1, 4><<<blocks, 128, 0, c->stream>>>(b); break;
          case 2: step3d_f32_kernel<2, 4><<<blocks, 128, 0, c->stream>>>(b); break;
          case 3: step3d_f32_kernel<3, 4><<<blocks, 128, 0, c->stream>>>(b); break;
          default: step3d_f32_kernel<4, 4><<<blocks, 128, 0, c->stream>>>(b); break;
        }
      } else {
        switch (c->g.order) {
          case 1: step3d_f32_kernel<1, 0><<<blocks, 128, 0, c->stream>>>(b); break;
          case 2: step3d_f32_kernel<2, 0><<<blocks, 128, 0, c->stream>>>(b); break;
          case 3: step3d_f32_kernel<3, 0><<<blocks, 128, 0, c->stream>>>(b); break;
          default: step3d_f32_kernel<4, 0><<<blocks, 128, 0, c->stream>>>(b); break;
        }
      }
      const sllbm_status s = cuda3(c, cudaGetLastError(), "step3d_f32_kernel");
      if (s != SLLBM_OK) return s;
      c->cur ^= 1;
    }
    return SLLBM_OK;
  }
  for (int k = 0; k < nsteps; ++k) {
    a.src = c->state[c->cur];
    a.dst = c->state[c->cur ^ 1];
    switch (c->g.order) {
      case 1: step3d_f64_kernel<1><<<blocks, 128, 0, c->stream>>>(a); break;
      case 2: step3d_f64_kernel<2><<<blocks, 128, 0, c->stream>>>(a); break;
      case 3: step3d_f64_kernel<3><<<blocks, 128, 0, c->stream>>>(a); break;
      default: step3d_f64_kernel<4><<<blocks, 128, 0, c->stream>>>(a); break;
    }
    const sllbm_status s = cuda3(c, cudaGetLastError(), "step3d_f64_kernel");
    if (s != SLLBM_OK) return s;
    c->cur ^= 1;
  }
  return SLLBM_OK;
}

const char* sllbm3d_step_kernel_name(const sllbm3d_ctx* c) {
  if (!c) return "";
  return !c->f32 ? "plain_f64" : (c->tiled ? "stream3d" : "gather_f32");
}

sllbm_status sllbm3d_moments(sllbm3d_ctx* c, double* rho, double* u, double* v, double* w, double* T) {
  if (!c) return SLLBM_ERR_ARG;
  if (!c->initialized) return fail3(c, SLLBM_ERR_STATE, "init first");
  Field3Args a{};
  a.orho = rho;
  a.ou = u;
  a.ov = v;
  a.ow = w;
  a.oT = T;
  a.state = c->state[c->cur];
  a.state32 = c->f32 ? pairs(c, c->cur) : nullptr;
  a.lay = c->lay;
  a.nx = c->ax.nv;
  a.ny = c->ay.nv;
  a.nv = c->nv;
  a.cs = c->cs;
  a.K = 2.0 * c->p.cv - 3.0;
  a.cv = c->p.cv;
  a.npop = c->npop;
  a.flag = c->flag;
  moments3d_kernel<<<blocks_for(c->nv, 128), 128, 0, c->stream>>>(a);
  sllbm_status s = cuda3(c, cudaGetLastError(), "moments3d_kernel");
  if (s != SLLBM_OK) return s;
  int flag = 0;
  s = cuda3(c, cudaMemcpyAsync(&flag, c->flag, sizeof(int), cudaMemcpyDeviceToHost, c->stream), "cudaMemcpyAsync");
  if (s == SLLBM_OK) s = cuda3(c, cudaStreamSynchronize(c->stream), "cudaStreamSynchronize");
  if (s != SLLBM_OK) return s;
  if (flag & 4) return fail3(c, SLLBM_ERR_CUDA, "a staging copy of the 3D stream kernel timed out");
  return (flag & 1) ? fail3(c, SLLBM_ERR_UNSTABLE, "non-positive or non-finite density or temperature") : SLLBM_OK;
}

sllbm_status sllbm3d_get_state(sllbm3d_ctx* c, double* dst) {
  if (!c || !dst) return fail3(c, SLLBM_ERR_ARG, "null pointer");
  if (c->f32) {
    convert3d_kernel<<<dim3(blocks_for(c->nv, 256 * kConvPer), kQ3), 256, 0, c->stream>>>(
        pairs(c, c->cur), c->lay, dst, c->ax.nv, c->ay.nv, (unsigned)c->nv, c->npop, 2.0 * c->p.cv - 3.0, c->cs, 1);
    return cuda3(c, cudaGetLastError(), "convert3d_kernel");
  }
  return cuda3(c, cudaMemcpyAsync(dst, c->state[c->cur], state_doubles(c) * sizeof(double), cudaMemcpyDeviceToDevice,
                                  c->stream), "cudaMemcpyAsync");
}

sllbm_status sllbm3d_set_state(sllbm3d_ctx* c, const double* src) {
  if (!c || !src) return fail3(c, SLLBM_ERR_ARG, "null pointer");
  if (c->f32) {
    convert3d_kernel<<<dim3(blocks_for(c->nv, 256 * kConvPer), kQ3), 256, 0, c->stream>>>(
        pairs(c, c->cur), c->lay, const_cast<double*>(src), c->ax.nv, c->ay.nv, (unsigned)c->nv, c->npop,
        2.0 * c->p.cv - 3.0, c->cs, 0);
    sllbm_status s = cuda3(c, cudaGetLastError(), "convert3d_kernel");
    if (s == SLLBM_OK) s = cuda3(c, fill_ghosts3d(c), "ghost3d_kernel");
    if (s == SLLBM_OK) c->initialized = true;
    return s;
  }
  const sllbm_status s = cuda3(c, cudaMemcpyAsync(c->state[c->cur], src, state_doubles(c) * sizeof(double),
                                                  cudaMemcpyDeviceToDevice, c->stream), "cudaMemcpyAsync");
  if (s == SLLBM_OK) c->initialized = true;
  return s;
}

const char* sllbm3d_last_error(const sllbm3d_ctx* c) { return c ? c->err.c_str() : "null context"; }

}  // extern "C"
