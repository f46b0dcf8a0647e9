// Plain FP64 SLLBM step on full populations: the accuracy and speed baseline of the FP32 paths.
// Moments (Sec. II), the fourth-order equilibrium (Sec. II.A) and BGK (Eq. streaming_fg).
//
// step_tile_f64_kernel (uniform grids that fill its tiles, Pr = 1): tiles of 32 x 4 vertices, sum factorisation through
// shared memory.  step_plain_f64_kernel (the rest): one thread per vertex, (p+1)^2 gathers per
// velocity plane from global memory with FP64 weights.
#include "kernels.h"

namespace sllbm {

namespace {

// The FP64 pipe (two operations a clock and SM) bounds the step, so the tile kernel is built to
// need few of them: per value and axis p + 1 multiply-adds (the y pass runs on the tile's columns
// and the halo, 40 for 32 at p = 4) in place of (p + 1)^2 + p + 1, none for components at rest (copied),
// moments through row and column sums, and the equilibrium with the parts that mirrored velocities
// share formed once: about 750 a vertex at p = 4 in place of 2200.  513 x 513 vertices, p = 4:
// 982 -> 470 us a step.  The tables and windows are those of the grid's own stencils (any boundary, per-vertex
// weights); the next plane's window is loaded into registers while one is worked on.
constexpr int kFX = 32, kFY = 4, kFN = kFX * kFY;   // tile; threads, one vertex each
constexpr int kFElems = 6;                          // window elements a thread stages per population

struct F64Window {
  int ox, oy, W, H;   // origin relative to the tile origin, columns and rows
};

template <int P>
size_t f64_tile_smem(const F64Window& w) {
  return sizeof(double) * ((size_t)2 * kQ * kFN + 2 * w.W * w.H + 2 * kFY * w.W + kQ1 * (kFX + kFY) * (P + 1)) +
         sizeof(int) * kQ1 * (kFX + kFY);
}

template <int P>
__global__ void __launch_bounds__(kFN, 3) step_tile_f64_kernel(const __grid_constant__ StepArgs a,
                                                               const __grid_constant__ F64Window win) {
  extern __shared__ double f64_smem[];
  const int W = win.W, HW = win.H * W;
  double* F = f64_smem;                        // [2][25][kFN] interpolated populations
  double* S = F + 2 * kQ * kFN;                // [2][H][W] window of the plane
  double* T = S + 2 * HW;                      // [2][kFY][W] after the y pass
  double* WX = T + 2 * kFY * W;                // [5][kFX][P + 1]
  double* WY = WX + kQ1 * kFX * (P + 1);       // [5][kFY][P + 1]
  int* XO = reinterpret_cast<int*>(WY + kQ1 * kFY * (P + 1));   // [5][kFX] window column of the stencil
  int* YO = XO + kQ1 * kFX;                    // [5][kFY] window row
  const int tid = threadIdx.x, lane = tid & 31, row = tid >> 5;
  const int tiles_x = (a.nx + kFX - 1) / kFX;
  const int tx0 = (int)(blockIdx.x % tiles_x) * kFX, ty0 = (int)(blockIdx.x / tiles_x) * kFY;
  const int x = tx0 + lane, y = ty0 + row;
  const int npop = a.cp.npop;
  for (int e = tid; e < kQ1 * (kFX + kFY); e += kFN) {   // tables (nodes past the grid clamped)
    const bool isx = e < kQ1 * kFX;
    const int r = isx ? e : e - kQ1 * kFX, c = r / (isx ? kFX : kFY), j = r - c * (isx ? kFX : kFY);
    const int n = isx ? min(tx0 + j, a.nx - 1) : min(ty0 + j, a.ny - 1);
    const double* w = (isx ? a.wx64 + (size_t)(c * a.nx + n) * (P + 1) : a.wy64 + (size_t)(c * a.ny + n) * (P + 1));
    (isx ? XO : YO)[r] = isx ? n + a.offx[c * a.nx + n] - tx0 - win.ox : n + a.offy[c * a.ny + n] - ty0 - win.oy;
    for (int k = 0; k <= P; ++k) (isx ? WX : WY)[r * (P + 1) + k] = w[k];
  }
  // the window elements this thread stages, as offsets in a plane
  ptrdiff_t at[kFElems];
#pragma unroll
  for (int j = 0; j < kFElems; ++j) {
    const int e = min(tid + j * kFN, HW - 1), r = e / W, c = e - r * W;
    int gx = tx0 + win.ox + c, gy = ty0 + win.oy + r;
    gx = a.periodic_x ? wrap_index(gx, a.nx, 1) : min(max(gx, 0), a.nx - 1);
    gy = a.periodic_y ? wrap_index(gy, a.ny, 1) : min(max(gy, 0), a.ny - 1);
    at[j] = (ptrdiff_t)gy * a.pitch + (ptrdiff_t)gx * a.xs;
  }
  const double* src = static_cast<const double*>(a.src);
  double nf[kFElems], ng[kFElems];
  auto load = [&](int i) {
    const double* pl = src + (size_t)i * a.plane_stride;
#pragma unroll
    for (int j = 0; j < kFElems; ++j) {
      if (j * kFN >= HW) break;
      nf[j] = __ldg(pl + at[j]);
      if (npop == 2) ng[j] = __ldg(pl + a.ps + at[j]);
    }
  };
  load(0);
  double rho = 0.0, jx = 0.0, e2 = 0.0, G = 0.0, C[kQ1];
#pragma unroll
  for (int b = 0; b < kQ1; ++b) C[b] = 0.0;
  // y-pass units (population, row, column), the uneven last round on other warps in every other block
  const int u0 = (tid + (blockIdx.x & 1) * (kFN / 2)) % kFN, units = npop * kFY * W;
#pragma unroll 1
  for (int ia = 0; ia < kQ1; ++ia) {
    double R = 0.0;
#pragma unroll
    for (int ib = 0; ib < kQ1; ++ib) {
      const int i = kQ1 * ia + ib;
#pragma unroll
      for (int j = 0; j < kFElems; ++j) {   // (every thread is past the y pass of the plane before)
        const int e = tid + j * kFN;
        if (e < HW) {
          S[e] = nf[j];
          if (npop == 2) S[HW + e] = ng[j];
        }
      }
      if (i + 1 < kQ) load(i + 1);
      __syncthreads();   // window staged; every thread is past the x pass of the plane before
      for (int u = u0; u < units; u += kFN) {
        const int r = u / W, c = u - r * W, ty = r & (kFY - 1), pop = r / kFY;
        const double* col = S + pop * HW + c;
        if (ib == 0) {   // at rest along y: the vertex's own row
          T[r * W + c] = col[(ty - win.oy) * W];
        } else {
          const double* w = WY + (ib * kFY + ty) * (P + 1);
          col += YO[ib * kFY + ty] * W;
          double acc = w[0] * col[0];
#pragma unroll
          for (int k = 1; k <= P; ++k) acc += w[k] * col[k * W];
          T[r * W + c] = acc;
        }
      }
      __syncthreads();   // T complete
      {
        const double *tf = T + row * W, *tg = tf + kFY * W;
        double f, g = 0.0;
        if (ia == 0) {   // at rest along x: the vertex's own column
          f = tf[lane - win.ox];
          if (npop == 2) g = tg[lane - win.ox];
        } else {
          const double* w = WX + (ia * kFX + lane) * (P + 1);
          const int o = XO[ia * kFX + lane];
          f = w[0] * tf[o];
          if (npop == 2) g = w[0] * tg[o];
#pragma unroll
          for (int k = 1; k <= P; ++k) {
            f += w[k] * tf[o + k];
            if (npop == 2) g += w[k] * tg[o + k];
          }
        }
        F[i * kFN + tid] = f;
        F[(kQ + i) * kFN + tid] = g;
        R += f;
        C[ib] += f;
        G += g;
      }
    }
    const double c = a.cs.xi[ia];
    rho += R;
    jx += c * R;
    e2 += c * c * R;
  }
  if (x >= a.nx || y >= a.ny) return;   // no barrier follows
  double jy = 0.0;
#pragma unroll
  for (int b = 1; b < kQ1; ++b) {
    jy += a.cs.xi[b] * C[b];
    e2 += a.cs.xi[b] * a.cs.xi[b] * C[b];
  }
  e2 += G;
  const double inv = 1.0 / rho, ux = jx * inv, uy = jy * inv;
  const double theta_k = (e2 - rho * (ux * ux + uy * uy)) * inv / (2.0 * a.cp.cv);
  const double theta = a.cp.iso ? 1.0 : theta_k, q = theta - 1.0;
  if (a.mom) {
    const long long v = (long long)y * a.nx + x;
    a.mom[v] = (float)rho;
    a.mom[a.nv + v] = (float)ux;
    a.mom[2 * a.nv + v] = (float)uy;
    a.mom[3 * a.nv + v] = (float)theta_k;
  }
  const double x2 = ux * ux, y2 = uy * uy, q3 = 3.0 * q, q6 = 6.0 * q, qq = q3 * q;
  const double ax[5] = {1.0, ux, x2 + q, ux * (x2 + q3), x2 * (x2 + q6) + qq};
  const double ay[5] = {1.0, uy, y2 + q, uy * (y2 + q3), y2 * (y2 + q6) + qq};
  double X[5][3];   // rho A_k(u_x) he[k][a]; the nodes are 0, +s, +l, -s, -l
#pragma unroll
  for (int k = 0; k <= 4; ++k)
#pragma unroll
    for (int c = 0; c < 3; ++c) X[k][c] = (c == 0 && k % 2) ? 0.0 : rho * (ax[k] * a.cs.he[k][c]);
  const double om = a.cp.omega, Kt = a.cp.K * theta;
  double* dst = static_cast<double*>(a.dst) + (ptrdiff_t)y * a.pitch + (ptrdiff_t)x * a.xs;
  auto relax = [&](int ia, int ib, double e) {   // e = f^eq / w_a
    const int i = kQ1 * ia + ib;
    const double feq = a.cs.w[ia] * e, f = F[i * kFN + tid];
    dst[(size_t)i * a.plane_stride] = f - om * (f - feq);
    if (npop == 2) {
      const double g = F[(kQ + i) * kFN + tid];
      dst[(size_t)i * a.plane_stride + a.ps] = g - om * (g - Kt * feq);
    }
  };
#pragma unroll
  for (int b = 0; b < kQ1; ++b) {
    double Sw[5];   // w_b sum_{l <= m} A_l(u_y) he[l][b]
    Sw[0] = a.cs.w[b];
#pragma unroll
    for (int m = 1; m <= 4; ++m) Sw[m] = (b == 0 && m % 2) ? Sw[m - 1] : Sw[m - 1] + a.cs.w[b] * a.cs.he[m][b] * ay[m];
    relax(0, b, X[0][0] * Sw[4] + X[2][0] * Sw[2] + X[4][0] * Sw[0]);
#pragma unroll
    for (int c = 1; c <= 2; ++c) {
      const double ev = X[0][c] * Sw[4] + X[2][c] * Sw[2] + X[4][c] * Sw[0], od = X[1][c] * Sw[3] + X[3][c] * Sw[1];
      relax(c, b, ev + od);
      relax(c + 2, b, ev - od);
    }
  }
  if (!(rho > 0.0 && theta > 0.0 && isfinite(rho) && isfinite(theta))) atomicOr(a.flag, 1);
}

// Whether the tiles are filled well enough: vertices past the grid cost as much as others, so on grids of
// a few columns (or rows) the gathers are faster.  The lines are where the two cross on grids of 4,800 and
// 24,000 rows (7 x 20000 vertices, p = 1: 306 us a step by gathers, 723 in tiles; 16 x 24000, p = 4: 1569 and 1228);
// the gathers' longer start is worth some 12,000 vertices at p <= 2 (24000 x 5, p = 1: 263 and 210).
// Tiles that are all resident at once (three blocks an SM) wait for latency, not for the pipe, and are the
// shorter way at any filling (6 x 480, p = 1: 38 us and 60; 12 x 1820: 70 and 79; at p = 1 the third block of
// fewer than 12 columns is not: 8 x 1820 69 and 55).
bool tile_f64_pays(const StepArgs& a) {
  const long long tiles = (long long)((a.nx + kFX - 1) / kFX) * ((a.ny + kFY - 1) / kFY);
  int dev = 0, n_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return true;   // (the launch reports the error)
  const double least[5] = {1.0, 0.65, 0.58, 0.49, 0.41};
  return tiles <= (a.P == 1 && a.nx < 12 ? 2LL : 3LL) * n_sm || (double)a.nv + (a.P <= 2 ? 12400.0 : 0.0) >= least[a.P] * (double)(tiles * kFN);
}

// The tile kernel takes the step: a uniform grid, Pr = 1, and a window a block can stage.
bool tile_f64_window(const StepArgs& a, F64Window* w) {
  if (a.mapped || a.cp.pr_on || a.cs.nq1 != kQ1) return false;
  *w = F64Window{a.offx_min, a.offy_min, kFX + a.offx_max - a.offx_min, kFY + a.offy_max - a.offy_min};
  // (the window holds each vertex itself: components at rest have offsets in [-p, 0] and ends in [0, p])
  return w->ox <= 0 && w->oy <= 0 && a.offx_max >= 0 && a.offy_max >= 0 && w->W * w->H <= kFElems * kFN && tile_f64_pays(a);
}

}  // namespace

template <int P, bool Mapped, bool PR>
__global__ void __launch_bounds__(128) step_plain_f64_kernel(const __grid_constant__ StepArgs a) {
  const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= a.nv) return;
  const int ix = (int)(v % a.nx), iy = (int)(v / a.nx);
  const double* src = static_cast<const double*>(a.src);
  double* dst = static_cast<double*>(a.dst);
  const int npop = a.cp.npop;
  double f[kQ], g[kQ];
#pragma unroll 1
  for (int i = 0; i < kQ; ++i) {
    const int ia = i / 5, ib = i % 5;
    int sx, sy;
    double wx[P + 1], wy[P + 1];
    if (Mapped) {
      const long long d = (long long)i * a.nv + v;
      sx = a.dcx[d] * P;
      sy = a.dcy[d] * P;
      lagrange_basis<P, double>(a.nodes, a.dr64[d], wx);
      lagrange_basis<P, double>(a.nodes, a.ds64[d], wy);
    } else {
      sx = ix + a.offx[ia * a.nx + ix];
      sy = iy + a.offy[ib * a.ny + iy];
#pragma unroll
      for (int k = 0; k <= P; ++k) {
        wx[k] = a.wx64[(ia * a.nx + ix) * (P + 1) + k];
        wy[k] = a.wy64[(ib * a.ny + iy) * (P + 1) + k];
      }
    }
    double accf = 0.0, accg = 0.0;
    const double* pf = src + (size_t)i * a.plane_stride;
    const double* pg = pf + a.ps;
#pragma unroll
    for (int kb = 0; kb <= P; ++kb) {
      const size_t r = (size_t)wrap_index(sy + kb, a.ny, a.periodic_y) * a.pitch;
      double axf = 0.0, axg = 0.0;
#pragma unroll
      for (int ka = 0; ka <= P; ++ka) {
        const size_t o = r + (size_t)wrap_index(sx + ka, a.nx, a.periodic_x) * a.xs;
        axf += wx[ka] * __ldg(pf + o);
        if (npop == 2) axg += wx[ka] * __ldg(pg + o);
      }
      accf += wy[kb] * axf;
      accg += wy[kb] * axg;
    }
    f[i] = accf;
    g[i] = accg;
  }
  // moments
  double rho = 0.0, jx = 0.0, jy = 0.0, e2 = 0.0;
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    const double cx = a.cs.xi[i / 5], cy = a.cs.xi[i % 5];
    rho += f[i];
    jx += f[i] * cx;
    jy += f[i] * cy;
    e2 += f[i] * (cx * cx + cy * cy) + (npop == 2 ? g[i] : 0.0);
  }
  const double ux = jx / rho, uy = jy / rho;
  const double theta_k = (e2 - rho * (ux * ux + uy * uy)) / (2.0 * a.cp.cv * rho);
  const double theta = a.cp.iso ? 1.0 : theta_k;
  if (a.mom) {
    const long long v = (long long)iy * a.nx + ix;
    a.mom[v] = (float)rho;
    a.mom[a.nv + v] = (float)ux;
    a.mom[2 * a.nv + v] = (float)uy;
    a.mom[3 * a.nv + v] = (float)theta_k;
  }
  const double q = theta - 1.0;
  EqFactors<double> e;
  eq_factors<double>(a.cs.he, ux, uy, q, e);
  const double om = a.cp.omega;
  const size_t o = (size_t)iy * a.pitch + (size_t)ix * a.xs;
  // Pr != 1 (Sec. II.C): non-equilibrium centred third moments of f and g (xxx, xxy, xyy, yyy)
  double qf[4] = {0.0, 0.0, 0.0, 0.0}, qg[4] = {0.0, 0.0, 0.0, 0.0};
  if (PR) {
#pragma unroll 1
    for (int i = 0; i < kQ; ++i) {
      const int ia = i / 5, ib = i % 5;
      const double feq = a.cs.w[ia] * a.cs.w[ib] * rho * (1.0 + eq_em1<double>(e, ia, ib));
      const double df = f[i] - feq, dg = npop == 2 ? g[i] - a.cp.K * theta * feq : 0.0;
      const double cx = a.cs.xi[ia] - ux, cy = a.cs.xi[ib] - uy;
      const double m[4] = {cx * cx * cx, cx * cx * cy, cx * cy * cy, cy * cy * cy};
      for (int k = 0; k < 4; ++k) {
        qf[k] += df * m[k];
        qg[k] += dg * m[k];
      }
    }
  }
#pragma unroll
  for (int ia = 0; ia < kQ1; ++ia)
#pragma unroll
    for (int ib = 0; ib < kQ1; ++ib) {
      const int i = 5 * ia + ib;
      const double feq = a.cs.w[ia] * a.cs.w[ib] * rho * (1.0 + eq_em1<double>(e, ia, ib));
      // quasi-equilibrium: w_a w_b (Q_xxx h3(a) + Q_xxy h2(a) h1(b) + Q_xyy h1(a) h2(b) + Q_yyy h3(b))
      double sf = 0.0, sg = 0.0;
      if (PR) {
        const double wab = a.cs.w[ia] * a.cs.w[ib];
        const double h[4] = {a.cs.he[3][ia], a.cs.he[2][ia] * a.cs.he[1][ib],
                             a.cs.he[1][ia] * a.cs.he[2][ib], a.cs.he[3][ib]};
        for (int k = 0; k < 4; ++k) {
          sf += qf[k] * h[k];
          sg += qg[k] * h[k];
        }
        sf *= a.cp.cpr * wab;
        sg *= a.cp.cpr * wab;
      }
      dst[(size_t)i * a.plane_stride + o] = f[i] - om * (f[i] - feq) + sf;
      if (npop == 2) {
        const double geq = a.cp.K * theta * feq;
        dst[(size_t)i * a.plane_stride + a.ps + o] = g[i] - om * (g[i] - geq) + sg;
      }
    }
  if (!(rho > 0.0 && theta > 0.0 && isfinite(rho) && isfinite(theta))) atomicOr(a.flag, 1);
}

template <int P>
static cudaError_t launch_p(const StepArgs& a, cudaStream_t s) {
  F64Window win;
  if (tile_f64_window(a, &win)) {
    const size_t smem = f64_tile_smem<P>(win);
    const cudaError_t e =
        cudaFuncSetAttribute(step_tile_f64_kernel<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const long long tiles = (long long)((a.nx + kFX - 1) / kFX) * ((a.ny + kFY - 1) / kFY);
    step_tile_f64_kernel<P><<<(unsigned)tiles, kFN, smem, s>>>(a, win);
    return cudaGetLastError();
  }
  const int threads = 128;
  const unsigned blocks = (unsigned)((a.nv + threads - 1) / threads);
  if (a.mapped)
    a.cp.pr_on ? step_plain_f64_kernel<P, true, true><<<blocks, threads, 0, s>>>(a)
               : step_plain_f64_kernel<P, true, false><<<blocks, threads, 0, s>>>(a);
  else
    a.cp.pr_on ? step_plain_f64_kernel<P, false, true><<<blocks, threads, 0, s>>>(a)
               : step_plain_f64_kernel<P, false, false><<<blocks, threads, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_step_plain_f64(const StepArgs& a, cudaStream_t s) {
  switch (a.P) {
    case 1: return launch_p<1>(a, s);
    case 2: return launch_p<2>(a, s);
    case 3: return launch_p<3>(a, s);
    case 4: return launch_p<4>(a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace sllbm
