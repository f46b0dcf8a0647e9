// Fused step of a short list of vertices of a uniform grid, one warp per vertex: the vertices next
// to zero-gradient boundaries, whose stencils differ from the cell-periodic pattern of the fused
// uniform kernel.  Lane i < 25 carries velocity i: it gathers the (p+1)^2 stencil of its plane from
// global memory, the moments are warp sums (butterfly shuffles, so every lane holds them), and
// each lane forms and relaxes its own equilibrium value.  FP32 arithmetic, (f, g) pairs, the same
// difference form, deviation form and residual correction as the fused kernel
// (collide_deviation_f32).
//
// What bounds it is latency: the list has one row or column of vertices per clamped side (16
// vertices on the 8193 x 8 strip, 2,000 at most: more go to the fused kernel's edge tiles), so a thread per
// vertex (25 dependent gathers and the collision in one thread) left the chip idle for 43 us on
// that strip, longer than the fused kernel beside it; a warp per vertex has all 25 gathers in
// flight at once.  The launch overlaps the fused kernel's last tiles (programmatic dependent
// launch): it reads what that kernel reads, written by steps that ended before it began, and
// writes other vertices.  It ends after that kernel has ended (pdl_wait at the end), so that
// whatever follows this launch follows both.
#include "tma.cuh"

namespace sllbm {

namespace {

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
  return v;
}

constexpr int kFixThreads = 64;   // two vertices a block

template <int P, typename Store, bool PR>
__global__ void __launch_bounds__(kFixThreads) step_fixup_kernel(const __grid_constant__ StepArgs a) {
  const int lane = threadIdx.x & 31;
  const long long e = (long long)blockIdx.x * (kFixThreads / 32) + (threadIdx.x >> 5);
  if (e >= a.nlist) {   // whole warps
    pdl_wait();
    return;
  }
  const int v = a.vlist[e];
  const int iy = v / a.nx, ix = v - iy * a.nx;
  const bool on = lane < kQ;
  const int i = on ? lane : 0, ia = i / kQ1, ib = i - kQ1 * ia;
  const float xa = a.cs.xif[ia], xb = a.cs.xif[ib];
  float2 fg;   // (f, g) deviations after streaming
  {
    const int sx = ix + __ldg(a.offx + ia * a.nx + ix), sy = iy + __ldg(a.offy + ib * a.ny + iy);
    const float* wx = a.wx + (size_t)(ia * a.nx + ix) * (P + 1);
    const float* wy = a.wy + (size_t)(ib * a.ny + iy) * (P + 1);
    const Store* pl = static_cast<const Store*>(a.src) + (size_t)i * a.plane_stride;
    int col[P + 1];
#pragma unroll
    for (int k = 0; k <= P; ++k) col[k] = 2 * wrap_index(sx + k, a.nx, a.periodic_x);
    float2 rows[P + 1];
#pragma unroll
    for (int kb = 0; kb <= P; ++kb) {
      const Store* row = pl + (ptrdiff_t)wrap_index(sy + kb, a.ny, a.periodic_y) * a.pitch;
      const float2 base = ld_pair(row + col[0]);
      float2 acc = base;
#pragma unroll
      for (int ka = 1; ka <= P; ++ka) acc = fma2(bcast2(__ldg(wx + ka)), sub2(ld_pair(row + col[ka]), base), acc);
      rows[kb] = acc;
    }
    fg = rows[0];
#pragma unroll
    for (int kb = 1; kb <= P; ++kb) fg = fma2(bcast2(__ldg(wy + kb)), sub2(rows[kb], rows[0]), fg);
  }
  const bool two = a.cp.npop == 2;
  if (!on) fg = make_float2(0.f, 0.f);
  if (!two) fg.y = 0.f;
  // moments (Sec. II) of the deviations
  const float xa2 = xa * xa, xb2 = xb * xb;
  const float drho = warp_sum(fg.x), jx = warp_sum(xa * fg.x), jy = warp_sum(xb * fg.x);
  const float a2 = warp_sum((xa2 + xb2) * fg.x), G = warp_sum(fg.y);
  const float rho = 1.f + drho, inv_rho = __frcp_rn(rho);
  const float ux = jx * inv_rho, uy = jy * inv_rho;
  const float qk = (a2 + G - rho * (ux * ux + uy * uy) - 2.f * a.cp.cvf * drho) * inv_rho * a.cp.inv2cvf;
  const float q = a.cp.iso ? 0.f : qk;
  const float wa = a.cs.wf[ia], wb = a.cs.wf[ib], w = wa * wb;
  // Pr != 1: w_a w_b (Q_xxx h3(a) + Q_xxy h2(a) h1(b) + Q_xyy h1(a) h2(b) + Q_yyy h3(b)) of the
  // non-equilibrium centred third moments (the lattice-weight part added in closed form)
  float2 qe = make_float2(0.f, 0.f);
  if constexpr (PR) {
    const float cx = xa - ux, cy = xb - uy;
    const float m[4] = {cx * cx * cx, cx * cx * cy, cx * cy * cy, cy * cy * cy};
    const float lat[4] = {-3.f * ux - ux * ux * ux, -uy - ux * ux * uy, -ux - ux * uy * uy, -3.f * uy - uy * uy * uy};
    const float h[4] = {a.cs.hef[3][ia], a.cs.hef[2][ia] * a.cs.hef[1][ib], a.cs.hef[1][ia] * a.cs.hef[2][ib],
                        a.cs.hef[3][ib]};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float qf = warp_sum(on ? m[k] * fg.x : 0.f) + lat[k];
      const float qg = warp_sum(on ? m[k] * fg.y : 0.f) + a.cp.Kf * lat[k];
      qe.x = fmaf(qf, h[k], qe.x);
      qe.y = fmaf(qg, h[k], qe.y);
    }
    const float c = a.cp.cprf * w;
    qe = make_float2(c * qe.x, c * qe.y);
  }
  // f^eq - w = w (drho + rho (S_4(b) + sum_k X_k(a) (1 + S_{4-k}(b))))
  float X[5], S[5];
  X[1] = ux * a.cs.hef[1][ia];
  X[2] = (ux * ux + q) * a.cs.hef[2][ia];
  X[3] = ux * (ux * ux + 3.f * q) * a.cs.hef[3][ia];
  X[4] = (ux * ux * (ux * ux + 6.f * q) + 3.f * q * q) * a.cs.hef[4][ia];
  S[0] = 0.f;
  S[1] = uy * a.cs.hef[1][ib];
  S[2] = S[1] + (uy * uy + q) * a.cs.hef[2][ib];
  S[3] = S[2] + uy * (uy * uy + 3.f * q) * a.cs.hef[3][ib];
  S[4] = S[3] + (uy * uy * (uy * uy + 6.f * q) + 3.f * q * q) * a.cs.hef[4][ib];
  float em1 = S[4];
#pragma unroll
  for (int k = 1; k <= 4; ++k) em1 = fmaf(X[k], 1.f + S[4 - k], em1);
  const float ef = w * fmaf(rho, em1, drho);
  const float eg = a.cp.Kf * ((1.f + q) * ef + q * w);   // g^eq - K w
  const float om = a.cp.omegaf;
  float2 d = sub2(make_float2(ef, two ? eg : 0.f), fg);
  if (!on) d = make_float2(0.f, 0.f);
  float2 out = fma2(bcast2(om), d, fg);
  // residual moments of f^eq - f (FP32 rounding of the equilibrium), removed at the velocities
  // (s, 0) (i = 5), (0, s) (i = 1) and the rest velocity, the energy on g at rest
  const float r0 = warp_sum(d.x), r1 = warp_sum(xa * d.x), r2 = warp_sum(xb * d.x);
  const float r3 = warp_sum((xa2 + xb2) * d.x + d.y);   // d.y is 0 with one population
  const float inv_s = a.cs.inv_xi1f;
  const float d1 = r1 * inv_s, d2 = r2 * inv_s, d0 = r0 - d1 - d2;
  const float de = r3 - a.cs.xi1sqf * (d1 + d2);
  if (lane == 0) out.x -= om * d0;
  if (lane == 5) out.x -= om * d1;
  if (lane == 1) out.x -= om * d2;
  if (two) {
    if (lane == 0) out.y -= om * de;
  } else if (!a.cp.iso) {   // one population: along (+-s, 0), -2 at rest
    const float ee = om * 0.5f * de * inv_s * inv_s;
    if (lane == 5 || lane == 15) out.x -= ee;
    if (lane == 0) out.x += 2.f * ee;
  }
  if constexpr (PR) out = make_float2(out.x + qe.x, out.y + qe.y);
  if (!two) out.y = 0.f;   // one population: the g slots stay zero
  if (lane == 0) {
    if (!((rho > 0.f) && (q > -1.f) && isfinite(rho) && isfinite(q))) atomicOr(a.flag, 1);
    if (a.mom) {
      VertexMoments vm;
      vm.rho = rho;
      vm.ux = ux;
      vm.uy = uy;
      vm.theta = 1.f + qk;
      store_moments(a.mom, a.nv, v, vm);
    }
  }
  if (on) {
    Store* dst = static_cast<Store*>(a.dst) + (size_t)i * a.plane_stride;
    store_images(a.ghost, ix, iy, [&](int xx, int yy) {
      st_pair(dst + (ptrdiff_t)yy * a.pitch + 2 * (ptrdiff_t)xx, out);
    });
  }
  pdl_wait();
}

template <int P, typename Store>
cudaError_t launch_p(const StepArgs& a, cudaStream_t s) {
  const unsigned blocks = (unsigned)((a.nlist + kFixThreads / 32 - 1) / (kFixThreads / 32));
  return a.cp.pr_on ? launch_dependent(step_fixup_kernel<P, Store, true>, dim3(blocks), dim3(kFixThreads), 0, s, true, a)
                    : launch_dependent(step_fixup_kernel<P, Store, false>, dim3(blocks), dim3(kFixThreads), 0, s, true, a);
}

template <typename Store>
cudaError_t launch_store(const StepArgs& a, cudaStream_t s) {
  switch (a.P) {
    case 1: return launch_p<1, Store>(a, s);
    case 2: return launch_p<2, Store>(a, s);
    case 3: return launch_p<3, Store>(a, s);
    case 4: return launch_p<4, Store>(a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_step_fixup(const StepArgs& a, int store, cudaStream_t s) {
  if (!a.vlist || a.nlist <= 0 || a.mapped || a.xs != 2 || a.ps != 1) return cudaErrorInvalidValue;
  if (store == kStoreBF16) return launch_store<__nv_bfloat16>(a, s);
  return launch_store<float>(a, s);
}

}  // namespace sllbm
