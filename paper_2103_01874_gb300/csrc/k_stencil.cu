// Point-wise kernels of the projection: rho_0 = min(rho) (text after Eq. (32)),
// the velocity correction of Eq. (33), and the device-side refinement control.
#include "dfloat.cuh"
#include "ppe_internal.h"
#include "pdl.cuh"
#include "stencil.cuh"
#include "correct.cuh"

namespace ppe {

__global__ void k_init_scalars(DevScalars* sc, double rho0, double tol, int keep_rho0, double* out_p,
                               double* out_u, double* out_v, double* out_w) {
  pdl_enter();
  if (threadIdx.x == 0) init_scalars(sc, rho0, tol, keep_rho0, out_p, out_u, out_v, out_w);
}

__global__ void __launch_bounds__(256) k_rho_min(const double* __restrict__ rho, size_t n, DevScalars* sc) {
  pdl_enter();
  rho_min_body(rho, n, sc, blockIdx.x, gridDim.x);
}

// Eq. (33) after the solve, from the explicitly split velocity u_pre written by
// the right-hand-side kernel:  u^{n+1} = u_pre - (dt/rho_0) G p^{n+1}.
// One thread per (i, j, k) with 0 <= j <= ny: x and z faces of cell (i, j, k)
// (j < ny) and the y face j; wall faces keep v_pre (= v*).  p is read as pairs
// (pdf) or as FP64 (p64); with both given, p64 receives p in FP64.
__global__ void __launch_bounds__(256) k_correct_pre(GridDev g, double dt, const df* __restrict__ upre,
                                                     const df* __restrict__ vpre, const df* __restrict__ wpre,
                                                     const df* __restrict__ pdf, double* p64, const DevScalars* sc,
                                                     double* u_out, double* v_out, double* w_out) {
  pdl_enter();
  const uint32_t nx = (uint32_t)g.nx, ny = (uint32_t)g.ny;
  const uint32_t total = (uint32_t)g.nz * (ny + 1) * nx;
  const StencilConst K = sc->K;
  auto P = [&](size_t c) -> df { return pdf ? pdf[c] : d2df(p64[c]); };
  constexpr int U = 2;  // faces per thread per round, loads issued first
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t t0 = blockIdx.x * blockDim.x + threadIdx.x; t0 < total; t0 += U * stride) {
    df vp[U], up[U], wp[U], p0[U], pym[U], pxm[U], pzm[U];
    size_t cc[U];
    int jj[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t t = t0 + u * stride;
      jj[u] = -1;
      if (t >= total) continue;
      const uint32_t r = fdiv(t, g.fd_nx);
      const int i = (int)(t - r * nx);
      const int k = (int)fdiv(r, g.fd_nyp1);
      const int j = (int)(r - (uint32_t)k * (ny + 1));
      jj[u] = j;
      vp[u] = vpre[t];
      if (j < (int)ny) {
        const Nbr n = neighbours(g, i, j, k);
        cc[u] = n.c;
        up[u] = upre[n.c];
        wp[u] = wpre[n.c];
        p0[u] = P(n.c);
        pxm[u] = P(n.xm);
        pzm[u] = P(n.zm);
        pym[u] = (j > 0) ? P(n.c - nx) : p0[u];
      } else if (g.top_open) {
        p0[u] = P(((size_t)k * ny + (ny - 1)) * nx + i);  // the top cell below the open face
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int j = jj[u];
      if (j < 0) continue;
      const uint32_t t = t0 + u * stride;
      if (j == (int)ny && g.top_open) {  // open top: the ghost -p of the cell below
        v_out[t] = df2d(df_subz(vp[u], df_mulz(K.gy, df_subz(df_neg(p0[u]), p0[u]))));
        continue;
      }
      if (j == 0 || j == (int)ny) {
        v_out[t] = df2d(vp[u]);
        if (j == (int)ny) continue;
      } else {
        v_out[t] = df2d(df_subz(vp[u], df_mulz(K.gy, df_subz(p0[u], pym[u]))));
      }
      const size_t c = cc[u];
      u_out[c] = df2d(df_subz(up[u], df_mulz(K.gx, df_subz(p0[u], pxm[u]))));
      w_out[c] = df2d(df_subz(wp[u], df_mulz(K.gz, df_subz(p0[u], pzm[u]))));
      if (pdf && p64) p64[c] = df2d(p0[u]);
    }
  }
}

// Eq. (33) from the raw inputs:  u^{n+1} = u* - (dt/rho_0)(G p - beta_f G p_hat),
// using 1/rho_f - 1/rho_0 = -beta_f/rho_0.  In-place (u_out == u) is allowed:
// every thread reads u*, v*, w* only at the faces it writes.  All of a thread's
// inputs (the cell and its three lower neighbours, the three velocities) are
// read before its first store: the outputs may alias the velocities, so loads
// written after a store cannot move above it, and three rounds of latency per
// cell were what the kernel waited for.
template <int RULE>
__global__ void __launch_bounds__(256) k_correct_full(GridDev g, StencilIn in, const DevScalars* sc, double* u_out,
                                                      double* v_out, double* w_out) {
  pdl_enter();
  const uint32_t nx = (uint32_t)g.nx, ny = (uint32_t)g.ny;
  const uint32_t total = (uint32_t)g.nz * (ny + 1) * nx;
  const StencilConst K = sc->K;
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    const uint32_t r = fdiv(t, g.fd_nx);
    const int i = (int)(t - r * nx);
    const int k = (int)fdiv(r, g.fd_nyp1);
    const int j = (int)(r - (uint32_t)k * (ny + 1));
    const double vs = in.v[t];
    if (j == g.ny) {  // top face: a wall keeps v*
      if (!g.top_open) {
        v_out[t] = vs;
        continue;
      }
      // open top: the face between the top cell and its ghost (-p, -p_hat, same density)
      const uint32_t ct = ((uint32_t)k * ny + (ny - 1)) * nx + i;
      const df pt = d2df(in.p[ct]), ht = phat_df(in.pn, in.pnm1, ct), rt = rho_cell<RULE>(d2df(__ldg(in.rho + ct)), K);
      const df b = beta_cells<RULE, false>(rt, rt, K);
      const df gp = df_subz(df_neg(pt), pt), gh = df_subz(df_neg(ht), ht);
      v_out[t] = df2d(df_subz(d2df(vs), df_mulz(K.gy, df_subz(gp, df_mulz(b, gh)))));
      continue;
    }
    const Nbr n = neighbours(g, i, j, k);
    const size_t at[4] = {n.c, n.xm, j > 0 ? n.c - nx : n.c, n.zm};
    double p[4], a[4], b[4], q[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      p[m] = in.p[at[m]];
      a[m] = __ldg(in.pn + at[m]);
      b[m] = __ldg(in.pnm1 + at[m]);
      q[m] = __ldg(in.rho + at[m]);
    }
    const double us = in.u[n.c], ws = in.w[n.c];
    const df p0 = d2df(p[0]), h0 = phat_of(a[0], b[0]), r0 = rho_cell<RULE>(d2df(q[0]), K);
    auto corrected = [&](double v, int m, const df& gk) {
      const df bf = beta_cells<RULE, false>(rho_cell<RULE>(d2df(q[m]), K), r0, K);
      const df gp = df_subz(p0, d2df(p[m])), gh = df_subz(h0, phat_of(a[m], b[m]));
      return df2d(df_subz(d2df(v), df_mulz(gk, df_subz(gp, df_mulz(bf, gh)))));
    };
    const double un = corrected(us, 1, K.gx), vn = j > 0 ? corrected(vs, 2, K.gy) : vs, wn = corrected(ws, 3, K.gz);
    u_out[n.c] = un;
    v_out[t] = vn;
    w_out[n.c] = wn;
  }
}

__global__ void __launch_bounds__(256) k_df_to_d(const df* __restrict__ a, double* out, size_t n) {
  pdl_enter();
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    out[i] = df2d(a[i]);
}

__global__ void k_refine_check(DevScalars* sc, int smax, int off, cudaGraphConditionalHandle handle,
                               int use_handle) {
  pdl_enter();
  if (threadIdx.x != 0) return;
  const int cont = refine_decide(sc, smax, off);
  if (use_handle) cudaGraphSetConditional(handle, cont);
}

__global__ void __launch_bounds__(256, 4) k_correct_check(GridDev g, const df* __restrict__ upre,
                                                       const df* __restrict__ vpre, const df* __restrict__ wpre,
                                                       const df* __restrict__ pdf, const df* __restrict__ fdf,
                                                       DevScalars* sc) {
  pdl_enter();
  correct_check_tile(g, upre, vpre, wpre, pdf, fdf, sc, blockIdx.x, gridDim.x);
}

__global__ void k_make_const(GridDev g, DevScalars* sc, double dt) {
  pdl_enter();
  if (threadIdx.x == 0) sc->K = make_const(g, read_rho0(sc), dt);
}

__global__ void k_set_rho0(DevScalars* sc, double rho0) {
  pdl_enter();
  if (threadIdx.x == 0) sc->rho0_bits = (unsigned long long)__double_as_longlong(rho0);
}

// Eq. (31): S = -(1 - C) comp_g - C comp_l + mdot (1/rho_g - 1/rho_l) in pairs;
// zero in under-resolved interface cells (mask set, 0 < C < 1); the one-fluid
// density rho = rho_g (1 - C) + rho_l C when rho is given.  C's range tests
// run on the FP64 bit pattern (C >= 0).
__global__ void __launch_bounds__(256) k_div_constraint(size_t n, const double* __restrict__ C,
                                                        const double* __restrict__ comp_g,
                                                        const double* __restrict__ comp_l,
                                                        const double* __restrict__ mdot,
                                                        const double* __restrict__ rho_g,
                                                        const double* __restrict__ rho_l,
                                                        const unsigned char* __restrict__ mask, double* S,
                                                        double* rho) {
  pdl_enter();
  const df one = {1.0f, 0.0f};
  for (size_t c = blockIdx.x * (size_t)blockDim.x + threadIdx.x; c < n; c += (size_t)gridDim.x * blockDim.x) {
    const double cd = __ldg(C + c);
    const df vc = d2df(cd);
    const df rg = d2df(__ldg(rho_g + c)), rl = d2df(__ldg(rho_l + c));
    const df omc = df_subz(one, vc);  // 1 - C
    const df s = df_addz(df_subz(df_neg(df_mulz(omc, d2df(__ldg(comp_g + c)))), df_mulz(vc, d2df(__ldg(comp_l + c)))),
                         df_mulz(d2df(__ldg(mdot + c)), df_subz(df_recip(rg), df_recip(rl))));
    const unsigned long long cb = (unsigned long long)__double_as_longlong(cd);
    const bool interface_cell = cb > 0ull && cb < 0x3FF0000000000000ull;  // 0 < C < 1
    S[c] = (mask && mask[c] && interface_cell) ? 0.0 : df2d(s);
    if (rho) rho[c] = df2d(df_addz(df_mulz(rg, omc), df_mulz(rl, vc)));
  }
}

namespace {
unsigned grid_for(size_t total, size_t cap) {
  size_t b = (total + 255) / 256;
  if (b > cap) b = cap;
  if (b == 0) b = 1;
  return (unsigned)b;
}
// One wave of 256-thread CTAs: the SMs times the CTAs of `kernel` resident per
// SM (taken once per kernel).  The grid-stride correction kernels launched
// this way keep every resident slot busy to the end; several waves of short
// CTAs measured slower (230 against 216 us at 256^3 for the correction check:
// the slots refill unevenly between waves).
template <auto kernel>
size_t one_wave() {
  static const size_t ctas = [] {
    int dev = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                  cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 256, 0) != cudaSuccess || per_sm < 1) {
      cudaGetLastError();
      return (size_t)152 * 4;
    }
    return (size_t)sms * (size_t)per_sm;
  }();
  return ctas;
}
}  // namespace

cudaError_t launch_div_constraint(size_t n, const double* C, const double* comp_g, const double* comp_l,
                                  const double* mdot, const double* rho_g, const double* rho_l,
                                  const unsigned char* mask, double* S, double* rho, cudaStream_t st) {
  launch_pdl(k_div_constraint, grid_for(n, (size_t)152 * 16), 256, 0, st, n, C, comp_g, comp_l, mdot, rho_g, rho_l, mask,
             S, rho);
  return cudaGetLastError();
}

cudaError_t launch_init_scalars(DevScalars* sc, double rho0, double tol, int keep_rho0, cudaStream_t st,
                                double* out_p, double* out_u, double* out_v, double* out_w) {
  launch_pdl(k_init_scalars, 1, 32, 0, st, sc, rho0, tol, keep_rho0, out_p, out_u, out_v, out_w);
  return cudaGetLastError();
}

cudaError_t launch_set_rho0(DevScalars* sc, double rho0, cudaStream_t st) {
  launch_pdl(k_set_rho0, 1, 32, 0, st, sc, rho0);
  return cudaGetLastError();
}

cudaError_t launch_make_const(const GridDev& g, DevScalars* sc, double dt, cudaStream_t st) {
  launch_pdl(k_make_const, 1, 32, 0, st, g, sc, dt);
  return cudaGetLastError();
}

cudaError_t launch_rho_min(const double* rho, size_t n, DevScalars* sc, cudaStream_t st) {
  launch_pdl(k_rho_min, grid_for(n, 152 * 8), 256, 0, st, rho, n, sc);
  return cudaGetLastError();
}

cudaError_t launch_correct_pre(const GridDev& g, double dt, const df* upre, const df* vpre, const df* wpre,
                               const df* pdf, double* p64, const DevScalars* sc, double* u_out, double* v_out,
                               double* w_out, cudaStream_t st) {
  const size_t total = (size_t)g.nz * (g.ny + 1) * g.nx;
  launch_pdl(k_correct_pre, grid_for(total, one_wave<k_correct_pre>()), 256, 0, st, g, dt, upre, vpre, wpre, pdf, p64, sc,
             u_out, v_out, w_out);
  return cudaGetLastError();
}

cudaError_t launch_correct_full(const GridDev& g, const StencilIn& in, const DevScalars* sc, double* u_out,
                                double* v_out, double* w_out, cudaStream_t st) {
  const size_t total = (size_t)g.nz * (g.ny + 1) * g.nx;
  if (in.face_rule == 0)
    launch_pdl(k_correct_full<0>, grid_for(total, one_wave<k_correct_full<0>>()), 256, 0, st, g, in, sc, u_out, v_out,
               w_out);
  else
    launch_pdl(k_correct_full<1>, grid_for(total, one_wave<k_correct_full<1>>()), 256, 0, st, g, in, sc, u_out, v_out,
               w_out);
  return cudaGetLastError();
}

cudaError_t launch_correct_check(const GridDev& g, const df* upre, const df* vpre, const df* wpre, const df* pdf,
                                 const df* fdf, DevScalars* sc, cudaStream_t st) {
  const size_t total = (size_t)g.nz * (g.ny + 1) * g.nx;
  launch_pdl(k_correct_check, grid_for(total, one_wave<k_correct_check>()), 256, 0, st, g, upre, vpre, wpre, pdf, fdf, sc);
  return cudaGetLastError();
}

cudaError_t launch_df_to_d(const df* a, double* out, size_t n, cudaStream_t st) {
  launch_pdl(k_df_to_d, grid_for(n, (size_t)152 * 32), 256, 0, st, a, out, n);
  return cudaGetLastError();
}

cudaError_t launch_refine_check(DevScalars* sc, int smax, int off, cudaGraphConditionalHandle handle,
                                int use_handle, cudaStream_t st) {
  launch_pdl(k_refine_check, 1, 32, 0, st, sc, smax, off, handle, use_handle);
  return cudaGetLastError();
}

}  // namespace ppe
