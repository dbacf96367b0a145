// Finite-volume operators of the uniform staggered (MAC) mesh used by the
// split pressure-gradient projection (Sec. 5 of the paper: velocities on face
// centres, pressure and density at cell centres; Eqs. (32)-(34)), in pair
// (double-float) arithmetic.
//
//   G q on the x face i      = (q_i - q_{i-1}) / dx          periodic in x, z
//   G q on the y face j      = (q_j - q_{j-1}) / dy,  0 on the walls j = 0, ny
//   D a at cell (i,j,k)      = (a_{i+1} - a_i)/dx + (b_{j+1} - b_j)/dy + (c_{k+1} - c_k)/dz
//   L = D G                  the 7-point Laplacian with homogeneous Neumann walls
//   rho_f                    0.5 (rho_L + rho_R) (arithmetic) or 2/(1/rho_L + 1/rho_R)
//   beta_f = 1 - rho_0/rho_f the coefficient of the explicit split term, Eq. (34)
#pragma once
#include "dfloat.cuh"
#include "ppe_internal.h"

namespace ppe {

__device__ __forceinline__ double read_rho0(const DevScalars* sc) {
  return __longlong_as_double((long long)sc->rho0_bits);
}

// Stencil constants (struct StencilConst in ppe_internal.h) from rho_0 and dt:
// the only FP64 arithmetic of a call besides the boundary conversions, done
// once by one thread (k_make_const).
__device__ __forceinline__ StencilConst make_const(const GridDev& g, double rho0, double dt) {
  StencilConst K;
  K.c = d2df(rho0 / dt);
  K.g = d2df(dt / rho0);
  K.r0h = d2df(0.5 * rho0);
  K.r02 = d2df(2.0 * rho0);
  K.idx = d2df(g.idx);
  K.idy = d2df(g.idy);
  K.idz = d2df(g.idz);
  K.gx = d2df(dt / rho0 * g.idx);
  K.gy = d2df(dt / rho0 * g.idy);
  K.gz = d2df(dt / rho0 * g.idz);
  K.lx = d2df(g.idx * g.idx);
  K.ly = d2df(g.idy * g.idy);
  K.lz = d2df(g.idz * g.idz);
  K.cx = d2df(rho0 / dt * g.idx);
  K.cy = d2df(rho0 / dt * g.idy);
  K.cz = d2df(rho0 / dt * g.idz);
  return K;
}

// What a stencil keeps per cell for the face densities: rho itself
// (arithmetic rule) or (rho_0/2)/rho (harmonic rule: beta_f is 1 minus the sum
// of the two cells' values, so the reciprocal is taken once per cell instead
// of at each of its six faces).
template <int RULE>
__device__ __forceinline__ df rho_cell(df rho, const StencilConst& K) {
  if (RULE == 0) return rho;
  return df_mulz(K.r0h, df_recipz(rho));
}

// beta_f = 1 - rho_0/rho_f from two cells' rho_cell values (unnormalised pair).
// Arithmetic rule: t = 2 rho_0/(a + b) as y + e/(a + b) with y = fl(2 rho_0 rcp(a + b))
// and e = 2 rho_0 - (a + b) y from two fused multiply-adds (the correction of
// a quotient by its remainder; relative error that of the seed squared,
// ~2^-46, as a Newton step's), so neither the reciprocal nor its product with
// 2 rho_0 is formed as a pair: 17 operations against 26.
// TAME: rho_0 is the minimum of rho, hence t <= 1 (up to its last bit) and
// 1 - t needs only the fast two-sum; a rho_0 given by the caller may be larger.
template <int RULE, bool TAME>
__device__ __forceinline__ df beta_cells(df a, df b, const StencilConst& K) {
  const df s = df_addz(a, b);
  float y, tl;  // t = y + tl
  if (RULE == 0) {
    const float rc = rcp_seed(s.hi);
    y = mul_rn(K.r02.hi, rc);
    const float e = fmaf(-s.hi, y, K.r02.hi) + fmaf(-s.lo, y, K.r02.lo);
    tl = mul_rn(e, rc);
  } else {
    y = s.hi;
    tl = s.lo;
  }
  const df d = TAME ? fast_two_sum(1.0f, -y) : two_sum(1.0f, -y);
  return {d.hi, d.lo - tl};
}

// Explicitly split velocity of one face (Eq. (33) without its G p^{n+1} term),
//   u_pre = u*_f + (dt/rho_0)(1/h) beta_f (p_hat_R - p_hat_L),  gh = (dt/rho_0)/h.
// It is also the face quantity of the right-hand side: by Eq. (34)
//   f = (rho_0/dt) (D u_pre - S),
// so no separate flux is formed (an earlier form kept Q~ = beta Delta p_hat +
// (rho_0/dt) h u* and u_pre = gh Q~: one pair product more per face).  Left
// unnormalised (the lazy operations of dfloat.cuh): the divergence, the
// correction's subtraction and its conversion to FP64 take it so.
template <int RULE, bool TAME>
__device__ __forceinline__ df face_upre(df rl, df rh, df pl, df ph, df us, df gh, const StencilConst& K) {
  return df_addz(us, df_mulz(df_mulz(beta_cells<RULE, TAME>(rl, rh, K), df_subz(ph, pl)), gh));
}

// p_hat = 2 p^n - p^{n-1} (Eq. (32)): one FP64 fused multiply-add (a single
// rounding, on the FP64 pipe, which these kernels leave otherwise idle), then
// one split into a pair
__device__ __forceinline__ df phat_of(double pn, double pnm1) { return d2df(fma(2.0, pn, -pnm1)); }

__device__ __forceinline__ df phat_df(const double* pn, const double* pnm1, size_t c) {
  return phat_of(__ldg(pn + c), __ldg(pnm1 + c));
}

struct Nbr {
  size_t c, xp, xm, zp, zm;
};

__device__ __forceinline__ Nbr neighbours(const GridDev& g, int i, int j, int k) {
  Nbr n;
  const size_t nx = (size_t)g.nx, ny = (size_t)g.ny;
  const int ip = (i + 1 == g.nx) ? 0 : i + 1;
  const int im = (i == 0) ? g.nx - 1 : i - 1;
  const int kp = (k + 1 == g.nz) ? 0 : k + 1;
  const int km = (k == 0) ? g.nz - 1 : k - 1;
  n.c = ((size_t)k * ny + j) * nx + i;
  n.xp = n.c - i + ip;
  n.xm = n.c - i + im;
  n.zp = ((size_t)kp * ny + j) * nx + i;
  n.zm = ((size_t)km * ny + j) * nx + i;
  return n;
}

__device__ __forceinline__ void block_max_to(unsigned long long* slot, float v) {
  // v >= 0; reduce over the warp in FP32, one FP64 atomic per warp with a
  // non-zero maximum (all lanes must call).  The maxima only steer the
  // refinement stop test and the reports, so the float hi part suffices.
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0 && v > 0.0f) atomicMax(slot, (unsigned long long)__double_as_longlong((double)v));
}

// Reduction of two per-thread pair values over the CTA (a fixed shuffle tree,
// then the warps in index order); thread 0 stores the pair of totals in *out.
// Every thread of the CTA must call it (blockDim.x a multiple of 32, <= 1024).
__device__ __forceinline__ void block_pair_sums(df a, df b, double2* out) {
  __shared__ df red_s[2][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  a = df_norm(a);
  b = df_norm(b);
  for (int o = 16; o > 0; o >>= 1) {
    a = df_add(a, {__shfl_down_sync(0xffffffffu, a.hi, o), __shfl_down_sync(0xffffffffu, a.lo, o)});
    b = df_add(b, {__shfl_down_sync(0xffffffffu, b.hi, o), __shfl_down_sync(0xffffffffu, b.lo, o)});
  }
  if (lane == 0) {
    red_s[0][wid] = a;
    red_s[1][wid] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a = red_s[0][0];
    b = red_s[1][0];
    for (int w = 1; w < nw; ++w) {
      a = df_add(a, red_s[0][w]);
      b = df_add(b, red_s[1][w]);
    }
    *out = make_double2(df2d(a), df2d(b));
  }
}

// Sum of part[0..n) in an order that depends only on n and blockDim.x (thread
// t takes t, t + blockDim.x, ... in turn; then a fixed shuffle and warp tree).
// Every thread of the CTA must call it; thread 0 gets the totals.
__device__ __forceinline__ void sum_parts_fixed(const double2* part, int n, double* tx, double* ty) {
  __shared__ double red_p[2][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  double x = 0.0, y = 0.0;
  // each thread adds its entries i = threadIdx.x + m blockDim.x in order of m;
  // eight loads are issued before their additions (the order is unchanged)
  constexpr int U = 8;
  for (int i0 = threadIdx.x; i0 < n; i0 += U * blockDim.x) {
    double2 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * blockDim.x;
      v[u] = i < n ? __ldcg(part + i) : make_double2(0.0, 0.0);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * blockDim.x;
      if (i < n) {
        x += v[u].x;
        y += v[u].y;
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    x += __shfl_down_sync(0xffffffffu, x, o);
    y += __shfl_down_sync(0xffffffffu, y, o);
  }
  if (lane == 0) {
    red_p[0][wid] = x;
    red_p[1][wid] = y;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    x = red_p[0][0];
    y = red_p[1][0];
    for (int w = 1; w < nw; ++w) {
      x += red_p[0][w];
      y += red_p[1][w];
    }
    *tx = x;
    *ty = y;
  }
}

// Totals of the per-CTA partial sums of the current call, formed by one CTA
// (all threads) in a kernel that runs after their producers (the kernel
// boundary orders the accesses): the sum of f from the forward x transform,
// the sum of p from the inverse one and the wall flux from the wall tiles of
// the right-hand side (lower and upper wall of each chunk of planes).  The
// three totals share one pass of loads and one tree, in an order that depends
// only on their counts and blockDim.x (thread t takes t, t + blockDim.x, ... in
// turn): a dependent loop over the chunks and two trees one after the other
// held the z pass of a small grid back (32^3: 10 us of it).
__device__ __forceinline__ void finish_sums(DevScalars* sc, const GridDev& g) {
  __shared__ double red_f[3][32];
  const size_t nynz = (size_t)g.ny * g.nz;
  const double2* const part = sc->part;
  const int xp = sc->x_parts, pp = sc->p_parts, nt = sc->rhs_tiles, nc = sc->rhs_chunks;
  const int wp = nt > 0 ? (nt > 1 ? 2 * nc : nc) : 0;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  auto walls = [&](int i) -> const double2* {  // chunk by chunk, lower then upper wall
    return nt > 1 ? part + (size_t)(i >> 1) * nt + (i & 1) * (nt - 1) : part + i;
  };
  double v[3] = {0.0, 0.0, 0.0};
  const int most = max(xp, max(pp, wp));
  constexpr int U = 2;  // loads issued before their additions (the order is unchanged; more cost the z pass registers)
  for (int i0 = threadIdx.x; i0 < most; i0 += U * blockDim.x) {
    double a[U][3];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * blockDim.x;
      a[u][0] = i < xp ? __ldcg(&part[nynz + i].x) : 0.0;
      a[u][1] = i < pp ? __ldcg(&part[2 * nynz + i].x) : 0.0;
      a[u][2] = i < wp ? __ldcg(&walls(i)->x) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * blockDim.x;
      if (i < xp) v[0] += a[u][0];
      if (i < pp) v[1] += a[u][1];
      if (i < wp) v[2] += a[u][2];
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
    for (int q = 0; q < 3; ++q) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
  }
  if (lane == 0) {
#pragma unroll
    for (int q = 0; q < 3; ++q) red_f[q][wid] = v[q];
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int w = 1; w < nw; ++w) {
#pragma unroll
    for (int q = 0; q < 3; ++q) v[q] += red_f[q][w];
  }
  const double fs = v[0], ps = v[1];
  // the sum of the p the last inverse x transform formed: the next correction's
  // zero mode is -sum(p)/ny, which adds -mean(p) to p after the inverse transforms
  // (DCT-III unscaled in its zero mode, z and x inverses scaled by 1/(nx nz))
  if (pp > 0) {
    sc->zmode = -ps / (double)g.ny;
    sc->p_parts = 0;
  }
  if (nt > 0) {
    sc->wall_flux = v[2];
    sc->rhs_ran = 1;
  }
  if (xp > 0) {
    // A mean below 2^-40 ||f||_inf is rounding noise of a compatible right-hand
    // side (its last bits depend on how the cells were grouped into CTAs); it is
    // not subtracted, which keeps the refinement's result independent of the
    // tile shapes.
    const double mean = fs / ((double)g.nx * (double)g.ny * (double)g.nz);
    const double fmax = __longlong_as_double((long long)sc->fmax_bits);
    sc->f_sum = fs;
    // (an open top has no zero mode: nothing is dropped, nothing left out)
    sc->f_mean = (!g.top_open && fabs(mean) > 0x1p-40 * fmax) ? d2df(mean) : df{0.0f, 0.0f};
    sc->f_ran = 1;
  }
}

}  // namespace ppe
