// Right-hand side of the split pressure Poisson equation, Eq. (34).
//
//   f = D[beta_f G p_hat] + (rho_0/dt)(D u* - S),  beta_f = 1 - rho_0/rho_f,
//   p_hat = 2 p^n - p^{n-1}                                        (Eq. (32))
//
// Written per face as u_pre_f = u*_f + (dt/rho_0) beta_f (G p_hat)_f, the explicitly
// split velocity of Eq. (33) (since 1/rho_f - 1/rho_0 = -beta_f/rho_0,
// u^{n+1}_f = u_pre_f - (dt/rho_0) (G p^{n+1})_f), so that
//   f = (rho_0/dt) (D u_pre - S).
// This kernel stores u_pre and f, leaving only the pressure-gradient term for
// the kernel that runs after the solve.
//
// Arithmetic: p_hat is formed by one FP64 fused multiply-add; it and the other
// FP64 inputs are split into float pairs with integer operations (dfloat.cuh)
// and every face and cell value is formed in pair arithmetic.
//
// Blocking: a CTA owns `tj` consecutive y-lines for a chunk of `kc` z-planes and
// marches upward in z.  Grids up to 512 wide take the column-stack form
// (rhs.cuh), wider ones the general march below: each thread owns fixed (i, j)
// columns of the tile and keeps in registers the next plane's p_hat and rho
// and the value of the lower z face of its cells; shared memory holds the
// current plane's p_hat and rho (the tj lines plus one halo line on each side)
// and the x- and y-face values.  Each input value is converted once per CTA
// (plus halo lines), each face is evaluated once.  f is written as float pairs
// (the forward x transform reads it back, k_xfwd) and/or as FP64.
#include "dfloat.cuh"
#include "ppe_internal.h"
#include "pdl.cuh"
#include "stencil.cuh"
#include "rhs.cuh"

namespace ppe {

// CPT: columns per thread (tj * nx <= CPT * kRhsThreads); RULE: face density
// rule (0 arithmetic, 1 harmonic); PROJ: the projection's outputs (f as pairs
// and u_pre, v_pre, w_pre always written, f as FP64 when given) or, with
// PROJ = false, f as FP64 only (ppe_rhs)
template <int CPT, int RULE, bool PROJ>
__global__ void __launch_bounds__(kRhsThreads, CPT == 4 ? 2 : 1)
    k_rhs_march(GridDev g, StencilIn in, DevScalars* sc, RhsOut out, int tj, int kc) {
  pdl_enter();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nx = g.nx, ny = g.ny, nz = g.nz;
  const int ntile = (ny + tj - 1) / tj;
  const int jt = blockIdx.x % ntile, kci = blockIdx.x / ntile;
  const int j0 = jt * tj, k0 = kci * kc;
  const int steps = min(kc, nz - k0);
  const int nl = tj + 2;  // lines of the current plane held in shared memory (with halos)

  // shared: current plane p_hat and rho (nl lines), x-face and y-face values
  df* P = reinterpret_cast<df*>(smem_raw);  // [nl][nx]
  df* R = P + nl * nx;                      // [nl][nx]
  df* QX = R + nl * nx;                     // [tj][nx]
  df* QY = QX + tj * nx;                    // [tj+1][nx]

  const StencilConst K = sc->K;  // formed once per call by k_make_const
  // 32-bit element offsets (grids up to 1024^3 stay below 2^32)
  const uint32_t plane = (uint32_t)ny * (uint32_t)nx;
  const uint32_t vplane = (uint32_t)(ny + 1) * (uint32_t)nx;
  const int ncol = tj * nx;

  // this thread's columns (i, jj), fixed for the whole march
  int ci[CPT], cj[CPT];
  bool cv[CPT];
#pragma unroll
  for (int u = 0; u < CPT; ++u) {
    const int c = threadIdx.x + u * kRhsThreads;
    cj[u] = (int)fdiv((uint32_t)c, g.fd_nx);
    ci[u] = c - cj[u] * nx;
    cv[u] = c < ncol && j0 + cj[u] < ny;
  }
  // registers: p_hat, rho of the plane above the current one; Q of the lower z face
  df P1[CPT], R1[CPT], QZ[CPT];

  auto cell = [&](int kk, int j, int i) -> uint32_t { return (uint32_t)kk * plane + (uint32_t)(j * nx + i); };
  auto wrapk = [&](int kk) { return kk < 0 ? kk + nz : (kk >= nz ? kk - nz : kk); };  // kk in [-nz, 2 nz)

  auto face = [&](df rl, df rh, df pl, df ph, df us, df gh) {
    return face_upre<RULE, false>(rl, rh, pl, ph, us, gh, K);
  };

  // own columns of plane kk into (pv, rv)
  auto load_cols = [&](int kk, df* pv, df* rv) {
    kk = wrapk(kk);
    double a[CPT], b[CPT], r[CPT];
#pragma unroll
    for (int u = 0; u < CPT; ++u) {
      a[u] = 0.0; b[u] = 0.0; r[u] = 1.0;
      if (cv[u]) {
        const uint32_t c = cell(kk, j0 + cj[u], ci[u]);
        a[u] = __ldg(in.pn + c);
        b[u] = __ldg(in.pnm1 + c);
        r[u] = __ldg(in.rho + c);
      }
    }
#pragma unroll
    for (int u = 0; u < CPT; ++u) {
      pv[u] = phat_of(a[u], b[u]);  // p_hat = 2 p^n - p^{n-1}
      rv[u] = rho_cell<RULE>(d2df(r[u]), K);
    }
  };
  // halo lines j0-1 and j0+tj of plane kk into shared lines 0 and nl-1
  auto load_halo = [&](int kk) {
    kk = wrapk(kk);
    for (int idx = threadIdx.x; idx < 2 * nx; idx += kRhsThreads) {
      const int h = idx >= nx, i = idx - h * nx;
      const int j = h ? j0 + tj : j0 - 1;
      const int l = h ? nl - 1 : 0;
      df pv = {0.0f, 0.0f}, rv = {1.0f, 0.0f};
      if (j >= 0 && j < ny) {
        const uint32_t c = cell(kk, j, i);
        pv = phat_of(__ldg(in.pn + c), __ldg(in.pnm1 + c));
        rv = rho_cell<RULE>(d2df(__ldg(in.rho + c)), K);
      }
      P[l * nx + i] = pv;
      R[l * nx + i] = rv;
    }
  };
  // z face kf (between planes kf-1 and kf) of own columns from (pl, rl) below and (ph, rh) above
  auto z_face = [&](int kf, const df* pl, const df* rl, const df* ph, const df* rh, bool owned, df* q) {
    kf = wrapk(kf);
    double ws[CPT];
#pragma unroll
    for (int u = 0; u < CPT; ++u) ws[u] = cv[u] ? __ldg(in.w + cell(kf, j0 + cj[u], ci[u])) : 0.0;
#pragma unroll
    for (int u = 0; u < CPT; ++u) {
      q[u] = {0.0f, 0.0f};
      if (!cv[u]) continue;
      q[u] = face(rl[u], rh[u], pl[u], ph[u], d2df(ws[u]), K.gz);
      if (PROJ && owned) out.wpre[cell(kf, j0 + cj[u], ci[u])] = q[u];
    }
  };

  // raw next-step loads, issued a phase ahead of their use
  double us_[CPT], ss_[CPT], ws_[CPT];
  auto load_step = [&](int k) {  // u* and S of plane k, w* of face k+1, own columns
    const int kw = wrapk(k + 1);
#pragma unroll
    for (int u = 0; u < CPT; ++u) {
      us_[u] = cv[u] ? __ldg(in.u + cell(k, j0 + cj[u], ci[u])) : 0.0;
      ss_[u] = cv[u] ? __ldg(in.S + cell(k, j0 + cj[u], ci[u])) : 0.0;
      ws_[u] = cv[u] ? __ldg(in.w + cell(kw, j0 + cj[u], ci[u])) : 0.0;
    }
  };

  // prologue: plane k0 in shared memory (own lines from registers, halos
  // loaded), face k0 from planes k0-1 and k0, plane k0+1 in registers
  {
    df P0[CPT], R0[CPT];
    load_cols(k0 - 1, P1, R1);
    load_cols(k0, P0, R0);
    z_face(k0, P1, R1, P0, R0, true, QZ);
#pragma unroll
    for (int u = 0; u < CPT; ++u)
      if (threadIdx.x + u * kRhsThreads < ncol) {
        P[(cj[u] + 1) * nx + ci[u]] = P0[u];
        R[(cj[u] + 1) * nx + ci[u]] = R0[u];
      }
    load_halo(k0);
    load_cols(k0 + 1, P1, R1);
    load_step(k0);
  }
  __syncthreads();

  float vmax = 0.0f, smax = 0.0f, wmax = 0.0f;
  df wsum = {0.0f, 0.0f};  // wall flux v*(ny) - v*(0) of this CTA's wall faces
  for (int st = 0; st < steps; ++st) {
    const int k = k0 + st;
    const bool more = st + 1 < steps;
    // raw p^n, p^{n-1}, rho of plane k+2 (own columns): in flight during A and B
    double rp[CPT], rm[CPT], rr[CPT];
    if (more) {
      const int k2 = wrapk(k + 2);
#pragma unroll
      for (int u = 0; u < CPT; ++u) {
        rp[u] = 0.0; rm[u] = 0.0; rr[u] = 1.0;
        if (cv[u]) {
          const uint32_t c = cell(k2, j0 + cj[u], ci[u]);
          rp[u] = __ldg(in.pn + c);
          rm[u] = __ldg(in.pnm1 + c);
          rr[u] = __ldg(in.rho + c);
        }
      }
    }
    // ---- phase A: faces of plane k (x, y from shared; z face k+1 from registers)
#pragma unroll
    for (int u = 0; u < CPT; ++u) {
      if (threadIdx.x + u * kRhsThreads >= ncol) continue;
      df q = {0.0f, 0.0f};
      if (cv[u]) {
        const int r = (cj[u] + 1) * nx;
        const int i = ci[u], im = (i == 0) ? nx - 1 : i - 1;
        q = face(R[r + im], R[r + i], P[r + im], P[r + i], d2df(us_[u]), K.gx);
        if (PROJ) out.upre[cell(k, j0 + cj[u], i)] = q;
      }
      QX[cj[u] * nx + ci[u]] = q;
    }
    {
      constexpr int UY = 4;
      const int ny_faces = (tj + 1) * nx;
      for (int b0 = 0; b0 < ny_faces; b0 += UY * kRhsThreads) {
        double vv[UY];
#pragma unroll
        for (int u = 0; u < UY; ++u) {
          const int idx = b0 + u * kRhsThreads + threadIdx.x;
          const int jf = (int)fdiv((uint32_t)idx, g.fd_nx), i = idx - jf * nx;
          vv[u] = (idx < ny_faces && j0 + jf <= ny)
                      ? __ldg(in.v + ((uint32_t)k * vplane + (uint32_t)((j0 + jf) * nx + i))) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < UY; ++u) {
          const int idx = b0 + u * kRhsThreads + threadIdx.x;
          if (idx >= ny_faces) continue;
          const int jf = (int)fdiv((uint32_t)idx, g.fd_nx), i = idx - jf * nx;
          const int j = j0 + jf;  // face between cells j-1 and j
          df q = {0.0f, 0.0f};
          if (j <= ny) {
            const uint32_t cvv = (uint32_t)k * vplane + (uint32_t)(j * nx + i);
            const df vs = d2df(vv[u]);
            const bool own = (jf < tj) || (j == ny);
            if (j == ny && g.top_open) {  // open top: p = 0 on the face, ghost -p_hat above
              const int rl = jf * nx + i;
              q = face(R[rl], R[rl], P[rl], df_neg(P[rl]), vs, K.gy);
            } else if (j == 0 || j == ny) {  // wall: u_pre = v*
              q = vs;
              wsum = (j == ny) ? df_addz(wsum, vs) : df_subz(wsum, vs);
              wmax = fmaxf(wmax, fabsf(vs.hi));
            } else {
              const int rl = jf * nx + i, rh = (jf + 1) * nx + i;
              q = face(R[rl], R[rh], P[rl], P[rh], vs, K.gy);
            }
            if (PROJ && own) out.vpre[cvv] = q;
          }
          QY[idx] = q;
        }
      }
    }
    df QZup[CPT];
#pragma unroll
    for (int u = 0; u < CPT; ++u) {
      QZup[u] = {0.0f, 0.0f};
      if (!cv[u]) continue;
      const int r = (cj[u] + 1) * nx + ci[u];
      QZup[u] = face(R[r], R1[u], P[r], P1[u], d2df(ws_[u]), K.gz);
      if (PROJ && k + 1 < k0 + steps) out.wpre[cell(wrapk(k + 1), j0 + cj[u], ci[u])] = QZup[u];
    }
    __syncthreads();
    // ---- phase B: cells of plane k
#pragma unroll
    for (int u = 0; u < CPT; ++u) {
      if (!cv[u]) continue;
      const int i = ci[u], jj = cj[u];
      const int ip = (i + 1 == nx) ? 0 : i + 1;
      // f = (rho_0/dt) (D u_pre - S)
      const df dxq = df_mulz(df_subz(QX[jj * nx + ip], QX[jj * nx + i]), K.cx);
      const df dyq = df_mulz(df_subz(QY[(jj + 1) * nx + i], QY[jj * nx + i]), K.cy);
      const df dzq = df_mulz(df_subz(QZup[u], QZ[u]), K.cz);
      const uint32_t c = cell(k, j0 + jj, i);
      const df sv = d2df(ss_[u]);
      const df f = df_norm(df_subz(df_addz(df_addz(dxq, dyq), dzq), df_mulz(K.c, sv)));
      smax = fmaxf(smax, fabsf(sv.hi));
      if (PROJ) out.fdf[c] = f;
      if (!PROJ || out.f64) out.f64[c] = df2d(f);
      vmax = fmaxf(vmax, fabsf(f.hi));
      QZ[u] = QZup[u];
    }
    if (more) {
      load_step(k + 1);  // next step's u*, S, w*: in flight during the rest of this step
      __syncthreads();
      // ---- phase C: plane k+1 becomes current; plane k+2 (loaded above) into registers
#pragma unroll
      for (int u = 0; u < CPT; ++u)
        if (threadIdx.x + u * kRhsThreads < ncol) {
          P[(cj[u] + 1) * nx + ci[u]] = P1[u];
          R[(cj[u] + 1) * nx + ci[u]] = R1[u];
        }
      load_halo(k + 1);
#pragma unroll
      for (int u = 0; u < CPT; ++u) {
        P1[u] = phat_of(rp[u], rm[u]);
        R1[u] = rho_cell<RULE>(d2df(rr[u]), K);
      }
      __syncthreads();
    }
  }
  block_max_to(&sc->fmax_bits, vmax);
  block_max_to(&sc->smax_bits, smax);
  block_max_to(&sc->wallv_bits, wmax);
  // wall tiles: the CTA's wall flux, totalled in a fixed order by a later
  // kernel (finish_sums), so no grid-wide fence here
  if (j0 == 0 || j0 + tj >= ny) block_pair_sums(wsum, df{0.0f, 0.0f}, sc->part + blockIdx.x);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    sc->rhs_tiles = ntile;
    sc->rhs_chunks = (nz + kc - 1) / kc;
  }
}

__global__ void k_finish_sums(GridDev g, DevScalars* sc) {
  pdl_enter();
  finish_sums(sc, g);
}

// Column-stack form of the march (rhs.cuh): one CTA of BT threads at most per
// tile.  What bounds it: instruction issue and the latency of a step's loads
// (528 warp instructions per 32 cells, 683 before, at 71 % issue; raw values
// prefetched into shared memory, whole stacks per CTA).  256^3, projection outputs: 371 -> 305
// us (1.61 GB moved, 5.3 TB/s); 384 x 256 x 384 (the general march before):
// 1248 -> 690; 192^3 (a quarter of the threads idle before): 201 -> 132; 128^3:
// 66 -> 45.  The register budget (80 a thread for S <= 2: three CTAs of 256 threads
// or two of 384 per SM) keeps the loads of the next plane in flight; a CTA of
// up to 512 threads runs alone on its SM.
template <int S, int RULE, bool PROJ, int BT, int NXC>
__global__ void __launch_bounds__(BT, BT == 256 ? (S <= 2 ? 3 : (S == 4 ? 2 : 1)) : (BT == 384 && S <= 2 ? 2 : 1))
    k_rhs_stack(GridDev g, StencilIn in, DevScalars* sc, RhsOut out, int kc) {
  pdl_enter();
  rhs_stack_tile<S, RULE, PROJ, NXC>(g, in, sc, out, kc, blockIdx.x);
}


namespace {
// Stacks of a launch: those that fill its grid best, within the block bound of
// the instance of this nx (two at least where it gives a thread one halo cell).
// Eight lines a thread: 256 threads at most, whose registers and raw slots
// (129 KB) an SM holds.
int launch_stacks(int nx, int ny, int S) {
  if (S == 8) return stacks_of(nx, ny, S, 1, 256);
  const int s0 = stacks_of(nx);
  return stacks_of(nx, ny, S, s0 > 1 ? 2 : 1, stack_bound(stack_threads(nx, s0)));
}
size_t stack_smem(int nx, int stacks, int S) {
  const size_t tj = (size_t)stacks * S, nl = tj + 2;
  return sizeof(df) * (2 * nl * nx + tj * nx) + sizeof(double) * rhs_slots(S, 2) * stack_threads(nx, stacks);
}
}  // namespace

// Lines per tile: the stack form (nx <= 512) has launch_stacks stacks of
// `lines` lines each; the general form has `lines` lines.
int rhs_tile_lines(int nx, int ny, int lines) {
  return nx <= kRhsStackNx ? launch_stacks(nx, ny, lines) * lines : lines;
}

size_t rhs_smem(int nx, int ny, int lines) {
  if (nx <= kRhsStackNx) return stack_smem(nx, launch_stacks(nx, ny, lines), lines);
  const size_t tj = lines, nl = tj + 2;
  return sizeof(df) * (2 * nl * nx + tj * nx + (tj + 1) * nx);
}

// Planes per CTA of the column-stack form at S = 2.  A CTA marches kc planes
// after a prologue worth about one and a half; with N CTAs on `slots` resident
// places the march takes (N / slots + 1/2) (kc + 3/2) steps, and where one wave
// holds them all, kc + 3/2 longer steps, the shorter the emptier the SMs
// (measured over kc = 1 .. 32 at 32^3 .. 384 x 256 x 384: within 4 % of the best
// of each, except 12 % on 48 x 192 x 32; the fixed kc = 8 before cost 32^3 24
// instead of 10 us, 64^3 24 instead of 14).
int rhs_planes(int nx, int ny, int nz) {
  if (nx > kRhsStackNx) return nz < 8 ? nz : 8;
  const int stacks = launch_stacks(nx, ny, 2), threads = stack_threads(nx, stacks);
  const int bound = stack_bound(threads);
  const double slots = 152.0 * (bound == 512 ? 1 : 65536 / (80 * threads));
  const int ntile = (ny + 2 * stacks - 1) / (2 * stacks);
  int best = 1;
  double least = 0.0;
  for (int kc = 1; kc <= 12 && kc <= nz; ++kc) {
    const double w = ntile * ((nz + kc - 1) / kc) / slots;
    const double t = (w <= 1.0 ? 0.75 + 0.7 * w : w + 0.5) * (kc + 1.5);
    if (kc == 1 || t < least) {
      least = t;
      best = kc;
    }
  }
  return best;
}

int rhs_max_lines(int nx) {
  if (nx <= kRhsThreads) return kRhsMaxCols;
  int tj = 8;
  while (tj > 1 && tj * nx > kRhsThreads * kRhsMaxCols) tj /= 2;
  return tj;
}

namespace {
// Calls f(kernel) with the column-stack instance for (S, rule, proj, nx).
// The default S = 2 has instances with nx compiled in for the widths 2^a and
// 3 2^a that are whole warps, up to 384: their CTAs are whole stacks (threads =
// stacks * nx) and offsets are immediates.  Without and with them (projection,
// min rho_0, cubes; 384 x 256 x 128): 32 11.6 -> 9.7 us, 64 16 -> 14, 96 36 -> 27,
// 128 59 -> 49, 192 170 -> 136, 256 371 -> 304, 384 291 -> 243; ppe_rhs: 128
// 55 -> 45, 192 164 -> 131, 256 364 -> 305 (the form with a flux per face took
// 349).  An instance would buy 4 % at 144 (93 -> 89), 2 % at 512 (349 -> 341) and
// 2 us at 48 (12.6 -> 10.7), for four kernels of build each.  The other heights
// take any nx.
template <int S, int RULE, bool PROJ, class F>
void stack_instance(int nx, int threads, F&& f) {
  if constexpr (S == 2) {
#define PPE_NX(N) \
    case N: return f(k_rhs_stack<2, RULE, PROJ, stack_bound(stack_threads(N, stacks_of(N))), N>);
    switch (nx) {
      PPE_NX(32) PPE_NX(64) PPE_NX(96) PPE_NX(128) PPE_NX(192) PPE_NX(256) PPE_NX(384)
      default: break;
    }
#undef PPE_NX
  }
  if constexpr (S < 8) {
    if constexpr (S <= 2)
      if (threads > 256 && threads <= 384) return f(k_rhs_stack<S, RULE, PROJ, 384, 0>);
    if (threads > 256) return f(k_rhs_stack<S, RULE, PROJ, 512, 0>);
  }
  f(k_rhs_stack<S, RULE, PROJ, 256, 0>);
}

template <int S, class F>
void stack_kernel(int nx, int threads, int rule, bool proj, F&& f) {
  if (rule == 0) {
    if (proj) stack_instance<S, 0, true>(nx, threads, f);
    else stack_instance<S, 0, false>(nx, threads, f);
  } else {
    if (proj) stack_instance<S, 1, true>(nx, threads, f);
    else stack_instance<S, 1, false>(nx, threads, f);
  }
}
}  // namespace

cudaError_t launch_rhs(const GridDev& g, const StencilIn& in, DevScalars* sc, double* f64, df* fdf, df* upre,
                       df* vpre, df* wpre, int tj, int kc, cudaStream_t st) {
  RhsOut o;
  o.f64 = f64;
  o.fdf = fdf;
  o.upre = upre;
  o.vpre = vpre;
  o.wpre = wpre;
  const int tile = rhs_tile_lines(g.nx, g.ny, tj);
  const int ntile = (g.ny + tile - 1) / tile;
  const int nchunk = (g.nz + kc - 1) / kc;
  const size_t sm = rhs_smem(g.nx, g.ny, tj);
  const int grid = ntile * nchunk;
  const bool proj = fdf != nullptr;
  if (proj && !(upre && vpre && wpre)) return cudaErrorInvalidValue;
  if (!proj && !f64) return cudaErrorInvalidValue;
  if (g.nx <= kRhsStackNx) {
    // column-stack form: tj is the stack height S
    const int threads = stack_threads(g.nx, launch_stacks(g.nx, g.ny, tj));
    cudaError_t e = cudaSuccess;
    auto go = [&](auto kernel) {
      e = allow_smem(kernel, sm);
      if (e == cudaSuccess) e = launch_pdl(kernel, grid, threads, sm, st, g, in, sc, o, kc);
    };
    switch (tj) {
      case 1: stack_kernel<1>(g.nx, threads, in.face_rule, proj, go); break;
      case 2: stack_kernel<2>(g.nx, threads, in.face_rule, proj, go); break;
      case 4: stack_kernel<4>(g.nx, threads, in.face_rule, proj, go); break;
      case 8: stack_kernel<8>(g.nx, threads, in.face_rule, proj, go); break;
      default: return cudaErrorInvalidValue;
    }
    return e != cudaSuccess ? e : cudaGetLastError();
  }
  const int cpt = tj * g.nx <= 4 * kRhsThreads ? 4 : 8;
  cudaError_t e = cudaSuccess;
  auto go = [&](auto kernel) {
    e = allow_smem(kernel, sm);
    if (e == cudaSuccess) e = launch_pdl(kernel, grid, kRhsThreads, sm, st, g, in, sc, o, tj, kc);
  };
  // instance table: [cpt][rule][proj]
#define PPE_RHS_CASE(C)                                                        \
  if (cpt == C) {                                                              \
    if (in.face_rule == 0) {                                                   \
      if (proj) go(k_rhs_march<C, 0, true>); else go(k_rhs_march<C, 0, false>); \
    } else {                                                                   \
      if (proj) go(k_rhs_march<C, 1, true>); else go(k_rhs_march<C, 1, false>); \
    }                                                                          \
  }
  PPE_RHS_CASE(4)
  PPE_RHS_CASE(8)
#undef PPE_RHS_CASE
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_finish_sums(const GridDev& g, DevScalars* sc, cudaStream_t st) {
  launch_pdl(k_finish_sums, 1, 256, 0, st, g, sc);
  return cudaGetLastError();
}

// The per-CTA maximum minus an instance's static shared memory (the reduction
// scratch, the same in every instance of a form).
size_t rhs_smem_limit(int nx) {
  cudaFuncAttributes a;
  const cudaError_t e = nx <= kRhsStackNx ? cudaFuncGetAttributes(&a, k_rhs_stack<1, 0, false, 256, 0>)
                                          : cudaFuncGetAttributes(&a, k_rhs_march<4, 0, false>);
  return e == cudaSuccess ? kSmemPerCta - a.sharedSizeBytes : 0;
}

}  // namespace ppe
