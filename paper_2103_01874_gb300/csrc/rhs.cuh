// Column-stack form of the right-hand side of Eq. (34) as a device function
// of the tile index, shared by its own kernel (k_rhs.cu) and the persistent
// batched kernel (k_batch.cu).  The arithmetic is described in k_rhs.cu.
#pragma once
#include "async.cuh"
#include "dfloat.cuh"
#include "ppe_internal.h"
#include "stencil.cuh"

namespace ppe {

constexpr int kRhsThreads = 256;  // the general march and the persistent batch
constexpr int kRhsMaxCols = 8;    // columns per thread: tj * nx <= 2048
constexpr int kRhsStackNx = 512;  // widest grid of the column-stack form

// Threads of a CTA of s stacks, and the block bound of its instance.
__host__ __device__ constexpr int stack_threads(int nx, int s) { return (s * nx + 31) / 32 * 32; }
__host__ __device__ constexpr int stack_bound(int threads) { return threads <= 256 ? 256 : threads <= 384 ? 384 : 512; }
// Work per SM of CTAs of s stacks of S lines on a grid of ny lines (ny = 0: an
// endless one): the threads that the launch bounds allow at work (an nx that
// does not divide the block leaves the rest of it idle: 192 of 256 threads at
// nx = 192, 144 at nx = 144), times the share of the tiles' lines that exist,
// each stack's halo lines weighing about a tenth of its work.
__host__ __device__ constexpr double stack_score(int nx, int ny, int S, int s) {
  const int threads = stack_threads(nx, s);
  const int ctas = stack_bound(threads) == 512 ? 1 : 65536 / (80 * threads);
  const int tile = s * S, lines = ny > 0 ? (ny + tile - 1) / tile * tile : 0;
  return ctas * s * nx / (1.0 + 0.1 / s) * (lines ? (double)ny / lines : 1.0);
}
// Stacks per CTA of the column-stack form, at least `least`, of `most` threads.
__host__ __device__ constexpr int stacks_of(int nx, int ny = 0, int S = 1, int least = 1, int most = 384) {
  int best = least;
  double score = -1.0;
  for (int s = least; stack_threads(nx, s) <= most || s == least; ++s) {
    const double v = stack_score(nx, ny, S, s);
    if (v > score) {
      score = v;
      best = s;
    }
  }
  return best;
}

struct RhsOut {
  double* f64;   // optional: f as FP64
  df* fdf;       // optional: f as pairs (kept for the residual)
  df* upre;      // optional: u_pre on x faces  [nz][ny][nx]
  df* vpre;      //           v_pre on y faces  [nz][ny+1][nx]
  df* wpre;      //           w_pre on z faces  [nz][ny][nx]
};

// Raw input values of a thread, fetched a phase or more ahead of their use.
// SMEM: they wait in shared memory (8-byte cp.async into slots of the thread's
// own, so that no barrier is needed to reuse one): kept in registers they left
// room for neither the halo's nor a second plane's loads at 80 registers a
// thread, and load latency (long scoreboard 3.7 of 9.5 cycles per instruction)
// held the march at 55 % issue; taller stacks spilled (four lines: 256^3 513
// -> 405 us, 192^3 283 -> 179, 144^3 143 -> 102).  The persistent batch keeps
// registers (k_batch.cu).
template <int NS, bool SMEM>
struct RawSlots {
  double* own;  // slot i at own[i * blockDim.x]
  double reg[SMEM ? 1 : NS];
  __device__ __forceinline__ void fetch(int i, const double* p, bool ok, double other) {
    if (SMEM) {
      if (ok) cp_async<8>(own + i * (int)blockDim.x, p);
    } else {
      reg[i] = ok ? __ldg(p) : other;
    }
  }
  // (the slot's last fetch has been waited for)
  __device__ __forceinline__ double get(int i, bool ok, double other) const {
    if (SMEM) return ok ? own[i * (int)blockDim.x] : other;
    return reg[i];
  }
  __device__ __forceinline__ void commit() {
    if (SMEM) cp_async_commit();
  }
  // all but the two newest commits have landed
  __device__ __forceinline__ void wait2() {
    if (SMEM) cp_async_wait_group<2>();
  }
};
// Slots: u*, w*, S of S lines, v* of S + 1 faces, (p^n, p^{n-1}, rho) of S lines
// and of hn halo cells.
__host__ __device__ constexpr int rhs_slots(int S, int hn) { return 3 * S + (S + 1) + 3 * S + 3 * hn; }

// Column-stack form of the march for nx <= 512 (the same face and cell
// arithmetic as k_rhs_march, bit for bit).  The CTA's threads form nstk =
// blockDim.x / nx stacks; thread (s, i) owns x position i of the S consecutive
// lines s*S .. s*S + S - 1 of the tile (tile height nstk * S lines).  The own
// lines' p_hat and rho_cell of the current plane stay in registers, so the
// thread evaluates the y faces below, between and above its lines from
// registers (only the line below and the line above its stack come from
// shared memory, as do the x neighbours), and the y-face values never go
// through shared memory; the x faces are exchanged through shared memory for
// the cell divergence.  Faces between two stacks are evaluated by both (same
// bits).
// SM: raw values in shared memory (RawSlots).
// NXC: nx where it is compiled in (0: any): line and row offsets become
// immediates, so one address per array and plane serves the S lines.
// INT: the tile and its halo lines lie strictly inside the walls (no wall or
// open-top face, every line in range) and rho_0 is the minimum of rho, so the
// boundary branches and the general form of 1 - rho_0/rho_f drop out.
template <int S, int RULE, bool PROJ, bool INT, int NXC, bool SM>
__device__ __forceinline__ void rhs_stack_body(const GridDev& g, const StencilIn& in, DevScalars* sc,
                                               const RhsOut& out, int kc, uint32_t bid) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nx = NXC ? NXC : g.nx, ny = g.ny, nz = g.nz;
  const int nstk = (int)blockDim.x / nx;
  const int tj = nstk * S;  // lines per tile
  const int ntile = (ny + tj - 1) / tj;
  const int jt = (int)(bid % ntile), kci = (int)(bid / ntile);
  const int j0 = jt * tj, k0 = kci * kc;
  const int steps = min(kc, nz - k0);
  const int nl = tj + 2;

  df* P = reinterpret_cast<df*>(smem_raw);  // [nl][nx]: row r holds tile line r - 1
  df* R = P + nl * nx;                      // [nl][nx]
  df* QX = R + nl * nx;                     // [tj][nx]

  const StencilConst K = sc->K;
  const uint32_t plane = (uint32_t)ny * (uint32_t)nx;
  const uint32_t vplane = (uint32_t)(ny + 1) * (uint32_t)nx;

  const int stk = NXC ? (int)threadIdx.x / NXC : (int)fdiv((uint32_t)threadIdx.x, g.fd_nx);
  const int i = (int)threadIdx.x - stk * nx;
  const bool active = (NXC && NXC % 32 == 0) || stk < nstk;  // (such CTAs are whole stacks)
  const int jb = stk * S;                    // first own line (tile coordinates)
  const int im = (i == 0) ? nx - 1 : i - 1;
  const int ip = (i + 1 == nx) ? 0 : i + 1;
  bool cv[S];
#pragma unroll
  for (int l = 0; l < S; ++l) cv[l] = active && (INT || j0 + jb + l < ny);
  bool fv[S + 1];
#pragma unroll
  for (int f = 0; f <= S; ++f) fv[f] = active && (INT || j0 + jb + f <= ny);

  const uint32_t own = (uint32_t)((j0 + jb) * nx + i);  // the first own line within a plane
  auto wrapk = [&](int kk) { return kk < 0 ? kk + nz : (kk >= nz ? kk - nz : kk); };  // kk in [-nz, 2 nz)
  auto at = [&](int kk) -> uint32_t { return (uint32_t)kk * plane + own; };          // own cell of line 0

  constexpr int HN = (NXC > 0 && stacks_of(NXC) > 1) ? 1 : 2;  // a thread's halo cells (such CTAs have two stacks or more)
  RawSlots<rhs_slots(S, HN), SM> raw;
  raw.own = reinterpret_cast<double*>(QX + tj * nx) + threadIdx.x;
  constexpr int S_U = 0, S_W = S, S_S = 2 * S, S_V = 3 * S, S_P = 4 * S + 1, S_H = 7 * S + 1;

  // own lines of one plane, read and converted at once (prologue)
  auto load_cols = [&](int kk, df* pv, df* rv) {
    const uint32_t c = at(wrapk(kk));
    const double *pa = in.pn + c, *pb = in.pnm1 + c, *pr = in.rho + c;
    double a[S], b[S], r[S];
#pragma unroll
    for (int l = 0; l < S; ++l) {
      a[l] = cv[l] ? __ldg(pa + l * nx) : 0.0;
      b[l] = cv[l] ? __ldg(pb + l * nx) : 0.0;
      r[l] = cv[l] ? __ldg(pr + l * nx) : 1.0;
    }
#pragma unroll
    for (int l = 0; l < S; ++l) {
      pv[l] = phat_of(a[l], b[l]);  // p_hat = 2 p^n - p^{n-1}
      rv[l] = rho_cell<RULE>(d2df(r[l]), K);
    }
  };
  auto fetch_cols = [&](int kk) {
    const uint32_t c = at(wrapk(kk));
    const double *pa = in.pn + c, *pb = in.pnm1 + c, *pr = in.rho + c;
#pragma unroll
    for (int l = 0; l < S; ++l) {
      raw.fetch(S_P + 3 * l, pa + l * nx, cv[l], 0.0);
      raw.fetch(S_P + 3 * l + 1, pb + l * nx, cv[l], 0.0);
      raw.fetch(S_P + 3 * l + 2, pr + l * nx, cv[l], 1.0);
    }
  };
  auto take_cols = [&](df* pv, df* rv) {
#pragma unroll
    for (int l = 0; l < S; ++l) {
      pv[l] = phat_of(raw.get(S_P + 3 * l, cv[l], 0.0), raw.get(S_P + 3 * l + 1, cv[l], 0.0));
      rv[l] = rho_cell<RULE>(d2df(raw.get(S_P + 3 * l + 2, cv[l], 1.0)), K);
    }
  };
  // halo lines j0-1 and j0+tj of plane kk (a thread's one or two cells) for
  // shared rows 0 and nl-1
  bool hv[HN];
  uint32_t hoff[HN];  // offset within a plane
  int hrow[HN];       // offset within the rows (-1: none)
#pragma unroll
  for (int q = 0; q < HN; ++q) {
    const int idx = (int)threadIdx.x + q * (int)blockDim.x;
    const int up = idx >= nx;
    const int j = up ? j0 + tj : j0 - 1;
    const bool in2 = idx < 2 * nx;
    hv[q] = in2 && (INT || (j >= 0 && j < ny));
    hoff[q] = (uint32_t)(j * nx + idx - up * nx);
    hrow[q] = in2 ? idx + up * (nl - 2) * nx : -1;
  }
  auto fetch_halo = [&](int kk) {
    const uint32_t kb = (uint32_t)wrapk(kk) * plane;
#pragma unroll
    for (int q = 0; q < HN; ++q) {
      const uint32_t c = kb + hoff[q];
      raw.fetch(S_H + 3 * q, in.pn + c, hv[q], 0.0);
      raw.fetch(S_H + 3 * q + 1, in.pnm1 + c, hv[q], 0.0);
      raw.fetch(S_H + 3 * q + 2, in.rho + c, hv[q], 1.0);
    }
  };
  auto store_halo = [&]() {
#pragma unroll
    for (int q = 0; q < HN; ++q) {
      if (hrow[q] < 0) continue;
      P[hrow[q]] = phat_of(raw.get(S_H + 3 * q, hv[q], 0.0), raw.get(S_H + 3 * q + 1, hv[q], 0.0));
      R[hrow[q]] = rho_cell<RULE>(d2df(raw.get(S_H + 3 * q + 2, hv[q], 1.0)), K);
    }
  };
  auto store_rows = [&](const df* pv, const df* rv) {
    if (!active) return;
#pragma unroll
    for (int l = 0; l < S; ++l) {
      P[(jb + l + 1) * nx + i] = pv[l];
      R[(jb + l + 1) * nx + i] = rv[l];
    }
  };
  auto face = [&](df rl, df rh, df pl, df ph, df us, df gh) {
    return face_upre<RULE, INT>(rl, rh, pl, ph, us, gh, K);
  };

  // u* of plane k, w* of face k+1 (own lines), v* of the y faces jb .. jb+S
  auto fetch_velocity = [&](int k) {
    const double *pu = in.u + at(k), *pw = in.w + at(wrapk(k + 1));
    const double* pv = in.v + ((uint32_t)k * vplane + own);
#pragma unroll
    for (int l = 0; l < S; ++l) {
      raw.fetch(S_U + l, pu + l * nx, cv[l], 0.0);
      raw.fetch(S_W + l, pw + l * nx, cv[l], 0.0);
    }
#pragma unroll
    for (int f = 0; f <= S; ++f) raw.fetch(S_V + f, pv + f * nx, fv[f], 0.0);
  };
  auto fetch_S = [&](int k) {
    const double* ps = in.S + at(k);
#pragma unroll
    for (int l = 0; l < S; ++l) raw.fetch(S_S + l, ps + l * nx, cv[l], 0.0);
  };

  df PC[S], RC[S], P1[S], R1[S], UZ[S];  // UZ: u_pre of the lower z face
  // prologue: plane k0 current (registers and shared rows), face k0, plane k0+1
  // in registers; in flight: the first step's velocities, its S, and the
  // planes that its phase C takes (own lines k0+2, halo k0+1)
  {
    df Pm[S], Rm[S];
    double w0[S];
    fetch_halo(k0);
    raw.commit();
    fetch_velocity(k0);
    raw.commit();
    fetch_S(k0);
    raw.commit();
    const double* pw = in.w + at(k0);
#pragma unroll
    for (int l = 0; l < S; ++l) w0[l] = cv[l] ? __ldg(pw + l * nx) : 0.0;
    load_cols(k0 - 1, Pm, Rm);
    load_cols(k0, PC, RC);
    load_cols(k0 + 1, P1, R1);
#pragma unroll
    for (int l = 0; l < S; ++l) {
      UZ[l] = {0.0f, 0.0f};
      if (!cv[l]) continue;
      UZ[l] = face(Rm[l], RC[l], Pm[l], PC[l], d2df(w0[l]), K.gz);
      if (PROJ) out.wpre[at(k0) + l * nx] = UZ[l];
    }
    store_rows(PC, RC);
    raw.wait2();
    store_halo();
    if (steps > 1) {
      fetch_cols(k0 + 2);
      fetch_halo(k0 + 1);
    }
    raw.commit();
  }
  __syncthreads();

  float vmax = 0.0f, smax = 0.0f, wmax = 0.0f;
  df wsum = {0.0f, 0.0f};  // wall flux v*(ny) - v*(0) of this CTA's wall faces
  for (int st = 0; st < steps; ++st) {
    const int k = k0 + st;
    const bool more = st + 1 < steps;
    const uint32_t ck = at(k);
    // ---- phase A: x faces (shared x neighbour), y faces and the upper z face (registers)
    raw.wait2();  // (in flight behind it: S of this plane, the planes of phase C)
    df UXo[S], UY[S + 1], UZup[S];
#pragma unroll
    for (int l = 0; l < S; ++l) {
      UXo[l] = {0.0f, 0.0f};
      if (!cv[l]) continue;
      const int r = (jb + l + 1) * nx;
      UXo[l] = face(R[r + im], RC[l], P[r + im], PC[l], d2df(raw.get(S_U + l, cv[l], 0.0)), K.gx);
      if (PROJ) out.upre[ck + l * nx] = UXo[l];
    }
    if (active) {
#pragma unroll
      for (int l = 0; l < S; ++l) QX[(jb + l) * nx + i] = UXo[l];
    }
    df* const vrow = out.vpre + ((uint32_t)k * vplane + own);
#pragma unroll
    for (int f = 0; f <= S; ++f) {  // face between tile lines jb+f-1 and jb+f
      UY[f] = {0.0f, 0.0f};
      const int j = j0 + jb + f;
      if (!fv[f]) continue;
      const df vs = d2df(raw.get(S_V + f, fv[f], 0.0));
      // a face belongs to the stack holding the line above it; the top wall to
      // the stack holding line ny - 1
      const bool mine = INT ? (f < S) : ((f < S && j < ny) || (j == ny && f >= 1));
      if (!INT && j == ny && g.top_open) {  // open top: p = 0 on the face, ghost -p_hat above
        const df rl = (f == 0) ? R[(jb) * nx + i] : RC[f > 0 ? f - 1 : 0];
        const df pl = (f == 0) ? P[(jb) * nx + i] : PC[f > 0 ? f - 1 : 0];
        UY[f] = face(rl, rl, pl, df_neg(pl), vs, K.gy);
      } else if (!INT && (j == 0 || j == ny)) {  // wall: u_pre = v*
        UY[f] = vs;
        if (mine) {
          wsum = (j == ny) ? df_addz(wsum, vs) : df_subz(wsum, vs);
          wmax = fmaxf(wmax, fabsf(vs.hi));
        }
      } else {
        const df rl = (f == 0) ? R[(jb) * nx + i] : RC[f > 0 ? f - 1 : 0];
        const df pl = (f == 0) ? P[(jb) * nx + i] : PC[f > 0 ? f - 1 : 0];
        const df rh = (f == S) ? R[(jb + S + 1) * nx + i] : RC[f < S ? f : 0];
        const df ph = (f == S) ? P[(jb + S + 1) * nx + i] : PC[f < S ? f : 0];
        UY[f] = face(rl, rh, pl, ph, vs, K.gy);
      }
      if (PROJ && mine) vrow[f * nx] = UY[f];
    }
    {
      df* const wrow = out.wpre + at(wrapk(k + 1));
#pragma unroll
      for (int l = 0; l < S; ++l) {
        UZup[l] = {0.0f, 0.0f};
        if (!cv[l]) continue;
        UZup[l] = face(RC[l], R1[l], PC[l], P1[l], d2df(raw.get(S_W + l, cv[l], 0.0)), K.gz);
        if (PROJ && more) wrow[l * nx] = UZup[l];
      }
    }
    if (more) fetch_velocity(k + 1);
    raw.commit();
    __syncthreads();
    // ---- phase B: cells of plane k, f = (rho_0/dt) (D u_pre - S)
    raw.wait2();
#pragma unroll
    for (int l = 0; l < S; ++l) {
      if (!cv[l]) continue;
      const df dx = df_mulz(df_subz(QX[(jb + l) * nx + ip], UXo[l]), K.cx);
      const df dy = df_mulz(df_subz(UY[l + 1], UY[l]), K.cy);
      const df dz = df_mulz(df_subz(UZup[l], UZ[l]), K.cz);
      const uint32_t c = ck + l * nx;
      const df sv = d2df(raw.get(S_S + l, cv[l], 0.0));
      const df f = df_norm(df_subz(df_addz(df_addz(dx, dy), dz), df_mulz(K.c, sv)));
      smax = fmaxf(smax, fabsf(sv.hi));
      if (PROJ) out.fdf[c] = f;
      if (!PROJ || out.f64) out.f64[c] = df2d(f);
      vmax = fmaxf(vmax, fabsf(f.hi));
      UZ[l] = UZup[l];
    }
    if (more) fetch_S(k + 1);
    raw.commit();
    if (more) {
      // ---- phase C: plane k+1 becomes current, plane k+2 next.  Phase B reads
      // only QX, so the rows can be rewritten without a barrier; the barrier
      // below orders them before the next phase A.
      raw.wait2();
#pragma unroll
      for (int l = 0; l < S; ++l) {
        PC[l] = P1[l];
        RC[l] = R1[l];
      }
      store_rows(PC, RC);
      store_halo();
      take_cols(P1, R1);
      if (st + 2 < steps) {
        fetch_cols(k + 3);
        fetch_halo(k + 2);
      }
      raw.commit();
      __syncthreads();
    }
  }
  block_max_to(&sc->fmax_bits, vmax);
  block_max_to(&sc->smax_bits, smax);
  block_max_to(&sc->wallv_bits, wmax);
  if (j0 == 0 || j0 + tj >= ny) block_pair_sums(wsum, df{0.0f, 0.0f}, sc->part + bid);
  if (bid == 0 && threadIdx.x == 0) {
    sc->rhs_tiles = ntile;
    sc->rhs_chunks = (nz + kc - 1) / kc;
  }
}

// One tile (CTA index bid) of the column-stack march: the interior form when
// the tile and its halo lines lie strictly inside the walls and rho_0 is the
// minimum of rho (in.min_rho0).  With a caller's rho_0 every tile takes the
// boundary form (256^3: 360 us against 304; the form with a flux per face took
// 375 with either).  A third body in the same kernel, interior with the general
// difference, brings that to 319 but costs the usual case registers: 384 x 256 x
// 128 243 -> 256 us, 144^3 93 -> 97, and 128^3 with a caller's rho_0 55 -> 58.
template <int S, int RULE, bool PROJ, int NXC = 0, bool SM = true>
__device__ __forceinline__ void rhs_stack_tile(const GridDev& g, const StencilIn& in, DevScalars* sc,
                                               const RhsOut& out, int kc, uint32_t bid) {
  const int tj = ((int)blockDim.x / (NXC ? NXC : g.nx)) * S;
  const int ntile = (g.ny + tj - 1) / tj;
  const int j0 = (int)(bid % ntile) * tj;
  if (in.min_rho0 && j0 > 0 && j0 + tj < g.ny)  // uniform over the CTA
    rhs_stack_body<S, RULE, PROJ, true, NXC, SM>(g, in, sc, out, kc, bid);
  else
    rhs_stack_body<S, RULE, PROJ, false, NXC, SM>(g, in, sc, out, kc, bid);
}

}  // namespace ppe
