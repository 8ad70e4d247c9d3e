// FP32 sweeps of the dimensionally split step (the method: sweep_kernels.cuh), without shared memory.
//
// A sweep is bound by instruction issue.  Tiles of 64x16 and 32x32 cells kept everything in shared memory between
// barriers and formed each MC slope three times and each shock detector twice (KH 1030x770 52.9 us per step).  Here a cell's
// values stay in registers and each is formed once (42.0 us):
//  - along y a thread marches up a column, two rows at a time, the rows below in registers;
//  - along x a warp takes 64 cells of a row, two a lane, 56 of them its own, and lanes exchange what their neighbours
//    need by shuffles;
// and the two faces of a thread are solved as a pair (riemann_pair).  KH 1024^2: 490 and 575 instructions per zone, at
// 68 % of the issue slots along x (20 warps an SM) and 61 % along y (16 warps; segments of 14 rows).
#pragma once

#include "ctu_march.cuh"
#include "ctu_kernels.cuh"

namespace hydro {

constexpr int SWEEP_NT = 128;  // threads of a block
// Blocks resident on an SM: 128 registers along y (three blocks of 151 registers: KH 2048^2 160.9 us per step against
// 152.8, 1030x770 40.3 against 42.0), 102 along x (four blocks: 153.9 and 44.0).
constexpr int SWEEP_Y_BLOCKS = 4, SWEEP_X_BLOCKS = 5;
// Most rows of a thread's or warp's piece.  Along y the six rows below and above a piece are converted twice (2048^2
// 166 us with 16 rows, 157 with 32, 154 with 64); along x nothing is.
constexpr int SWEEP_Y_ROWS = 64, SWEEP_X_ROWS = 12;

// Slopes, limited by xi, or the parabola, and the traced states of one cell in the face frame (rho, u_normal,
// u_transverse, p): ql at its upper face, qr at its lower one.  qm, qp: the neighbours; mm, m0, mp: the MC slopes of the
// three; kv: the component gravity acts on.
template <int MODE>
__device__ __forceinline__ void sweep_trace(const KParams& P, const SP<float>& s, float sigma, float hdtg, int kv, float xi,
                                            const float qm[4], const float q[4], const float qp[4], const float mm[4],
                                            const float m0[4], const float mp[4], float ql[4], float qr[4]) {
  const Waves<float> w(s, q[0], q[3]);
  if constexpr ((MODE & RECON_PPM) != 0) {
    float eL[4], eR[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) ppm_edges_mc<float>(qm[k], q[k], qp[k], mm[k], m0[k], mp[k], xi, eL[k], eR[k]);
    trace_ppm<float>(s, sigma, q, eL, eR, w, ql, qr);
  } else {
    float dl[4], dr[4], dd[4], dq[4];
    sub4(q, qm, dl);
    sub4(qp, q, dr);
    sub4(qp, qm, dd);
    slope4(s.limiter, xi, dl, dr, dd, mm, m0, mp, dq);
    trace<float>(s, sigma, q, dq, w, ql, qr);
  }
  if (P.use_grav) {
    ql[kv] = ql[kv] + hdtg;
    qr[kv] = qr[kv] + hdtg;
  }
}

// MC slope of a cell from its neighbours.
__device__ __forceinline__ void sweep_mc(const float qm[4], const float q[4], const float qp[4], float m[4]) {
  float dl[4], dr[4], dd[4];
  sub4(q, qm, dl);
  sub4(qp, q, dr);
  sub4(qp, qm, dd);
  mc4(dl, dr, dd, m);
}

// The viscous part of a face's flux F (face frame), from the states and normal velocities of its two cells.
__device__ __forceinline__ void sweep_viscosity(const SP<float>& s, float unl, float unr, const float Ul[4],
                                                const float Ur[4], float F[4]) {
  float d[4];
  sub4(Ul, Ur, d);
  axpy4(s.cvisc * fmaxf(0.0f, unl - unr), d, F);
}

// A new cell (conserved order): its CFL value (FUSED) or its state's check, and the store.
template <bool FUSED>
__device__ __forceinline__ void sweep_check(const SP<float>& s, const float Un[4], int check_state, float& cmin,
                                            TileCounters& cnt) {
  if constexpr (FUSED) {
    cfl_value(s, Un[0], Un[1], Un[2], Un[3], cmin, cnt.flags);  // the next step's constraint (Eq. 6)
  } else if (check_state) {
    if (!finite4(Un[0], Un[1], Un[2], Un[3])) {
      cnt.flags |= STATUS_NONFINITE;
    } else {
      const float ke = M<float>::dv(0.5f * (Un[1] * Un[1] + Un[2] * Un[2]), Un[0]);
      if (!(Un[0] > 0.0f) || !(Un[3] - ke > 0.0f)) cnt.flags |= STATUS_NEGATIVE;
    }
  }
}

__device__ __forceinline__ void sweep_factors(const StepScalars& sc_host, const StepScalars* sc_dev,
                                              StepFactors<float>& f) {
  if (sc_dev)
    f.load_ordered(sc_dev);
  else
    f.load(sc_host);
}

// The sweep along y: thread t takes column t % nx of segment t / nx, nh rows (even) of the interior.
template <bool FUSED, int MODE>
__global__ void __launch_bounds__(SWEEP_NT, SWEEP_Y_BLOCKS)
    sweep_y_kernel(KParams P, const float* __restrict__ Uin, float* __restrict__ Uout, StepScalars sc_host,
                   const StepScalars* __restrict__ sc_dev, DevScratch* __restrict__ scr, int check_state,
                   StepScalars* __restrict__ sc_next, double tmax, int nh) {
  step_begin();
  SP<float> s;
  s.load(P);
  StepFactors<float> f;
  sweep_factors(sc_host, sc_dev, f);
  const float sigma = f.sigy;
  const unsigned int t = blockIdx.x * SWEEP_NT + threadIdx.x;
  const int seg = (int)(t / (unsigned int)P.nx), i = P.ng + (int)(t % (unsigned int)P.nx);
  const int j0 = P.ng + seg * nh, n = min(nh, P.ng + P.ny - j0);
  const size_t plane = (size_t)P.NY * P.pitch;
  TileCounters cnt;
  float cmin = FLT_MAX;
  if (n > 0) {
    // conserved values of a row, in the face frame (rho, m_y, m_x, E), raw
    auto fetch = [&](int row, float u[4]) {
      row = min(row, P.ng + P.ny + 3);
      const float* a = Uin + (size_t)map_index(row, P.ng, P.ny, P.bc[2], P.bc[3]) * P.pitch + i;
      u[0] = ld_ordered(a);
      u[2] = ld_ordered(a + plane);
      u[1] = ld_ordered(a + 2 * plane);
      u[3] = ld_ordered(a + 3 * plane);
    };
    // what a side's condition makes of them
    auto side = [&](int row, float u[4]) {
      if (!P.bc_general) return;
      row = min(row, P.ng + P.ny + 3);
      const int bc = ghost_bc(row, P.ng, P.ny, P.bc[2], P.bc[3]);
      if (bc == 2) u[1] = -u[1];
      if (bc == 3) {
        const int d = row - map_index(row, P.ng, P.ny, P.bc[2], P.bc[3]);
        u[3] = hydrostatic_energy(P.gm1, __dmul_rn(__dmul_rn((double)u[0], P.grav), __dmul_rn((double)d, P.dy)), u[0],
                                  u[2], u[1], u[3]);
      }
    };
    auto prim = [&](int row, float u[4], float q[4]) {
      side(row, u);
      cons_to_prim(s, u[0], u[1], u[2], u[3], q[0], q[1], q[2], q[3]);
    };
    // carried over the rows c, c + 1 of an iteration: primitives of rows c - 1 .. c + 2, MC slopes and chi of c - 1 and c,
    // the traced state of row c - 1 at its upper face, the flux at face c - 3/2, U of row c - 1, rows on their way
    float qa[4], qb[4], qc[4], qd[4], ma[4], mb[4], lp[4] = {1, 0, 0, 1}, fp[4] = {0, 0, 0, 0}, up[4] = {1, 0, 0, 1};
    float n0[4], n1[4], chia = 1, chib = 1;
    {
      float u[6][4], q0[4], q1[4];
#pragma unroll
      for (int k = 0; k < 6; ++k) fetch(j0 - 4 + k, u[k]);
      fetch(j0 + 2, n0);
      fetch(j0 + 3, n1);
      prim(j0 - 4, u[0], q0);
      prim(j0 - 3, u[1], q1);
      prim(j0 - 2, u[2], qa);
      prim(j0 - 1, u[3], qb);
      prim(j0, u[4], qc);
      prim(j0 + 1, u[5], qd);
      sweep_mc(q1, qa, qb, ma);
      sweep_mc(qa, qb, qc, mb);
      if (s.flatten) {
        chia = flatten_chi<float>(q0[3], q1[3], qb[3], qc[3], q1[1], qb[1], s.small_pres);
        chib = flatten_chi<float>(q1[3], qa[3], qc[3], qd[3], qa[1], qc[1], s.small_pres);
      }
    }
#pragma unroll 1
    for (int c = j0 - 1; c <= j0 + n; c += 2) {
      float qe[4], qf[4], mc[4], md[4];
      prim(c + 3, n0, qe);
      prim(c + 4, n1, qf);
      fetch(c + 5, n0);
      fetch(c + 6, n1);
      float uc[4], ud[4];
      fetch(c, uc);
      fetch(c + 1, ud);
      sweep_mc(qb, qc, qd, mc);
      sweep_mc(qc, qd, qe, md);
      float xc = 1.0f, xd = 1.0f;
      if (s.flatten) {
        const float chic = flatten_chi<float>(qa[3], qb[3], qd[3], qe[3], qb[1], qd[1], s.small_pres);
        const float chid = flatten_chi<float>(qb[3], qc[3], qe[3], qf[3], qc[1], qe[1], s.small_pres);
        xc = fminf(chib, qc[3] - qa[3] >= 0.0f ? chia : chic);
        xd = fminf(chic, qd[3] - qb[3] >= 0.0f ? chib : chid);
        chia = chic;
        chib = chid;
      }
      float lc[4], rc[4], ld[4], rd[4], F[4], G[4];
      sweep_trace<MODE>(P, s, sigma, f.hdtg, 1, xc, qa, qb, qc, ma, mb, mc, lc, rc);
      sweep_trace<MODE>(P, s, sigma, f.hdtg, 1, xd, qb, qc, qd, mb, mc, md, ld, rd);
      const bool w0 = c >= j0, w1 = c + 1 <= P.ng + P.ny && (c + 1 < j0 + n || j0 + n == P.ng + P.ny);
      face_pair<MODE>(s, lp, rc, w0, F, lc, rd, w1, G, cnt);
      side(c, uc);
      side(c + 1, ud);
      if (s.cvisc > 0.0f) {
        sweep_viscosity(s, qa[1], qb[1], up, uc, F);
        sweep_viscosity(s, qb[1], qc[1], uc, ud, G);
      }
      // new rows c - 1 and c
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = c - 1 + h;
        if (row < j0 || row >= j0 + n) continue;
        const float* u = h ? uc : up;
        float d[4], Un[4];
        if (h)
          sub4(F, G, d);
        else
          sub4(fp, F, d);
        Un[0] = u[0] + sigma * d[0];
        Un[1] = u[2] + sigma * d[2];
        Un[2] = u[1] + sigma * d[1];
        Un[3] = u[3] + sigma * d[3];
        if (P.use_grav) {
          // the time-centred gravity sources, once per step, from the state this sweep starts from
          Un[2] = Un[2] + f.hdtg * (u[0] + Un[0]);
          Un[3] = Un[3] + f.hdtg * (u[1] + Un[2]);
        }
        float* o = Uout + (size_t)row * P.pitch + i;
#pragma unroll
        for (int k = 0; k < 4; ++k) o[k * plane] = Un[k];
        sweep_check<FUSED>(s, Un, check_state, cmin, cnt);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        qa[k] = qc[k];
        qb[k] = qd[k];
        qc[k] = qe[k];
        qd[k] = qf[k];
        ma[k] = mc[k];
        mb[k] = md[k];
        lp[k] = ld[k];
        fp[k] = G[k];
        up[k] = ud[k];
      }
    }
    // a face between two segments counts once
    const unsigned int solves = n + (j0 + n == P.ng + P.ny ? 1 : 0);
    cnt.solves += solves;
    if (face_kind(MODE) != FACE_HLLC) cnt.iters += solves;
  }
  flush_counters(cnt, scr);
  if constexpr (FUSED) finish_fused_step(P, cmin, sc_dev, sc_next, scr, tmax, 1u, gridDim.x);
}

// The sweep along x: warp w takes chunk w % chunks of nv cells (even, at most 56) in `rows` rows of the interior, two
// cells a lane and four cells of halo on each side.  vec: two neighbouring cells of an even column lie on 8 bytes.
template <bool FUSED, int MODE>
__global__ void __launch_bounds__(SWEEP_NT, SWEEP_X_BLOCKS)
    sweep_x_kernel(KParams P, const float* __restrict__ Uin, float* __restrict__ Uout, StepScalars sc_host,
                   const StepScalars* __restrict__ sc_dev, DevScratch* __restrict__ scr, int check_state,
                   StepScalars* __restrict__ sc_next, double tmax, int nv, int chunks, int rows, int vec) {
  step_begin();
  SP<float> s;
  s.load(P);
  StepFactors<float> f;
  sweep_factors(sc_host, sc_dev, f);
  const float sigma = f.sigx;
  const unsigned int item = (blockIdx.x * SWEEP_NT + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int j0 = P.ng + (int)(item / (unsigned int)chunks) * rows, n = min(rows, P.ng + P.ny - j0);
  const int i0 = P.ng + (int)(item % (unsigned int)chunks) * nv, cols = min(nv, P.ng + P.nx - i0);
  const int ea = 2 * lane, eb = ea + 1, ga = i0 - 4 + ea;  // the lane's cells in the chunk, and the first one's column
  const int hi = P.ng + P.nx + 3;
  const int gac = min(ga, hi), gbc = min(ga + 1, hi);
  const int ca = map_index(gac, P.ng, P.nx, P.bc[0], P.bc[1]), cb = map_index(gbc, P.ng, P.nx, P.bc[0], P.bc[1]);
  const bool flip_a = P.bc_general && ghost_bc(gac, P.ng, P.nx, P.bc[0], P.bc[1]) == 2;
  const bool flip_b = P.bc_general && ghost_bc(gbc, P.ng, P.nx, P.bc[0], P.bc[1]) == 2;
  const bool pairs = vec && i0 - 4 >= P.ng && i0 + 60 <= P.ng + P.nx;  // all 64 cells are interior
  const bool on_a = ea >= 4 && ea < 4 + cols, on_b = eb >= 4 && eb < 4 + cols;
  const bool end = i0 + cols == P.ng + P.nx;  // a face between two chunks counts once
  const bool face_a = on_a || (end && ea == 4 + cols), face_b = on_b || (end && eb == 4 + cols);
  const size_t plane = (size_t)P.NY * P.pitch;
  TileCounters cnt;
  float cmin = FLT_MAX;
  float na[4], nb[4];
  auto fetch = [&](int row) {
    const float* r = Uin + (size_t)row * P.pitch;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (pairs) {
        const float2 v = ld_ordered2(r + k * plane + ga);
        na[k] = v.x;
        nb[k] = v.y;
      } else {
        na[k] = ld_ordered(r + k * plane + ca);
        nb[k] = ld_ordered(r + k * plane + cb);
      }
    }
  };
  auto left = [](float v) { return __shfl_up_sync(0xffffffffu, v, 1); };
  auto right = [](float v) { return __shfl_down_sync(0xffffffffu, v, 1); };
  if (n > 0) fetch(j0);
#pragma unroll 1
  for (int j = j0; j < j0 + n; ++j) {
    float ua[4], ub[4], qa[4], qb[4], ql[4], qr[4], ma[4], mb[4], ml[4], mr[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      ua[k] = na[k];
      ub[k] = nb[k];
    }
    if (j + 1 < j0 + n) fetch(j + 1);
    if (flip_a) ua[1] = -ua[1];
    if (flip_b) ub[1] = -ub[1];
    cons_to_prim(s, ua[0], ua[1], ua[2], ua[3], qa[0], qa[1], qa[2], qa[3]);
    cons_to_prim(s, ub[0], ub[1], ub[2], ub[3], qb[0], qb[1], qb[2], qb[3]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      ql[k] = left(qb[k]);
      qr[k] = right(qa[k]);
    }
    sweep_mc(ql, qa, qb, ma);
    sweep_mc(qa, qb, qr, mb);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      ml[k] = left(mb[k]);
      mr[k] = right(ma[k]);
    }
    float xa = 1.0f, xb = 1.0f;
    if (s.flatten) {
      const float pl2 = left(qa[3]), pr2 = right(qb[3]);
      const float chia = flatten_chi<float>(pl2, ql[3], qb[3], qr[3], ql[1], qb[1], s.small_pres);
      const float chib = flatten_chi<float>(ql[3], qa[3], qr[3], pr2, qa[1], qr[1], s.small_pres);
      const float chil = left(chib), chir = right(chia);
      xa = fminf(chia, qb[3] - ql[3] >= 0.0f ? chil : chib);
      xb = fminf(chib, qr[3] - qa[3] >= 0.0f ? chia : chir);
    }
    float la[4], ra[4], lb[4], rb[4], ll[4], F[4], G[4], d[4];
    sweep_trace<MODE>(P, s, sigma, f.hdtg, 2, xa, ql, qa, qb, ml, ma, mb, la, ra);
    sweep_trace<MODE>(P, s, sigma, f.hdtg, 2, xb, qa, qb, qr, ma, mb, mr, lb, rb);
#pragma unroll
    for (int k = 0; k < 4; ++k) ll[k] = left(lb[k]);
    face_pair<MODE>(s, ll, ra, face_a, F, la, rb, face_b, G, cnt);
    if (s.cvisc > 0.0f) {
      float ul[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) ul[k] = left(ub[k]);
      sweep_viscosity(s, ql[1], qa[1], ul, ua, F);
      sweep_viscosity(s, qa[1], qb[1], ua, ub, G);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float H = right(F[k]);
      ua[k] = ua[k] + sigma * (F[k] - G[k]);
      ub[k] = ub[k] + sigma * (G[k] - H);
    }
    float* o = Uout + (size_t)j * P.pitch + ga;
    if (vec && on_a && on_b) {
#pragma unroll
      for (int k = 0; k < 4; ++k) *reinterpret_cast<float2*>(o + k * plane) = make_float2(ua[k], ub[k]);
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (on_a) o[k * plane] = ua[k];
        if (on_b) o[k * plane + 1] = ub[k];
      }
    }
    if (on_a) sweep_check<FUSED>(s, ua, check_state, cmin, cnt);
    if (on_b) sweep_check<FUSED>(s, ub, check_state, cmin, cnt);
  }
  const unsigned int solves = n > 0 ? n * ((face_a ? 1 : 0) + (face_b ? 1 : 0)) : 0;
  cnt.solves += solves;
  if (face_kind(MODE) != FACE_HLLC) cnt.iters += solves;
  flush_counters(cnt, scr);
  if constexpr (FUSED) finish_fused_step(P, cmin, sc_dev, sc_next, scr, tmax, 1u, gridDim.x);
}

// Rows for each of `slots` pieces that run at once, in as many rounds as keep a piece at most `most` rows.
inline int sweep_share(int ny, long long slots, int most) {
  slots = slots > 1 ? slots : 1;
  const long long rounds = (ny + slots * most - 1) / (slots * most);
  return (int)((ny + slots * rounds - 1) / (slots * rounds));
}

// One sweep (dir 0: along x).  sc_next == NULL: a plain sweep; otherwise the fused second sweep of a step.
template <int MODE>
cudaError_t launch_sweep_f32(const KParams& P, const float* Uin, float* Uout, int dir, const StepScalars& sc_host,
                             const StepScalars* sc_dev, DevScratch* scr, int check_state, StepScalars* sc_next,
                             double tmax, cudaStream_t stream) {
  int nsm = 0;
  const cudaError_t e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  const auto kx = sc_next ? sweep_x_kernel<true, MODE> : sweep_x_kernel<false, MODE>;
  const auto ky = sc_next ? sweep_y_kernel<true, MODE> : sweep_y_kernel<false, MODE>;
  if (dir == 1) {
    int nh = sweep_share(P.ny, (long long)nsm * SWEEP_Y_BLOCKS * SWEEP_NT / P.nx, SWEEP_Y_ROWS);
    nh += nh & 1;
    // not shorter than eight rows while that leaves the SMs one and a half blocks each: what short segments repeat is
    // time that other streams' kernels lose (KH 512^2, us per step alone / four at once: 4 rows 22.9 / 59.4, 8 rows 23.7 /
    // 50.4; 384^2 2 and 4 rows 18.0 / 46.3 and 38.1, 6 rows 19.4 / 34.9)
    while (nh < 8 && 2 * (long long)((P.ny + nh + 1) / (nh + 2)) * P.nx >= 3ll * nsm * SWEEP_NT) nh += 2;
    const long long total = (long long)((P.ny + nh - 1) / nh) * P.nx;
    return launch_step_kernel(ky, dim3((unsigned int)((total + SWEEP_NT - 1) / SWEEP_NT)), SWEEP_NT, (size_t)0, stream, P,
                              Uin, Uout, sc_host, sc_dev, scr, check_state, sc_next, tmax, nh);
  }
  int chunks = (P.nx + 55) / 56;
  int nv = (P.nx + chunks - 1) / chunks;
  nv += nv & 1;
  chunks = (P.nx + nv - 1) / nv;
  const int rows = sweep_share(P.ny, (long long)nsm * SWEEP_X_BLOCKS * (SWEEP_NT / 32) / chunks, SWEEP_X_ROWS);
  const long long warps = (long long)chunks * ((P.ny + rows - 1) / rows);
  const int vec = P.ng % 2 == 0 && P.pitch % 2 == 0 && (size_t)Uin % 8 == 0 && (size_t)Uout % 8 == 0;
  return launch_step_kernel(kx, dim3((unsigned int)((warps + SWEEP_NT / 32 - 1) / (SWEEP_NT / 32))), SWEEP_NT, (size_t)0,
                            stream, P, Uin, Uout, sc_host, sc_dev, scr, check_state, sc_next, tmax, nv, chunks, rows,
                            vec);
}

}  // namespace hydro
