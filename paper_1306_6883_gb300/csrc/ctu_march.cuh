// The FP32 CTU step (paper §3.2; CTU construction §3.1) in strips: a block takes a strip of up to 120 columns and
// marches up its rows, one thread a column, with the stages of ctu_tile.cuh applied to one row after another.
//
// Why: the FP32 step is bound by instruction issue, and a 32x16 tile repeats the work of its halo (1.9 times the
// conversions, 1.2 times the tracing and the hat solves) and forms each MC slope three times and each shock detector
// twice.  A strip loads, converts and traces a row once, keeps what it needs of the rows below in registers and rings
// of rows, takes a column's own slopes and fluxes along y from the row before and a neighbour's along x from an
// exchange row, and has no item arithmetic.  Sedov 4096^2, one step: 64.3 -> 39.5 warp instructions per zone, 1.09 ->
// 0.74 ms (ncu); at 74 % issue with 16 warps an SM, where the tile had 79 % with 36.  The bound is still issue (ALU 42 %,
// FMA pipe 48 %, shared memory 11 % of their rates).  KH 1024^2, in segments of 16 rows: 52.2 and 69 %.
//
// What makes it so:
//  - all threads of a block run all of every row's work, on copies of the edge columns outside the halo, so the loop
//    has no divergent regions (with a branch per stage and role: 59.4 instructions per zone, 63 % issue);
//  - the two face solves of a stage run as a pair (riemann_pair), since four warps to a scheduler do not cover one
//    solve's chain of dependent operations;
//  - three barriers a row, with every exchange row written between one pair of them and read between the next;
//  - 128 registers: four strips of 128 threads an SM.  The two-shock and the learned step spill nothing, HLLC and PPM 4
//    bytes, ensembles (batch_march_kernel, whose members' parameters take registers) 36 to 48 (96 registers for five
//    strips spilled 340: Sedov 4096^2 1.22 ms; two threads a column, one for each direction, at 80 registers: KH 2048^2
//    317 us against 231).
//
// Row c is traced while row c + 3 arrives; the hat solves are row c's x faces and the y face c - 1/2 between the rows c -
// 1 and c, the final ones the x faces of row c - 1 and the same y face, and the row updated is c - 1.  Results do not
// depend on where a grid is cut into strips.
#pragma once

#include <float.h>

#include "ctu_tile.cuh"

namespace hydro {

// One component quadruple per column in shared memory.
__device__ __forceinline__ void q_ld(const float4* a, int i, float v[4]) {
  const float4 t = a[i];
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void q_st(float4* a, int i, const float v[4]) {
  a[i] = make_float4(v[0], v[1], v[2], v[3]);
}

// A strip's registers (128 a thread) let 512 threads share an SM: four strips of 128 columns.
constexpr int MARCH_MAX_THREADS = 128, MARCH_SM_THREADS = 512;
constexpr int MARCH_ROWS = 6;  // rows of primitives and of U^n a strip holds: c - 2 .. c + 3 around the traced row c

// Shared memory of a strip of `threads` columns: the two row rings, five exchange rows of quadruples (MC slopes,
// left states, hat fluxes, corrected left states, final fluxes) and six scalar rows (four of pressures, chi, the
// y difference of v); a learned step's strip also four rows of notes (ctu_march).
__host__ __device__ constexpr size_t march_bytes(int threads, bool learned = false) {
  return sizeof(float) * (size_t)threads * (4 * (2 * MARCH_ROWS + 5) + (learned ? 10 : 6));
}

// energy of a ghost cell of a hydrostatic side (bc_cell) from its edge cell's values and its distance in cells
static __device__ __noinline__ float hydrostatic_energy(double gm1, double gdy, float rho_, float mx_, float my_, float E) {
  const double rho = (double)rho_, mx = (double)mx_, my = (double)my_;
  const double ke = __ddiv_rn(__dmul_rn(0.5, __dadd_rn(__dmul_rn(mx, mx), __dmul_rn(my, my))), rho);
  const double pe = __dmul_rn(gm1, __dsub_rn((double)E, ke));
  const double pg = __dadd_rn(pe, gdy);
  return (float)__dadd_rn(__ddiv_rn(pg, gm1), ke);
}

// Two face solves of a thread; the faces that count (n0, n1) add their iterations past the first to cnt.iters.
// slow: as for riemann_pair.
template <int MODE, typename Slow>
__device__ __forceinline__ void face_pair(const SP<float>& s, const float a[4], const float b[4], bool n0, float F[4],
                                          const float c[4], const float d[4], bool n1, float G[4], TileCounters& cnt,
                                          Slow&& slow) {
  if constexpr (face_kind(MODE) == FACE_HLLC) {
    hllc(s, a, b, F);
    hllc(s, c, d, G);
  } else {
    riemann_pair(s, a, b, n0, F, c, d, n1, G, cnt.iters, cnt.nonconv, slow);
  }
}
template <int MODE>
__device__ __forceinline__ void face_pair(const SP<float>& s, const float a[4], const float b[4], bool n0, float F[4],
                                          const float c[4], const float d[4], bool n1, float G[4], TileCounters& cnt) {
  face_pair<MODE>(s, a, b, n0, F, c, d, n1, G, cnt, [](bool&, bool&) {});
}

// Work area of a learned step (learned_work_bytes, all zero between steps).  For each row of 32x16 tiles, four words of
// which a launch uses those of its first row (the list's length, the next tile to take, the blocks that are done, -);
// then for each tile what its cells are in the strips (count: solves in the high word, iterations past the first in the
// low one; status flags with LISTED; FLT_MAX's bits less those of the least CFL value; solves that did not converge),
// and the list of the tiles to be stepped with the network, a band's part beginning at its first tile.
constexpr int LEARNED_TX = 32, LEARNED_TY = 16;
struct LearnedWork {
  static constexpr unsigned int LISTED = 0x80000000u;
  unsigned int* counters;
  unsigned long long* count;
  unsigned int *state, *slack, *nonconv;
  int* list;
  int tx;
  __device__ __forceinline__ LearnedWork(int nx, int ny, unsigned int* w, int by0) {
    tx = (nx + LEARNED_TX - 1) / LEARNED_TX;
    const int ty = (ny + LEARNED_TY - 1) / LEARNED_TY;
    const size_t n = (size_t)tx * ty;
    counters = w + 4 * (size_t)by0;
    count = reinterpret_cast<unsigned long long*>(w + 4 * (size_t)ty);
    state = reinterpret_cast<unsigned int*>(count + n);
    slack = state + n;
    nonconv = slack + n;
    list = reinterpret_cast<int*>(nonconv + n) + (size_t)by0 * tx;
  }
  static constexpr size_t words(size_t tx, size_t ty) { return 4 * ty + 6 * tx * ty; }
};

// What a strip's warp hands in for the tile row ty (counted over the grid of nx by ny cells) of its cells: the lanes'
// counts (at most 2^7 solves each, of maxiter iterations), status flags and least CFL value to the tiles of the columns
// col they belong to (at most two tiles, from left to right), and to the list, each once, the tiles of the columns x - 1,
// x and x + 1 where left, own and right say so.
static __device__ __noinline__ void hand_in(int nx, int ny, unsigned int* work, int by0, int ty, int col, int x, bool left,
                                            bool own, bool right, TileCounters cnt, int maxiter, float cmin) {
  const LearnedWork w(nx, ny, work, by0);
  const int t = col / LEARNED_TX;
  const size_t row = (size_t)ty * w.tx;
  const int t0 = __shfl_sync(0xffffffffu, t, 0), t1 = __shfl_sync(0xffffffffu, t, 31);
  const bool first = t == t0;
  const unsigned int slack = 0x7f7fffffu - __float_as_uint(cmin);
  const unsigned int s0 = __reduce_max_sync(0xffffffffu, first ? slack : 0u);
  const unsigned int s1 = __reduce_max_sync(0xffffffffu, first ? 0u : slack);
  unsigned long long c0, c1;
  if (maxiter < 256) {  // solves (a warp's in 12 bits) and iterations in one sum
    const unsigned int c = cnt.solves | cnt.iters << 12;
    const unsigned int p0 = __reduce_add_sync(0xffffffffu, first ? c : 0u);
    const unsigned int p1 = __reduce_add_sync(0xffffffffu, first ? 0u : c);
    c0 = (unsigned long long)(p0 & 0xfffu) << 32 | p0 >> 12;
    c1 = (unsigned long long)(p1 & 0xfffu) << 32 | p1 >> 12;
  } else {
    c0 = (unsigned long long)__reduce_add_sync(0xffffffffu, first ? cnt.solves : 0u) << 32 |
         __reduce_add_sync(0xffffffffu, first ? cnt.iters : 0u);
    c1 = (unsigned long long)__reduce_add_sync(0xffffffffu, first ? 0u : cnt.solves) << 32 |
         __reduce_add_sync(0xffffffffu, first ? 0u : cnt.iters);
  }
  if ((threadIdx.x & 31) == 0) {
    if (s0) atomicMax(&w.slack[row + t0], s0);
    if (s1) atomicMax(&w.slack[row + t1], s1);
    if (c0) atomicAdd(&w.count[row + t0], c0);
    if (c1) atomicAdd(&w.count[row + t1], c1);
  }
  if (cnt.flags) atomicOr(&w.state[row + t], cnt.flags);
  if (cnt.nonconv) atomicAdd(&w.nonconv[row + t], cnt.nonconv);
  auto put = [&](int k) {
    if (!(atomicOr(&w.state[row + k], LearnedWork::LISTED) & LearnedWork::LISTED))
      w.list[atomicAdd(&w.counters[0], 1u)] = (int)row + k;
  };
  if (own) put(t);
  if (left && !(own && (x - 1) / LEARNED_TX == t)) put((x - 1) / LEARNED_TX);
  if (right && !(own && (x + 1) / LEARNED_TX == t)) put((x + 1) / LEARNED_TX);
}

// Steps the strip of nv columns (nv + 8 <= blockDim.x) and nh rows whose first interior cell is (i0, j0), padded
// indices; smem holds march_bytes(blockDim.x).  MODE, FUSED, cfl_min as for ctu_tile.
//
// FACE_LEARNED: the strip solves from the acoustic start.  The tiles that hold a cell whose update reads a strong face,
// one past the gate of mlp whose first iteration makes no small step (one of the cell's own faces, or a hat face that
// corrects their states), go on the list of work, to be stepped with the network by a second launch, which overwrites
// them; so the strip leaves a strong face after that iteration.  Every strip that has a cell solves all those faces, so
// the list does not depend on how the grid is cut.  What the strip counts, its status flags and CFL values go to the
// tiles' records (hand_in), of which the second launch takes those of the tiles that were not listed.  The network
// itself in the strip would hold up all its later rows (a blast's front kept strips for 1 ms).  Strong faces are noted
// per column and iteration c, as bit c mod 32 of a word for each of the four solves, and handed in at the end of each
// tile row (KH 3000^2: 448 us per plain step, 463 learned, 11 of them the second launch).
template <int MODE, bool FUSED>
__device__ __forceinline__ void ctu_march(const KParams& P, const SP<float>& s, const StepFactors<float>& f,
                                          const float* __restrict__ Uin, float* __restrict__ Uout, int i0, int nv, int j0,
                                          int nh, unsigned char* smem, TileCounters& cnt, float* cfl_min,
                                          const MlpBlob* mlp = nullptr, unsigned int* work = nullptr, int by0 = 0) {
  static_assert(face_kind(MODE) != FACE_HARVEST, "the harvest steps in tiles");
  constexpr bool GATED = face_kind(MODE) == FACE_LEARNED;
  const int W = blockDim.x, x = threadIdx.x;  // column of the strip, its halo and copies of the last column past it
  const int xl1 = x > 0 ? x - 1 : 0, xr1 = x < W - 1 ? x + 1 : W - 1;
  float4* const ring_q = reinterpret_cast<float4*>(smem);
  float4* const ring_u = ring_q + MARCH_ROWS * W;
  float4* const x_mc = ring_u + MARCH_ROWS * W;
  float4* const x_l = x_mc + W;
  float4* const x_hat = x_l + W;
  float4* const x_lc = x_hat + W;
  float4* const x_flux = x_lc + W;
  float* const ring_p = reinterpret_cast<float*>(x_flux + W);
  float* const x_chi = ring_p + 4 * W;
  float* const x_dv = x_chi + W;
  uint2* const x_note = reinterpret_cast<uint2*>(x_dv + W);  // FACE_LEARNED: own column's only

  const int gi = i0 - 4 + (x < nv + 7 ? x : nv + 7);
  const int col = FUSED ? map_index(gi, P.ng, P.nx, P.bc[0], P.bc[1]) : (gi < P.NX ? gi : P.NX - 1);
  const bool flip_x = FUSED && P.bc_general && ghost_bc(gi, P.ng, P.nx, P.bc[0], P.bc[1]) == 2;
  const bool on_trace = x >= 3 && x <= nv + 4, on_xface = x >= 4 && x <= nv + 4, on_cell = x >= 4 && x <= nv + 3;
  const size_t plane = (size_t)P.NY * P.pitch;
  const float sigx = f.sigx, sigy = f.sigy, hx = f.hx, hy = f.hy;

  auto fetch = [&](int row, float u[4]) {
    const int r = FUSED ? map_index(row, P.ng, P.ny, P.bc[2], P.bc[3]) : (row < P.NY ? row : P.NY - 1);
    const float* a = Uin + (size_t)r * P.pitch + col;
#pragma unroll
    for (int k = 0; k < 4; ++k) u[k] = ld_ordered(a + k * plane);
  };
  auto slot = [](int newest, int back) { return newest >= back ? newest - back : newest - back + MARCH_ROWS; };
  // a fetched row into ring slot sl; returns its primitives
  auto put = [&](int row, int sl, float un[4], float q[4]) {
    if (FUSED && P.bc_general) {
      const int ybc = ghost_bc(row, P.ng, P.ny, P.bc[2], P.bc[3]);
      if (flip_x) un[1] = -un[1];
      if (ybc == 2) un[2] = -un[2];
      if (ybc == 3) {
        const int d = row - map_index(row, P.ng, P.ny, P.bc[2], P.bc[3]);
        un[3] = hydrostatic_energy(P.gm1, __dmul_rn(__dmul_rn((double)un[0], P.grav), __dmul_rn((double)d, P.dy)),
                                      un[0], un[1], un[2], un[3]);
      }
    }
    cons_to_prim(s, un[0], un[1], un[2], un[3], q[0], q[1], q[2], q[3]);
    q_st(ring_q + sl * W, x, q);
    q_st(ring_u + sl * W, x, un);
    ring_p[(row & 3) * W + x] = q[3];
  };
  // MC slopes and chi along x of the row in slot sl (own primitives q)
  auto slopes_x = [&](int row, int sl, const float q[4]) {
    const float4* rq = ring_q + sl * W;
    float qL[4], qR[4], dl[4], dr[4], d2[4], m[4];
    q_ld(rq, xl1, qL);
    q_ld(rq, xr1, qR);
    sub4(q, qL, dl);
    sub4(qR, q, dr);
    sub4(qR, qL, d2);
    mc4(dl, dr, d2, m);
    q_st(x_mc, x, m);
    if (s.flatten) {
      const float* p1 = ring_p + (row & 3) * W;
      x_chi[x] = flatten_chi<float>(p1[x > 1 ? x - 2 : 0], qL[3], qR[3], p1[x < W - 2 ? x + 2 : W - 1], qL[1], qR[1],
                                s.small_pres);
    }
  };

  // carried from row to row (c: the row being traced)
  float my0[4], my1[4];         // MC slopes along y of rows c - 1, c
  float chi0 = 1, chi1 = 1;     // chi along y of rows c - 1, c
  // traced states of row c - 1 (before the first row, any valid state)
  float yl_c[4] = {1, 0, 0, 1}, xl_c[4] = {1, 0, 0, 1}, xr_c[4] = {1, 0, 0, 1};
  float fyh[4] = {0, 0, 0, 0};  // hat flux at face c - 3/2
  float ylc[4] = {1, 0, 0, 1};  // corrected state of row c - 1 at its upper face
  float fy0[4] = {0, 0, 0, 0};  // final flux at face c - 3/2
  float un[4];                  // U of row c + 4, on its way
  float du_c = 0, ddu_c = 0, ddv_c = 0;  // row c - 1: u_i - u_{i-1}, u_{i+1} - u_{i-1}, v_{j+1} - v_{j-1}
  // rows j0 - 4 .. j0 + 1, and the slopes of row j0 - 1 along x, of rows j0 - 2 and j0 - 1 along y
  {
    float q[4], u[6][4];
#pragma unroll
    for (int k = 0; k < 6; ++k) fetch(j0 - 4 + k, u[k]);  // all in flight at once
    fetch(j0 + 2, un);
#pragma unroll
    for (int k = 0; k < 6; ++k) put(j0 - 4 + k, k, u[k], q);
    __syncthreads();
    float a[4][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) q_ld(ring_q + (k + 1) * W, x, a[k]);  // rows j0 - 3 .. j0
    float p0[4], p5[4];
    q_ld(ring_q, x, p0);
    q_ld(ring_q + 5 * W, x, p5);
    float dl[4], dr[4], dd[4];
    sub4(a[1], a[0], dl);
    sub4(a[2], a[1], dr);
    sub4(a[2], a[0], dd);
    mc4(dl, dr, dd, my0);
    sub4(a[3], a[2], dl);
    sub4(a[3], a[1], dd);
    mc4(dr, dl, dd, my1);
    if (s.flatten) {
      chi0 = flatten_chi<float>(p0[3], a[0][3], a[2][3], a[3][3], a[0][2], a[2][2], s.small_pres);
      chi1 = flatten_chi<float>(a[0][3], a[1][3], a[3][3], p5[3], a[1][2], a[3][2], s.small_pres);
    }
    slopes_x(j0 - 1, 3, a[2]);
    __syncthreads();
  }
  // FACE_LEARNED: strong faces among the pair k of solves (0: hat faces along x and y, 1: final ones along y and x) of
  // iteration c
  auto strong = [&](int k, int c, bool sx, bool sy) {
    if (sx || sy) {
      uint2 v = x_note[k * W + x];
      v.x |= sx ? 1u << (c & 31) : 0u;
      v.y |= sy ? 1u << (c & 31) : 0u;
      x_note[k * W + x] = v;
    }
  };
  if constexpr (GATED) x_note[x] = x_note[W + x] = make_uint2(0, 0);
  int c_in = j0;  // first row c whose solves have not been handed in
  int s3 = 0;  // ring slot of row c + 3
#pragma unroll 1
  for (int c = j0 - 1; c <= j0 + nh; ++c) {
    const int s0 = slot(s3, 3), s1 = slot(s3, 2), sm = slot(s3, 4);  // slots of rows c, c + 1, c - 1
    float q3[4], qb[4], xr[4], yl[4], yr[4], xl[4];
    float du, ddu, ddv, dly;
    // ---- row c + 3 into the rings; slopes and tracing of row c
    put(c + 3, s3, un, q3);
    if (c < j0 + nh) fetch(c + 4, un);
    {
      float qm[4], qa[4], qc[4], qL[4], qR[4], mL[4], m0[4], mR[4];
      q_ld(ring_q + sm * W, x, qm);
      q_ld(ring_q + s0 * W, x, qa);
      q_ld(ring_q + s1 * W, x, qb);
      q_ld(ring_q + slot(s3, 1) * W, x, qc);
      q_ld(ring_q + s0 * W, xl1, qL);
      q_ld(ring_q + s0 * W, xr1, qR);
      q_ld(x_mc, xl1, mL);
      q_ld(x_mc, x, m0);
      q_ld(x_mc, xr1, mR);
      float my2[4], dhi[4], dlo[4], dd[4], dl[4], dr[4], d2[4], dlm[4], d2y[4];
      sub4(qb, qa, dhi);
      sub4(qc, qb, dlo);
      sub4(qc, qa, dd);
      mc4(dhi, dlo, dd, my2);
      sub4(qa, qL, dl);
      sub4(qR, qa, dr);
      sub4(qR, qL, d2);
      sub4(qa, qm, dlm);
      sub4(qb, qm, d2y);
      du = dl[1];
      ddu = d2[1];
      ddv = d2y[2];
      dly = dlm[2];
      float xi = 1.0f;
      if (s.flatten) {
        const float chi2 = flatten_chi<float>(qm[3], qa[3], qc[3], q3[3], qa[2], qc[2], s.small_pres);
        const float xix = fminf(x_chi[x], x_chi[d2[3] >= 0.0f ? xl1 : xr1]);
        const float xiy = fminf(chi1, d2y[3] >= 0.0f ? chi0 : chi2);
        xi = fminf(xix, xiy);
        chi0 = chi1;
        chi1 = chi2;
      }
      const Waves<float> w(s, qa[0], qa[3]);
      if constexpr ((MODE & RECON_PPM) != 0) {
        float eL[4], eR[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) ppm_edges_mc<float>(qL[k], qa[k], qR[k], mL[k], m0[k], mR[k], xi, eL[k], eR[k]);
        trace_ppm<float>(s, sigx, qa, eL, eR, w, xl, xr);
#pragma unroll
        for (int k = 0; k < 4; ++k) ppm_edges_mc<float>(qm[k], qa[k], qb[k], my0[k], my1[k], my2[k], xi, eL[k], eR[k]);
        const float qy[4] = {qa[0], qa[2], qa[1], qa[3]}, eLy[4] = {eL[0], eL[2], eL[1], eL[3]},
                eRy[4] = {eR[0], eR[2], eR[1], eR[3]};
        trace_ppm<float>(s, sigy, qy, eLy, eRy, w, yl, yr);
      } else {
        float dq[4];
        slope4(s.limiter, xi, dl, dr, d2, mL, m0, mR, dq);
        trace<float>(s, sigx, qa, dq, w, xl, xr);
        slope4(s.limiter, xi, dlm, dhi, d2y, my0, my1, my2, dq);
        const float qy[4] = {qa[0], qa[2], qa[1], qa[3]}, dqy[4] = {dq[0], dq[2], dq[1], dq[3]};
        trace<float>(s, sigy, qy, dqy, w, yl, yr);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        my0[k] = my1[k];
        my1[k] = my2[k];
      }
      if (P.use_grav) {  // half-step gravity on v: transverse in x, normal in y
        xl[2] = xl[2] + f.hdtg;
        xr[2] = xr[2] + f.hdtg;
        yl[1] = yl[1] + f.hdtg;
        yr[1] = yr[1] + f.hdtg;
      }
      q_st(x_l, x, xl);
      x_dv[x] = ddv_c;  // of row c - 1, for that row's final x faces
    }
    __syncthreads();
    // ---- hat solves: x faces of row c, y face c - 1/2; transverse correction of row c - 1's x states; MC slopes
    // and chi along x of row c + 1
    float fxh[4];
    {
      float a[4], F[4];
      q_ld(x_l, xl1, a);
      const bool on_y = on_trace && c >= j0;
      face_pair<MODE>(s, a, xr, on_xface, fxh, yl_c, yr, on_y, F, cnt, [&](bool& ok0, bool& ok1) {
        if constexpr (GATED) {
          const float ratio = __ldg(&mlp->gate_ratio), u4 = __ldg(&mlp->gate_u4);
          const bool sx = !ok0 & on_xface & strong_face(a, xr, ratio, u4);
          const bool sy = !ok1 & on_y & strong_face(yl_c, yr, ratio, u4);
          strong(0, c, sx, sy);
          ok0 |= sx;
          ok1 |= sy;
        }
      });
      q_st(x_hat, x, fxh);
      const float G[4] = {F[0], F[2], F[1], F[3]};
      float d[4];
      sub4(G, fyh, d);
      correct_state(s, xl_c[0], xl_c[1], xl_c[2], xl_c[3], d, hy, a);
      q_st(x_lc, x, a);
      correct_state(s, xr_c[0], xr_c[1], xr_c[2], xr_c[3], d, hy, a);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        xr_c[k] = a[k];
        fyh[k] = G[k];
      }
      slopes_x(c + 1, s1, qb);
    }
    __syncthreads();
    // ---- transverse correction of row c's y states (face frame: rho, v, u, p); final solves: y face c - 1/2, x
    // faces of row c - 1
    float gx[4], gy[4], um[4];
    {
      float d[4], g[4], a[4], yrc[4], ylc_new[4], lc[4];
      q_ld(x_hat, xr1, g);
      sub4(g, fxh, d);
      correct_state(s, yr[0], yr[2], yr[1], yr[3], d, hx, a);
      yrc[0] = a[0]; yrc[1] = a[2]; yrc[2] = a[1]; yrc[3] = a[3];
      correct_state(s, yl[0], yl[2], yl[1], yl[3], d, hx, a);
      ylc_new[0] = a[0]; ylc_new[1] = a[2]; ylc_new[2] = a[1]; ylc_new[3] = a[3];
      q_ld(x_lc, xl1, lc);
      float F[4];
      const bool on_y = on_cell && c >= j0, on_x = on_xface && c > j0;
      face_pair<MODE>(s, ylc, yrc, on_y, F, lc, xr_c, on_x, gx, cnt, [&](bool& ok0, bool& ok1) {
        if constexpr (GATED) {
          const float ratio = __ldg(&mlp->gate_ratio), u4 = __ldg(&mlp->gate_u4);
          const bool sy = !ok0 & on_y & strong_face(ylc, yrc, ratio, u4);
          const bool sx = !ok1 & on_x & strong_face(lc, xr_c, ratio, u4);
          strong(1, c, sy, sx);
          ok0 |= sy;
          ok1 |= sx;
        }
      });
      gy[0] = F[0]; gy[1] = F[2]; gy[2] = F[1]; gy[3] = F[3];
      q_ld(ring_u + sm * W, x, um);
      if (s.cvisc > 0.0f) {
        float ua[4], ul[4], dux[4], duy[4], divx, divy;
        q_ld(ring_u + s0 * W, x, ua);
        q_ld(ring_u + sm * W, xl1, ul);
        sub4(um, ua, duy);
        sub4(ul, um, dux);
        divy = dly * s.idy + (ddu + ddu_c) * (0.25f * s.idx);
        divx = du_c * s.idx + (x_dv[xl1] + ddv_c) * (0.25f * s.idy);
        axpy4(s.cvisc * fmaxf(0.0f, -divy * s.dy), duy, gy);
        axpy4(s.cvisc * fmaxf(0.0f, -divx * s.dx), dux, gx);
      }
      q_st(x_flux, x, gx);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        ylc[k] = ylc_new[k];
        yl_c[k] = yl[k];
        xl_c[k] = xl[k];
        xr_c[k] = xr[k];
      }
      du_c = du;
      ddu_c = ddu;
      ddv_c = ddv;
    }
    __syncthreads();
    // ---- update of row c - 1
    if (c > j0 && on_cell) {
      float fx1[4], Un[4];
      q_ld(x_flux, x + 1, fx1);
#pragma unroll
      for (int h = 0; h < 4; h += 2) {
        const float2 dx = sub2(f2(gx[h], gx[h + 1]), f2(fx1[h], fx1[h + 1]));
        const float2 dy = sub2(f2(fy0[h], fy0[h + 1]), f2(gy[h], gy[h + 1]));
        const float2 n = add2(f2(um[h], um[h + 1]), fma2(f2(sigx), dx, mul2(f2(sigy), dy)));
        Un[h] = n.x;
        Un[h + 1] = n.y;
      }
      if (P.use_grav) {
        Un[2] = Un[2] + f.hdtg * (um[0] + Un[0]);
        Un[3] = Un[3] + f.hdtg * (um[2] + Un[2]);
      }
      float* o = Uout + (size_t)(c - 1) * P.pitch + (i0 - 4 + x);
#pragma unroll
      for (int k = 0; k < 4; ++k) o[k * plane] = Un[k];
      if constexpr (FUSED) {
        cfl_value(s, Un[0], Un[1], Un[2], Un[3], *cfl_min, cnt.flags);
      } else if (!finite4(Un[0], Un[1], Un[2], Un[3])) {
        cnt.flags |= STATUS_NONFINITE;
      } else {
        const float ke = M<float>::dv(0.5f * (Un[1] * Un[1] + Un[2] * Un[2]), Un[0]);
        if (!(Un[0] > 0.0f) || !(Un[3] - ke > 0.0f)) cnt.flags |= STATUS_NEGATIVE;
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) fy0[k] = gy[k];
    if constexpr (GATED) {
      if (c > j0 && ((c - P.ng) % LEARNED_TY == 0 || c == j0 + nh)) {  // row c - 1 ends a tile row or the strip
        // its rows r0 .. c - 1 read the hat faces along x of iterations r0 - 1 to c and those along y of r0 to c, the final
        // faces along y of r0 to c and along x of r0 + 1 to c; the next rows read those from c - 1 on again
        const int n = (c - 1 - P.ng) % LEARNED_TY, r0 = c - 1 - n > j0 ? c - 1 - n : j0;
        auto bits = [&](int from) {  // iterations from .. c
          const unsigned int all = (2u << (c - from)) - 1u;
          return __funnelshift_l(all, all, from & 31);
        };
        const uint2 h = x_note[x], g = x_note[W + x];
        const unsigned int keep = 1u << (c & 31) | 1u << ((c - 1) & 31);
        x_note[x] = make_uint2(h.x & keep, h.y & keep);
        x_note[W + x] = make_uint2(g.x & keep, g.y & keep);
        const bool hy = (h.y & bits(r0)) != 0, mine = (g.x & bits(r0)) != 0;
        const bool both = ((h.x & bits(r0 - 1)) | (g.y & bits(r0 + 1))) != 0 || hy;
        // a row c from j0 on has on_xface twice, on_trace and on_cell; row j0 - 1's x faces make up for row j0's
        cnt.solves = (unsigned int)(c + 1 - c_in) * ((on_xface ? 2 : 0) + (on_trace ? 1 : 0) + (on_cell ? 1 : 0));
        const int k = x < 4 ? 0 : x > nv + 3 ? nv - 1 : x - 4;  // the strip's column this thread's faces belong to
        hand_in(P.nx, P.ny, work, by0, (c - 1 - P.ng) / LEARNED_TY, i0 - P.ng + k, i0 - P.ng + x - 4,
                both && x >= 5 && x <= nv + 4, (both || mine) && on_cell, hy && x >= 3 && x <= nv + 2, cnt, s.maxiter,
                FUSED ? *cfl_min : FLT_MAX);
        cnt = TileCounters();
        if constexpr (FUSED) *cfl_min = FLT_MAX;
        c_in = c + 1;
      }
    }
    s3 = s3 + 1 == MARCH_ROWS ? 0 : s3 + 1;
  }
  // every face above counted once; the iterations past the first were added as they ran
  if constexpr (!GATED) {
    const unsigned int solves = (on_xface ? 2 * nh + 2 : 0) + (on_trace ? nh + 1 : 0) + (on_cell ? nh + 1 : 0);
    cnt.solves += solves;
    if (face_kind(MODE) != FACE_HLLC) cnt.iters += solves;
  }
}

}  // namespace hydro
