// Kernels and launches of the FP32 step in marching strips (ctu_march.cuh), with the rule that chooses between
// strips and tiles.
#pragma once

#include "ctu_kernels.cuh"
#include "ctu_march.cuh"

namespace hydro {

// Work area of a learned step: the 32x16 tiles of the strips that met a strong face.  For each tile row, four words of
// which a launch uses those of its first row (the list's length, the next tile to take, the blocks that are done, -);
// then the list, a band's part beginning at its first tile; then a mark for each tile.  All zero between steps.
struct LearnedWork {
  unsigned int* counters;
  int* list;
  unsigned int* mark;
  int tx;
  __device__ __forceinline__ LearnedWork(const KParams& P, unsigned int* w, int by0) {
    tx = (P.nx + F32_TX - 1) / F32_TX;
    const int ty = (P.ny + F32_TY - 1) / F32_TY;
    counters = w + 4 * by0;
    list = (int*)(w + 4 * ty) + (size_t)by0 * tx;
    mark = w + 4 * ty + (size_t)tx * ty;
  }
};

// Puts the tiles that overlap a strip's cells [i0, i0 + nv) x [j0, j0 + nh) on the list, each once.
__device__ __forceinline__ void list_strip(const KParams& P, unsigned int* work, int by0, int i0, int nv, int j0,
                                           int nh) {
  const LearnedWork w(P, work, by0);
  const int bx0 = (i0 - P.ng) / F32_TX, bx1 = (i0 - P.ng + nv - 1) / F32_TX;
  const int r0 = (j0 - P.ng) / F32_TY, r1 = (j0 - P.ng + nh - 1) / F32_TY;
  const int n = (bx1 - bx0 + 1) * (r1 - r0 + 1);
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const int t = (r0 + k / (bx1 - bx0 + 1)) * w.tx + bx0 + k % (bx1 - bx0 + 1);
    if (atomicExch(&w.mark[t], 1u) == 0u) w.list[atomicAdd(&w.counters[0], 1u)] = t;
  }
}

template <int MODE>
__global__ void __launch_bounds__(MARCH_MAX_THREADS, MARCH_SM_THREADS / MARCH_MAX_THREADS)
    march_step_kernel(KParams P, const float* __restrict__ Uin, float* __restrict__ Uout, StepScalars sc_host,
                      const StepScalars* __restrict__ sc_dev, DevScratch* __restrict__ scr, int nv, int nh,
                      const MlpBlob* __restrict__ mlp, unsigned int* __restrict__ work) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  SP<float> s;
  s.load(P);
  StepFactors<float> f;
  f.load(sc_dev ? *sc_dev : sc_host);
  TileCounters cnt;
  const int i0 = P.ng + blockIdx.x * nv, j0 = P.ng + blockIdx.y * nh;
  const int cols = min(nv, P.ng + P.nx - i0), n = min(nh, P.ng + P.ny - j0);
  if (ctu_march<MODE, false>(P, s, f, Uin, Uout, i0, cols, j0, n, smem_raw, cnt, mlp)) {
    cnt = TileCounters();  // the strip's tiles count instead
    list_strip(P, work, 0, i0, cols, j0, n);
  }
  flush_counters(cnt, scr);
}

// The fused step (see ctu_step_fused_kernel) over rows [row0, row0 + rows) of the interior, which may be one band of
// a step whose bands run as launches of their own.
template <int MODE>
__global__ void __launch_bounds__(MARCH_MAX_THREADS, MARCH_SM_THREADS / MARCH_MAX_THREADS)
    march_step_fused_kernel(KParams P, const float* __restrict__ Uin, float* __restrict__ Uout,
                            const StepScalars* __restrict__ sc_cur, StepScalars* __restrict__ sc_next,
                            DevScratch* __restrict__ scr, double tmax, int row0, int rows, int nv, int nh,
                            const MlpBlob* __restrict__ mlp, unsigned int* __restrict__ work) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  step_begin();
  SP<float> s;
  s.load(P);
  StepFactors<float> f;
  f.load_ordered(sc_cur);
  TileCounters cnt;
  float cmin = FLT_MAX;
  const int i0 = P.ng + blockIdx.x * nv, j0 = P.ng + row0 + blockIdx.y * nh;
  const int cols = min(nv, P.ng + P.nx - i0), n = min(nh, P.ng + row0 + rows - j0);
  if (sf_zero(ld_ordered(&sc_cur->dt))) {  // a step of length zero: copy (ctu_step_fused_kernel)
    const size_t plane = (size_t)P.NY * P.pitch;
    if ((int)threadIdx.x < cols) {
      for (int j = 0; j < n; ++j) {
        const size_t o = (size_t)(j0 + j) * P.pitch + i0 + threadIdx.x;
        float u[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) Uout[o + k * plane] = u[k] = ld_ordered(Uin + o + k * plane);
        cfl_value(s, u[0], u[1], u[2], u[3], cmin, cnt.flags);
      }
    }
  } else if (ctu_march<MODE, true>(P, s, f, Uin, Uout, i0, cols, j0, n, smem_raw, cnt, mlp, &cmin)) {
    cnt = TileCounters();  // the strip's tiles count instead
    cmin = FLT_MAX;
    list_strip(P, work, row0 / F32_TY, i0, cols, j0, n);
  }
  flush_counters(cnt, scr);
  // a strip counts its rows, so that the bands of a step may cut it into segments of their own height; a learned step
  // is finished by the launch over the listed tiles
  finish_fused_step<face_kind(MODE) != FACE_LEARNED>(P, cmin, sc_cur, sc_next, scr, tmax, (unsigned int)n, gridDim.x * (unsigned int)P.ny);
}

// The listed tiles of a learned step, from the network's proposals (blocks take them from the list until it is empty),
// and for a fused step its end.  by0, rows: the tile rows of the launch (a band of the step, or all).  Bound by the chain
// of stages of the few tiles it has.  Sedov 8192^2 learned, one step: 4.73 ms with all tiles in the tile kernel, 3.40 in
// strips with this launch; with the network called from the strip's loop the strips on the blast's front took 1 ms each.
template <bool FUSED>
__global__ void __launch_bounds__(320, 3)
    learned_tiles_kernel(KParams P, const float* __restrict__ Uin, float* __restrict__ Uout, StepScalars sc_host,
                         const StepScalars* __restrict__ sc_dev, StepScalars* __restrict__ sc_next,
                         DevScratch* __restrict__ scr, double tmax, const __grid_constant__ CUtensorMap tmap, int use_tma,
                         int by0, int rows, const MlpBlob* __restrict__ mlp, unsigned int* __restrict__ work) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ int cur;
  const LearnedWork w(P, work, by0);
  TileCounters cnt;
  float cmin = FLT_MAX;
  const unsigned int n = *(volatile unsigned int*)&w.counters[0];
  if (n > 0) {
    SP<float> s;
    s.load(P);
    StepFactors<float> f;
    f.load(sc_dev ? *sc_dev : sc_host);
    while (true) {
      if (threadIdx.x == 0) {
        const unsigned int k = atomicAdd(&w.counters[1], 1u);
        cur = k < n ? w.list[k] : -1;
        if (cur >= 0) w.mark[cur] = 0u;
      }
      __syncthreads();
      const int t = cur;
      if (t < 0) break;
      ctu_tile<float, F32_TX, F32_TY, 320, FACE_LEARNED, FUSED, true>(P, s, f, Uin, Uout, t % w.tx, t / w.tx, smem_raw,
                                                                      cnt, FaceHook{}, mlp, &cmin,
                                                                      use_tma ? &tmap : nullptr);
      __syncthreads();  // the tile's last shared-memory reads finish before the next tile's loads
    }
  }
  flush_counters(cnt, scr);
  if constexpr (FUSED)
    finish_fused_step(P, cmin, sc_dev, sc_next, scr, tmax, (unsigned int)rows,
                      gridDim.x * (unsigned int)((P.ny + F32_TY - 1) / F32_TY));
  if (threadIdx.x == 0 && atomicAdd(&w.counters[2], 1u) == gridDim.x - 1u)
    w.counters[0] = w.counters[1] = w.counters[2] = 0u;
}

// Strips of a grid: nv columns and nh rows each, `threads` a block.  nh == 0: the grid is stepped in tiles.
struct StripShape {
  int nv, nh, threads;
};

// What a step costs in us: strips waves * (row * nh + 9) + base - 9 (a row takes a strip `row` us with one strip on the SM
// or with four; the rest is the rows loaded ahead, the launch and the tail), tiles 10 + tile * waves, where tiles share
// the SMs evenly, so that waves are counted in fractions.  Tiles on reflecting or hydrostatic sides take 2.5 times as
// long (bc_cell_clamped).
struct StepCost {
  double row, base, tile;
};
inline StepCost step_cost(const KParams& P) {
  if (P.reconstruction == 1) return P.riemann_solver == 1 ? StepCost{4.0, 13.0, 17.0} : StepCost{5.1, 14.5, 19.0};
  return P.riemann_solver == 1 ? StepCost{3.15, 12.0, 14.0} : StepCost{4.3, 14.0, 16.4};
}

// The strips of the grid on nsm SMs: the width (64, 96 or 128 threads, four columns of halo on each side) and the number
// of rows that fill the SMs' strips evenly, in one wave where that takes at most 64 rows (in more, the SMs even out
// strips of unlike cost: Sedov 4096^2 776 us per step in three or four waves, 860 in two, 1048 in one).  The step takes
// the cheaper of strips and tiles, and tiles where the segments would be under five rows (their two halo rows are then
// 40 % of the work, and the solves counted are twice a tile's).  Measured (us per step, tiles / strips):
//   two-shock, PLM   512^2 29.0 / 34.4, 600x500 32.6 / 37.1, 700x500 33.7 / 35.0, RT 317x951 39.3 / 36.3, 800x640 43.8 /
//                    46.4, 1000x800 65.9 / 65.7, KH 1024^2 79.4 / 78.0, 1300x1500 147 / 137, Sedov 2048^2 310 / 292
//   HLLC             512^2 26.5 / 27.8, 700x500 30.9 / 28.3, 800x640 40.5 / 37.0, KH 1024^2 68.8 / 56.4
//   two-shock, PPM   512^2 32.9 / 39.6, 800x640 50.6 / 53.7, 1000x700 69.8 / 75.9, KH 1024^2 92.3 / 90.5, 1300x1500 171 / 158
inline StripShape strip_shape(const KParams& P, int nsm) {
  constexpr int MAX_ROWS = 64;
  const StepCost k = step_cost(P);
  const int nx = P.nx, ny = P.ny;
  StripShape best{0, 0, 0};
  double best_cost = 0.0;
  for (int threads = MARCH_MAX_THREADS; threads >= 64; threads -= 32) {
    const int n = (nx + threads - 9) / (threads - 8);  // strips across
    const long long slots = (long long)nsm * (MARCH_SM_THREADS / threads);
    long long waves = 1, m = slots / n > 1 ? slots / n : 1;  // segments per strip
    while ((ny + m - 1) / m > MAX_ROWS) {
      ++waves;
      m = slots * waves / n > 1 ? slots * waves / n : 1;
      if (waves > (1 << 20)) break;
    }
    const int nh = (int)((ny + m - 1) / m);
    const double cost = (double)waves * (k.row * nh + 9.0) + k.base - 9.0;
    if (best.nh == 0 || cost < best_cost) {
      best = StripShape{(nx + n - 1) / n, nh, threads};
      best_cost = cost;
    }
  }
  const long long tx = (nx + F32_TX - 1) / F32_TX, ty = (ny + F32_TY - 1) / F32_TY;
  const double tiles = (double)(tx * ty) + (P.bc_general ? 3.0 * (double)(tx + ty) : 0.0);
  const double tile_cost = 10.0 + k.tile * tiles / (HYDRO_F32_MINB * (double)nsm);
  if (best.nh < 5 || best_cost >= tile_cost) best.nh = 0;
  return best;
}

// The shape for a launch (nh == 0: tiles).  The withheld-copy test (hydro_test_drop_tile_copies) steps in tiles,
// whose loads it is about.  A learned step's strips give up where they meet a strong face and cost a second launch, of
// tiles three to an SM, so they need many waves of tiles to gain (us per step, tiles / strips, KH and quad problems:
// 600x500 35.9 / 44.1 and 40.7 / 76.8, 1000^2 88 / 89 and 100 / 121, 1900^2 278 / 243 and 305 / 302).
constexpr int LEARNED_STRIP_WAVES = 16;

inline cudaError_t choose_strips(const KParams& P, StripShape* shape, bool learned = false) {
  *shape = StripShape{0, 0, 0};
  if (P.tma_test_drop) return cudaSuccess;
  int nsm = 0;
  const cudaError_t e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  const long long tiles = (long long)((P.nx + F32_TX - 1) / F32_TX) * ((P.ny + F32_TY - 1) / F32_TY);
  if (!learned || tiles >= (long long)LEARNED_STRIP_WAVES * HYDRO_F32_MINB * nsm) *shape = strip_shape(P, nsm);
  return cudaSuccess;
}

template <int MODE>
cudaError_t launch_march_step(const StripShape& sh, const KParams& P, const float* Uin, float* Uout,
                              const StepScalars& sc_host, const StepScalars* sc_dev, DevScratch* scr,
                              cudaStream_t stream, const MlpBlob* mlp = nullptr, unsigned int* work = nullptr) {
  static std::atomic<unsigned long long> attr_done{0};
  const cudaError_t e = smem_attr_once(march_step_kernel<MODE>, march_bytes(MARCH_MAX_THREADS), attr_done);
  if (e != cudaSuccess) return e;
  const dim3 grid((P.nx + sh.nv - 1) / sh.nv, (P.ny + sh.nh - 1) / sh.nh);
  march_step_kernel<MODE><<<grid, sh.threads, march_bytes(sh.threads), stream>>>(
      P, Uin, Uout, sc_host, sc_dev, scr, sh.nv, sh.nh, mlp, work);
  return cudaGetLastError();
}

// band: tile rows of F32_TY cells (band.y <= 0: the whole step).  The segments of a band are short, since a band is a
// fraction of the step and what counts is when its last row is done (KH 1024^2 chained host step, five bands: 188 us
// with 4 rows, 194 with 8, 209 with 2; 8192^2 7.66 ms with 16 or 32, 7.72 with 8, and with the learned start 7.74 and
// 8.13; 4096^2 2.00, 2.03 with 32).
template <int MODE>
cudaError_t launch_march_step_fused(const StripShape& sh, const KParams& P, const float* Uin, float* Uout,
                                    const StepScalars* sc_cur, StepScalars* sc_next, DevScratch* scr, double tmax,
                                    cudaStream_t stream, int2 band, const MlpBlob* mlp = nullptr,
                                    unsigned int* work = nullptr) {
  static std::atomic<unsigned long long> attr_done{0};
  const cudaError_t e = smem_attr_once(march_step_fused_kernel<MODE>, march_bytes(MARCH_MAX_THREADS), attr_done);
  if (e != cudaSuccess) return e;
  const int row0 = band.y > 0 ? band.x * F32_TY : 0;
  const int rows = band.y > 0 ? min(band.y * F32_TY, P.ny - row0) : P.ny;
  const int nh = band.y <= 0 ? sh.nh : sh.nh < 32 ? 4 : 16;
  if (row0 < 0 || rows <= 0 || row0 + rows > P.ny) return cudaErrorInvalidValue;
  const dim3 grid((P.nx + sh.nv - 1) / sh.nv, (rows + nh - 1) / nh);
  return launch_step_kernel(march_step_fused_kernel<MODE>, grid, sh.threads, march_bytes(sh.threads), stream, P, Uin, Uout,
                            sc_cur, sc_next, scr, tmax, row0, rows, sh.nv, nh, mlp, work);
}

// A learned step of a grid that runs in strips: the strips, then the tiles they listed (three to an SM).
template <bool FUSED>
cudaError_t launch_learned_tiles(const KParams& P, const float* Uin, float* Uout, const StepScalars& sc_host,
                                 const StepScalars* sc_dev, StepScalars* sc_next, DevScratch* scr, double tmax,
                                 const CUtensorMap* tmap, cudaStream_t stream, int2 band, const MlpBlob* mlp,
                                 unsigned int* work) {
  static std::atomic<unsigned long long> attr_done{0};
  const size_t smem = TileLayout<float, F32_TX, F32_TY>::bytes;
  cudaError_t e = smem_attr_once(learned_tiles_kernel<FUSED>, smem, attr_done);
  int nsm = 0;
  if (e == cudaSuccess) e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  const int ty = (P.ny + F32_TY - 1) / F32_TY, by0 = band.y > 0 ? band.x : 0, rows = band.y > 0 ? band.y : ty;
  learned_tiles_kernel<FUSED><<<3 * nsm, 320, smem, stream>>>(P, Uin, Uout, sc_host, sc_dev, sc_next, scr, tmax,
                                                             tmap ? *tmap : CUtensorMap{}, tmap ? 1 : 0, by0, rows, mlp,
                                                             work);
  return cudaGetLastError();
}

}  // namespace hydro
