// Kernels and launches of the FP32 step in marching strips (ctu_march.cuh), with the rule that chooses between
// strips and tiles.
#pragma once

#include "ctu_kernels.cuh"
#include "ctu_march.cuh"

namespace hydro {

static_assert(LEARNED_TX == F32_TX && LEARNED_TY == F32_TY, "the listed tiles are those of learned_tiles_kernel");

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
  ctu_march<MODE, false>(P, s, f, Uin, Uout, i0, cols, j0, n, smem_raw, cnt, nullptr, mlp, work);
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
  } else {
    ctu_march<MODE, true>(P, s, f, Uin, Uout, i0, cols, j0, n, smem_raw, cnt, &cmin, mlp, work, row0 / LEARNED_TY);
  }
  flush_counters(cnt, scr);
  // a strip counts its rows, so that the bands of a step may cut it into segments of their own height; a learned step
  // is finished by the launch over the listed tiles
  finish_fused_step<face_kind(MODE) != FACE_LEARNED>(P, cmin, sc_cur, sc_next, scr, tmax, (unsigned int)n,
                                                     gridDim.x * (unsigned int)P.ny);
}

// The second launch of a learned step: the listed tiles from the network's proposals (blocks take them from the list
// until it is empty), which overwrite the strips' cells; the records of the tiles that were not listed; and for a fused
// step its end.  by0, rows: the tile rows of the launch (a band of the step, or all).  Bound by the chain of stages of
// the few tiles it has (11 us without any, 38 with those of a blast's front; ncu).  Sedov 8192^2 learned, one step: 4.73 ms
// with all tiles in the tile kernel, 3.07 in strips with this launch (3.40 when a strip tested every face's gate and
// gave up at the first strong one, and the list depended on the cut); with the network called from the strip's loop the
// strips on the blast's front took 1 ms each.
// Two blocks an SM: with three the registers (64) spilled 136 bytes in the chain (Sedov 3000^2 503 us per step, 488 with
// two; 2200x2100 298 and 282).
template <bool FUSED>
__global__ void __launch_bounds__(320, 2)
    learned_tiles_kernel(KParams P, const float* __restrict__ Uin, float* __restrict__ Uout, StepScalars sc_host,
                         const StepScalars* __restrict__ sc_dev, StepScalars* __restrict__ sc_next,
                         DevScratch* __restrict__ scr, double tmax, const __grid_constant__ CUtensorMap tmap, int use_tma,
                         int by0, int rows, const MlpBlob* __restrict__ mlp, unsigned int* __restrict__ work) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ int cur;
  step_begin();
  const LearnedWork w(P.nx, P.ny, work, by0);
  TileCounters cnt;
  float cmin = FLT_MAX;
  const unsigned int n = *(volatile unsigned int*)&w.counters[0];
  if (n > 0) {
    SP<float> s;
    s.load(P);
    StepFactors<float> f;
    if (sc_dev)
      f.load_ordered(sc_dev);
    else
      f.load(sc_host);
    while (true) {
      if (threadIdx.x == 0) {
        const unsigned int k = atomicAdd(&w.counters[1], 1u);
        cur = k < n ? w.list[k] : -1;
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
  const int first = by0 * w.tx, tiles = rows * w.tx;
  for (int k = first + blockIdx.x * blockDim.x + threadIdx.x; k < first + tiles; k += gridDim.x * blockDim.x) {
    const unsigned int state = w.state[k];
    if (!(state & LearnedWork::LISTED)) {
      const unsigned long long c = w.count[k];
      cnt.flags |= state;
      cnt.solves += (unsigned int)(c >> 32);
      cnt.iters += (unsigned int)(c >> 32) + (unsigned int)c;
      cnt.nonconv += w.nonconv[k];
      cmin = fminf(cmin, __uint_as_float(0x7f7fffffu - w.slack[k]));
    }
    w.state[k] = w.slack[k] = w.nonconv[k] = 0u;
    w.count[k] = 0ull;
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
// whose loads it is about.  A learned step's strong faces cost a second launch, so its strips need many waves of tiles
// to gain (us per step, tiles / strips, KH, quadrants and Sedov: 1000^2 84.5 / 73.6, 101 / 123 and 82.3 / 128; 1500x1300
// 148 / 123, 169 / 181 and 144 / 185; 1900^2 268 / 199, 292 / 274 and 256 / 282, with three blocks of the second launch
// an SM).
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
  constexpr bool LEARNED = face_kind(MODE) == FACE_LEARNED;
  static std::atomic<unsigned long long> attr_done{0};
  const cudaError_t e = smem_attr_once(march_step_kernel<MODE>, march_bytes(MARCH_MAX_THREADS, LEARNED), attr_done);
  if (e != cudaSuccess) return e;
  const dim3 grid((P.nx + sh.nv - 1) / sh.nv, (P.ny + sh.nh - 1) / sh.nh);
  march_step_kernel<MODE><<<grid, sh.threads, march_bytes(sh.threads, LEARNED), stream>>>(
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
  constexpr bool LEARNED = face_kind(MODE) == FACE_LEARNED;
  static std::atomic<unsigned long long> attr_done{0};
  const cudaError_t e = smem_attr_once(march_step_fused_kernel<MODE>, march_bytes(MARCH_MAX_THREADS, LEARNED), attr_done);
  if (e != cudaSuccess) return e;
  const int row0 = band.y > 0 ? band.x * F32_TY : 0;
  const int rows = band.y > 0 ? min(band.y * F32_TY, P.ny - row0) : P.ny;
  const int nh = band.y <= 0 ? sh.nh : sh.nh < 32 ? 4 : 16;
  if (row0 < 0 || rows <= 0 || row0 + rows > P.ny) return cudaErrorInvalidValue;
  const dim3 grid((P.nx + sh.nv - 1) / sh.nv, (rows + nh - 1) / nh);
  return launch_step_kernel(march_step_fused_kernel<MODE>, grid, sh.threads, march_bytes(sh.threads, LEARNED), stream, P,
                            Uin, Uout, sc_cur, sc_next, scr, tmax, row0, rows, sh.nv, nh, mlp, work);
}

// A learned step of a grid that runs in strips: the strips, then the tiles they listed (two to an SM).
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
  return launch_step_kernel(learned_tiles_kernel<FUSED>, dim3(2 * nsm), 320, smem, stream, P, Uin, Uout, sc_host, sc_dev,
                            sc_next, scr, tmax, tmap ? *tmap : CUtensorMap{}, tmap ? 1 : 0, by0, rows, mlp, work);
}

}  // namespace hydro
