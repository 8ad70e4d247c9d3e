// Kernels and launches of the FP32 step in marching strips (ctu_march.cuh), with the rule that chooses between
// strips and tiles.
#pragma once

#include "ctu_kernels.cuh"
#include "ctu_march.cuh"

namespace hydro {
// A strip's registers (128 a thread) let 512 threads share an SM: four strips of 128 columns.
constexpr int MARCH_MAX_THREADS = 128, MARCH_SM_THREADS = 512;

template <int MODE>
__global__ void __launch_bounds__(MARCH_MAX_THREADS, MARCH_SM_THREADS / MARCH_MAX_THREADS)
    march_step_kernel(KParams P, const float* __restrict__ Uin, float* __restrict__ Uout, StepScalars sc_host,
                      const StepScalars* __restrict__ sc_dev, DevScratch* __restrict__ scr, int nv, int nh) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  SP<float> s;
  s.load(P);
  StepFactors<float> f;
  f.load(sc_dev ? *sc_dev : sc_host);
  TileCounters cnt;
  const int i0 = P.ng + blockIdx.x * nv, j0 = P.ng + blockIdx.y * nh;
  ctu_march<MODE, false>(P, s, f, Uin, Uout, i0, min(nv, P.ng + P.nx - i0), j0, min(nh, P.ng + P.ny - j0), smem_raw,
                            cnt);
  flush_counters(cnt, scr);
}

// The fused step (see ctu_step_fused_kernel) over rows [row0, row0 + rows) of the interior, which may be one band of
// a step whose bands run as launches of their own.
template <int MODE>
__global__ void __launch_bounds__(MARCH_MAX_THREADS, MARCH_SM_THREADS / MARCH_MAX_THREADS)
    march_step_fused_kernel(KParams P, const float* __restrict__ Uin, float* __restrict__ Uout,
                            const StepScalars* __restrict__ sc_cur, StepScalars* __restrict__ sc_next,
                            DevScratch* __restrict__ scr, double tmax, int row0, int rows, int nv, int nh) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  SP<float> s;
  s.load(P);
  StepFactors<float> f;
  f.load(*sc_cur);
  TileCounters cnt;
  float cmin = FLT_MAX;
  const int i0 = P.ng + blockIdx.x * nv, j0 = P.ng + row0 + blockIdx.y * nh;
  const int cols = min(nv, P.ng + P.nx - i0), n = min(nh, P.ng + row0 + rows - j0);
  if (sf_zero(sc_cur->dt)) {  // a step of length zero: copy (ctu_step_fused_kernel)
    const size_t plane = (size_t)P.NY * P.pitch;
    if ((int)threadIdx.x < cols) {
      for (int j = 0; j < n; ++j) {
        const size_t o = (size_t)(j0 + j) * P.pitch + i0 + threadIdx.x;
        float u[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) Uout[o + k * plane] = u[k] = Uin[o + k * plane];
        cfl_value(s, u[0], u[1], u[2], u[3], cmin, cnt.flags);
      }
    }
  } else {
    ctu_march<MODE, true>(P, s, f, Uin, Uout, i0, cols, j0, n, smem_raw, cnt, &cmin);
  }
  flush_counters(cnt, scr);
  // a strip counts its rows, so that the bands of a step may cut it into segments of their own height
  finish_fused_step(P, cmin, sc_cur, sc_next, scr, tmax, (unsigned int)n, gridDim.x * (unsigned int)P.ny);
}

// Strips of a grid: nv columns and nh rows each, `threads` a block.  nh == 0: the grid is stepped in tiles.
struct StripShape {
  int nv, nh, threads;
};

// The strips of an nx x ny grid on nsm SMs: the width (64, 96 or 128 threads, four columns of halo on each side) and
// the number of rows that fill the SMs' strips evenly, in one wave where that takes at most 64 rows (in more, the SMs
// even out strips of unlike cost: Sedov 4096^2 776 us per step in three or four waves, 860 in two, 1048 in one).  A row
// takes a strip 3 to 4 us with one strip on the SM or with four, and each strip has six rows to load and two rows of
// halo beside its own, so a step takes about 4 nh + 9 us a wave; a wave of three 32x16 tiles per SM is 16 us.  The
// step takes the cheaper of the two, and tiles where the segments would be under five rows (their two halo rows are
// then 40 % of the work, and the solves counted are twice a tile's).  Measured (us per step, tiles / strips): KH 64^2 16.8 / 15.1 (tiles),
// 256^2 16.8 / 20.8 (tiles), 512^2 30.9 / 31.7 (tiles), 700x500 35.3 / 33.7, 1024^2 80.4 / 71.3, 1500x1300 139.8 / 116,
// 2048^2 287 / 234, RT 317x951 39.6 / 36.2, Sedov 4096^2 1073 / 776.
inline StripShape strip_shape(int nx, int ny, int nsm) {
  constexpr int MAX_ROWS = 64;
  StripShape best{0, 0, 0};
  long long best_cost = 0;
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
    const long long cost = waves * (4 * nh + 9);
    if (best.nh == 0 || cost < best_cost) {
      best = StripShape{(nx + n - 1) / n, nh, threads};
      best_cost = cost;
    }
  }
  const long long tiles = (long long)((nx + F32_TX - 1) / F32_TX) * ((ny + F32_TY - 1) / F32_TY);
  const long long tile_waves = (tiles + HYDRO_F32_MINB * (long long)nsm - 1) / (HYDRO_F32_MINB * (long long)nsm);
  if (best.nh < 5 || best_cost >= 16 * tile_waves) best.nh = 0;
  return best;
}

// The shape for a launch (nh == 0: tiles).  The withheld-copy test (hydro_test_drop_tile_copies) steps in tiles,
// whose loads it is about.
inline cudaError_t choose_strips(const KParams& P, StripShape* shape) {
  *shape = StripShape{0, 0, 0};
  if (P.tma_test_drop) return cudaSuccess;
  int dev = 0, nsm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) *shape = strip_shape(P.nx, P.ny, nsm);
  return e;
}

template <int MODE>
cudaError_t launch_march_step(const StripShape& sh, const KParams& P, const float* Uin, float* Uout,
                              const StepScalars& sc_host, const StepScalars* sc_dev, DevScratch* scr,
                              cudaStream_t stream) {
  static std::atomic<unsigned long long> attr_done{0};
  const cudaError_t e = smem_attr_once(march_step_kernel<MODE>, march_bytes(MARCH_MAX_THREADS), attr_done);
  if (e != cudaSuccess) return e;
  const dim3 grid((P.nx + sh.nv - 1) / sh.nv, (P.ny + sh.nh - 1) / sh.nh);
  march_step_kernel<MODE><<<grid, sh.threads, march_bytes(sh.threads), stream>>>(
      P, Uin, Uout, sc_host, sc_dev, scr, sh.nv, sh.nh);
  return cudaGetLastError();
}

// band: tile rows of F32_TY cells (band.y <= 0: the whole step).  The segments of a band are short, since a band is a
// fraction of the step and what counts is when its last row is done (KH 1024^2 chained host step, five bands: 188 us
// with 4 rows, 194 with 8, 209 with 2; 4096^2: 2025 with 8, 2050 with 4).
template <int MODE>
cudaError_t launch_march_step_fused(const StripShape& sh, const KParams& P, const float* Uin, float* Uout,
                                    const StepScalars* sc_cur, StepScalars* sc_next, DevScratch* scr, double tmax,
                                    cudaStream_t stream, int2 band) {
  static std::atomic<unsigned long long> attr_done{0};
  const cudaError_t e =
      smem_attr_once(march_step_fused_kernel<MODE>, march_bytes(MARCH_MAX_THREADS), attr_done);
  if (e != cudaSuccess) return e;
  const int row0 = band.y > 0 ? band.x * F32_TY : 0;
  const int rows = band.y > 0 ? min(band.y * F32_TY, P.ny - row0) : P.ny;
  const int nh = band.y <= 0 ? sh.nh : sh.nh < 32 ? 4 : 8;
  if (row0 < 0 || rows <= 0 || row0 + rows > P.ny) return cudaErrorInvalidValue;
  const dim3 grid((P.nx + sh.nv - 1) / sh.nv, (rows + nh - 1) / nh);
  march_step_fused_kernel<MODE><<<grid, sh.threads, march_bytes(sh.threads), stream>>>(
      P, Uin, Uout, sc_cur, sc_next, scr, tmax, row0, rows, sh.nv, nh);
  return cudaGetLastError();
}

}  // namespace hydro
