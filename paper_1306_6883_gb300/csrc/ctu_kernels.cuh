// Single-problem CTU step kernels and their launch templates: one CTA per tile (the tile itself is in
// ctu_tile.cuh).  Instantiated for FP32 in k_ctu.cu and for FP64 in k_ctu_f64.cu, which is compiled without
// multiply-add contraction.
#pragma once
#include <float.h>

#include <algorithm>
#include <atomic>
#include <utility>

#include "ctu_tile.cuh"
#include "hydro_kernels.h"

namespace hydro {

// Per-block reduction of the tile counters into the context's scratch: warp shuffles, then one thread adds
// the block's sums (one atomic per counter and block; per-warp atomics on the same words cost ~4 % of a
// KH 1024^2 step).  Called by every thread of the block (at most 512 threads).
__device__ __forceinline__ void flush_counters(TileCounters& cnt, DevScratch* scr) {
  if (cnt.nonconv) cnt.flags |= STATUS_NONCONV;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    cnt.solves += __shfl_xor_sync(0xffffffffu, cnt.solves, off);
    cnt.iters += __shfl_xor_sync(0xffffffffu, cnt.iters, off);
    cnt.nonconv += __shfl_xor_sync(0xffffffffu, cnt.nonconv, off);
    cnt.flags |= __shfl_xor_sync(0xffffffffu, cnt.flags, off);
  }
  __shared__ unsigned int part[16][4];
  if ((threadIdx.x & 31) == 0) {
    const int w = threadIdx.x >> 5;
    part[w][0] = cnt.solves;
    part[w][1] = cnt.iters;
    part[w][2] = cnt.nonconv;
    part[w][3] = cnt.flags;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long solves = 0, iters = 0, nonconv = 0;
    unsigned int flags = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      solves += part[w][0];
      iters += part[w][1];
      nonconv += part[w][2];
      flags |= part[w][3];
    }
    atomicAdd(&scr->stats[0], solves);
    atomicAdd(&scr->stats[1], iters);
    if (nonconv) atomicAdd(&scr->stats[2], nonconv);
    if (flags) atomicOr(&scr->status, flags);
  }
}

// End of a fused step for one block: its CFL minimum into the step's accumulator and its share into the step's
// count; the block that completes the count (total) advances the time by this step's dt and writes the next step's
// factors.  LAST false: the count is left to a later launch of the step.
template <bool LAST = true, typename R>
__device__ __forceinline__ void finish_fused_step(const KParams& P, R cmin, const StepScalars* sc_cur,
                                                  StepScalars* sc_next, DevScratch* scr, double tmax,
                                                  unsigned int share, unsigned int total) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const R o = __shfl_xor_sync(0xffffffffu, cmin, off);
    cmin = M<R>::mnp(o, cmin);
  }
  __shared__ R wmin[16];
  __shared__ bool last;
  if ((threadIdx.x & 31) == 0) wmin[threadIdx.x >> 5] = cmin;
  __syncthreads();
  if (threadIdx.x == 0) {
    R b = wmin[0];
    for (int k = 1; k < (int)(blockDim.x >> 5); ++k) b = wmin[k] < b ? wmin[k] : b;
    atomicMin(&scr->dtn_min_bits, (unsigned long long)__double_as_longlong((double)b));
    __threadfence();
    last = LAST && atomicAdd(&scr->step_blocks_done, share) + share == total;
  }
  __syncthreads();
  if (LAST && last && threadIdx.x == 0) {
    __threadfence();
    const unsigned long long bits =
        atomicExch(&scr->dtn_min_bits, (unsigned long long)__double_as_longlong(DBL_MAX));
    const double t = scr->t + ld_ordered(&sc_cur->dt);
    scr->t = t;
    scr->nsteps = scr->nsteps + 1;
    double dt = P.cfl * __longlong_as_double((long long)bits);
    if (tmax > 0.0) {
      const double left = tmax - t;
      dt = dt > left ? left : dt;
      dt = dt < 0.0 ? 0.0 : dt;
    }
    scr->dt = dt;
    *sc_next = make_step_scalars(dt, P.dx, P.dy, P.grav);
    scr->step_blocks_done = 0u;
  }
}

// Tile of the single-problem FP32 kernels (overridable at compile time for tile sweeps; the TMA box of the
// state buffers is encoded for it).  Measured on KH
// 1024^2 and Sedov 2048^2 at 256 threads: 32x16 (3 CTAs per SM) beats 30x16 (warp-aligned rows but a ragged
// last tile on power-of-two grids), 30x8 and 14x16 by 1-2%, and 30x24/384, 62x8 and 30x32/512 (fewer warps
// per SM) by 4-40%.  With 384 threads (36 warps per SM at 56 registers) 32x16 gains another 6-8%; more
// threads per tile force spills or fewer tiles per SM and lose.
#ifndef HYDRO_F32_TX
#define HYDRO_F32_TX 32
#endif
#ifndef HYDRO_F32_TY
#define HYDRO_F32_TY 16
#endif
#ifndef HYDRO_F32_NT
#define HYDRO_F32_NT 384
#endif
constexpr int F32_TX = HYDRO_F32_TX, F32_TY = HYDRO_F32_TY, F32_NT = HYDRO_F32_NT;

#ifndef HYDRO_F32_MINB
#define HYDRO_F32_MINB 3
#endif
// The FP32 tile of grids so small that all its tiles run at once, three to an SM: such a step takes as long as one
// block's chain of stages, which is shortest where each thread has one item per stage.  Measured per step, 16x8 at
// 384 threads / 32x16 (KH, us): 64^2 9.3 / 15.1, 192^2 (two tiles an SM / one) 10.6 / 15.2, 224^2 (three / one) 11.8 /
// 15.1, 256^2 (four, so two rounds / one) 14.9 / 15.2, 384^2 (eight / two) 23.9 / 18.3.  16x8 at 192 threads takes
// 10.6 at 64^2 and 12.4 at 224^2, 32x8 at 384 11.7 and 13.5, 8x8 at 256 9.1 and 14.2 (five to an SM).
constexpr int F32_SMALL_TX = 16, F32_SMALL_TY = 8;

// Tiles of the FP64 kernels.  Their time is the SM's one FP64 unit, so a tile's cost is its FP64 instructions,
// and what counts is the halo (for large grids) or how many SMs have a tile at all (for small ones).  Measured on
// KH 1024^2 per step / Sod 128^2 host loop per step: 16x16 at 384 threads, two per SM 2.75 ms / 155 us; at 256
// threads, three per SM 2.95 / 204; 32x8 at 384 2.74 / 155; 32x16 at 512, one per SM 2.84 / 267; 16x8 at 384
// 3.72 / 109; 16x8 at 192 3.32 / 119; 8x8 at 256 4.06 / 119.  A 16x8 tile costs 0.68 of a 16x16 one in both
// columns, so a step takes the shape with the smaller (tiles per SM, rounded up) x cost: 16x8 while its tiles
// find an SM each that 16x16 ones would leave idle.
constexpr int F64_TX = 16, F64_TY = 16, F64_NT = 384, F64_TY_SMALL = 8;

// Resident blocks per SM the register allocator must allow: shared memory admits three tiles per SM in FP32
// (three blocks of 384 threads need <= 56 registers) and in FP64 two of 16x16 (<= 85 registers, at which the two-shock
// step spills 64 bytes beside the arguments of its out-of-line solver: 0.9 % of the instructions of a KH 512^2 step are
// local loads and stores); the small FP64 tile runs one to an SM.
template <typename R, int TY>
constexpr int min_blocks() {
  return is_f32<R>() ? HYDRO_F32_MINB : TY == F64_TY ? 2 : 1;
}

template <typename R, int TX, int TY, int NT, int MODE>
__global__ void __launch_bounds__(NT, min_blocks<R, TY>()) ctu_step_kernel(KParams P, const R* __restrict__ Uin, R* __restrict__ Uout,
                                                      StepScalars sc_host, const StepScalars* __restrict__ sc_dev,
                                                      DevScratch* __restrict__ scr, FaceHook hook,
                                                      const __grid_constant__ CUtensorMap tmap, int use_tma) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  // the network's weights are read from global memory (L1/L2-resident) only by warps whose gate opens,
  // which is rare in smooth flow, so no CTA pays to stage them
  const MlpBlob* wsm = face_kind(MODE) == FACE_LEARNED ? hook.mlp : nullptr;
  SP<R> s;
  s.load(P);
  StepFactors<R> f;
  f.load(sc_dev ? *sc_dev : sc_host);
  TileCounters cnt;
  ctu_tile<R, TX, TY, NT, MODE>(P, s, f, Uin, Uout, blockIdx.x, blockIdx.y, smem_raw, cnt, hook, wsm, nullptr,
                                use_tma ? &tmap : nullptr);
  flush_counters(cnt, scr);
}

// Raises a kernel's dynamic shared-memory limit once per device (function attributes belong to the device's
// context); later calls on the same device only test a bit.  Devices beyond 63 set it on every call.
template <typename K>
cudaError_t smem_attr_once(K kernel, size_t smem, std::atomic<unsigned long long>& done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
  if (bit && (done.load(std::memory_order_relaxed) & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess && bit) done.fetch_or(bit, std::memory_order_relaxed);
  return e;
}

template <typename R, int TX, int TY, int NT, int MODE>
cudaError_t launch_ctu_step(const KParams& P, const R* Uin, R* Uout, const StepScalars& sc_host,
                            const StepScalars* sc_dev, DevScratch* scr, const FaceHook& hook, const CUtensorMap* tmap,
                            cudaStream_t stream) {
  const size_t smem = TileLayout<R, TX, TY>::bytes;
  static std::atomic<unsigned long long> attr_done{0};
  cudaError_t e = smem_attr_once(ctu_step_kernel<R, TX, TY, NT, MODE>, smem, attr_done);
  if (e != cudaSuccess) return e;
  dim3 grid((P.nx + TX - 1) / TX, (P.ny + TY - 1) / TY);
  ctu_step_kernel<R, TX, TY, NT, MODE><<<grid, NT, smem, stream>>>(P, Uin, Uout, sc_host, sc_dev, scr, hook,
                                                                    tmap ? *tmap : CUtensorMap{}, tmap ? 1 : 0);
  return cudaGetLastError();
}

// Fused steps follow one another on a stream, one launch each.  Their kernels are launched so that the next one's
// blocks are placed as soon as every block of this one has exited, and wait there for what it wrote (step_begin, the
// kernel's first statement): launch and flush then overlap (us per step: KH 64^2 FP32 11.0 -> 9.4, 384^2 21.1 -> 18.4,
// split 512^2 27.3 -> 22.9, KH 64^2 FP64 77.0 -> 74.1).  Blocks placed any earlier hold SMs that another stream's
// kernels could use, and unevenly, since SMs that are done first take more than their share.  Let in when this one's
// blocks had begun, with shared memory padded to hold an SM to its even share, four KH 256^2 solvers on streams of
// their own took 36.4 us per step (22.6 now, 24.7 without overlap); let in before the blocks' last reductions,
// unpadded, FP64 192^2 alone took 154 (126 now).  What the step before wrote is read with ld_ordered.
__device__ __forceinline__ void step_begin() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

inline cudaError_t sm_count(int* nsm) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  return e == cudaSuccess ? cudaDeviceGetAttribute(nsm, cudaDevAttrMultiProcessorCount, dev) : e;
}

// Launches a fused step's kernel.
template <typename... Params, typename... Args>
cudaError_t launch_step_kernel(void (*kernel)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t stream,
                               Args&&... args) {
  // a captured step keeps plain dependencies: graphs that a program edits or queries see the edges they always had
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  const cudaError_t e = cudaStreamIsCapturing(stream, &cap);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned int)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &attr;
  cfg.numAttrs = cap == cudaStreamCaptureStatusNone ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// Fused step: the tile reads ghost cells through the boundary map and folds the CFL constraint of its new
// cells into a block minimum; the last block to finish advances the time by this step's dt and writes
// the next step's factors, so a run needs one launch per step and no ghost-fill or dt pass.  A step may be
// split into launches over bands of tile rows (by0: the band's first tile row; nblocks: the tiles of the
// whole step), which run concurrently; the last block of all of them finishes the step.
template <typename R, int TX, int TY, int NT, int MODE = FACE_PLAIN>
__global__ void __launch_bounds__(NT, min_blocks<R, TY>()) ctu_step_fused_kernel(KParams P, const R* __restrict__ Uin,
                                                            R* __restrict__ Uout, const StepScalars* __restrict__ sc_cur,
                                                            StepScalars* __restrict__ sc_next,
                                                            DevScratch* __restrict__ scr, double tmax,
                                                            const __grid_constant__ CUtensorMap tmap, int use_tma,
                                                            int by0, unsigned int nblocks,
                                                            const MlpBlob* __restrict__ mlp) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  step_begin();
  // FACE_LEARNED: the network's weights (read from global memory by the warps whose gate opens)
  const MlpBlob* wsm = face_kind(MODE) == FACE_LEARNED ? mlp : nullptr;
  SP<R> s;
  s.load(P);
  StepFactors<R> f;
  f.load_ordered(sc_cur);
  TileCounters cnt;
  R cmin = is_f32<R>() ? (R)FLT_MAX : (R)DBL_MAX;
  const int by = by0 + (int)blockIdx.y;
  if (sf_zero(ld_ordered(&sc_cur->dt))) {
    // a step of length zero (the run has reached tmax) leaves the state as it is: copy the tile's interior
    // cells and take their CFL constraint as a step would (the next dt is then clamped to 0 again)
    const size_t plane = (size_t)P.NY * P.pitch;
    for (int e = threadIdx.x; e < TX * TY; e += NT) {
      const int gi = P.ng + blockIdx.x * TX + e % TX, gj = P.ng + by * TY + e / TX;
      if (gi >= P.ng + P.nx || gj >= P.ng + P.ny) continue;
      const size_t o = (size_t)gj * P.pitch + gi;
      R u[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) Uout[o + k * plane] = u[k] = ld_ordered(Uin + o + k * plane);
      cfl_value(s, u[0], u[1], u[2], u[3], cmin, cnt.flags);
    }
  } else {
    ctu_tile<R, TX, TY, NT, MODE, true>(P, s, f, Uin, Uout, blockIdx.x, by, smem_raw, cnt, FaceHook{}, wsm,
                                        &cmin, use_tma ? &tmap : nullptr);
  }
  flush_counters(cnt, scr);
  finish_fused_step(P, cmin, sc_cur, sc_next, scr, tmax, 1u, nblocks);
}

// band: tile rows [band.x, band.x + band.y) of the step (band.y <= 0: all of them).  mlp: the network of
// MODE FACE_LEARNED (device).
template <typename R, int TX, int TY, int NT, int MODE = FACE_PLAIN>
cudaError_t launch_ctu_step_fused(const KParams& P, const R* Uin, R* Uout, const StepScalars* sc_cur,
                                  StepScalars* sc_next, DevScratch* scr, double tmax, const CUtensorMap* tmap,
                                  cudaStream_t stream, int2 band = make_int2(0, 0), const MlpBlob* mlp = nullptr) {
  const size_t smem = TileLayout<R, TX, TY>::bytes;
  static std::atomic<unsigned long long> attr_done{0};
  cudaError_t e = smem_attr_once(ctu_step_fused_kernel<R, TX, TY, NT, MODE>, smem, attr_done);
  if (e != cudaSuccess) return e;
  const int tx = (P.nx + TX - 1) / TX, ty = (P.ny + TY - 1) / TY;
  const int y0 = band.y > 0 ? band.x : 0, ny = band.y > 0 ? band.y : ty;
  if (y0 < 0 || ny <= 0 || y0 + ny > ty) return cudaErrorInvalidValue;
  dim3 grid(tx, ny);
  return launch_step_kernel(ctu_step_fused_kernel<R, TX, TY, NT, MODE>, grid, NT, smem, stream, P, Uin, Uout,
                            sc_cur, sc_next, scr, tmax, tmap ? *tmap : CUtensorMap{}, tmap ? 1 : 0, y0,
                            (unsigned int)tx * (unsigned int)ty, mlp);
}

// Whether an FP64 step takes 16x8 tiles instead of 16x16 ones (see F64_TY_SMALL).
inline cudaError_t f64_small_tile(const KParams& P, bool* small) {
  int nsm = 0;
  const cudaError_t e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  auto rounds = [&](int ty) {
    const long long n = (long long)((P.nx + F64_TX - 1) / F64_TX) * ((P.ny + ty - 1) / ty);
    return (n + nsm - 1) / nsm;
  };
  *small = 17 * rounds(F64_TY_SMALL) < 25 * rounds(F64_TY);
  return cudaSuccess;
}

template <int MODE>
cudaError_t launch_ctu_step_f64(const KParams& P, const double* Uin, double* Uout, const StepScalars& sc_host,
                                const StepScalars* sc_dev, DevScratch* scr, cudaStream_t stream) {
  bool small = false;
  const cudaError_t e = f64_small_tile(P, &small);
  if (e != cudaSuccess) return e;
  const auto launch = small ? launch_ctu_step<double, F64_TX, F64_TY_SMALL, F64_NT, MODE>
                            : launch_ctu_step<double, F64_TX, F64_TY, F64_NT, MODE>;
  return launch(P, Uin, Uout, sc_host, sc_dev, scr, FaceHook{}, nullptr, stream);
}

// A band of a step (band.y > 0) counts tile rows of 16 cells (fused_tile_height).
template <int MODE>
cudaError_t launch_ctu_step_fused_f64(const KParams& P, const double* Uin, double* Uout, const StepScalars* sc_cur,
                                      StepScalars* sc_next, DevScratch* scr, double tmax, cudaStream_t stream,
                                      int2 band) {
  bool small = false;
  const cudaError_t e = band.y > 0 ? cudaSuccess : f64_small_tile(P, &small);
  if (e != cudaSuccess) return e;
  const auto launch = small ? launch_ctu_step_fused<double, F64_TX, F64_TY_SMALL, F64_NT, MODE>
                            : launch_ctu_step_fused<double, F64_TX, F64_TY, F64_NT, MODE>;
  return launch(P, Uin, Uout, sc_cur, sc_next, scr, tmax, nullptr, stream, band, nullptr);
}

// Whether an FP32 step in tiles takes the small ones (see F32_SMALL_TX).  The withheld-copy test
// (hydro_test_drop_tile_copies) keeps the large ones, which load through the tensor map.
inline cudaError_t f32_small_tile(const KParams& P, bool* small) {
  int nsm = 0;
  const cudaError_t e = sm_count(&nsm);
  const long long n =
      (long long)((P.nx + F32_SMALL_TX - 1) / F32_SMALL_TX) * ((P.ny + F32_SMALL_TY - 1) / F32_SMALL_TY);
  *small = !P.tma_test_drop && n <= (long long)HYDRO_F32_MINB * nsm;
  return e;
}

template <int MODE, int NT = F32_NT>
cudaError_t launch_ctu_step_f32(const KParams& P, const float* Uin, float* Uout, const StepScalars& sc_host,
                                const StepScalars* sc_dev, DevScratch* scr, const FaceHook& hook,
                                const CUtensorMap* tmap, cudaStream_t stream) {
  bool small = false;
  const cudaError_t e = f32_small_tile(P, &small);
  if (e != cudaSuccess) return e;
  if (small)
    return launch_ctu_step<float, F32_SMALL_TX, F32_SMALL_TY, NT, MODE>(P, Uin, Uout, sc_host, sc_dev, scr, hook,
                                                                        nullptr, stream);
  return launch_ctu_step<float, F32_TX, F32_TY, NT, MODE>(P, Uin, Uout, sc_host, sc_dev, scr, hook, tmap, stream);
}

// A band of a step (band.y > 0) counts tile rows of F32_TY cells.
template <int MODE, int NT = F32_NT>
cudaError_t launch_ctu_step_fused_f32(const KParams& P, const float* Uin, float* Uout, const StepScalars* sc_cur,
                                      StepScalars* sc_next, DevScratch* scr, double tmax, const CUtensorMap* tmap,
                                      cudaStream_t stream, int2 band, const MlpBlob* mlp = nullptr) {
  bool small = false;
  const cudaError_t e = band.y > 0 ? cudaSuccess : f32_small_tile(P, &small);
  if (e != cudaSuccess) return e;
  if (small)
    return launch_ctu_step_fused<float, F32_SMALL_TX, F32_SMALL_TY, NT, MODE>(P, Uin, Uout, sc_cur, sc_next, scr, tmax,
                                                                              nullptr, stream, band, mlp);
  return launch_ctu_step_fused<float, F32_TX, F32_TY, NT, MODE>(P, Uin, Uout, sc_cur, sc_next, scr, tmax, tmap, stream,
                                                                band, mlp);
}

}  // namespace hydro
