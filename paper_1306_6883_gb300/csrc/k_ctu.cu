// Single-problem CTU step: the FP32 instantiations (strips or tiles, march_kernels.cuh) and the precision dispatch
// (FP64 in k_ctu_f64.cu).
#include "march_kernels.cuh"

namespace hydro {

int f32_tile_x() { return F32_TX; }
int f32_tile_y() { return F32_TY; }

cudaError_t ctu_step_fused(int precision, const KParams& P, const void* Uin, void* Uout, const StepScalars* sc_cur,
                           StepScalars* sc_next, DevScratch* scr, double tmax, const CUtensorMap* tmap,
                           cudaStream_t stream, int2 band, const MlpBlob* mlp, unsigned int* learned_work) {
  if (mlp != nullptr && (precision == 0 || P.reconstruction == 1 || P.riemann_solver == 1)) return cudaErrorInvalidValue;
  if (P.reconstruction == 1)
    return ctu_step_fused_ppm(precision, P, Uin, Uout, sc_cur, sc_next, scr, tmax, tmap, stream, band);
  if (P.riemann_solver == 1)
    return ctu_step_fused_hllc(precision, P, Uin, Uout, sc_cur, sc_next, scr, tmax, tmap, stream, band);
  if (precision == 0)
    return ctu_step_fused_f64(P, (const double*)Uin, (double*)Uout, sc_cur, sc_next, scr, tmax, stream, band);
  const float* in = (const float*)Uin;
  float* out = (float*)Uout;
  StripShape sh;
  const cudaError_t e = choose_strips(P, &sh, mlp != nullptr);
  if (e != cudaSuccess) return e;
  if (mlp != nullptr) {
    if (sh.nh && learned_work) {
      const cudaError_t el = launch_march_step_fused<FACE_LEARNED>(sh, P, in, out, sc_cur, sc_next, scr, tmax, stream,
                                                                   band, mlp, learned_work);
      if (el != cudaSuccess) return el;
      return launch_learned_tiles<true>(P, in, out, StepScalars{}, sc_cur, sc_next, scr, tmax, tmap, stream, band, mlp,
                                        learned_work);
    }
    // 320 threads (64 registers at 3 CTAs per SM): at 384 threads (56 registers) the gate test in the face
    // loops, together with the pass over the queued faces, makes the allocator spill inside the loops
    return launch_ctu_step_fused_f32<FACE_LEARNED, 320>(P, in, out, sc_cur, sc_next, scr, tmax, tmap, stream, band, mlp);
  }
  if (sh.nh) return launch_march_step_fused<FACE_PLAIN>(sh, P, in, out, sc_cur, sc_next, scr, tmax, stream, band);
  return launch_ctu_step_fused_f32<FACE_PLAIN>(P, in, out, sc_cur, sc_next, scr, tmax, tmap, stream, band);
}

int fused_tile_height(int precision) { return precision == 0 ? F64_TY : F32_TY; }

int fused_tile_rows(int precision, const KParams& P) {
  const int th = fused_tile_height(precision);
  return (P.ny + th - 1) / th;
}

cudaError_t ctu_step(int precision, const KParams& P, const void* Uin, void* Uout, const StepScalars& sc_host,
                     const StepScalars* sc_dev, DevScratch* scr, cudaStream_t stream, int mode, const FaceHook* hook,
                     const CUtensorMap* tmap) {
  if (P.reconstruction == 1) return ctu_step_ppm(precision, P, Uin, Uout, sc_host, sc_dev, scr, stream, tmap);
  if (P.riemann_solver == 1) return ctu_step_hllc(precision, P, Uin, Uout, sc_host, sc_dev, scr, stream, tmap);
  if (precision == 0) return ctu_step_f64(P, (const double*)Uin, (double*)Uout, sc_host, sc_dev, scr, stream);
  const FaceHook h = hook ? *hook : FaceHook{};
  const float* in = (const float*)Uin;
  float* out = (float*)Uout;
  StripShape sh{0, 0, 0};
  if (mode != FACE_HARVEST) {  // the harvest samples faces by their place in a tile
    const cudaError_t e = choose_strips(P, &sh, mode == FACE_LEARNED);
    if (e != cudaSuccess) return e;
  }
  if (sh.nh && mode == FACE_LEARNED && h.learned_work) {
    const cudaError_t e = launch_march_step<FACE_LEARNED>(sh, P, in, out, sc_host, sc_dev, scr, stream, h.mlp,
                                                          h.learned_work);
    if (e != cudaSuccess) return e;
    return launch_learned_tiles<false>(P, in, out, sc_host, sc_dev, nullptr, scr, 0.0, tmap, stream, make_int2(0, 0),
                                       h.mlp, h.learned_work);
  }
  if (sh.nh && mode != FACE_LEARNED) return launch_march_step<FACE_PLAIN>(sh, P, in, out, sc_host, sc_dev, scr, stream);
  switch (mode) {
    case FACE_HARVEST:
      return launch_ctu_step<float, F32_TX, F32_TY, F32_NT, FACE_HARVEST>(P, in, out, sc_host, sc_dev, scr, h, tmap,
                                                                           stream);
    case FACE_LEARNED:
      return launch_ctu_step_f32<FACE_LEARNED>(P, in, out, sc_host, sc_dev, scr, h, tmap, stream);
    default:
      return launch_ctu_step_f32<FACE_PLAIN>(P, in, out, sc_host, sc_dev, scr, h, tmap, stream);
  }
}

cudaError_t step_cut(int precision, const KParams& P, bool learned, int cut[3]) {
  StripShape sh{0, 0, 0};
  bool small = false;
  cudaError_t e = precision == 0 ? f64_small_tile(P, &small) : choose_strips(P, &sh, learned);
  if (e == cudaSuccess && precision != 0 && !sh.nh) e = f32_small_tile(P, &small);
  cut[0] = sh.nh > 0;
  cut[1] = sh.nh ? sh.nv : precision == 0 ? F64_TX : small ? F32_SMALL_TX : F32_TX;
  cut[2] = sh.nh ? sh.nh : precision == 0 ? (small ? F64_TY_SMALL : F64_TY) : small ? F32_SMALL_TY : F32_TY;
  return e;
}

size_t learned_work_bytes(const KParams& P) {
  const size_t tx = (P.nx + F32_TX - 1) / F32_TX, ty = (P.ny + F32_TY - 1) / F32_TY;
  return sizeof(unsigned int) * LearnedWork::words(tx, ty);
}

}  // namespace hydro
