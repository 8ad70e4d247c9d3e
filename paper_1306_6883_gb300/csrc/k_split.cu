// FP32 sweeps of the dimensionally split variant and the precision dispatch.
#include "sweep_march.cuh"

namespace hydro {

cudaError_t split_sweep(int precision, const KParams& P, const void* Uin, void* Uout, int dir,
                        const StepScalars& sc_host, const StepScalars* sc_dev, DevScratch* scr, int check_state,
                        StepScalars* sc_next, double tmax, cudaStream_t stream) {
  if (P.reconstruction == 1) return split_sweep_ppm(precision, P, Uin, Uout, dir, sc_host, sc_dev, scr, check_state,
                                                    sc_next, tmax, stream);
  if (precision == 0)
    return split_sweep_f64(P, (const double*)Uin, (double*)Uout, dir, sc_host, sc_dev, scr, check_state, sc_next, tmax, stream);
  const float* in = (const float*)Uin;
  float* out = (float*)Uout;
  if (P.riemann_solver == 1)
    return launch_sweep_f32<FACE_HLLC>(P, in, out, dir, sc_host, sc_dev, scr, check_state, sc_next, tmax, stream);
  return launch_sweep_f32<FACE_PLAIN>(P, in, out, dir, sc_host, sc_dev, scr, check_state, sc_next, tmax, stream);
}

}  // namespace hydro
