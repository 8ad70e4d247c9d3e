// FP64 instantiations of the single-problem CTU step with the HLLC solver.  Compiled with -fmad=false: every
// multiply and add rounds on its own, in source order, like the plain C implementation of the method.
#include "ctu_kernels.cuh"

namespace hydro {

cudaError_t ctu_step_hllc_f64(const KParams& P, const double* Uin, double* Uout, const StepScalars& sc_host,
                              const StepScalars* sc_dev, DevScratch* scr, cudaStream_t stream) {
  return launch_ctu_step_f64<FACE_HLLC>(P, Uin, Uout, sc_host, sc_dev, scr, stream);
}

cudaError_t ctu_step_fused_hllc_f64(const KParams& P, const double* Uin, double* Uout, const StepScalars* sc_cur,
                                    StepScalars* sc_next, DevScratch* scr, double tmax, cudaStream_t stream,
                                    int2 band) {
  return launch_ctu_step_fused_f64<FACE_HLLC>(P, Uin, Uout, sc_cur, sc_next, scr, tmax, stream, band);
}

}  // namespace hydro
