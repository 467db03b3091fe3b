// bcm_pcg_res64.cu -- the on-chip PCG (bcm_pcg_res.cuh) on FP64 vectors.
#include "bcm_pcg_res.cuh"

namespace bcm {

cudaError_t launch_pcg_resident64(const Ctx& x, const SolveParams& prm, bool* launched) {
  ResPlan P;
  const cudaError_t e = res_plan<double>(x, &P, launched);
  if (e != cudaSuccess || !*launched) return e;
  if (P.nt == 256) return res_launch<double, 256, 1, 0>(x, prm, P);
#define BCM_RES(GEOv, Mv) \
  if (P.geo == GEOv && P.m == Mv) return res_launch<double, 512, Mv, GEOv>(x, prm, P);
  BCM_RES(0, 1) BCM_RES(0, 2) BCM_RES(0, 4)
  BCM_RES(8, 4) BCM_RES(8, 6)
  BCM_RES(16, 4) BCM_RES(16, 6)
#undef BCM_RES
  return cudaErrorInvalidValue;
}

}  // namespace bcm
