// bcm_pcg_res32.cu -- the on-chip PCG (bcm_pcg_res.cuh) on FP32 vectors, the inner solve of
// the mixed precisions, and the form's entry point.
#include "bcm_pcg_res.cuh"

namespace bcm {

size_t res_words_bytes(int n_sims) {
  return sizeof(WordLine) * 3 * (size_t)(kResBlocks + n_sims);
}

static cudaError_t res32(const Ctx& x, const SolveParams& prm, bool* launched) {
  ResPlan P;
  const cudaError_t e = res_plan<float>(x, &P, launched);
  if (e != cudaSuccess || !*launched) return e;
  if (P.nt == 256) return res_launch<float, 256, 1, 0>(x, prm, P);
#define BCM_RES(GEOv, Mv) \
  if (P.geo == GEOv && P.m == Mv) return res_launch<float, 512, Mv, GEOv>(x, prm, P);
  BCM_RES(0, 1) BCM_RES(0, 2) BCM_RES(0, 4) BCM_RES(0, 8)
  BCM_RES(8, 4) BCM_RES(8, 8) BCM_RES(8, 14)
  BCM_RES(16, 4) BCM_RES(16, 8) BCM_RES(16, 14)
#undef BCM_RES
  return cudaErrorInvalidValue;
}

// The on-chip PCG when the grid allows it (at most kMaxPersistentSims sims, vectors that
// fit); *launched says whether it ran.
cudaError_t launch_pcg_resident(const Ctx& x, const SolveParams& prm, bool* launched) {
  *launched = false;
  if (x.g.n_sims > kMaxPersistentSims || x.g.n_cubes < 1) return cudaSuccess;
  return x.solve64 ? launch_pcg_resident64(x, prm, launched) : res32(x, prm, launched);
}

}  // namespace bcm
