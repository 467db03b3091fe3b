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

cudaError_t pcg_resident_fits(const Ctx& x, bool* fits) {
  *fits = false;
  if (x.g.n_sims > kMaxPersistentSims || x.g.n_cubes < 1) return cudaSuccess;
  ResPlan P;
  return x.solve64 ? res_plan<double>(x, &P, fits) : res_plan<float>(x, &P, fits);
}

// The on-chip PCG when the grid allows it (at most kMaxPersistentSims sims, vectors that
// fit); *launched says whether it ran.  A device that refuses the cooperative launch runs
// another form.
cudaError_t launch_pcg_resident(const Ctx& x, const SolveParams& prm, bool* launched) {
  *launched = false;
  if (x.g.n_sims > kMaxPersistentSims || x.g.n_cubes < 1) return cudaSuccess;
  const cudaError_t e = x.solve64 ? launch_pcg_resident64(x, prm, launched) : res32(x, prm, launched);
  if (e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorNotSupported) return e;
  (void)cudaGetLastError();
  *launched = false;
  return cudaSuccess;
}

}  // namespace bcm

extern "C" int bcm_onchip_shape(int cells_per_edge, int n_cubes, int n_sims, int max_level, int fp64,
                                int n_sms, size_t smem_bytes, int32_t* out) {
  using namespace bcm;
  if (!out || n_cubes < 1 || n_sims < 1 || n_sims > n_cubes || n_sms < 1 ||
      (cells_per_edge != 4 && cells_per_edge != 8 && cells_per_edge != 16))
    return 0;
  Ctx x{};
  x.B = cells_per_edge;
  x.g.n_cubes = n_cubes;
  x.g.n_sims = n_sims;
  x.g.max_level = max_level;
  ResPlan P{};
  if (n_sims > kMaxPersistentSims || !(fp64 ? res_shape<double>(x, n_sms, smem_bytes, &P)
                                            : res_shape<float>(x, n_sms, smem_bytes, &P)))
    return 0;
  const int32_t v[6] = {1 << P.sh.lk, P.grid, P.sh.ipb, P.nt, P.m, P.geo};
  for (int i = 0; i < 6; ++i) out[i] = v[i];
  return 1;
}
