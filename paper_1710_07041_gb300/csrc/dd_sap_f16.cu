// Schwarz kernel instances for __half storage (see dd_sap.cu).
#include "dd_sap_run.cuh"

namespace dd {
int sap_run_f16(const SapLattice *L, int nl, const dd_sap_params &p, const RhsPtrs &rp,
                const SapWork *ax, cudaStream_t st) {
  return sap_variants<__half>(L, nl, p, rp, ax, st);
}
}  // namespace dd
