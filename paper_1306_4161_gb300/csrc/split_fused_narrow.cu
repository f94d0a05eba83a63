// The product kernel that recombines (split_fused.cuh) with tiles of 64 columns.
#include "internal.h"

namespace hs {
namespace {
constexpr int TN = 64;
}
}  // namespace hs
#include "split_fused.cuh"

namespace hs {

int launch_fused_narrow(int w, int S, const CUtensorMap &tA, const CUtensorMap &tB, FusedParams &p,
                        int nbands, cudaStream_t s) {
  return launch_fused_kernel(w, S, tA, tB, p, nbands, s);
}

}  // namespace hs
