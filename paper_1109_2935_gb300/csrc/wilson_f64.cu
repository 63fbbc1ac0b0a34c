// Wilson-clover stencil instantiations for P64 storage (kernel template in wilson.cuh).
#include "wilson_split.cuh"
#include "internal.h"

namespace dirac {
void launch_wilson_p64(int recon, bool fullm, const WilsonArg& a, cudaStream_t st) {
  if (!launch_wilson_split64(recon, fullm, a, st)) launch_wilson_prec<P64>(recon, fullm, a, st);
}
}  // namespace dirac
