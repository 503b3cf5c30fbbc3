// One group of the persistent kernel's instantiations.  Compiled once per group with
//   SJ_INST_NAME (one of the mega_kernel_* functions), SJ_INST_HD, SJ_INST_TRACE
#include "sj_mega.cuh"

namespace sj {

MegaKernel SJ_INST_NAME(int ns) {
  constexpr bool TR = SJ_INST_TRACE != 0;
  if (ns == 4) return k_verify_mega<SJ_INST_HD, 4, TR>;
  if (ns == 6) return k_verify_mega<SJ_INST_HD, 6, TR>;
  return k_verify_mega<SJ_INST_HD, 8, TR>;
}

}  // namespace sj
