// One compiled variant of the whole-pass kernel per object file: FWD_HD, FWD_FAM, FWD_ATT, FWD_ONE, FWD_SHARE (see Spec) come from the
// build, which compiles this file once for each: in parallel, and a variant's code does not depend on the others.
#if FWD_ATT == 0
#define STAIRS_WAIT_SLOW __forceinline__
#endif
#include "../../include/stairs.h"
#include "megakernel.cuh"

#define FWD_NAME3(a, b, c, d, e) forward_##a##_##b##_##c##_##d##_##e
#define FWD_NAME2(a, b, c, d, e) FWD_NAME3(a, b, c, d, e)

namespace stairs {
namespace mk {
const void* FWD_NAME2(FWD_HD, FWD_FAM, FWD_ATT, FWD_ONE, FWD_SHARE)() {
  return (const void*)k_forward<Spec<FWD_HD, FWD_FAM, FWD_ATT, FWD_ONE != 0, FWD_SHARE != 0>>;
}
}  // namespace mk
}  // namespace stairs
