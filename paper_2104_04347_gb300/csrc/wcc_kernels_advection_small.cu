// Many half-steps of a small mesh in one launch, advection system.
#define WCC_SYSTEM ::wcc::ADVECTION
#define WCC_KERNELS_PART 4
#include "wcc_kernels.inc"
