// Many half-steps of a small mesh in one launch, burgers system.
#define WCC_SYSTEM ::wcc::BURGERS
#define WCC_KERNELS_PART 4
#include "wcc_kernels.inc"
