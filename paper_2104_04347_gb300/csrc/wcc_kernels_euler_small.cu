// Many half-steps of a small mesh in one launch, euler system.
#define WCC_SYSTEM ::wcc::EULER
#define WCC_KERNELS_PART 4
#include "wcc_kernels.inc"
