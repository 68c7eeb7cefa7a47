// Variants for windows of 1089 to 2176 samples (20-s cadence).
#include "umi_variants.h"
UMI_DEFINE_VARIANT(32, 48, 2)
UMI_DEFINE_VARIANT(32, 56, 2)
UMI_DEFINE_VARIANT(32, 68, 2)
