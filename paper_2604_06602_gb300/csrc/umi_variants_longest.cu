// Variants for the longest windows (W up to 4096).
#include "umi_variants.h"
UMI_DEFINE_VARIANT(32, 92, 1)
UMI_DEFINE_VARIANT(32, 112, 1)
UMI_DEFINE_VARIANT(32, 128, 1)
