// Variants for short windows (W <= 52): one lane per window.
#include "umi_variants.h"
UMI_DEFINE_VARIANT(1, 8, 4)
UMI_DEFINE_VARIANT(1, 16, 4)
UMI_DEFINE_VARIANT(1, 26, 4)
UMI_DEFINE_VARIANT(1, 32, 3)
UMI_DEFINE_VARIANT(1, 40, 3)
UMI_DEFINE_VARIANT(1, 52, 2)
