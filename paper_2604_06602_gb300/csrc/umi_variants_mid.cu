// Variants for windows of 193 to 384 samples (TESS 2-min, 200-s images): the
// autotuner picks among lane-group widths 4 to 32.
#include "umi_variants.h"
UMI_DEFINE_VARIANT(4, 56, 2)
UMI_DEFINE_VARIANT(4, 68, 2)
UMI_DEFINE_VARIANT(8, 40, 2)
UMI_DEFINE_VARIANT(8, 46, 2)
UMI_DEFINE_VARIANT(8, 46, 3)
UMI_DEFINE_VARIANT(8, 48, 2)
UMI_DEFINE_VARIANT(16, 24, 4)
UMI_DEFINE_VARIANT(32, 12, 4)
