// The box-sum sweep on BF16 images.
#include "sweep_box.cuh"

TNLM_BOX_ENTRY(launch_box_big, kBig, true, __nv_bfloat16)
TNLM_BOX_ENTRY(launch_box_small, kSmall, true, __nv_bfloat16)
