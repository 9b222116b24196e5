// The box-sum sweep on BF16 images with values apart from the weights' sources.
#include "sweep_box.cuh"

TNLM_BOX_ENTRY(launch_box_apart_big, kBig, false, __nv_bfloat16)
TNLM_BOX_ENTRY(launch_box_apart_small, kSmall, false, __nv_bfloat16)
