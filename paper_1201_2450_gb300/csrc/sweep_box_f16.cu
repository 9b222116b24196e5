// The box-sum sweep on FP16 images.
#include "sweep_box.cuh"

TNLM_BOX_ENTRY(launch_box_big, kBig, true, __half)
TNLM_BOX_ENTRY(launch_box_small, kSmall, true, __half)
