// The box-sum sweep on FP32 images.
#include "sweep_box.cuh"

TNLM_BOX_ENTRY(launch_box_big, kBig, true, float)
TNLM_BOX_ENTRY(launch_box_small, kSmall, true, float)
