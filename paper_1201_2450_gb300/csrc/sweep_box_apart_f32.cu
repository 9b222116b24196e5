// The box-sum sweep on FP32 images with values apart from the weights' sources.
#include "sweep_box.cuh"

TNLM_BOX_ENTRY(launch_box_apart_big, kBig, false, float)
TNLM_BOX_ENTRY(launch_box_apart_small, kSmall, false, float)
