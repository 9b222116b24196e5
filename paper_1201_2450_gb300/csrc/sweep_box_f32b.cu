// The second launch shape of the box-sum sweep on FP32 images, and the grouped sweep.
#include "sweep_box.cuh"

TNLM_BOX_ENTRY(launch_box_big2, kBig2, true, float)

namespace tnlm {

bool launch_box_grouped(int d, int M, const GroupSweep *probs, int nprob, long long total, unsigned long long *counter,
                        int sms, cudaStream_t st, cudaError_t *err)
{
#define TNLM_GROUP_CASE(DD, MM)                                                                                       \
    if (d == DD && M == MM)                                                                                           \
        return box::launch_grouped<box::Tile<DD, MM, box::kBig2>, box::Tile<DD, MM, box::kSmall>>(probs, nprob, total, \
                                                                                                  counter, sms, st, err);
    TNLM_GROUP_CASE(1, 1)
    TNLM_GROUP_CASE(1, 2)
    TNLM_GROUP_CASE(1, 3)
    TNLM_GROUP_CASE(2, 1)
    TNLM_GROUP_CASE(2, 2)
    TNLM_GROUP_CASE(2, 3)
#undef TNLM_GROUP_CASE
    return false;
}

bool box_grouped_tiles(int d, int M, int nx, int ny, int nz, int np, int *ntx, int *nty, int *ntz, long long *items)
{
#define TNLM_GTILE_CASE(DD, MM)                                                                                      \
    if (d == DD && M == MM)                                                                                          \
        return box::grouped_tiles<box::Tile<DD, MM, box::kBig2>, box::Tile<DD, MM, box::kSmall>>(nx, ny, nz, np, ntx, \
                                                                                                 nty, ntz, items);
    TNLM_GTILE_CASE(1, 1)
    TNLM_GTILE_CASE(1, 2)
    TNLM_GTILE_CASE(1, 3)
    TNLM_GTILE_CASE(2, 1)
    TNLM_GTILE_CASE(2, 2)
    TNLM_GTILE_CASE(2, 3)
#undef TNLM_GTILE_CASE
    return false;
}

}  // namespace tnlm
