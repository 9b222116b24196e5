// The energy kernels on BF16 images.
#include "energy_box.cuh"

namespace tnlm {

bool launch_energy_box_bf16(int d, int M, int nx, int ny, int nz, int np, const uint16_t *a, const uint16_t *f,
                            float h, float *lam, float *t1, float *grad, double *jpart, long long *nblk,
                            cudaStream_t st, cudaError_t *err)
{
    using B = __nv_bfloat16;
    const float c2 = (float)(1.4426950408889634 / (2.0 * (double)h * (double)h));
    return box::launch_energy<B>(d, M, nx, ny, nz, np, reinterpret_cast<const B *>(a), reinterpret_cast<const B *>(f),
                                 c2, lam, t1, grad, jpart, nblk, st, err);
}

}  // namespace tnlm
