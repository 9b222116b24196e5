// The box-sum block of the energy and pair kernels: a thread holds 2 x BZ
// outputs in (y, z) as FP32x2 pairs along y, the lanes span x.
#pragma once

#include "sweep_tile.cuh"

namespace tnlm {
namespace box {

template <class T>
__device__ __forceinline__ void stage_clamped(float *dst, const T *__restrict__ src, int ox, int oy, int oz,
                                              int ex, int ey, int ez, int nx, int ny, int nz, int tid, int nthr)
{
    const int n = ex * ey * ez;
    for (int t = tid; t < n; t += nthr) {
        const int lx = t % ex, ly = (t / ex) % ey, lz = t / (ex * ey);
        const int gx = clampi(ox + lx, nx), gy = clampi(oy + ly, ny), gz = clampi(oz + lz, nz);
        dst[t] = ld(src + ((long long)gz * ny + gy) * nx + gx);
    }
}

// The block: a warp's 32 lanes span x (lanes d .. 31 - d are outputs, the others supply the x halo) and sum along x with
// shuffles; each thread holds BY x BZ outputs in (y, z) and sums along z and y in registers.  The images of the neighbour
// phase are staged in shared memory; the thread's own patch block of phase i stays in registers for all offsets.
template <int D_, int M_, int BY, int BZ, int WY_, int WZ_>
struct BoxCfg {
    static constexpr int WY = WY_, WZ = WZ_;        // warps per CTA along y and z
    static constexpr int NT = 32 * WY * WZ;
    static constexpr int TXO = 32 - 2 * D_;         // outputs per warp row
    static constexpr int TY = WY * BY, TZ = WZ * BZ;
    static constexpr int SY = BY + 2 * D_, SZ = BZ + 2 * D_;
    static constexpr int AJX = 32 + 2 * M_, AJY = TY + 2 * (M_ + D_), AJZ = TZ + 2 * (M_ + D_);
    static constexpr int VJX = 32 + 2 * M_, VJY = TY + 2 * M_, VJZ = TZ + 2 * M_;
    static constexpr size_t SMEM = sizeof(float) * ((size_t)AJX * AJY * AJZ + (size_t)VJX * VJY * VJZ);
};

__device__ __forceinline__ float2 shfl_up2(float2 v, int d)
{
    return make_float2(__shfl_up_sync(0xffffffffu, v.x, d), __shfl_up_sync(0xffffffffu, v.y, d));
}
__device__ __forceinline__ float2 shfl_down2(float2 v, int d)
{
    return make_float2(__shfl_down_sync(0xffffffffu, v.x, d), __shfl_down_sync(0xffffffffu, v.y, d));
}

// x box sum over the warp lanes of a pair of values (two y rows)
template <int D_>
__device__ __forceinline__ float2 xbox2(float2 b)
{
    if constexpr (D_ == 0) {
        return b;
    } else if constexpr (D_ == 1) {
        return __fadd2_rn(__fadd2_rn(shfl_up2(b, 1), b), shfl_down2(b, 1));
    } else if constexpr (D_ == 2) {
        const float2 p = __fadd2_rn(b, shfl_down2(b, 1));  // b(x) + b(x+1)
        return __fadd2_rn(__fadd2_rn(shfl_up2(p, 2), p), shfl_down2(b, 2));
    } else {
        float2 acc = b;
#pragma unroll
        for (int t = 1; t <= D_; ++t) acc = __fadd2_rn(acc, __fadd2_rn(shfl_up2(b, t), shfl_down2(b, t)));
        return acc;
    }
}

// z box sums of BZ = 4 outputs from the differences t of their 4 + 2 D rows, the middle rows shared (sweep_tile.cuh).
template <int D_, int BZ, int SZ, int SP>
__device__ __forceinline__ void zsums(const float2 (&t)[SZ], float2 (&b)[BZ][SP], int p)
{
    static_assert(BZ == 4 && SZ == BZ + 2 * D_, "four outputs");
    if constexpr (D_ == 1) {
#pragma unroll
        for (int k = 0; k < BZ; k += 2) {
            const float2 m = __ffma2_rn(t[k + 2], t[k + 2], __fmul2_rn(t[k + 1], t[k + 1]));
            b[k][p] = __ffma2_rn(t[k], t[k], m);
            b[k + 1][p] = __ffma2_rn(t[k + 3], t[k + 3], m);
        }
    } else {
        const float2 core = __ffma2_rn(t[4], t[4], __fmul2_rn(t[3], t[3]));
        const float2 q1 = __ffma2_rn(t[1], t[1], __ffma2_rn(t[2], t[2], core));
        const float2 q2 = __ffma2_rn(t[6], t[6], __ffma2_rn(t[5], t[5], core));
        b[0][p] = __ffma2_rn(t[0], t[0], q1);
        b[1][p] = __ffma2_rn(t[5], t[5], q1);
        b[2][p] = __ffma2_rn(t[2], t[2], q2);
        b[3][p] = __ffma2_rn(t[7], t[7], q2);
    }
}

// Block shapes: (warps along y, warps along z, output rows per thread along z).
template <int V> struct BoxShape;
template <> struct BoxShape<0> { static constexpr int WY = 4, WZ = 2, BZ = 4; };  // 256 threads, tile 8 x 8
template <> struct BoxShape<2> { static constexpr int WY = 4, WZ = 2, BZ = 2; };  // 256 threads, tile 8 x 4

}  // namespace box
}  // namespace tnlm
