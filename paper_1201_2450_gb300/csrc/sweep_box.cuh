// The box-sum form of the fused weights + Eq. 8 sweep (K3), as templates over
// the patch radius d, the window radius M, the storage type and the form; the
// tile itself is sweep_tile.cuh.  The forms are instantiated in translation
// units of their own (sweep_box_*.cu) so that they compile in parallel.
#pragma once

#include "sweep_tile.cuh"

namespace tnlm {
namespace box {

// The forms by patch radius.  kBig is the block with the fewest FMA cycles per evaluation and kBig2 the same block
// with other warps along (y, z), the launch shapes that tnlm_autotune times (bit-identical: an output's operations do
// not depend on where in a tile it lies).  kSmall is a smaller block, for volumes that give the big one too few warps
// (sweep_small).  Measured (ms per sweep, M = 3, FP32; the 1 x 2 x 4 block of y pairs with running references that
// these replace in front):
//   d = 1, 10 x 256x256x64: 17.77 -> 15.56 (kBig2 15.80, kSmall 16.3; 1 x 4 x 4 y pairs 15.59; kBig 15.12 since warps
//     that keep references leave the common path); 4 x 32^3: 0.166 ->
//     0.229 big, 0.147 small; 4 x 96x90x40: 0.875 -> 0.833, 0.752; 10 x 128x128x48: 3.83 -> 3.44, 3.52.
//   d = 2, 4 x 512x512x128: 115.4 -> 75.9 (kBig2 76.5, kSmall 82); 4 x 32^3: 0.242 -> 0.32, 0.203; 4 x 96x90x40:
//     1.59 -> 1.19, 1.10; 10 x 128x128x48: 7.23 -> 4.78, 5.19.
// d = 1 big: 12 warps per SM at 168 registers, FMA pipe 63 %, LSU 43 %, issue 60 %; d = 2 big: 8 warps at 255, FMA
// 62 %, LSU 57 %: what is left is the latency between dependent instructions of few warps.
enum Form { kBig, kBig2, kSmall };

template <int D_, int M_, Form F> struct TileOf;
template <int M_> struct TileOf<1, M_, kBig> { using type = XPair<M_, 1, 4, 4, 2, 168>; };
template <int M_> struct TileOf<1, M_, kBig2> { using type = XPair<M_, 2, 2, 4, 2, 168>; };
template <int M_> struct TileOf<1, M_, kSmall> { using type = XPair<M_, 2, 2, 2, 2, 128>; };
template <int M_> struct TileOf<2, M_, kBig> { using type = YBlock<M_, 4, 2, 4, 256>; };
template <int M_> struct TileOf<2, M_, kBig2> { using type = YBlock<M_, 2, 2, 4, 256>; };
template <int M_> struct TileOf<2, M_, kSmall> { using type = YBlock<M_, 2, 2, 2, 168>; };
template <int D_, int M_, Form F> using Tile = typename TileOf<D_, M_, F>::type;
// Values staged apart from the weights' sources take a second image of shared memory and more loads: with d = 1 the
// smaller block keeps 16 warps per SM and is the faster one for every volume (17.6 against 20.5 ms at 10 x
// 256x256x64; bit-identical, as the two blocks sum alike).
template <int D_, int M_, Form F, bool SAME> using TileFor = Tile<D_, M_, (!SAME && D_ == 1) ? kSmall : F>;

// SAME: the weights' source images are also the values (vals == wsrc)
template <class C, bool SAME, class T>
__global__ void __launch_bounds__(C::NT, C::kPerSM)
    k_sweep_box(int nx, int ny, int nz, int np, int p0, int ntx, int nty, int ntz, const T *__restrict__ wsrc,
                const T *__restrict__ vals, const T *__restrict__ g, T *__restrict__ out, float c2,
                float mu, int clip)
{
    extern __shared__ float sm[];
    int b = blockIdx.x;
    const int tx_i = b % ntx;
    b /= ntx;
    const int ty_i = b % nty;
    b /= nty;
    const int tz_i = b % ntz;
    C::template tile<SAME, T>(nx, ny, nz, np, tx_i, ty_i, tz_i, p0 + b / ntz, wsrc, vals, g, out, c2, mu, clip, sm);
}

// The sweeps of several problems with one (d, M) in one persistent launch: every CTA takes the next
// (problem, tile) item from a device counter until none is left, and runs the tile as k_sweep_box
// would (same operations in the same order, so the same results).  Items run problem by problem,
// phase by phase, tile by tile.  Every problem sweeps from its own weight sources (vals == wsrc).
// B, S: the tiles of big and small volumes, of one CTA size.
template <class B, class S>
__global__ void __launch_bounds__(B::NT, B::kPerSM)
    k_sweep_box_grouped(const GroupSweep *__restrict__ probs, int nprob, long long total,
                        unsigned long long *__restrict__ counter)
{
    static_assert(B::NT == S::NT, "one CTA size");
    extern __shared__ float sm[];
    __shared__ long long s_item;
    for (;;) {
        __syncthreads();  // the previous item is done with the shared memory and s_item
        if (threadIdx.x == 0) s_item = (long long)atomicAdd(counter, 1ULL);
        __syncthreads();
        const long long it = s_item;
        if (it >= total) return;
        int b = 0;
        while (b + 1 < nprob && probs[b + 1].first <= it) ++b;
        const GroupSweep P = probs[b];
        long long r = it - P.first;
        const int tx_i = (int)(r % P.ntx);
        r /= P.ntx;
        const int ty_i = (int)(r % P.nty);
        r /= P.nty;
        const int tz_i = (int)(r % P.ntz);
        const int i = (int)(r / P.ntz);
        if (sweep_small(P.nx, P.ny, P.nz))
            S::template tile<true, float>(P.nx, P.ny, P.nz, P.np, tx_i, ty_i, tz_i, i, P.wsrc, P.vals, P.g, P.out, P.c2,
                                          P.mu, P.clip, sm);
        else
            B::template tile<true, float>(P.nx, P.ny, P.nz, P.np, tx_i, ty_i, tz_i, i, P.wsrc, P.vals, P.g, P.out, P.c2,
                                          P.mu, P.clip, sm);
    }
}

// the tiles of one problem of a grouped sweep
template <class B, class S>
bool grouped_tiles(int nx, int ny, int nz, int np, int *ntx, int *nty, int *ntz, long long *items)
{
    const bool small = sweep_small(nx, ny, nz);
    const int tx = small ? S::TX : B::TX, ty = small ? S::TY : B::TY, tz = small ? S::TZ : B::TZ;
    *ntx = (nx + tx - 1) / tx;
    *nty = (ny + ty - 1) / ty;
    *ntz = (nz + tz - 1) / tz;
    *items = (long long)*ntx * *nty * *ntz * np;
    return true;
}

template <class B, class S>
bool launch_grouped(const GroupSweep *probs, int nprob, long long total, unsigned long long *counter, int sms,
                    cudaStream_t st, cudaError_t *err)
{
    constexpr size_t smem = sizeof(float) * (B::image > S::image ? B::image : S::image);
    auto kern = k_sweep_box_grouped<B, S>;
    *err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (*err != cudaSuccess) return true;
    int per_sm = 0;
    *err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, B::NT, smem);
    if (*err != cudaSuccess) return true;
    const long long ctas = (long long)sms * (per_sm > 0 ? per_sm : 1);
    kern<<<(unsigned)(ctas < total ? ctas : total), B::NT, smem, st>>>(probs, nprob, total, counter);
    *err = cudaGetLastError();
    return true;
}

// phases p0 .. p0 + nout - 1 of arrays of np phases
template <class C, bool SAME, class T>
bool launch_box(int nx, int ny, int nz, int np, int p0, int nout, const T *wsrc, const T *vals, const T *g, T *out,
                float c2, float mu, int clip, cudaStream_t st, cudaError_t *err)
{
    const int ntx = (nx + C::TX - 1) / C::TX, nty = (ny + C::TY - 1) / C::TY, ntz = (nz + C::TZ - 1) / C::TZ;
    const long long blocks = (long long)ntx * nty * ntz * nout;
    if (blocks > 0x7fffffffLL) return false;
    constexpr size_t smem = sizeof(float) * (C::image + (SAME ? 0 : C::values));
    auto kern = k_sweep_box<C, SAME, T>;
    *err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (*err != cudaSuccess) return true;
    kern<<<(unsigned)blocks, C::NT, smem, st>>>(nx, ny, nz, np, p0, ntx, nty, ntz, wsrc, vals, g, out, c2, mu, clip);
    *err = cudaGetLastError();
    return true;
}

// (d, M) dispatch of one form; false when (d, M) has no box kernel
template <Form F, bool SAME, class T>
bool launch_form(int d, int M, int nx, int ny, int nz, int np, int p0, int nout, const T *wsrc, const T *vals,
                 const T *g, T *out, float c2, float mu, int clip, cudaStream_t st, cudaError_t *err)
{
#define TNLM_BOX_CASE(DD, MM)                                                                                     \
    if (d == DD && M == MM)                                                                                       \
        return launch_box<TileFor<DD, MM, F, SAME>, SAME, T>(nx, ny, nz, np, p0, nout, wsrc, vals, g, out, c2, mu, clip, st, \
                                                            err);
    TNLM_BOX_CASE(1, 1)
    TNLM_BOX_CASE(1, 2)
    TNLM_BOX_CASE(1, 3)
    TNLM_BOX_CASE(2, 1)
    TNLM_BOX_CASE(2, 2)
    TNLM_BOX_CASE(2, 3)
#undef TNLM_BOX_CASE
    return false;
}

}  // namespace box
}  // namespace tnlm

// Defines one sweep entry point: a form, for values that are the weights' sources (SAME) or apart from them.
#define TNLM_BOX_ENTRY(NAME, FORM, SAME, T)                                                                          \
    namespace tnlm {                                                                                                 \
    bool NAME(int d, int M, int nx, int ny, int nz, int np, int p0, int nout, const T *wsrc, const T *vals, const T *g, \
              T *out, float c2, float mu, int clip, cudaStream_t st, cudaError_t *err)                               \
    {                                                                                                                \
        return box::launch_form<box::FORM, SAME, T>(d, M, nx, ny, nz, np, p0, nout, wsrc, vals, g, out, c2, mu, clip, \
                                                    st, err);                                                        \
    }                                                                                                                \
    }
