// One tile of the box-sum sweep (K3), by the whole CTA: the weights of Eq. 9
// toward both neighbour phases fused with the Eq. 8 combination.  For a fixed
// window offset delta the patch distance is a separable box sum,
//   D_delta(x) = sum_{o in [-d,d]^3} s_delta(x + o),
//   s_delta(z) = (a_i(clamp z) - a_j(clamp(z + delta)))^2,
// the definition of Eq. 3 / Eq. 9 regrouped (clamping depends on z only).  A
// warp spans x (its outer lanes or outputs are the x halo) and each thread
// holds a block of outputs whose patch block of phase i stays in registers;
// the neighbour phase is staged in shared memory per direction, negated (so
// that a difference is one addition), and slides through registers along dz.
// The z sums start from squares by FMA and share their middle rows between
// outputs: 4 operations for 2 outputs of a 3-row sum, 10 for 4 outputs of a
// 5-row sum.  FP32x2 pairs halve the issue slots; the FMA pipe is what binds,
// so the two forms take the block that needs fewest of its cycles per pair
// evaluation with shuffles and loads (the LSU) below that:
//   XPair, d = 1: 2 (x) x 4 (y) x 2 (z) outputs, pairs along x: 12.0 FMA-pipe
//     cycles and 8.3 LSU cycles per evaluation and warp (the 1 x 2 x 4 block
//     of pairs along y: 15 and 12.9);
//   YBlock, d = 2: 1 x 4 x 4 outputs, pairs along y: 17.3 and 16.
//
// Normalisation is online.  The weights are 2^(m - t), t = D log2(e) / 2h^2,
// against a running reference m that starts at the first candidate and moves
// only when a candidate beats it by 2^kRescale.  The window columns (dy, dx)
// are taken (0, 0) first: every output in the volume then has a reference, and
// an output whose reference is at most kRescale (its best match so far weighs
// at least 2^-kRescale of a perfect one) changes to the reference 0, which no
// candidate can beat (t >= 0).  Each output decides for itself, so results do
// not depend on the tiling; a warp whose outputs all did runs the other
// columns without the test and without the references.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <cfloat>
#include <cmath>
#include <type_traits>

#include "tnlm_internal.cuh"

namespace tnlm {
namespace box {

// lazy-rescale threshold (log2 units): every weight and sum stays below
// 2^kRescale times the candidate count and the normaliser above 2^-kRescale
constexpr float kRescale = 64.f;

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ int clampi(int a, int n) { return a < 0 ? 0 : (a >= n ? n - 1 : a); }

__device__ __forceinline__ float ld(const float *p) { return __ldg(p); }
__device__ __forceinline__ float ld(const __nv_bfloat16 *p) { return __bfloat162float(__ldg(p)); }
__device__ __forceinline__ float ld(const __half *p) { return __half2float(__ldg(p)); }
__device__ __forceinline__ void st(float *p, float v) { *p = v; }
__device__ __forceinline__ void st(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }
__device__ __forceinline__ void st(__half *p, float v) { *p = __float2half_rn(v); }

// One candidate pair against the running references (the general form): lazily rescaled online sums.
__device__ __forceinline__ void add_checked(float2 D, float2 nc2, float c2, bool ok0, bool ok1, float2 v, float2 &mref,
                                            float2 &N, float2 &Z)
{
    float2 a = __ffma2_rn(D, nc2, mref);  // log2 weights vs the references
    if (!ok0) a.x = -FLT_MAX;
    if (!ok1) a.y = -FLT_MAX;
    if (fmaxf(a.x, a.y) > kRescale) {
        if (a.x > kRescale) {  // candidate beats the reference by 2^kRescale: move it
            const float sc = ex2(-a.x);
            N.x *= sc;
            Z.x *= sc;
            mref.x = D.x * c2;
            a.x = 0.f;
        }
        if (a.y > kRescale) {
            const float sc = ex2(-a.y);
            N.y *= sc;
            Z.y *= sc;
            mref.y = D.y * c2;
            a.y = 0.f;
        }
    }
    const float2 e = make_float2(ex2(a.x), ex2(a.y));
    N = __ffma2_rn(e, v, N);
    Z = __fadd2_rn(Z, e);
}

// add_checked without a branch: the same operations, with a scale of 1 where the reference stays.
__device__ __forceinline__ void add_straight(float2 D, float2 nc2, float c2, bool ok0, bool ok1, float2 v, float2 &mref,
                                             float2 &N, float2 &Z)
{
    float2 a = __ffma2_rn(D, nc2, mref);
    if (!ok0) a.x = -FLT_MAX;
    if (!ok1) a.y = -FLT_MAX;
    const bool mx = a.x > kRescale, my = a.y > kRescale;
    const float2 sc = make_float2(mx ? ex2(-a.x) : 1.f, my ? ex2(-a.y) : 1.f);
    const float2 m = __fmul2_rn(D, make_float2(c2, c2));
    N = __fmul2_rn(N, sc);
    Z = __fmul2_rn(Z, sc);
    mref = make_float2(mx ? m.x : mref.x, my ? m.y : mref.y);
    const float2 e = make_float2(mx ? 1.f : ex2(a.x), my ? 1.f : ex2(a.y));
    N = __ffma2_rn(e, v, N);
    Z = __fadd2_rn(Z, e);
}

// After the first column: the reference of an output whose best match is good enough becomes 0.
__device__ __forceinline__ void settle(float &mref, float &N, float &Z)
{
    if (mref <= kRescale) {
        const float sc = ex2(-mref);
        N *= sc;
        Z *= sc;
        mref = 0.f;
    }
}

// d = 1.  Lanes: two rows of 16 along x, 4 outputs in y apart; lane l of a row holds x = X0 - 1 + 2l and the next
// (30 outputs: the first and last of the 32 are the halo).  The staged rows keep even and odd x apart (RS, HO), so
// that a pair at any window offset is two conflict-free loads.
template <int M_, int WY_, int WZ_, int BY_, int BZ_, int REGS>
struct XPair {
    static constexpr int D = 1, M = M_, BY = BY_, BZ = BZ_;
    static constexpr int NT = 32 * WY_ * WZ_;
    static constexpr int TX = 30, TY = WY_ * 2 * BY, TZ = WZ_ * BZ;
    static constexpr int SY = BY + 2, SZ = BZ + 2;
    static constexpr int AX = 32 + 2 * M_, AY = TY + 2 * (M_ + 1), AZ = TZ + 2 * (M_ + 1);
    // BY RS = 16 (mod 32): the two rows of lanes do not clash
    static constexpr int RS = BY == 2 ? 40 : (AX <= 36 ? 36 : 44), HO = RS / 2;
    static constexpr int ROWS = AY * AZ;
    static constexpr int VY = TY + 2 * M_, VZ = TZ + 2 * M_;  // rows of values, where they are staged apart
    static constexpr size_t image = (size_t)RS * ROWS, values = (size_t)RS * VY * VZ;
    static constexpr int kPerSM = 65536 / (NT * REGS) > 0 ? 65536 / (NT * REGS) : 1;

    // rows from (y0, z0) on, NY x NZ of them
    template <int NY, int NZ, class T>
    static __device__ __forceinline__ void stage(float *dst, const T *__restrict__ src, int X0, int y0, int z0, int nx,
                                                 int ny, int nz, int tid)
    {
        for (int t = tid; t < AX * NY * NZ; t += NT) {
            const int lx = t % AX, r = t / AX, ly = r % NY, lz = r / NY;
            const int gx = clampi(X0 - 1 - M_ + lx, nx), gy = clampi(y0 + ly, ny), gz = clampi(z0 + lz, nz);
            dst[r * RS + (lx & 1) * HO + (lx >> 1)] = -ld(src + ((long long)gz * ny + gy) * nx + gx);
        }
    }

    // The sums and references of a thread's outputs, [z][y] pairs along x
    struct State {
        float2 N[BZ][BY], Z[BZ][BY], mref[BZ][BY];
    };

    // One direction: res += N / Z of the thread's outputs, [z][y] pairs along x.  Returns 0, or, for a block of 16 outputs and
    // several columns (APART) and a warp that does not settle, stops after the first column and returns the form (kRest, kRestFar) in which
    // unsettled() is to go on from its state.
    static constexpr bool APART = BY == 4 && M_ > 1;
    enum { kWhole, kRest, kRestFar };
    template <bool SAME, int PART>
    static __device__ __forceinline__ int direction(const float2 (&ai)[SZ][SY], const float *s_a, const float *s_v, int l,
                                                     int ry, int rz, int x, int yb, int zb, int nx, int ny, int nz,
                                                     float c2, bool zin, float2 (&res)[BZ][BY], State &state)
    {
        constexpr int S = 2 * M_ + 1;
        constexpr bool REST = PART != kWhole;
        float2 N[BZ][BY], Z[BZ][BY], mref[BZ][BY];
#pragma unroll
        for (int k = 0; k < BZ; ++k)
#pragma unroll
            for (int j = 0; j < BY; ++j) {
                N[k][j] = REST ? state.N[k][j] : make_float2(0.f, 0.f);
                Z[k][j] = REST ? state.Z[k][j] : make_float2(0.f, 0.f);
                mref[k][j] = REST ? state.mref[k][j] : make_float2(FLT_MAX, FLT_MAX);
            }
        const float2 nc2 = make_float2(-c2, -c2);
        auto column = [&](int dy, int dx, auto check_tag, auto zin_tag) {
            constexpr bool CHECK = decltype(check_tag)::value, ZIN = decltype(zin_tag)::value;
            const int px = dx + M_, odd = px & 1;
            const int row = (rz * AY + ry + dy + M_) * RS;
            const float *p0 = s_a + row + l + (odd ? HO + (px >> 1) : (px >> 1));
            const float *p1 = s_a + row + l + (odd ? (px >> 1) + 1 : HO + (px >> 1));
            const int vrow = (rz * VY + ry + dy + M_) * RS - row;
            const float *v0 = s_v + (p0 - s_a) + vrow, *v1 = s_v + (p1 - s_a) + vrow;
            const bool okx0 = (unsigned)(x + dx) < (unsigned)nx, okx1 = (unsigned)(x + 1 + dx) < (unsigned)nx;
            bool oky[BY];
            float2 bias[BY];  // log2 of the candidates' validity in x and y
#pragma unroll
            for (int j = 0; j < BY; ++j) {
                oky[j] = (unsigned)(yb + j + dy) < (unsigned)ny;
                bias[j] = make_float2(okx0 && oky[j] ? 0.f : -FLT_MAX, okx1 && oky[j] ? 0.f : -FLT_MAX);
            }
            // rows of the neighbour phase along z: a sliding window of SZ
            float2 aw[2 * M_ + SZ][SY], vw[SAME ? 1 : 2 * M_ + BZ][SAME ? 1 : BY];
            auto load_row = [&](int r) {
#pragma unroll
                for (int y = 0; y < SY; ++y) aw[r][y] = make_float2(p0[(r * AY + y) * RS], p1[(r * AY + y) * RS]);
                if constexpr (!SAME) {
                    if (r >= 1 && r <= 2 * M_ + BZ)
#pragma unroll
                        for (int y = 0; y < BY; ++y)
                            vw[r - 1][y] = make_float2(v0[((r - 1) * VY + y) * RS], v1[((r - 1) * VY + y) * RS]);
                }
            };
#pragma unroll
            for (int r = 0; r < SZ - 1; ++r) load_row(r);
#pragma unroll
            for (int q = 0; q < S; ++q) {  // q = dz + M
                load_row(q + SZ - 1);
                float2 b[BZ][SY];
#pragma unroll
                for (int y = 0; y < SY; ++y) {
                    float2 t[SZ];
#pragma unroll
                    for (int z = 0; z < SZ; ++z) t[z] = __fadd2_rn(ai[z][y], aw[q + z][y]);
#pragma unroll
                    for (int k = 0; k < BZ; k += 2) {
                        const float2 m = __ffma2_rn(t[k + 2], t[k + 2], __fmul2_rn(t[k + 1], t[k + 1]));
                        b[k][y] = __ffma2_rn(t[k], t[k], m);
                        b[k + 1][y] = __ffma2_rn(t[k + 3], t[k + 3], m);
                    }
                }
#pragma unroll
                for (int k = 0; k < BZ; ++k) {
                    const bool okz = ZIN || (unsigned)(zb + k + q - M_) < (unsigned)nz;
                    float2 o[BY];
#pragma unroll
                    for (int j = 0; j < BY; j += 2) {
                        const float2 m = __fadd2_rn(b[k][j + 1], b[k][j + 2]);
                        o[j] = __fadd2_rn(b[k][j], m);
                        o[j + 1] = __fadd2_rn(m, b[k][j + 3]);
                    }
#pragma unroll
                    for (int j = 0; j < BY; ++j) {
                        const float s = o[j].x + o[j].y;
                        const float2 Dv = make_float2(__shfl_up_sync(0xffffffffu, o[j].y, 1, 16) + s,
                                                      s + __shfl_down_sync(0xffffffffu, o[j].x, 1, 16));
                        float2 v;
                        if constexpr (SAME) v = aw[q + k + 1][j + 1];
                        else v = vw[q + k][j];
                        if constexpr (CHECK && PART == kRestFar) {
                            add_straight(Dv, nc2, c2, okz && okx0 && oky[j], okz && okx1 && oky[j], v, mref[k][j], N[k][j], Z[k][j]);
                        } else if constexpr (CHECK) {
                            add_checked(Dv, nc2, c2, okz && okx0 && oky[j], okz && okx1 && oky[j], v, mref[k][j], N[k][j], Z[k][j]);
                        } else {
                            const float2 a = __ffma2_rn(Dv, nc2, okz ? bias[j] : make_float2(-FLT_MAX, -FLT_MAX));
                            const float2 e = make_float2(ex2(a.x), ex2(a.y));
                            N[k][j] = __ffma2_rn(e, v, N[k][j]);
                            Z[k][j] = __fadd2_rn(Z[k][j], e);
                        }
                    }
                }
            }
        };
        constexpr int kCentre = M_ * S + M_;
        // the first column, and the others of a warp that did not settle
        for (int it = REST ? 1 : 0; it < S * S; ++it) {
            const int c = it == 0 ? kCentre : (it - 1 < kCentre ? it - 1 : it);
            column(c / S - M_, c % S - M_, std::true_type{}, std::false_type{});
            if (!REST && it == 0) {
                bool ok = true;  // every output of the warp that counts has the reference 0
#pragma unroll
                for (int k = 0; k < BZ; ++k)
#pragma unroll
                    for (int j = 0; j < BY; ++j) {
                        settle(mref[k][j].x, N[k][j].x, Z[k][j].x);
                        settle(mref[k][j].y, N[k][j].y, Z[k][j].y);
                        const bool in = yb + j < ny && zb + k < nz;
                        ok = ok && (!in || l == 0 || x >= nx || mref[k][j].x == 0.f) &&
                             (!in || l == 15 || x + 1 >= nx || mref[k][j].y == 0.f);
                    }
                const bool all = __all_sync(0xffffffffu, ok);
                if (APART && !all) {
                    float far = 0.f;
#pragma unroll
                    for (int k = 0; k < BZ; ++k)
#pragma unroll
                        for (int j = 0; j < BY; ++j) {
                            state.N[k][j] = N[k][j];
                            state.Z[k][j] = Z[k][j];
                            state.mref[k][j] = mref[k][j];
                            far = fmaxf(far, fmaxf(mref[k][j].x, mref[k][j].y));
                        }
                    return __any_sync(0xffffffffu, far > 2.f * kRescale && far < FLT_MAX) ? kRestFar : kRest;
                }
                if (all) {
                    if (zin) {
                        for (int b = 0; b < S * S; ++b)
                            if (b != kCentre) column(b / S - M_, b % S - M_, std::false_type{}, std::true_type{});
                    } else {
                        for (int b = 0; b < S * S; ++b)
                            if (b != kCentre) column(b / S - M_, b % S - M_, std::false_type{}, std::false_type{});
                    }
                    break;
                }
            }
        }
#pragma unroll
        for (int k = 0; k < BZ; ++k)
#pragma unroll
            for (int j = 0; j < BY; ++j) {
                res[k][j].x -= N[k][j].x / Z[k][j].x;  // the values were staged negated
                res[k][j].y -= N[k][j].y / Z[k][j].y;
            }
        return 0;
    }

    // this thread's patch block of phase i (clamped reads), kept for all offsets
    template <class T>
    static __device__ __forceinline__ void patch(float2 (&ai)[SZ][SY], const T *__restrict__ src, int x, int yb, int zb, int nx,
                                                 int ny, int nz)
    {
        const int x0 = clampi(x, nx), x1 = clampi(x + 1, nx);
#pragma unroll
        for (int z = 0; z < SZ; ++z)
#pragma unroll
            for (int y = 0; y < SY; ++y) {
                const T *r = src + ((long long)clampi(zb - 1 + z, nz) * ny + clampi(yb - 1 + y, ny)) * nx;
                ai[z][y] = make_float2(ld(r + x0), ld(r + x1));
            }
    }

    template <class T>
    static __device__ __noinline__ void read_patch(float2 (&ai)[SZ][SY], const T *__restrict__ src, int x, int yb, int zb, int nx,
                                                   int ny, int nz)
    {
        patch(ai, src, x, yb, zb, nx, ny, nz);
    }

    // The rest of a direction of a warp whose outputs did not all settle.  kRestFar, where some reference lies far above
    // what settles: tests without a branch, as some output of the warp moves its reference at nearly every candidate.  Out
    // of line, and with the patch block read again in it and after it, so that the registers of the other warps do not
    // depend on it.  6 x 128x128x48, noise sigma, M = 3 (tests in line / here): sigma = h 3.54 / 3.34 ms, 10 h 3.78 /
    // 3.36; the sweep without unsettled warps at 10 x 256x256x64 15.41 / 15.12 ms.  M = 1: 9 columns do not repay the call.
    template <bool SAME, int PART, class T>
    static __device__ __noinline__ void unsettled(const T *__restrict__ src, const float *s_a, const float *s_v, int l, int ry,
                                                  int rz, int x, int yb, int zb, int nx, int ny, int nz, float c2,
                                                  float2 (&res)[BZ][BY], State &state)
    {
        float2 ai[SZ][SY];
        patch(ai, src, x, yb, zb, nx, ny, nz);
        direction<SAME, PART>(ai, s_a, s_v, l, ry, rz, x, yb, zb, nx, ny, nz, c2, false, res, state);
    }

    template <bool SAME, class T>
    static __device__ __forceinline__ void tile(int nx, int ny, int nz, int np, int tx_i, int ty_i, int tz_i, int i,
                                                const T *__restrict__ wsrc, const T *__restrict__ vals,
                                                const T *__restrict__ g, T *__restrict__ out, float c2, float mu, int clip,
                                                float *sm)
    {
        float *s_a = sm, *s_v = SAME ? sm : sm + image;
        const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, l = lane & 15;
        const int X0 = tx_i * TX, Y0 = ty_i * TY, Z0 = tz_i * TZ;
        const int ry = ((warp % WY_) * 2 + (lane >> 4)) * BY, rz = (warp / WY_) * BZ;
        const int x = X0 - 1 + 2 * l, yb = Y0 + ry, zb = Z0 + rz;
        const long long nvox = (long long)nx * ny * nz;
        const bool zin = Z0 - M_ >= 0 && Z0 + TZ - 1 + M_ < nz;  // every candidate of the tile lies inside in z
        float2 ai[SZ][SY];
        patch(ai, wsrc + i * nvox, x, yb, zb, nx, ny, nz);
        float2 res[BZ][BY];
#pragma unroll
        for (int k = 0; k < BZ; ++k)
#pragma unroll
            for (int j = 0; j < BY; ++j) res[k][j] = make_float2(0.f, 0.f);
        for (int dir = 0; dir < 2; ++dir) {
            const int jp = dir == 0 ? (i + 1) % np : (i - 1 + np) % np;
            __syncthreads();
            stage<AY, AZ>(s_a, wsrc + jp * nvox, X0, Y0 - 1 - M_, Z0 - 1 - M_, nx, ny, nz, tid);
            if constexpr (!SAME) stage<VY, VZ>(s_v, vals + jp * nvox, X0, Y0 - M_, Z0 - M_, nx, ny, nz, tid);
            __syncthreads();
            State state;
            const int rest = direction<SAME, kWhole>(ai, s_a, s_v, l, ry, rz, x, yb, zb, nx, ny, nz, c2, zin, res, state);
            if (APART && rest != 0) {
                const T *src = wsrc + i * nvox;
                if (rest == kRest)
                    unsettled<SAME, kRest>(src, s_a, s_v, l, ry, rz, x, yb, zb, nx, ny, nz, c2, res, state);
                else
                    unsettled<SAME, kRestFar>(src, s_a, s_v, l, ry, rz, x, yb, zb, nx, ny, nz, c2, res, state);
                if (dir == 0) read_patch(ai, src, x, yb, zb, nx, ny, nz);
            }
        }
        const float inv = 1.f / (2.f + mu);
#pragma unroll
        for (int k = 0; k < BZ; ++k)
#pragma unroll
            for (int j = 0; j < BY; ++j)
                if (yb + j < ny && zb + k < nz) {
                    const long long o = i * nvox + ((long long)(zb + k) * ny + yb + j) * nx + x;
                    if (l > 0 && x < nx) {
                        float f = (mu * ld(g + o) + res[k][j].x) * inv;  // Eq. 8
                        if (clip) f = fmaxf(f, 0.f);                     // positivity (TNLM-R step 4)
                        st(out + o, f);
                    }
                    if (l < 15 && x + 1 < nx) {
                        float f = (mu * ld(g + o + 1) + res[k][j].y) * inv;
                        if (clip) f = fmaxf(f, 0.f);
                        st(out + o + 1, f);
                    }
                }
    }
};

// d = 2.  Lanes along x (28 outputs, 2 halo lanes either side), 4 x BZ outputs in (y, z) per thread, pairs along y.
template <int M_, int WY_, int WZ_, int BZ_, int REGS>
struct YBlock {
    static constexpr int D_ = 2, D = D_, M = M_, BY = 4, BZ = BZ_, BP = BY / 2;
    static_assert(BZ == 2 || BZ == 4, "z sums of two or four outputs");
    static constexpr int NT = 32 * WY_ * WZ_;
    static constexpr int TX = 32 - 2 * D_, TY = WY_ * BY, TZ = WZ_ * BZ;
    static constexpr int SP = (BY + 2 * D_) / 2, SZ = BZ + 2 * D_;  // y pairs and z rows of the patch block
    static constexpr int AX = 32 + 2 * M_, AY = TY + 2 * (M_ + D_), AZ = TZ + 2 * (M_ + D_);
    static constexpr int ROWS = AY * AZ;
    static constexpr int VY = TY + 2 * M_, VZ = TZ + 2 * M_;  // rows of values, where they are staged apart
    static constexpr size_t image = (size_t)AX * ROWS, values = (size_t)AX * VY * VZ;
    static constexpr int kPerSM = 65536 / (NT * REGS) > 0 ? 65536 / (NT * REGS) : 1;

    // rows from (y0, z0) on, NY x NZ of them
    template <int NY, int NZ, class T>
    static __device__ __forceinline__ void stage(float *dst, const T *__restrict__ src, int X0, int y0, int z0, int nx,
                                                 int ny, int nz, int tid)
    {
        for (int t = tid; t < AX * NY * NZ; t += NT) {
            const int lx = t % AX, r = t / AX, ly = r % NY, lz = r / NY;
            const int gx = clampi(X0 - D_ - M_ + lx, nx), gy = clampi(y0 + ly, ny), gz = clampi(z0 + lz, nz);
            dst[t] = -ld(src + ((long long)gz * ny + gy) * nx + gx);
        }
    }

    static __device__ __forceinline__ float2 xbox(float2 b)  // sums over x - d .. x + d
    {
        const unsigned F = 0xffffffffu;
        const float2 p = __fadd2_rn(b, make_float2(__shfl_down_sync(F, b.x, 1), __shfl_down_sync(F, b.y, 1)));
        const float2 u = make_float2(__shfl_up_sync(F, p.x, 2), __shfl_up_sync(F, p.y, 2));
        const float2 w = make_float2(__shfl_down_sync(F, b.x, 2), __shfl_down_sync(F, b.y, 2));
        return __fadd2_rn(__fadd2_rn(u, p), w);
    }

    // one direction: res += N / Z of the thread's outputs, [z][pair] pairs along y
    template <bool SAME>
    static __device__ __forceinline__ void direction(const float2 (&ai)[SZ][SP], const float *s_a, const float *s_v,
                                                     int lane, int ry, int rz, int x, int yb, int zb, int nx, int ny,
                                                     int nz, float c2, bool zin, float2 (&res)[BZ][BP])
    {
        constexpr int S = 2 * M_ + 1;
        float2 N[BZ][BP], Z[BZ][BP], mref[BZ][BP];
#pragma unroll
        for (int k = 0; k < BZ; ++k)
#pragma unroll
            for (int h = 0; h < BP; ++h) {
                N[k][h] = Z[k][h] = make_float2(0.f, 0.f);
                mref[k][h] = make_float2(FLT_MAX, FLT_MAX);
            }
        const float2 nc2 = make_float2(-c2, -c2);
        auto column = [&](int dy, int dx, auto check_tag, auto zin_tag) {
            constexpr bool CHECK = decltype(check_tag)::value, ZIN = decltype(zin_tag)::value;
            const float *pa = s_a + (rz * AY + ry + dy + M_) * AX + lane + dx + M_;
            const float *pv = s_v + (rz * VY + ry + dy + M_) * AX + lane + dx + M_;
            const bool okx = (unsigned)(x + dx) < (unsigned)nx;
            bool ok[BY];
            float2 bias[BP];
#pragma unroll
            for (int j = 0; j < BY; ++j) ok[j] = okx && (unsigned)(yb + j + dy) < (unsigned)ny;
#pragma unroll
            for (int h = 0; h < BP; ++h) bias[h] = make_float2(ok[2 * h] ? 0.f : -FLT_MAX, ok[2 * h + 1] ? 0.f : -FLT_MAX);
            float2 aw[2 * M_ + SZ][SP], vw[SAME ? 1 : 2 * M_ + BZ][SAME ? 1 : BP];
            auto load_row = [&](int r) {
#pragma unroll
                for (int p = 0; p < SP; ++p) {
                    const float *q = pa + (r * AY + 2 * p) * AX;
                    aw[r][p] = make_float2(q[0], q[AX]);
                }
                if constexpr (!SAME) {
                    if (r >= D_ && r < 2 * M_ + BZ + D_)
#pragma unroll
                        for (int h = 0; h < BP; ++h) {
                            const float *q = pv + ((r - D_) * VY + 2 * h) * AX;
                            vw[r - D_][h] = make_float2(q[0], q[AX]);
                        }
                }
            };
#pragma unroll
            for (int r = 0; r < SZ - 1; ++r) load_row(r);
#pragma unroll
            for (int q = 0; q < S; ++q) {  // q = dz + M
                load_row(q + SZ - 1);
                float2 b[BZ][SP];
#pragma unroll
                for (int p = 0; p < SP; ++p) {
                    float2 t[SZ];
#pragma unroll
                    for (int z = 0; z < SZ; ++z) t[z] = __fadd2_rn(ai[z][p], aw[q + z][p]);
                    if constexpr (BZ == 2) {
                        const float2 m = __ffma2_rn(t[3], t[3], __fmul2_rn(t[2], t[2]));
                        const float2 q1 = __ffma2_rn(t[1], t[1], __ffma2_rn(t[4], t[4], m));
                        b[0][p] = __ffma2_rn(t[0], t[0], q1);
                        b[1][p] = __ffma2_rn(t[5], t[5], q1);
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
#pragma unroll
                for (int k = 0; k < BZ; ++k) {
                    const bool okz = ZIN || (unsigned)(zb + k + q - M_) < (unsigned)nz;
                    const float core = b[k][1].y + b[k][2].x;
                    const float q1 = core + (b[k][0].y + b[k][1].x), q2 = core + (b[k][2].y + b[k][3].x);
                    const float2 o[BP] = {make_float2(b[k][0].x + q1, q1 + b[k][2].y), make_float2(b[k][1].x + q2, q2 + b[k][3].y)};
#pragma unroll
                    for (int h = 0; h < BP; ++h) {
                        const float2 Dv = xbox(o[h]);
                        float2 v;
                        if constexpr (SAME) v = aw[q + k + 2][h + 1];
                        else v = vw[q + k][h];
                        if constexpr (CHECK) {
                            add_checked(Dv, nc2, c2, okz && ok[2 * h], okz && ok[2 * h + 1], v, mref[k][h], N[k][h], Z[k][h]);
                        } else {
                            const float2 a = __ffma2_rn(Dv, nc2, okz ? bias[h] : make_float2(-FLT_MAX, -FLT_MAX));
                            const float2 e = make_float2(ex2(a.x), ex2(a.y));
                            N[k][h] = __ffma2_rn(e, v, N[k][h]);
                            Z[k][h] = __fadd2_rn(Z[k][h], e);
                        }
                    }
                }
            }
        };
        constexpr int kCentre = M_ * S + M_;
        for (int it = 0; it < S * S; ++it) {  // the first column, and the others of a warp that did not settle
            const int c = it == 0 ? kCentre : (it - 1 < kCentre ? it - 1 : it);
            column(c / S - M_, c % S - M_, std::true_type{}, std::false_type{});
            if (it == 0) {
                const bool out_x = lane >= D_ && lane < 32 - D_ && x < nx;
                bool ok = true;
#pragma unroll
                for (int k = 0; k < BZ; ++k)
#pragma unroll
                    for (int h = 0; h < BP; ++h) {
                        settle(mref[k][h].x, N[k][h].x, Z[k][h].x);
                        settle(mref[k][h].y, N[k][h].y, Z[k][h].y);
                        const bool in = out_x && zb + k < nz;
                        ok = ok && (!in || yb + 2 * h >= ny || mref[k][h].x == 0.f) &&
                             (!in || yb + 2 * h + 1 >= ny || mref[k][h].y == 0.f);
                    }
                if (__all_sync(0xffffffffu, ok)) {
                    if (zin) {
                        for (int b = 0; b < S * S; ++b)
                            if (b != kCentre) column(b / S - M_, b % S - M_, std::false_type{}, std::true_type{});
                    } else {
                        for (int b = 0; b < S * S; ++b)
                            if (b != kCentre) column(b / S - M_, b % S - M_, std::false_type{}, std::false_type{});
                    }
                    break;
                }
            }
        }
#pragma unroll
        for (int k = 0; k < BZ; ++k)
#pragma unroll
            for (int h = 0; h < BP; ++h) {
                res[k][h].x -= N[k][h].x / Z[k][h].x;  // the values were staged negated
                res[k][h].y -= N[k][h].y / Z[k][h].y;
            }
    }

    template <bool SAME, class T>
    static __device__ __forceinline__ void tile(int nx, int ny, int nz, int np, int tx_i, int ty_i, int tz_i, int i,
                                                const T *__restrict__ wsrc, const T *__restrict__ vals,
                                                const T *__restrict__ g, T *__restrict__ out, float c2, float mu, int clip,
                                                float *sm)
    {
        float *s_a = sm, *s_v = SAME ? sm : sm + image;
        const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
        const int X0 = tx_i * TX, Y0 = ty_i * TY, Z0 = tz_i * TZ;
        const int ry = (warp % WY_) * BY, rz = (warp / WY_) * BZ;
        const int x = X0 - D_ + lane, yb = Y0 + ry, zb = Z0 + rz;
        const long long nvox = (long long)nx * ny * nz;
        const bool zin = Z0 - M_ >= 0 && Z0 + TZ - 1 + M_ < nz;
        float2 ai[SZ][SP];
        {
            const T *src = wsrc + i * nvox;
            const int cx = clampi(x, nx);
#pragma unroll
            for (int z = 0; z < SZ; ++z)
#pragma unroll
                for (int p = 0; p < SP; ++p) {
                    const long long zo = (long long)clampi(zb - D_ + z, nz) * ny;
                    ai[z][p] = make_float2(ld(src + (zo + clampi(yb - D_ + 2 * p, ny)) * nx + cx),
                                           ld(src + (zo + clampi(yb - D_ + 2 * p + 1, ny)) * nx + cx));
                }
        }
        float2 res[BZ][BP];
#pragma unroll
        for (int k = 0; k < BZ; ++k)
#pragma unroll
            for (int h = 0; h < BP; ++h) res[k][h] = make_float2(0.f, 0.f);
        for (int dir = 0; dir < 2; ++dir) {
            const int jp = dir == 0 ? (i + 1) % np : (i - 1 + np) % np;
            __syncthreads();
            stage<AY, AZ>(s_a, wsrc + jp * nvox, X0, Y0 - D_ - M_, Z0 - D_ - M_, nx, ny, nz, tid);
            if constexpr (!SAME) stage<VY, VZ>(s_v, vals + jp * nvox, X0, Y0 - M_, Z0 - M_, nx, ny, nz, tid);
            __syncthreads();
            direction<SAME>(ai, s_a, s_v, lane, ry, rz, x, yb, zb, nx, ny, nz, c2, zin, res);
        }
        if (lane < D_ || lane >= 32 - D_ || x >= nx) return;
        const float inv = 1.f / (2.f + mu);
#pragma unroll
        for (int k = 0; k < BZ; ++k)
#pragma unroll
            for (int j = 0; j < BY; ++j)
                if (yb + j < ny && zb + k < nz) {
                    const long long o = i * nvox + ((long long)(zb + k) * ny + yb + j) * nx + x;
                    const float r = (j & 1) ? res[k][j / 2].y : res[k][j / 2].x;
                    float f = (mu * ld(g + o) + r) * inv;  // Eq. 8
                    if (clip) f = fmaxf(f, 0.f);           // positivity (TNLM-R step 4)
                    st(out + o, f);
                }
    }
};

}  // namespace box
}  // namespace tnlm
