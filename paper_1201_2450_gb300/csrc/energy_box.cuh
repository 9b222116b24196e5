// The TNLM half of the total energy and its gradient with frozen weights
// (see energy.cu for the formulas) on the box-sum machinery of the sweep: the
// same thread layout and separable patch sums.
//   pass 0, output x in phase i, candidates in phase i+1, x's own normaliser:
//     Lambda_i(x) = log2 Z_i(x),
//     T1_i(x) = sum_delta w (f_i(x) - f_{i+1}(x+delta)),
//     J_x = sum_delta w (f_i(x) - f_{i+1}(x+delta))^2 (FP64 block partials);
//   pass 1, output x in phase i, candidates y = x+delta in phase i-1, each
//     weighted by its own normaliser: w = 2^(-t - Lambda_{i-1}(y)) <= 1,
//     grad_i(x) += T1_i(x) + sum w (f_i(x) - f_{i-1}(y)).
// The patch sums are associated by the place of the output in its thread's
// block (y parity, z in its group of 2 or 4), so the distance of a pair in
// pass 1 equals the one behind Lambda to rounding only: w is off by about
// t 2^-24 of itself and w <= 1 holds to that.
// Every pair contributes its own difference f_i(x) - f_j(y), as in the scatter
// form of the gradient, so no term of size f has to cancel against another:
// near a fixed point of Eq. 8 (f close to its weighted means) the gradient is
// small against f and a form such as f (1 + sum w) - sum w f_j would lose the
// digits that matter.
// Bound by the FMA pipe, as the sweep is, with 8 to 16 warps per SM.  z sums shared between neighbouring outputs
// (zsums) serve both passes; pass 0 also runs all columns but the centre one without the reference test.  Measured
// per launch at 10 x 128^3, d = 1, M = 2, FP32: pass 0 2.68 -> 2.30 ms, pass 1 2.31 -> 2.20.
// Each storage type has a translation unit (energy_box*.cu), so that they compile side by side.
#pragma once

#include "box_block.cuh"

namespace tnlm {
namespace box {

template <int D_, int M_, int BZ, int WY_, int WZ_, bool INTERIOR, int PASS>
__device__ __forceinline__ void box_energy(const float2 (&ai)[BZ + 2 * D_][(2 + 2 * D_) / 2], const float *s_aj,
                                           const float *s_vj, const float *s_nl, const float2 (&fi)[BZ], int lane,
                                           int wy, int wz, int x, int yb, int zb, int nx, int ny, int nz, float c2,
                                           float2 (&o1)[BZ], float2 (&o2)[BZ], float2 (&o3)[BZ])
{
    constexpr int BY = 2;
    using C = BoxCfg<D_, M_, BY, BZ, WY_, WZ_>;
    constexpr int SP = C::SY / 2;
    float2 mref[BZ], N[BZ], Z[BZ], Q[BZ];
#pragma unroll
    for (int k = 0; k < BZ; ++k) {
        mref[k] = make_float2(FLT_MAX, FLT_MAX);
        N[k] = Z[k] = Q[k] = make_float2(0.f, 0.f);
    }
    const float2 nc2 = make_float2(-c2, -c2);
    auto column = [&](int dy, int dx, auto check_tag) {
        constexpr bool CHECK = decltype(check_tag)::value;
        const bool vy0 = INTERIOR || (unsigned)(yb + dy) < (unsigned)ny;
        const bool vy1 = INTERIOR || (unsigned)(yb + 1 + dy) < (unsigned)ny;
        {
            const bool vx = INTERIOR || (unsigned)(x + dx) < (unsigned)nx;
            const bool vxy0 = vx && vy0, vxy1 = vx && vy1;
            const float *paj = s_aj + (wy * BY + dy + M_) * C::AJX + lane + dx + M_;
            const int vo = (wy * BY + dy + M_) * C::VJX + lane + dx + M_;
            float2 aw[2 * M_ + C::SZ][SP];
            float2 vw[2 * M_ + BZ], lw[2 * M_ + BZ];
#pragma unroll
            for (int r = 0; r < C::SZ - 1; ++r)
#pragma unroll
                for (int p = 0; p < SP; ++p) {
                    const float *q0 = paj + ((wz * BZ + r) * C::AJY + 2 * p) * C::AJX;
                    aw[r][p] = make_float2(q0[0], q0[C::AJX]);
                }
#pragma unroll
            for (int r = 0; r < BZ - 1; ++r) {
                const int o = vo + (wz * BZ + r) * C::VJY * C::VJX;
                vw[r] = make_float2(s_vj[o], s_vj[o + C::VJX]);
                if (PASS == 1) lw[r] = make_float2(s_nl[o], s_nl[o + C::VJX]);
            }
#pragma unroll
            for (int q = 0; q <= 2 * M_; ++q) {  // q = dz + M
                {
                    const int r = q + C::SZ - 1;
#pragma unroll
                    for (int p = 0; p < SP; ++p) {
                        const float *q0 = paj + ((wz * BZ + r) * C::AJY + 2 * p) * C::AJX;
                        aw[r][p] = make_float2(q0[0], q0[C::AJX]);
                    }
                    const int rv = q + BZ - 1;
                    const int o = vo + (wz * BZ + rv) * C::VJY * C::VJX;
                    vw[rv] = make_float2(s_vj[o], s_vj[o + C::VJX]);
                    if (PASS == 1) lw[rv] = make_float2(s_nl[o], s_nl[o + C::VJX]);
                }
                float2 bz[BZ][SP];
#pragma unroll
                for (int p = 0; p < SP; ++p) {
                    float2 t[C::SZ];
#pragma unroll
                    for (int zz = 0; zz < C::SZ; ++zz)
                        t[zz] = __fadd2_rn(ai[zz][p], make_float2(-aw[q + zz][p].x, -aw[q + zz][p].y));
                    zsums<D_, BZ, C::SZ, SP>(t, bz, p);
                }
#pragma unroll
                for (int k = 0; k < BZ; ++k) {
                    float m = bz[k][0].y;
#pragma unroll
                    for (int yy = 2; yy <= 2 * D_; ++yy) m += (yy & 1) ? bz[k][yy / 2].y : bz[k][yy / 2].x;
                    const float2 yb2 = make_float2(bz[k][0].x + m, m + bz[k][SP - 1].y);
                    const float2 Dv = xbox2<D_>(yb2);
                    const bool vz = INTERIOR || (unsigned)(zb + k + q - M_) < (unsigned)nz;
                    if (PASS == 0) {
                        float2 a = CHECK ? __ffma2_rn(Dv, nc2, mref[k]) : __fmul2_rn(Dv, nc2);
                        if (!INTERIOR) {
                            if (!(vxy0 && vz)) a.x = -FLT_MAX;
                            if (!(vxy1 && vz)) a.y = -FLT_MAX;
                        }
                        if (CHECK && fmaxf(a.x, a.y) > kRescale) {
                            if (a.x > kRescale) {
                                const float sc = ex2(-a.x);
                                N[k].x *= sc;
                                Z[k].x *= sc;
                                Q[k].x *= sc;
                                mref[k].x = Dv.x * c2;
                                a.x = 0.f;
                            }
                            if (a.y > kRescale) {
                                const float sc = ex2(-a.y);
                                N[k].y *= sc;
                                Z[k].y *= sc;
                                Q[k].y *= sc;
                                mref[k].y = Dv.y * c2;
                                a.y = 0.f;
                            }
                        }
                        const float2 e = make_float2(ex2(a.x), ex2(a.y));
                        const float2 v = vw[q + k];
                        const float2 df = __fadd2_rn(fi[k], make_float2(-v.x, -v.y));
                        N[k] = __ffma2_rn(e, df, N[k]);
                        Z[k] = __fadd2_rn(Z[k], e);
                        Q[k] = __ffma2_rn(e, __fmul2_rn(df, df), Q[k]);
                    } else {
                        // weight of the candidate's own normalisation: 2^(-t - Lambda(y)) <= 1
                        float2 a = __ffma2_rn(Dv, nc2, lw[q + k]);
                        if (!INTERIOR) {
                            if (!(vxy0 && vz)) a.x = -FLT_MAX;
                            if (!(vxy1 && vz)) a.y = -FLT_MAX;
                        }
                        const float2 e = make_float2(ex2(a.x), ex2(a.y));
                        const float2 v = vw[q + k];
                        N[k] = __ffma2_rn(e, __fadd2_rn(fi[k], make_float2(-v.x, -v.y)), N[k]);
                    }
                }
            }
        }
    };
    constexpr int S = 2 * M_ + 1, kCentre = M_ * S + M_;
    if (PASS == 1) {  // the candidates' own normalisers: no running reference
        for (int c = 0; c < S * S; ++c) column(c / S - M_, c % S - M_, std::false_type{});
    } else {
        // the centre column first; then, as in the sweep, each output whose reference is good enough changes to the
        // reference 0, and a warp whose outputs all did runs the others without the test
        for (int it = 0; it < S * S; ++it) {
            const int c = it == 0 ? kCentre : (it - 1 < kCentre ? it - 1 : it);
            column(c / S - M_, c % S - M_, std::true_type{});
            if (it > 0) continue;
            bool ok = true;
            const bool out_x = lane >= D_ && lane < 32 - D_ && x < nx;
#pragma unroll
            for (int k = 0; k < BZ; ++k) {
                if (mref[k].x <= kRescale) {
                    const float sc = ex2(-mref[k].x);
                    N[k].x *= sc, Z[k].x *= sc, Q[k].x *= sc;
                    mref[k].x = 0.f;
                }
                if (mref[k].y <= kRescale) {
                    const float sc = ex2(-mref[k].y);
                    N[k].y *= sc, Z[k].y *= sc, Q[k].y *= sc;
                    mref[k].y = 0.f;
                }
                const bool in = out_x && zb + k < nz;
                ok = ok && (!in || yb >= ny || mref[k].x == 0.f) && (!in || yb + 1 >= ny || mref[k].y == 0.f);
            }
            if (__all_sync(0xffffffffu, ok)) {
                for (int b = 0; b < S * S; ++b)
                    if (b != kCentre) column(b / S - M_, b % S - M_, std::false_type{});
                break;
            }
        }
    }
#pragma unroll
    for (int k = 0; k < BZ; ++k) {
        if (PASS == 0) {
            o1[k] = make_float2(N[k].x / Z[k].x, N[k].y / Z[k].y);
            o2[k] = make_float2(log2f(Z[k].x) - mref[k].x, log2f(Z[k].y) - mref[k].y);
            o3[k] = make_float2(Q[k].x / Z[k].x, Q[k].y / Z[k].y);
        } else {
            o1[k] = N[k];
        }
    }
}

template <int D_, int M_, int BZ, int WY_, int WZ_, class T, int PASS>
__global__ void __launch_bounds__(BoxCfg<D_, M_, 2, BZ, WY_, WZ_>::NT)
    k_energy_box(int nx, int ny, int nz, int np, int ntx, int nty, int ntz, const T *__restrict__ a,
                 const T *__restrict__ f, float *__restrict__ lam, float *__restrict__ t1, float *__restrict__ grad,
                 double *__restrict__ jpart, float *__restrict__ qbar, float c2)
{
    constexpr int BY = 2;
    using C = BoxCfg<D_, M_, BY, BZ, WY_, WZ_>;
    extern __shared__ float sm[];
    float *s_aj = sm;
    float *s_vj = s_aj + C::AJX * C::AJY * C::AJZ;
    float *s_nl = s_vj + C::VJX * C::VJY * C::VJZ;  // pass 1: -Lambda of the neighbour phase
    __shared__ double ws[C::NT / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wy = warp % C::WY, wz = warp / C::WY;
    int b = blockIdx.x;
    const int tx_i = b % ntx;
    b /= ntx;
    const int ty_i = b % nty;
    b /= nty;
    const int tz_i = b % ntz;
    const int i = b / ntz;
    const int X0 = tx_i * C::TXO, Y0 = ty_i * C::TY, Z0 = tz_i * C::TZ;
    const int x = X0 - D_ + lane;
    const int yb = Y0 + wy * BY, zb = Z0 + wz * BZ;
    const long long nvox = (long long)nx * ny * nz;
    const bool interior = X0 - M_ >= 0 && X0 + C::TXO - 1 + M_ < nx && Y0 - M_ >= 0 && Y0 + C::TY - 1 + M_ < ny &&
                          Z0 - M_ >= 0 && Z0 + C::TZ - 1 + M_ < nz;
    const int jp = PASS == 0 ? (i + 1) % np : (i - 1 + np) % np;

    float2 ai[C::SZ][C::SY / 2];
    float2 fi[BZ];
    {
        const T *src = a + i * nvox, *fs = f + i * nvox;
        const int cx = clampi(x, nx);
#pragma unroll
        for (int zz = 0; zz < C::SZ; ++zz)
#pragma unroll
            for (int p = 0; p < C::SY / 2; ++p) {
                const long long zo = (long long)clampi(zb - D_ + zz, nz) * ny;
                ai[zz][p] = make_float2(ld(src + (zo + clampi(yb - D_ + 2 * p, ny)) * nx + cx),
                                        ld(src + (zo + clampi(yb - D_ + 2 * p + 1, ny)) * nx + cx));
            }
#pragma unroll
        for (int k = 0; k < BZ; ++k) {
            const long long zo = (long long)clampi(zb + k, nz) * ny;
            fi[k] = make_float2(ld(fs + (zo + clampi(yb, ny)) * nx + cx), ld(fs + (zo + clampi(yb + 1, ny)) * nx + cx));
        }
    }
    stage_clamped(s_aj, a + jp * nvox, X0 - D_ - M_, Y0 - D_ - M_, Z0 - D_ - M_, C::AJX, C::AJY, C::AJZ, nx, ny, nz,
                  tid, C::NT);
    stage_clamped(s_vj, f + jp * nvox, X0 - D_ - M_, Y0 - M_, Z0 - M_, C::VJX, C::VJY, C::VJZ, nx, ny, nz, tid, C::NT);
    if (PASS == 1) {
        const float *lj = lam + jp * nvox;
        const int ox = X0 - D_ - M_, oy = Y0 - M_, oz = Z0 - M_;
        for (int t = tid; t < C::VJX * C::VJY * C::VJZ; t += C::NT) {
            const int lx = t % C::VJX, ly = (t / C::VJX) % C::VJY, lz = t / (C::VJX * C::VJY);
            s_nl[t] = -__ldg(lj + ((long long)clampi(oz + lz, nz) * ny + clampi(oy + ly, ny)) * nx + clampi(ox + lx, nx));
        }
    }
    __syncthreads();
    float2 o1[BZ], o2[BZ], o3[BZ];
    if (interior)
        box_energy<D_, M_, BZ, WY_, WZ_, true, PASS>(ai, s_aj, s_vj, s_nl, fi, lane, wy, wz, x, yb, zb, nx, ny, nz, c2,
                                                     o1, o2, o3);
    else
        box_energy<D_, M_, BZ, WY_, WZ_, false, PASS>(ai, s_aj, s_vj, s_nl, fi, lane, wy, wz, x, yb, zb, nx, ny, nz, c2,
                                                      o1, o2, o3);
    double jsum = 0.0;
    if (lane >= D_ && lane < 32 - D_ && x < nx) {
#pragma unroll
        for (int j = 0; j < BY; ++j)
#pragma unroll
            for (int k = 0; k < BZ; ++k) {
                const int y = yb + j, z = zb + k;
                if (y < ny && z < nz) {
                    const long long o = i * nvox + ((long long)z * ny + y) * nx + x;
                    const float v1 = j == 0 ? o1[k].x : o1[k].y;
                    if (PASS == 0) {
                        const float v2 = j == 0 ? o2[k].x : o2[k].y, v3 = j == 0 ? o3[k].x : o3[k].y;
                        if (t1) t1[o] = v1;
                        lam[o] = v2;
                        if (qbar) qbar[o] = v3;  // weighted mean of q, for the gradient through the weights
                        jsum += (double)v3;
                    } else {
                        grad[o] += t1[o] + v1;
                    }
                }
            }
    }
    if (PASS == 0 && jpart) {
        for (int off = 16; off > 0; off >>= 1) jsum += __shfl_down_sync(0xffffffffu, jsum, off);
        if (lane == 0) ws[warp] = jsum;
        __syncthreads();
        if (tid == 0) {
            double s = 0.0;
            for (int w = 0; w < C::NT / 32; ++w) s += ws[w];
            jpart[blockIdx.x] = s;
        }
    }
}

template <int D_, int M_, class T>
bool launch_energy_dm(int nx, int ny, int nz, int np, const T *a, const T *f, float c2, float *lam, float *t1,
                      float *grad, double *jpart, long long *nblk, cudaStream_t st, cudaError_t *err)
{
    using S = BoxShape<0>;
    using C = BoxCfg<D_, M_, 2, S::BZ, S::WY, S::WZ>;
    const int ntx = (nx + C::TXO - 1) / C::TXO, nty = (ny + C::TY - 1) / C::TY, ntz = (nz + C::TZ - 1) / C::TZ;
    const long long blocks = (long long)ntx * nty * ntz * np;
    if (blocks > 0x7fffffffLL) return false;
    *nblk = blocks;
    const size_t smem = C::SMEM + sizeof(float) * (size_t)C::VJX * C::VJY * C::VJZ;
    auto k0 = k_energy_box<D_, M_, S::BZ, S::WY, S::WZ, T, 0>;
    auto k1 = k_energy_box<D_, M_, S::BZ, S::WY, S::WZ, T, 1>;
    if ((*err = cudaFuncSetAttribute(k0, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return true;
    if ((*err = cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return true;
    k0<<<(unsigned)blocks, C::NT, smem, st>>>(nx, ny, nz, np, ntx, nty, ntz, a, f, lam, t1, grad, jpart, nullptr, c2);
    if ((*err = cudaGetLastError()) != cudaSuccess) return true;
    k1<<<(unsigned)blocks, C::NT, smem, st>>>(nx, ny, nz, np, ntx, nty, ntz, a, f, lam, t1, grad, jpart, nullptr, c2);
    *err = cudaGetLastError();
    return true;
}

template <class T>
bool launch_energy(int d, int M, int nx, int ny, int nz, int np, const T *a, const T *f, float c2, float *lam,
                   float *t1, float *grad, double *jpart, long long *nblk, cudaStream_t st, cudaError_t *err)
{
#define TNLM_EBOX_CASE(DD, MM)                                                                                      \
    if (d == DD && M == MM) return launch_energy_dm<DD, MM, T>(nx, ny, nz, np, a, f, c2, lam, t1, grad, jpart, nblk, \
                                                                 st, err);
    TNLM_EBOX_CASE(1, 1)
    TNLM_EBOX_CASE(1, 2)
    TNLM_EBOX_CASE(1, 3)
    TNLM_EBOX_CASE(2, 1)
    TNLM_EBOX_CASE(2, 2)
    TNLM_EBOX_CASE(2, 3)
#undef TNLM_EBOX_CASE
    return false;
}

}  // namespace box
}  // namespace tnlm
