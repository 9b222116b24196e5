// The Eq. 8 sweep with the symmetric reuse of patch distances (Sec. 2.4): the
// distance between the patch of x in phase i and the patch of x + delta in
// phase i+1 is also the distance that the output x + delta of phase i+1
// needs for its candidate x in phase i (window offset -delta).  Per phase
// pair (i, i+1):
//   pass A (k_sweep_box_pa): the weights of phase i toward i+1 as in the
//     box-sum sweep, their normalised sum N/Z written to the output as a
//     partial result, and every patch distance written to a buffer G,
//     delta-major ([(2M+1)^3][voxel]);
//   pass B (k_pair_b): phase i+1 toward i from G -- only the exponentials
//     and sums, with the same online normalisation -- added to the partial
//     result of phase i+1, then the Eq. 8 combination and positivity.
// Two G buffers alternate around the ring of phases, so pass A of pair
// (i, i+1) can run while G of (i-1, i) is still to be read.  The distances
// read back are bitwise those pass A summed, up to the association of the
// y box sum (it depends on the row parity of the output within a thread's
// pair of rows), so the result agrees with the direct sweep to rounding.
#include "box_block.cuh"

namespace tnlm {
namespace box {

// One direction of the sweep for this thread's 2 x BZ outputs (y rows j = 0, 1
// are processed as FP32x2 pairs).  ai holds the thread's patch block of phase
// i as [z][y pair]; res accumulates N/Z per output.
// The window offsets are taken column by column, (dy, dx) = (0, 0) first and
// then the others in row-major order, dz ascending within a column.  The
// running reference of the online normalisation (mref = c2 D of the reference
// candidate, log2 units) moves only when a candidate beats it by more than
// 2^kRescale.  A candidate's log2 weight against the reference is
// a = mref - c2 D <= mref (D >= 0), so once every output of a warp has
// mref <= kRescale no later candidate can move it: after the first column the
// warp votes, and a warp that passed skips the test for the remaining
// columns (the same operations on every output otherwise, so the result does
// not depend on the vote).
// STORE: also write every patch distance of the thread's outputs to Gd[delta][voxel] (delta-major, delta =
// ((dz + M) S + dy + M) S + dx + M), for the phase-pair form of the sweep (k_pair_b reads them back).
template <int D_, int M_, int BZ, int WY_, int WZ_, bool INTERIOR, bool STORE = false>
__device__ __forceinline__ void box_direction(const float2 (&ai)[BZ + 2 * D_][(2 + 2 * D_) / 2], const float *s_aj,
                                              const float *s_vj, int lane, int wy, int wz, int x, int yb, int zb,
                                              int nx, int ny, int nz, float c2, float2 (&res)[BZ],
                                              float *__restrict__ Gd = nullptr, bool st0 = false, bool st1 = false)
{
    constexpr int BY = 2;
    using C = BoxCfg<D_, M_, BY, BZ, WY_, WZ_>;
    constexpr int SP = C::SY / 2;  // y pairs of the patch block
    constexpr int S = 2 * M_ + 1;
    float2 mref[BZ], N[BZ], Z[BZ];
#pragma unroll
    for (int k = 0; k < BZ; ++k) {
        mref[k] = make_float2(FLT_MAX, FLT_MAX);
        N[k] = make_float2(0.f, 0.f);
        Z[k] = make_float2(0.f, 0.f);
    }
    const float2 nc2 = make_float2(-c2, -c2);
    // the candidates of window column (dy, dx), dz = -M .. M
    auto column = [&](int dy, int dx, auto check_tag) {
        constexpr bool CHECK = decltype(check_tag)::value;
        const bool vy0 = INTERIOR || (unsigned)(yb + dy) < (unsigned)ny;
        const bool vy1 = INTERIOR || (unsigned)(yb + 1 + dy) < (unsigned)ny;
        const bool vx = INTERIOR || (unsigned)(x + dx) < (unsigned)nx;
        const bool vxy0 = vx && vy0, vxy1 = vx && vy1;
        const float *paj = s_aj + (wy * BY + dy + M_) * C::AJX + lane + dx + M_;
        const float *pvj = s_vj + (wy * BY + dy + M_) * C::VJX + lane + dx + M_;
        // neighbour-phase rows along z, a sliding window of SZ rows of y pairs
        float2 aw[2 * M_ + C::SZ][SP];
        float2 vw[2 * M_ + BZ];
#pragma unroll
        for (int r = 0; r < C::SZ - 1; ++r)
#pragma unroll
            for (int p = 0; p < SP; ++p) {
                const float *q0 = paj + ((wz * BZ + r) * C::AJY + 2 * p) * C::AJX;
                aw[r][p] = make_float2(q0[0], q0[C::AJX]);
            }
#pragma unroll
        for (int r = 0; r < BZ - 1; ++r) {
            const float *q0 = pvj + (wz * BZ + r) * C::VJY * C::VJX;
            vw[r] = make_float2(q0[0], q0[C::VJX]);
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
                const float *q1 = pvj + (wz * BZ + rv) * C::VJY * C::VJX;
                vw[rv] = make_float2(q1[0], q1[C::VJX]);
            }
            // squared differences and z box sums, per y pair
            float2 bz[BZ][SP];
#pragma unroll
            for (int p = 0; p < SP; ++p) {
                float2 sq[C::SZ];
#pragma unroll
                for (int zz = 0; zz < C::SZ; ++zz) {
                    const float2 t = __fadd2_rn(ai[zz][p], make_float2(-aw[q + zz][p].x, -aw[q + zz][p].y));
                    sq[zz] = __fmul2_rn(t, t);
                }
#pragma unroll
                for (int k = 0; k < BZ; ++k) {
                    float2 acc = sq[k];
#pragma unroll
                    for (int t = 1; t <= 2 * D_; ++t) acc = __fadd2_rn(acc, sq[k + t]);
                    bz[k][p] = acc;
                }
            }
#pragma unroll
            for (int k = 0; k < BZ; ++k) {
                // y box sums of the two output rows: row 0 sums y 0..2d, row 1 sums y 1..2d+1,
                // both direct sums sharing the middle rows m = y 1..2d
                float m = bz[k][0].y;
#pragma unroll
                for (int yy = 2; yy <= 2 * D_; ++yy) m += (yy & 1) ? bz[k][yy / 2].y : bz[k][yy / 2].x;
                const float2 yb2 = make_float2(bz[k][0].x + m, m + bz[k][SP - 1].y);
                const float2 Dv = xbox2<D_>(yb2);  // patch distances of outputs (0,k) and (1,k)
                if constexpr (STORE) {
                    const long long nvox = (long long)nx * ny * nz;
                    const int z = zb + k;
                    if (z < nz) {
                        float *gp = Gd + (long long)((q * S + dy + M_) * S + dx + M_) * nvox +
                                    ((long long)z * ny + yb) * nx + x;
                        if (st0) gp[0] = Dv.x;
                        if (st1) gp[nx] = Dv.y;
                    }
                }
                float2 a = __ffma2_rn(Dv, nc2, mref[k]);  // log2 weights vs the references
                const bool vz = INTERIOR || (unsigned)(zb + k + q - M_) < (unsigned)nz;
                if (!INTERIOR) {
                    if (!(vxy0 && vz)) a.x = -FLT_MAX;
                    if (!(vxy1 && vz)) a.y = -FLT_MAX;
                }
                if (CHECK && fmaxf(a.x, a.y) > kRescale) {  // rare: one test for both outputs of the pair
                    if (a.x > kRescale) {  // candidate beats the reference by 2^kRescale: move it
                        const float sc = ex2(-a.x);
                        N[k].x *= sc;
                        Z[k].x *= sc;
                        mref[k].x = Dv.x * c2;
                        a.x = 0.f;
                    }
                    if (a.y > kRescale) {
                        const float sc = ex2(-a.y);
                        N[k].y *= sc;
                        Z[k].y *= sc;
                        mref[k].y = Dv.y * c2;
                        a.y = 0.f;
                    }
                }
                const float2 e = make_float2(ex2(a.x), ex2(a.y));
                N[k] = __ffma2_rn(e, vw[q + k], N[k]);
                Z[k] = __fadd2_rn(Z[k], e);
            }
        }
    };
    constexpr int kCentre = M_ * S + M_;
    bool settled = false;  // every output of the warp has mref <= kRescale
    for (int it = 0; it < S * S; ++it) {
        const int c = it == 0 ? kCentre : (it - 1 < kCentre ? it - 1 : it);
        const int dy = c / S - M_, dx = c % S - M_;
        if (settled)
            column(dy, dx, std::false_type{});
        else
            column(dy, dx, std::true_type{});
        if (it == 0) {
            // this thread's outputs inside the volume (lanes d .. 31 - d; the others are the x
            // halo): the centre column holds the output itself, so each has a reference by now
            bool ok = true;
            if (lane >= D_ && lane < 32 - D_ && x < nx) {
#pragma unroll
                for (int k = 0; k < BZ; ++k) {
                    if (zb + k < nz) {
                        ok = ok && (yb >= ny || mref[k].x <= kRescale) && (yb + 1 >= ny || mref[k].y <= kRescale);
                    }
                }
            }
            settled = __all_sync(0xffffffffu, ok);
        }
    }
#pragma unroll
    for (int k = 0; k < BZ; ++k) {
        res[k].x += N[k].x / Z[k].x;
        res[k].y += N[k].y / Z[k].y;
    }
}

// Pass A: one direction (toward i+1) of the box-sum sweep for phase i, storing the distances.
template <int D_, int M_, int BY, int BZ, int WY_, int WZ_>
__global__ void __launch_bounds__(BoxCfg<D_, M_, BY, BZ, WY_, WZ_>::NT)
    k_sweep_box_pa(int nx, int ny, int nz, int np, int i, int ntx, int nty, const float *__restrict__ wsrc,
                   const float *__restrict__ vals, float *__restrict__ part, float *__restrict__ G, float c2)
{
    using C = BoxCfg<D_, M_, BY, BZ, WY_, WZ_>;
    extern __shared__ float sm[];
    float *s_aj = sm;
    float *s_vj = sm + C::AJX * C::AJY * C::AJZ;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wy = warp % C::WY, wz = warp / C::WY;
    int b = blockIdx.x;
    const int tx_i = b % ntx;
    b /= ntx;
    const int ty_i = b % nty;
    const int tz_i = b / nty;
    const int X0 = tx_i * C::TXO, Y0 = ty_i * C::TY, Z0 = tz_i * C::TZ;
    const int x = X0 - D_ + lane;
    const int yb = Y0 + wy * BY, zb = Z0 + wz * BZ;
    const long long nvox = (long long)nx * ny * nz;
    const bool interior = X0 - M_ >= 0 && X0 + C::TXO - 1 + M_ < nx && Y0 - M_ >= 0 && Y0 + C::TY - 1 + M_ < ny &&
                          Z0 - M_ >= 0 && Z0 + C::TZ - 1 + M_ < nz;
    float2 ai[C::SZ][C::SY / 2];
    {
        const float *src = wsrc + i * nvox;
        const int cx = clampi(x, nx);
#pragma unroll
        for (int zz = 0; zz < C::SZ; ++zz)
#pragma unroll
            for (int p = 0; p < C::SY / 2; ++p) {
                const long long zo = (long long)clampi(zb - D_ + zz, nz) * ny;
                ai[zz][p] = make_float2(__ldg(src + (zo + clampi(yb - D_ + 2 * p, ny)) * nx + cx),
                                        __ldg(src + (zo + clampi(yb - D_ + 2 * p + 1, ny)) * nx + cx));
            }
    }
    float2 res[BZ];
#pragma unroll
    for (int k = 0; k < BZ; ++k) res[k] = make_float2(0.f, 0.f);
    const int jp = (i + 1) % np;
    stage_clamped(s_aj, wsrc + jp * nvox, X0 - D_ - M_, Y0 - D_ - M_, Z0 - D_ - M_, C::AJX, C::AJY, C::AJZ, nx, ny, nz,
                  tid, C::NT);
    stage_clamped(s_vj, vals + jp * nvox, X0 - D_ - M_, Y0 - M_, Z0 - M_, C::VJX, C::VJY, C::VJZ, nx, ny, nz, tid,
                  C::NT);
    __syncthreads();
    const bool out_x = lane >= D_ && lane < 32 - D_ && x < nx;
    const bool st0 = out_x && yb < ny, st1 = out_x && yb + 1 < ny;
    if (interior)
        box_direction<D_, M_, BZ, WY_, WZ_, true, true>(ai, s_aj, s_vj, lane, wy, wz, x, yb, zb, nx, ny, nz, c2, res, G,
                                                         st0, st1);
    else
        box_direction<D_, M_, BZ, WY_, WZ_, false, true>(ai, s_aj, s_vj, lane, wy, wz, x, yb, zb, nx, ny, nz, c2, res,
                                                          G, st0, st1);
    if (out_x) {
#pragma unroll
        for (int j = 0; j < BY; ++j)
#pragma unroll
            for (int k = 0; k < BZ; ++k) {
                const int y = yb + j, z = zb + k;
                if (y < ny && z < nz) part[i * nvox + ((long long)z * ny + y) * nx + x] = j == 0 ? res[k].x : res[k].y;
            }
    }
}

// Pass B: output y of phase i toward phase i-1 from the distances of pair (i-1, i), in the candidate
// order and with the online normalisation of box_direction; adds N/Z to the partial result, then Eq. 8.
template <int M_>
__global__ void __launch_bounds__(256)
    k_pair_b(int nx, int ny, int nz, const float *__restrict__ G, const float *__restrict__ vprev,
             const float *__restrict__ g, float *__restrict__ out, float c2, float mu, int clip)
{
    constexpr int S = 2 * M_ + 1;
    const long long nvox = (long long)nx * ny * nz;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nvox) return;
    const int x = (int)(t % nx), y = (int)((t / nx) % ny), z = (int)(t / ((long long)nx * ny));
    float mref = FLT_MAX, N = 0.f, Z = 0.f;
    constexpr int kCentre = M_ * S + M_;
    for (int it = 0; it < S * S; ++it) {  // window columns (dy, dx): (0, 0) first, then row-major
        const int cc = it == 0 ? kCentre : (it - 1 < kCentre ? it - 1 : it);
        const int dy = cc / S - M_, dx = cc % S - M_;
        if ((unsigned)(y + dy) >= (unsigned)ny || (unsigned)(x + dx) >= (unsigned)nx) continue;
#pragma unroll
        for (int dz = -M_; dz <= M_; ++dz) {
            if ((unsigned)(z + dz) >= (unsigned)nz) continue;
            const long long c = ((long long)(z + dz) * ny + (y + dy)) * nx + (x + dx);  // candidate in phase i-1
            // its pair distance, stored by pass A at offset -delta
            const float D = __ldg(G + (long long)(((M_ - dz) * S + (M_ - dy)) * S + (M_ - dx)) * nvox + c);
            float a = fmaf(D, -c2, mref);
            if (a > kRescale) {
                const float sc = ex2(-a);
                N *= sc;
                Z *= sc;
                mref = D * c2;
                a = 0.f;
            }
            const float e = ex2(a);
            N = fmaf(e, __ldg(vprev + c), N);
            Z += e;
        }
    }
    const float r = out[t] + N / Z;
    float f = (mu * __ldg(g + t) + r) * (1.f / (2.f + mu));  // Eq. 8
    if (clip) f = fmaxf(f, 0.f);
    out[t] = f;
}

template <int D_, int M_>
tnlm_status pairs_dm(int nx, int ny, int nz, int np, const float *wsrc, const float *vals, const float *g, float *out,
                     float c2, float mu, int clip, float *G0, float *G1, cudaStream_t st)
{
    using S = BoxShape<2>;
    using C = BoxCfg<D_, M_, 2, S::BZ, S::WY, S::WZ>;
    const int ntx = (nx + C::TXO - 1) / C::TXO, nty = (ny + C::TY - 1) / C::TY, ntz = (nz + C::TZ - 1) / C::TZ;
    const long long blocks = (long long)ntx * nty * ntz;
    auto ka = k_sweep_box_pa<D_, M_, 2, S::BZ, S::WY, S::WZ>;
    TNLM_TRY_CUDA(cudaFuncSetAttribute(ka, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM));
    const long long nvox = (long long)nx * ny * nz;
    const unsigned nb = (unsigned)((nvox + 255) / 256);
    float *G[2] = {G0, G1};
    // pass A of pair (i, i+1) into G[i % 2]; pass B of phase i from G[(i - 1) % 2]; phase 0 last
    for (int i = 0; i < np; ++i) {
        ka<<<(unsigned)blocks, C::NT, C::SMEM, st>>>(nx, ny, nz, np, i, ntx, nty, wsrc, vals, out, G[i % 2], c2);
        TNLM_TRY_CUDA(cudaGetLastError());
        if (i > 0) {
            k_pair_b<M_><<<nb, 256, 0, st>>>(nx, ny, nz, G[(i - 1) % 2], vals + (i - 1) * nvox, g + i * nvox,
                                             out + i * nvox, c2, mu, clip);
            TNLM_TRY_CUDA(cudaGetLastError());
        }
    }
    k_pair_b<M_><<<nb, 256, 0, st>>>(nx, ny, nz, G[(np - 1) % 2], vals + (np - 1) * nvox, g, out, c2, mu, clip);
    TNLM_TRY_CUDA(cudaGetLastError());
    return TNLM_OK;
}

}  // namespace box

bool launch_sweep_pairs(int d, int M, int nx, int ny, int nz, int np, const float *wsrc, const float *vals,
                        const float *g, float *out, float h, float mu, int clip, float *G0, float *G1, cudaStream_t st,
                        tnlm_status *status)
{
    const float c2 = (float)(1.4426950408889634 / (2.0 * (double)h * (double)h));
#define TNLM_PAIRS_CASE(DD, MM)                                                                                    \
    if (d == DD && M == MM) {                                                                                      \
        *status = box::pairs_dm<DD, MM>(nx, ny, nz, np, wsrc, vals, g, out, c2, mu, clip, G0, G1, st);             \
        return true;                                                                                               \
    }
    TNLM_PAIRS_CASE(1, 1)
    TNLM_PAIRS_CASE(1, 2)
    TNLM_PAIRS_CASE(1, 3)
    TNLM_PAIRS_CASE(2, 1)
    TNLM_PAIRS_CASE(2, 2)
    TNLM_PAIRS_CASE(2, 3)
#undef TNLM_PAIRS_CASE
    return false;
}

}  // namespace tnlm
